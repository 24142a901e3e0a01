"""The last pass of a refresh over matrices with fewer than 512 rows: Gram matrix, factor and product in fp64, all such
matrices of a set in four launches.  Sizes at the edges of its 64 x 64 tiles and slabs of 256 rows, next to matrices that do
not take the pass."""
import pytest
import torch

pytestmark = pytest.mark.gpu

SETS = [
    ([(511, 640), (512, 64), (64, 200), (68, 96), (4, 8)], 500, "left"),
    ([(255, 264), (256, 264), (257, 264), (132, 72), (900, 136)], 128, "left"),
    ([(320, 328), (640, 104), (3000, 200), (1025, 64)], 68, "short_side"),
]


@pytest.mark.parametrize("shapes,rank,projection", SETS)
def test_short_bases_are_orthonormal_and_hold_the_leading_directions(shapes, rank, projection):
    from paper_2410_16029_b200.ngalore import NGaLore

    gen = torch.Generator(device="cuda").manual_seed(len(shapes) + rank)
    G = []
    for M, N in shapes:
        q = max(1, min(M, N, rank) // 4)
        A = torch.linalg.qr(torch.randn(M, q, generator=gen, device="cuda"))[0]
        B = torch.linalg.qr(torch.randn(N, q, generator=gen, device="cuda"))[0]
        s = 0.9 ** torch.arange(q, device="cuda")
        G.append(((A * s) @ B.T + 1e-5 * torch.randn(M, N, generator=gen, device="cuda")).bfloat16())
    opt = NGaLore(shapes, rank, 0, 0, projection=projection)
    opt.refresh_subspace(G)
    assert opt.poll_status()[0] == 0
    for i, g in enumerate(G):
        P = opt.get_subspace(i).double()
        r = P.shape[1]
        # An exact pass leaves the rounding of P's entries to fp32 and of the scaling to unit norm: 2^-24 of an entry each, at
        # most 4 * 2^-24 on an inner product of unit columns.  (Without it: 1e-5, see test_gpu_refresh_widths.py.)
        err = (P.T @ P - torch.eye(r, device="cuda")).abs().max().item()
        assert err <= (4 * 2.0 ** -24 if P.shape[0] < 512 else 1e-5), (i, err)
        # leading left singular vectors with a gap to the noise: sigma_j >= 0.9^k = 0.05 against at most the bf16 rounding of
        # G, 2^-9 |g| an entry, whose norm is below 2^-9 |G|_F (1.3e-2 for a spectrum 0.9^j), spread over min(M, N) directions
        g64 = g.double().T if opt.projects_right(i) else g.double()
        U, S, _ = torch.linalg.svd(g64, full_matrices=False)
        k = int((S > 0.2 * S[0]).sum())
        k = min(k, r)
        lost = (U[:, :k] - P @ (P.T @ U[:, :k])).norm(dim=0).max().item()
        assert lost <= 1e-3, (i, lost)
