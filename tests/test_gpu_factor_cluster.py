"""The factorisation with a cluster of CTAs to a matrix: sets of few wide matrices, two and four CTAs each, at widths around a
multiple of its blocks of 32, with narrow matrices among them.  The bound is what a refresh promises (see
test_gpu_refresh_widths.py); the planted directions are far above the noise."""
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("count,r", [(3, 420), (9, 260), (20, 288), (33, 320), (60, 292), (76, 292)])
def test_bases_of_few_wide_matrices(count, r):
    from paper_2410_16029_b200.ngalore import NGaLore

    gen = torch.Generator(device="cuda").manual_seed(count + r)
    shapes = [(1024 + 8 * (i % 3), 512) for i in range(count - 3)] + [(600, 8), (640, 72), (900, 136)]
    if count < 4:
        shapes = [(1024, 512), (640, 72), (2048, 424)]
    G, planted = [], []
    for M, N in shapes:
        q = min(6, N // 2)
        A = torch.linalg.qr(torch.randn(M, q, generator=gen, device="cuda"))[0]
        B = torch.linalg.qr(torch.randn(N, q, generator=gen, device="cuda"))[0]
        G.append((A @ B.T + 1e-4 * torch.randn(M, N, generator=gen, device="cuda")).bfloat16())
        planted.append(A)
    opt = NGaLore(shapes, r, 0, 0)
    opt.refresh_subspace(G)
    assert opt.poll_status()[0] == 0
    for i, A in enumerate(planted):
        P = opt.get_subspace(i).double()
        assert (P.T @ P - torch.eye(P.shape[1], device="cuda")).abs().max().item() <= 1e-5, i
        # bf16 rounding of G, 2^-9 of an entry: its singular vectors are within about that of the planted ones
        assert (A.double() - P @ (P.T @ A.double())).norm(dim=0).max().item() <= 2e-2, i
