"""The factorisation inside the refresh (Cholesky QR with R^-1 from one launch) at the basis widths where it changes
course: one block of 32 columns and less, block edges, the widest matrices whose blocks stay in shared memory (fp32 256,
fp64 160 columns), the widest whose operand rows do (fp64 672), and a set that mixes them."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


def _gradient(M, N, q, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    A = torch.linalg.qr(torch.randn(M, q, generator=g, device="cuda"))[0]
    B = torch.linalg.qr(torch.randn(N, q, generator=g, device="cuda"))[0]
    s = 0.8 ** torch.arange(q, device="cuda")
    return ((A * s) @ B.T + 1e-4 * torch.randn(M, N, generator=g, device="cuda")).to(torch.bfloat16), A


def _check(opt, i, A, r, q):
    """P orthonormal to 1e-5 (the accuracy the refresh promises) and its span holds the q planted directions: their
    singular values are at least 0.8^9 = 0.13 against a noise of at most 1e-4 (sqrt M + sqrt N) = 8e-3, so that the
    gradient's own singular vectors are within about 8e-3 / 0.13 of them (first-order bound), 6e-2."""
    P = opt.get_subspace(i).double()
    err = (P.T @ P - torch.eye(r, device="cuda", dtype=torch.float64)).abs().max().item()
    assert err <= 1e-5, (r, err)
    lost = (A.double() - P @ (P.T @ A.double())).norm(dim=0).max().item()
    assert lost <= 6e-2, (r, lost)


@pytest.mark.parametrize("r", [4, 28, 32, 36, 64, 128, 160, 164, 256, 260, 288, 672, 676, 872])
def test_basis_of_every_width(r):
    from paper_2410_16029_b200.ngalore import NGaLore

    q = min(10, r // 2)
    M, N = max(512, 2 * r), max(264, (r + 64) // 8 * 8)
    G, A = _gradient(M, N, q, r)
    opt = NGaLore([(M, N)], r, 0, 0)
    opt.refresh_subspace([G])
    _check(opt, 0, A, r, q)
    assert opt.poll_status()[0] == 0


def test_mixed_widths():
    from paper_2410_16029_b200.ngalore import NGaLore

    shapes = [(1024, 8), (600, 32), (1200, 128), (1024, 160), (700, 264), (2048, 520), (1400, 696), (1500, 1024)]
    made = [_gradient(M, N, min(10, N // 2), i) for i, (M, N) in enumerate(shapes)]
    opt = NGaLore(shapes, 676, 0, 0)
    opt.refresh_subspace([g for g, _ in made])
    for i, (M, N) in enumerate(shapes):
        r = min(676, M, N)
        _check(opt, i, made[i][1], r, min(10, N // 2))
    assert opt.poll_status()[0] == 0


@pytest.mark.parametrize("M,N,r", [(80072, 264, 64), (76904, 1560, 200)])
def test_tall_tiles(M, N, r):
    """Sets with at least two 256-row tiles of the products with G for every multiprocessor take such tiles (narrow bases,
    and wide ones with long products).  Rows that end in the first or in the second half of a tile; P orthonormal, its
    columns Ritz vectors of G (bounds as for smaller matrices: 1e-5 and 1e-4 of the larger diagonal entry) and the leading
    ones the planted singular vectors."""
    from paper_2410_16029_b200.ngalore import NGaLore

    gen = torch.Generator(device="cuda").manual_seed(M)
    q = 6
    U = torch.linalg.qr(torch.randn(M, q, generator=gen, device="cuda"))[0]
    V = torch.linalg.qr(torch.randn(N, q, generator=gen, device="cuda"))[0]
    G = ((U * 0.7 ** torch.arange(q, device="cuda")) @ V.T).add_(torch.randn(M, N, generator=gen, device="cuda"), alpha=2e-5).bfloat16()
    opt = NGaLore([(M, N)], r, 0, 0, ritz_columns=-1)
    opt.refresh_subspace([G])
    torch.cuda.synchronize()
    assert opt.poll_status()[0] == 0
    P = opt.get_subspace(0).double()
    G64 = G.double()
    if opt.projects_right(0):
        G64, U = G64.T, V
    assert (P.T @ P - torch.eye(r, device="cuda")).abs().max().item() <= 1e-5
    B = P.T @ G64
    C = B @ B.T
    d = torch.diagonal(C)
    off = (C - torch.diag(d)).abs() / torch.sqrt(torch.maximum(d[:, None], d[None, :]) * d[0])
    assert off.max().item() <= 1e-4
    # (the bf16 rounding of G, 2^-9 of an entry at most, tilts its singular vectors from the planted ones)
    assert (1.0 - (P[:, :q] * U.double()).sum(0).abs()).max().item() <= 1e-3
