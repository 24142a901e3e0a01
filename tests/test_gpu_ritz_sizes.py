"""The eigensolver of the refresh at the sizes where it changes course: one and two columns, widths around its warps,
panels and register tiles, around the widest matrix that fits shared memory (156), around each variant of the
back-transformation (128 | 256 | 512), odd widths, and a gradient of numerical rank far below the basis width (a
cluster of equal eigenvalues)."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


def _refresh(G, r, **kw):
    from paper_2410_16029_b200.ngalore import NGaLore

    opt = NGaLore([tuple(G.shape)], r, 0, 0, ritz_columns=-1, **kw)
    opt.refresh_subspace([G])
    torch.cuda.synchronize()
    P = opt.get_subspace(0).double().cpu().numpy()
    assert opt.poll_status()[0] == 0
    return P


def _planted(M, N, q, seed, noise):
    rng = np.random.default_rng(seed)
    U = np.linalg.qr(rng.standard_normal((M, q)))[0]
    V = np.linalg.qr(rng.standard_normal((N, q)))[0]
    G = (U * 0.7 ** np.arange(q)) @ V.T + noise * rng.standard_normal((M, N))
    return torch.from_numpy(G).to(torch.bfloat16).cuda()


def _check(P, G, r, q):
    """P is orthonormal, its columns are Ritz vectors (P^T G G^T P is diagonal: off-diagonal entries below 1e-4 of the
    larger of their two diagonal entries, the rounding of P to fp32 and of Q V to two bf16 parts, 2^-16 a product) in
    falling order, and the separated leading ones are singular vectors."""
    G64 = G.double().cpu().numpy()
    assert np.max(np.abs(P.T @ P - np.eye(r))) <= 1e-5
    B = P.T @ G64
    C = B @ B.T
    d = np.diag(C)
    off = np.abs(C - np.diag(d)) / np.sqrt(np.maximum.outer(d, d) * d[0])
    assert off.max() <= 1e-4, off.max()
    assert np.all(np.sqrt(d[1:]) <= np.sqrt(d[:-1]) * (1 + 1e-3) + 1e-6 * np.sqrt(d[0]))
    U, _, _ = np.linalg.svd(G64, full_matrices=False)
    assert np.max(1.0 - np.abs(np.sum(P[:, :q] * U[:, :q], axis=0))) <= 1e-3


@pytest.mark.parametrize("r", [1, 2, 3, 8, 15, 31, 32, 33, 64, 65, 100, 116, 127, 128, 132, 152, 156, 157, 160, 255, 256, 260, 511, 512, 516])
def test_columns_are_ritz_vectors(r):
    """r no multiple of 4 takes the plain path, the others the grouped one.  (Wide bases get twice as many rows as
    columns: the rounding of the two-part product with r columns averages out over the rows only, and at 552 x 512
    leaves P orthonormal to 4e-5, whatever diagonalises the small matrix.)"""
    M, N, q = max(r + 40, 160), max(r + 72, 168) // 8 * 8, max(1, min(6, r // 2))
    if r > 400:
        M = 2 * r
    G = _planted(M, N, q, 100 + r, 2e-4)
    _check(_refresh(G, r), G, r, q)


@pytest.mark.parametrize("r", [36, 132])
def test_more_matrices_than_sms(r):
    """A batch of 150: two CTAs of the reduction share an SM."""
    from paper_2410_16029_b200.ngalore import NGaLore

    M, N = r + 60, r + 76
    Gs = [_planted(M, N, 6, i, 2e-4) for i in range(3)]
    G = [Gs[i % 3].clone() for i in range(150)]
    opt = NGaLore([(M, N)] * 150, r, 0, 0)
    opt.refresh_subspace(G)
    torch.cuda.synchronize()
    for i in (0, 1, 2, 74, 148, 149):
        _check(opt.get_subspace(i).double().cpu().numpy(), G[i], r, 6)
    assert opt.poll_status()[0] == 0


@pytest.mark.parametrize("r", [30, 64, 256])
def test_gradient_of_low_rank(r):
    """Exactly rank 5 (integer factors, products exact in bf16): r - 5 eigenvalues are equal up to rounding."""
    rng = np.random.default_rng(7)
    A = rng.integers(-2, 3, (400, 5)).astype(np.float64)
    B = rng.integers(-2, 3, (5, 512)).astype(np.float64)
    G = torch.from_numpy(A @ B).to(torch.bfloat16).cuda()
    G64 = G.double().cpu().numpy()
    assert np.array_equal(G64, A @ B)
    P = _refresh(G, r)
    assert np.max(np.abs(P.T @ P - np.eye(r))) <= 1e-5
    R = G64 - P @ (P.T @ G64)
    assert np.linalg.norm(R) <= 1e-4 * np.linalg.norm(G64)


def test_widest_bases_beside_narrow_ones():
    """Above about 700 columns the factorisation of the Gram matrix of the vectors keeps its rows in global memory, for
    every matrix of the launch."""
    from paper_2410_16029_b200.ngalore import NGaLore

    shapes = [(1448, 800), (160, 48), (600, 200), (4, 160)]
    G = [_planted(M, N, min(M, N, 6), 700 + i, 2e-4) for i, (M, N) in enumerate(shapes)]
    opt = NGaLore(shapes, 724, 0, 0, ritz_columns=-1)
    opt.refresh_subspace(G)
    torch.cuda.synchronize()
    assert opt.poll_status()[0] == 0
    for i, (M, N) in enumerate(shapes):
        r = opt.rank(i)
        assert r == min(M, N, 724)
        _check(opt.get_subspace(i).double().cpu().numpy(), G[i] if not opt.projects_right(i) else G[i].T.contiguous(), r, min(r, 4))
