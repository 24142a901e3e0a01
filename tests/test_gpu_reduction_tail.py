"""The end of the tridiagonalisation, which keeps the last 128 columns (64 where two CTAs share an SM) in registers and hands them on every
32 columns: widths at and around each of its starts, odd ones (plain path, padded rows) among them, and after panels of eight."""
import pytest
import torch

from tests.test_gpu_ritz_sizes import _check, _planted, _refresh

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("r", [4, 5, 34, 63, 66, 95, 96, 97, 98, 126, 129, 131, 136, 137])
def test_columns_are_ritz_vectors(r):
    M, N, q = max(r + 40, 160), max(r + 72, 168) // 8 * 8, max(1, min(6, r // 2))
    G = _planted(M, N, q, 300 + r, 2e-4)
    _check(_refresh(G, r), G, r, q)


@pytest.mark.parametrize("r", [32, 64, 68, 76])
def test_more_matrices_than_sms(r):
    from paper_2410_16029_b200.ngalore import NGaLore

    M, N = r + 60, (r + 76) // 8 * 8
    Gs = [_planted(M, N, 6, 500 + i, 2e-4) for i in range(3)]
    G = [Gs[i % 3].clone() for i in range(150)]
    opt = NGaLore([(M, N)] * 150, r, 0, 0)
    opt.refresh_subspace(G)
    torch.cuda.synchronize()
    for i in (0, 1, 2, 74, 148, 149):
        _check(opt.get_subspace(i).double().cpu().numpy(), G[i], r, 6)
    assert opt.poll_status()[0] == 0
