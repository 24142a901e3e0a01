"""The factorisation of a refresh at numbers of 32-column blocks beside those of test_gpu_refresh_widths.py: three and four blocks, the
last whose blocks stay in shared memory and the first that do not, and a last block of a few columns."""
import pytest

from tests.test_gpu_refresh_widths import _check, _gradient

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("r", [68, 96, 100, 128, 132, 168, 192, 196, 416])
def test_basis_at_block_edges(r):
    from paper_2410_16029_b200.ngalore import NGaLore

    q = min(10, r // 2)
    M, N = max(512, 2 * r), max(264, (r + 64) // 8 * 8)
    G, A = _gradient(M, N, q, 1000 + r)
    opt = NGaLore([(M, N)], r, 0, 0)
    opt.refresh_subspace([G])
    _check(opt, 0, A, r, q)
    assert opt.poll_status()[0] == 0
