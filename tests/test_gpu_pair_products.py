"""Sets of wide bases with short products take 256 x 256 tiles on pairs of SMs: rows that end in either half of a tile, columns that end in
either CTA's half or in a tile of their own, a K that is no multiple of 64, and matrices with narrow bases among them."""
import pytest
import torch

from tests.test_gpu_refresh_widths import _check, _gradient

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("r,shapes", [
    (196, [(777, 520), (900, 264)]),
    (256, [(768, 768), (1024, 520)]),
    (256, [(768, 768), (3000, 264)]),       # (whose K of 3000 is split)
    (260, [(650, 584), (1100, 776), (640, 64)]),
])
def test_products_on_pairs(r, shapes):
    from paper_2410_16029_b200.ngalore import NGaLore

    made = [_gradient(M, N, min(10, r // 2, N // 2), 40 + i) for i, (M, N) in enumerate(shapes)]
    copies = 60 // len(shapes) + 1        # more than two 256 x 256 tiles for every SM
    G = [g.clone() for g, _ in made for _ in range(copies)]
    opt = NGaLore([s for s in shapes for _ in range(copies)], r, 0, 0)
    assert opt.debug_plan("refresh_products") == 2 and opt.debug_plan("refresh_splits") == int(max(M for M, _ in shapes) == 3000)
    opt.refresh_subspace(G)
    torch.cuda.synchronize()
    assert opt.poll_status()[0] == 0
    for i, (M, N) in enumerate(shapes):
        for k in (0, copies - 1):
            _check(opt, i * copies + k, made[i][1], min(r, M, N), min(10, r // 2, N // 2))
