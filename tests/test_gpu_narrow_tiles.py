"""Sets with few tiles take tiles of 128 or 64 columns in the projection and the back-projection: sets on either side of both lines (148
tiles of the narrower kind), widths that end inside a 64-column tile, K that is split, both projection rules, and the weight update
in groups.  Against the plain kernels, which add the same products in another order."""
import pytest
import torch

from tests.parity_util import TOL_UPDATE

pytestmark = pytest.mark.gpu


SETS = [
    ([(512, 1376)], 128, {}, 64, 0),
    ([(512, 1376)] * 6, 128, {}, 64, 0),
    ([(512, 1376)] * 7, 128, {}, 128, 0),
    ([(512, 1376)] * 24, 128, {}, 256, 0),
    ([(4000, 2048)], 256, {}, 128, 1),
    ([(6000, 720)], 200, {}, 64, 1),
    ([(1024, 4096)], 100, {"projection": "short_side"}, 64, 0),
    ([(4096, 1400)], 100, {"projection": "short_side"}, 64, 1),
    ([(32000, 1024)], 128, {}, 256, 1),
    ([(5000, 2000)] * 3, 128, {}, 256, 1),
]


@pytest.mark.skipif(not torch.cuda.is_available() or torch.cuda.get_device_properties(0).multi_processor_count != 148,
                    reason="the widths are those of 148 multiprocessors")
@pytest.mark.parametrize("shapes,r,kw,columns,splits", SETS)
def test_narrow_tiles_have_a_multiprocessor_each(shapes, r, kw, columns, splits):
    """With the pieces of a split K counted: where tiles would queue, they stay as wide as they are."""
    from paper_2410_16029_b200.ngalore import NGaLore

    opt = NGaLore(shapes, r, 2, 0, **kw)
    assert opt.debug_plan("projection_columns") == 256 or opt.debug_plan("projection_tiles") <= 148
    assert (opt.debug_plan("projection_columns"), opt.debug_plan("projection_splits")) == (columns, splits)


def _steps(shapes, r, gemm_impl, groups=0, **kw):
    from paper_2410_16029_b200.ngalore import NGaLore

    gen = torch.Generator(device="cuda").manual_seed(17)
    opt = NGaLore(shapes, r, 3, 0, lam=0.1, lr=1e-2, gemm_impl=gemm_impl, **kw)
    assert opt.debug_plan("projection_columns") < 256
    if groups:
        opt.set_update_groups(groups)
    for i, (M, N) in enumerate(shapes):
        rows = N if opt.projects_right(i) else M
        opt.set_subspace(i, torch.linalg.qr(torch.randn(rows, opt.rank(i), generator=gen, device="cuda"))[0])
    W = [torch.zeros(M, N, device="cuda") for M, N in shapes]
    for _ in range(4):
        opt.step(W, [torch.randn(M, N, generator=gen, device="cuda").bfloat16() for M, N in shapes])
    torch.cuda.synchronize()
    assert opt.poll_status()[0] == 0
    return W


@pytest.mark.parametrize("shapes,r,kw", [
    ([(512, 1376)], 128, {}),
    ([(512, 1376)] * 2, 128, {}),
    ([(512, 1376)] * 4, 128, {}),
    ([(512, 1376)] * 7, 128, {}),
    ([(128, 72), (130, 328), (257, 1000)], 40, {}),
    ([(4000, 200), (300, 136)], 64, {}),
    ([(4000, 1000)], 256, {}),
    ([(700, 264), (264, 696)], 100, {"projection": "short_side"}),
    ([(512, 1376)] * 3, 128, {"groups": 2}),
])
def test_steps_equal_those_of_the_plain_kernels(shapes, r, kw):
    kw = dict(kw)
    groups = kw.pop("groups", 0)
    want = _steps(shapes, r, 1, **kw)
    got = _steps(shapes, r, 0, groups, **kw)
    for i in range(len(shapes)):
        err = (torch.linalg.norm(got[i] - want[i]) / torch.linalg.norm(want[i])).item()
        assert err <= 0.1 * TOL_UPDATE, (i, err)
