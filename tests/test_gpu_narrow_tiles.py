"""Sets with few tiles take tiles of 128 or 64 columns in the projection and the back-projection: sets on either side of both lines (148
tiles of the narrower kind), widths that end inside a 64-column tile, K that is split, both projection rules, and the weight update
in groups.  Against the plain kernels, which add the same products in another order."""
import pytest
import torch

from tests.parity_util import TOL_UPDATE

pytestmark = pytest.mark.gpu


def _steps(shapes, r, gemm_impl, groups=0, **kw):
    from paper_2410_16029_b200.ngalore import NGaLore

    gen = torch.Generator(device="cuda").manual_seed(17)
    opt = NGaLore(shapes, r, 3, 0, lam=0.1, lr=1e-2, gemm_impl=gemm_impl, **kw)
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
