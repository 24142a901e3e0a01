"""A failed call stays its own.  A step that fails between its launches leaves no work counter or flag behind that the next step takes for its own.  beta1 = beta2 =
0, so that a step that ran in part and is taken again has the same result; K of the first matrix is split, so that its tiles add to
a ring slot that has to be cleared.  The bound is that of two orders of the same sums.  And a state that does not fit the device is
refused without an error left over for the next call on another."""
import pytest
import torch

from tests.parity_util import TOL_UPDATE

pytestmark = pytest.mark.gpu

SHAPES, R = [(4000, 264), (300, 136)], 32


def _run(phase, host, s=3, **kw):
    from paper_2410_16029_b200.ngalore import NGaLore, NGaLoreError

    gen = torch.Generator(device="cuda").manual_seed(5)
    opt = NGaLore(SHAPES, R, s, 0, lam=0.1, lr=1e-2, beta1=0.0, beta2=0.0, **kw)
    for i, (M, N) in enumerate(SHAPES):
        opt.set_subspace(i, torch.linalg.qr(torch.randn(M, R, generator=gen, device="cuda"))[0])
    W = [torch.zeros(M, N, device="cuda") for M, N in SHAPES]
    if host:
        W = [w.cpu().pin_memory() for w in W]
    for k in range(5):
        G = [torch.randn(M, N, generator=gen, device="cuda").bfloat16() for M, N in SHAPES]
        if host:
            G = [g.cpu().pin_memory() for g in G]
        step = opt.step_host if host else opt.step
        if phase is not None and k == 3:
            opt.debug_fail_step(phase)
            with pytest.raises(NGaLoreError):
                step(W, [g.neg() if not host else g.neg().pin_memory() for g in G])
            assert opt.step_count == k
        step(W, G)
    torch.cuda.synchronize()
    assert opt.poll_status()[0] == 0 and opt.step_count == 5
    return [w.cuda() for w in W]


@pytest.mark.parametrize("phase", [0, 1])
@pytest.mark.parametrize("host,kw", [(False, {}), (True, {}), (False, {"s": 0}), (False, {"gemm_impl": 1})])
def test_the_step_after_a_failed_one_is_a_regular_one(phase, host, kw):
    for got, want in zip(_run(phase, host, **kw), _run(None, host, **kw)):
        assert (torch.linalg.norm(got - want) / torch.linalg.norm(want)).item() <= 0.1 * TOL_UPDATE


def test_a_state_that_does_not_fit_leaves_no_error_for_the_next_step():
    from paper_2410_16029_b200.ngalore import NGaLore, NGaLoreError

    opt = NGaLore([(300, 136)], R, 3, 0)
    opt.set_subspace(0, torch.linalg.qr(torch.randn(300, R, device="cuda"))[0])
    with pytest.raises(NGaLoreError) as refused:
        NGaLore([(1 << 24, 1 << 24)], 512, 32, 0)      # a history of a terabyte
    assert refused.value.code == 2
    W = [torch.zeros(300, 136, device="cuda")]
    opt.step(W, [torch.randn(300, 136, device="cuda").bfloat16()])
    torch.cuda.synchronize()
    assert opt.poll_status()[0] == 0 and opt.step_count == 1 and W[0].abs().max().item() > 0
