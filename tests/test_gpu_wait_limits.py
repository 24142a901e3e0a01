"""A wait for weights that never come ends by itself, and before the waits of the same block that depend on it: those are abandoned after
two seconds, and with them whatever else the block has claimed.  The withheld matrix is the first of the list and has a tile for every
multiprocessor, so that the other one's tiles are behind it everywhere."""
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kw", [{}, {"history_bf16": True}])
def test_a_wait_for_weights_ends_by_itself_and_leaves_out_its_own_matrix_only(kw):
    from paper_2410_16029_b200.ngalore import NGaLore

    gen = torch.Generator(device="cuda").manual_seed(6)
    shapes = [(64, 20000), (64, 4096)]
    opts = [NGaLore(shapes, 64, 2, 0, lam=0.1, **kw) for _ in range(2)]
    Ws = [[torch.zeros(s, device="cuda") for s in shapes] for _ in opts]
    G = [[torch.randn(s, generator=gen, device="cuda").bfloat16() for s in shapes] for _ in range(4)]
    for o, W in zip(opts, Ws):
        for i in range(2):
            o.set_subspace(i, torch.eye(64, device="cuda"))
        for k in range(2):
            o.step(W, G[k])
    before = Ws[1][0].clone()
    opts[1].debug_withhold_solution(0, 0)      # (no limit but the kernel's own)
    begin, end = (torch.cuda.Event(enable_timing=True) for _ in range(2))
    begin.record()
    opts[1].step(Ws[1], G[2])
    end.record()
    opts[0].step(Ws[0], G[2])
    torch.cuda.synchronize()
    # one to three waits of 0.9 s on every multiprocessor, in turn (157 tiles on 148 of them); four million polls took up to 1.5 s a wait
    assert 890.0 < begin.elapsed_time(end) < 2700.0
    assert opts[1].poll_status() == (8, [8, 0])
    assert torch.equal(Ws[1][0], before) and torch.equal(Ws[1][1], Ws[0][1])
    for o, W in zip(opts, Ws):
        o.step(W, G[3])
    torch.cuda.synchronize()
    assert opts[1].poll_status() == (0, [0, 0]) and torch.equal(Ws[1][1], Ws[0][1]) and not torch.equal(Ws[1][0], before)
