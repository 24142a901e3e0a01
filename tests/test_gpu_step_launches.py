"""Steps queued one behind another, on both sides of the line below which the kernels of a step may start before their
predecessor has finished (32 back-projection tiles of 128 x 256 a multiprocessor: 4736 tiles on 148 of them).

What such launches can break is the order of reads and writes, between the kernels of a step, between two steps and
against the caller's own work in the stream; so queued and captured steps are compared with steps that are each waited
for.  Both add the same fp32 products, but the order of a few sums is not fixed, so the bound is a tenth of the parity
tolerance, as between two arrangements of one path.
"""
import pytest
import torch

from tests.parity_util import TOL_UPDATE

pytestmark = pytest.mark.gpu

M, N, R, S = 2048, 2048, 64, 3      # 128 tiles a matrix


def _run(n, how):
    """how: waited (for every step), queued, graph (captured on one stream), joined and joined-graph (the gradients of a
    step are written on a second stream, which the stepping stream waits for by an event just before the step; a wait
    ahead of the write makes sure that it comes late)."""
    from paper_2410_16029_b200.ngalore import NGaLore

    gen = torch.Generator(device="cuda").manual_seed(7)
    opt = NGaLore([(M, N)] * n, R, S, 0, lam=0.1, lr=1e-2)
    grads = [[torch.randn(M, N, generator=gen, device="cuda").bfloat16() for _ in range(3)] for _ in range(2)]
    P = torch.linalg.qr(torch.randn(M, R, generator=gen, device="cuda"))[0]
    for i in range(n):
        opt.set_subspace(i, P)
    buf = [torch.empty(M, N, device="cuda", dtype=torch.bfloat16) for _ in range(3)]
    G = [buf[i % 3] for i in range(n)]
    W = [torch.zeros(M, N, device="cuda") for _ in range(n)]

    def load(k):                            # the caller's own work between two steps, into the same buffers
        for i in range(3):
            buf[i].copy_(grads[k & 1][i])

    side = torch.cuda.Stream()

    def load_beside(k):
        main = torch.cuda.current_stream()
        side.wait_stream(main)
        with torch.cuda.stream(side):
            torch.cuda._sleep(2000000)      # about a millisecond
            load(k)
        main.wait_event(side.record_event())

    if how == "joined-graph":
        load(0)
        opt.step(W, G)
        torch.cuda.synchronize()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph):
            for k in (1, 0, 0):
                load_beside(k)
                opt.step(W, G)
        graph.replay()
    elif how == "joined":
        for k in (0, 1, 0, 0):
            load_beside(k)
            opt.step(W, G)
    elif how == "graph":
        load(0)
        opt.step(W, G)                      # binds the buffers
        load(1)
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph):
            opt.step(W, G)
            load(0)
            opt.step(W, G)
            opt.step(W, G)
            load(1)
        graph.replay()
    else:
        for k in (0, 1, 0, 0):
            load(k)
            opt.step(W, G)
            if how == "waited":
                torch.cuda.synchronize()
    torch.cuda.synchronize()
    assert opt.poll_status()[0] == 0
    return W


@pytest.mark.parametrize("n", [1, 37, 38])
def test_queued_and_captured_steps_equal_waited_ones(n):
    want = _run(n, "waited")
    for how in ("queued", "graph", "joined", "joined-graph"):
        got = _run(n, how)
        for i in range(n):
            err = (torch.linalg.norm(got[i] - want[i]) / torch.linalg.norm(want[i])).item()
            assert err <= 0.1 * TOL_UPDATE, (how, i, err)
