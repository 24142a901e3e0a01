"""The weights of the combination tiles: partial Gram rows from all CTAs, a solve in two parts, weights fetched ahead.  Ring lengths at
the edges of the kernel's instances, rings that fill and wrap, more matrices than CTAs, matrices of one tile and of many.  The plain
kernels (one launch a phase, one elimination over all slots) are the other side."""
import pytest
import torch

pytestmark = pytest.mark.gpu

FEW = [(96, 40), (256, 4096), (64, 8), (128, 1032)]
MANY = [(24, 16 + 8 * (i % 5)) for i in range(330)]


def _run(shapes, r, s, steps, **kw):
    from paper_2410_16029_b200.ngalore import NGaLore

    gen = torch.Generator(device="cuda").manual_seed(s)
    opt = NGaLore(shapes, r, s, 0, lam=0.1, lr=1e-2, **kw)
    for i, (M, N) in enumerate(shapes):
        opt.set_subspace(i, torch.linalg.qr(torch.randn(M, min(r, M, N), generator=gen, device="cuda"))[0])
    W = [torch.zeros(M, N, device="cuda") for M, N in shapes]
    common = [torch.randn(M, N, generator=gen, device="cuda") for M, N in shapes]
    for _ in range(steps):   # half of every gradient is shared, so that the Gram matrix is far from diagonal
        opt.step(W, [(x + torch.randn(x.shape, generator=gen, device="cuda")).bfloat16() for x in common])
    torch.cuda.synchronize()
    assert opt.poll_status()[0] == 0
    return W


@pytest.mark.parametrize("shapes", [FEW, MANY], ids=["few", "many"])
@pytest.mark.parametrize("s", [1, 2, 8, 9, 16, 17, 32])
def test_two_part_solve_agrees_with_the_plain_kernels(shapes, s):
    got, want = _run(shapes, 16, s, s + 3), _run(shapes, 16, s, s + 3, stream_impl=1)
    for x, y in zip(got, want):
        # Both sum the same fp32 products in other orders: 16 N products of size |R|^2 / (16 N) each, so K is off by at most
        # 2^-24 sqrt(16 N) |R|^2 / sqrt(16 N), and the weights by that over lambda c = 0.1 c, with |R|^2 = 2 * 16 N: 2e-5 N / c at
        # the shortest ring and widest matrix in the worst case, far less as sums of errors that are independent.
        assert (torch.linalg.norm(x - y) / torch.linalg.norm(y)).item() <= 1e-4


@pytest.mark.parametrize("s", [1, 2, 8, 9, 17, 32])
def test_two_unknowns_of_a_bf16_history(s):
    """Two rows are new every step (bf16 history): a set stepped as one state and matrix by matrix (other tiles, other sums)."""
    got = _run(FEW, 16, s, s + 3, history_bf16=True)
    want = _run(FEW, 16, s, s + 3, history_bf16=False)
    for x, y in zip(got, want):
        # independent halves of the gradients: the rounding of the history, 2^-9 of an entry, moves the update by about 3e-4
        # (measured for half-shared gradients); a wrong row or order is off by tenths
        assert (torch.linalg.norm(x - y) / torch.linalg.norm(y)).item() <= 5e-3
