"""As test_gpu_odd_chunks.py, with last tiles of one, three, five and seven 32-column chunks between full ones, so that both groups of warps have
chunks of them and the ring's slots change hands, in both lengths of the ring (r = 332: 93 % of the elements have a rank above 320): the same
bits with and without a pause after every step."""
import pytest
import torch

pytestmark = pytest.mark.gpu

SHAPES = [(1312, 256 * k + x) for k in (1, 3) for x in (96, 160, 224, 32, 256)] * 6 + [(1312, 32 * x) for x in (1, 1, 1, 3, 1, 5, 1, 7)] * 2


@pytest.mark.parametrize("r", [37, 332])
def test_weights_do_not_depend_on_the_order_of_loads(r):
    from paper_2410_16029_b200.ngalore import NGaLore

    gen = torch.Generator(device="cuda").manual_seed(r)
    sets = [[torch.randn(s, generator=gen, device="cuda").bfloat16() for s in SHAPES] for _ in range(3)]
    out = []
    for pause in (False, True):
        opt = NGaLore(SHAPES, r, 2, 0, lam=0.1)
        basis = {}
        for i in range(len(SHAPES)):
            rows, rank = opt.subspace_rows(i), opt.rank(i)
            if (rows, rank) not in basis:
                basis[rows, rank] = torch.linalg.qr(torch.randn(rows, rank, generator=torch.Generator(device="cuda").manual_seed(rank), device="cuda"))[0]
            opt.set_subspace(i, basis[rows, rank])
        W = [torch.zeros(s, device="cuda") for s in SHAPES]
        for k in range(120):
            opt.step(W, sets[k % 3])
            if pause:
                torch.cuda.synchronize()
        torch.cuda.synchronize()
        assert opt.poll_status()[0] == 0
        out.append(W)
        opt.close()
    assert all(torch.equal(a, b) for a, b in zip(*out))
