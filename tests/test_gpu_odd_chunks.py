"""The weight update of matrices whose last tile of columns has an odd number of 32-column chunks, many tiles a CTA, tens of steps
without a pause: the two groups of warps that take the chunks in turn over one ring of slots get the chunk they wait for, whatever order
the loads land in.  The other side waits for every step; K has two pieces at most, whose
sum is the same in either order, so the bits are the same."""
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("r,projection", [(37, "left"), (37, "short_side"), (332, "left")])
def test_weights_do_not_depend_on_the_order_of_loads(r, projection):
    from paper_2410_16029_b200.ngalore import NGaLore

    shapes = [(1312, 1312)] * 40 + [(1312, 4848)] * 14     # 32 and 240 columns in the last tile; 5 or 8 slots
    gen = torch.Generator(device="cuda").manual_seed(r)
    sets = [[torch.randn(s, generator=gen, device="cuda").bfloat16() for s in shapes] for _ in range(3)]
    out = []
    for pause in (False, True):
        opt = NGaLore(shapes, r, 2, 0, lam=0.1, projection=projection)
        basis = {}
        for i in range(len(shapes)):
            rows, rank = opt.subspace_rows(i), opt.rank(i)
            if (rows, rank) not in basis:
                basis[rows, rank] = torch.linalg.qr(torch.randn(rows, rank, generator=torch.Generator(device="cuda").manual_seed(rows), device="cuda"))[0]
            opt.set_subspace(i, basis[rows, rank])
        W = [torch.zeros(s, device="cuda") for s in shapes]
        for k in range(120):
            opt.step(W, sets[k % 3])
            if pause:
                torch.cuda.synchronize()
        torch.cuda.synchronize()
        assert opt.poll_status()[0] == 0
        out.append(W)
        opt.close()
    assert all(torch.equal(a, b) for a, b in zip(*out))
