"""The Gram row (with a bf16 history two rows), the solve and the combination of the stream kernel against 64 bits.  Ring lengths at the edges of
the kernel's instances, rings that fill and wrap, matrices of one tile and of many, more matrices than multiprocessors."""
import pytest

from tests.exact_step import largest_errors

pytestmark = pytest.mark.gpu

FEW = [(96, 40), (256, 4096), (64, 8), (128, 1032)]
MANY = [(24, 16 + 8 * (i % 5)) for i in range(200)]


@pytest.mark.parametrize("rounded", [False, True])
@pytest.mark.parametrize("shapes", [FEW, MANY], ids=["few", "many"])
@pytest.mark.parametrize("s", [1, 2, 8, 9, 16, 17, 32])
def test_natural_gradient_of_the_ring_as_it_is_kept(shapes, s, rounded):
    worst, scale = largest_errors(shapes, 16, s, s + 3 if shapes is FEW else min(s + 3, 20), rounded)
    assert worst <= 1.0 and scale <= 1.0
