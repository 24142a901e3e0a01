"""The binding's helper that checks and collects the pointers of a step's tensors."""
import ctypes

import pytest
import torch


def _collect(W, G, shapes, mode):
    import __graft_entry__ as entry

    entry.build()
    from paper_2410_16029_b200 import _bind

    n = len(shapes)
    flat = (ctypes.c_int64 * (2 * n))(*[x for s in shapes for x in s])
    w, g = (ctypes.c_void_p * n)(), (ctypes.c_void_p * n)()
    done = _bind.collect(W, G, n, ctypes.addressof(flat), ctypes.addressof(w), ctypes.addressof(g), mode)
    return done, list(w), list(g)


SHAPES = [(4, 8), (16, 2)]


def _tensors():
    return [torch.zeros(s) for s in SHAPES], [torch.zeros(s, dtype=torch.bfloat16) for s in SHAPES]


@pytest.mark.parametrize("mode", [0, 2])
@pytest.mark.parametrize("kind", [list, tuple])
def test_pointers_of_plain_tensors(mode, kind):
    W, G = _tensors()
    W[0] = torch.nn.Parameter(W[0])
    done, w, g = _collect(kind(W), kind(G), SHAPES, mode)
    assert done and w == [t.data_ptr() for t in W] and g == [t.data_ptr() for t in G]


def test_what_it_leaves_to_the_caller():
    class Sub(torch.Tensor):
        pass

    W, G = _tensors()
    assert not _collect(W[:1], G, SHAPES, 2)[0]
    assert not _collect(dict(enumerate(W)).values(), G, SHAPES, 2)[0]
    assert not _collect([W[0].as_subclass(Sub), W[1]], G, SHAPES, 2)[0]
    assert not _collect([W[0], 3], G, SHAPES, 0)[0]


def test_what_it_refuses():
    W, G = _tensors()
    with pytest.raises(AssertionError):
        _collect(W, G, SHAPES, 1)                     # not on a device
    with pytest.raises(AssertionError):
        _collect([W[0].t(), W[1]], G, SHAPES, 2)      # not contiguous
