"""What a step is given is refused before it reads or writes past its end: too few tensors, host buffers that are too small or of another type."""
import pytest
import torch

from tests.test_bind import SHAPES, _collect, _tensors


def _collected(W, G, shapes):
    return _collect(W, G, shapes, 2)


def _looked_at(W, G, shapes):
    from paper_2410_16029_b200.ngalore import _check_buffers

    _check_buffers(shapes, W, G, host=True)


SMALLER = [
    ("W", lambda t: t[:-1]),                        # fewer rows
    ("G", lambda t: t.flatten()[:-1]),
    ("W", lambda t: t.to(torch.bfloat16)),          # half the bytes
    ("W", lambda t: t.to(torch.float64)),
    ("G", lambda t: t.to(torch.float32)),
    ("G", lambda t: t.to(torch.float16)),           # the same bytes, other values
    ("G", lambda t: t.to(torch.int8)),
]


@pytest.mark.parametrize("look", [_collected, _looked_at])
@pytest.mark.parametrize("which", range(2))
@pytest.mark.parametrize("side,change", SMALLER)
def test_host_buffers_that_do_not_hold_the_matrix(look, which, side, change):
    W, G = _tensors()
    if side == "W":
        W[which] = change(W[which])
    else:
        G[which] = change(G[which])
    with pytest.raises(AssertionError):
        look(W, G, SHAPES)


@pytest.mark.parametrize("look", [_collected, _looked_at])
def test_host_buffers_that_do(look):
    W, G = _tensors()
    look(W, G, SHAPES)
    look([w.flatten() for w in W], [g.view(torch.int16) for g in G], SHAPES)
    look([torch.zeros(100) for _ in W], [g.view(torch.uint16) for g in G], SHAPES)


@pytest.mark.parametrize("host", [False, True])
def test_a_tensor_for_every_matrix(host):
    from paper_2410_16029_b200.ngalore import _check_buffers

    W, G = _tensors()
    _check_buffers(SHAPES, tuple(W), dict(enumerate(G)).values() if not host else G, host)
    for w, g in [(W[:1], G), (W, G[:1]), ([], [])]:
        with pytest.raises(AssertionError):
            _check_buffers(SHAPES, w, g, host)
