"""A set that one large matrix dominates: the rows that the warp which solves for it has to read are bounded in number, and the steps agree
with 64 bits."""
import pytest
import torch

from tests.exact_step import largest_errors

pytestmark = pytest.mark.gpu

LARGE = [(256, 40008)]
BEHIND = [(256, 264), (256, 70008)]


@pytest.mark.parametrize("s,kw,per_sm", [(3, {}, 6), (10, {}, 6), (17, {}, 6), (3, {"history_bf16": True}, 3),
                                         (10, {"history_bf16": True, "moments_bf16": True}, 3)])
@pytest.mark.parametrize("shapes", [LARGE, BEHIND], ids=["alone", "behind"])
def test_tiles_of_a_large_matrix_are_bounded(shapes, s, kw, per_sm):
    from paper_2410_16029_b200.ngalore import NGaLore

    most = per_sm * torch.cuda.get_device_properties(0).multi_processor_count
    opt = NGaLore(shapes, 256, s, 0, **kw)
    assert most // 3 <= opt.debug_plan("stream_tiles") <= most
    opt.close()


@pytest.mark.parametrize("s,rounded", [(3, False), (10, False), (17, False), (3, True), (10, True)])
def test_steps_of_a_large_matrix_agree_with_64_bits(s, rounded):
    worst, scale = largest_errors(BEHIND, 256, s, s + 2, rounded)
    assert worst <= 1.0 and scale <= 1.0


def test_rows_of_the_plain_kernels_are_not_held_beside_them():
    """A state holds the partial Gram rows that its kernels use: 16 bytes an entry in the stream kernel, and 8 more for the plain ones only."""
    from paper_2410_16029_b200.ngalore import NGaLore

    shapes, s = [(256, 24 * 1024)], 16          # 6 M elements, at least 700 tiles of 8192
    held = []
    for kw in ({}, {"stream_impl": 1}):
        opt = NGaLore(shapes, 256, s, 0, **kw)
        held.append((opt.device_bytes, opt.debug_plan("stream_tiles")))
        opt.close()
    assert held[0][1] == held[1][1] and held[1][0] - held[0][0] >= 8 * s * held[0][1]
