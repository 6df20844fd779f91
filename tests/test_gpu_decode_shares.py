"""Decodes in which CTAs have steps without a pixel, next to steps with some:
a grid larger than the first and last fronts of a picture, units narrower than
h + 1 (idle steps in every row), one tall unit beside short ones, and more than
64 units (the schedule's other form).  Equality with the coded images is exact.
"""
import pytest
import torch

from paper_2201_05213_gb300 import nlc as N

from gpu_util import images, make_codec, to_dev

pytestmark = pytest.mark.gpu

BATCHES = {
    "picture": [(61, 83)],
    "narrow": [(40, 1), (33, 2), (27, 3)],
    "tall": [(120, 9), (3, 5), (1, 1)],
    "many": [(1 + k % 9, 1 + k % 7) for k in range(70)] + [(40, 21)],
}


@pytest.mark.parametrize("prec", [N.NLC_FP32, N.NLC_BF16, N.NLC_BF16_SHEARED])
@pytest.mark.parametrize("name", sorted(BATCHES))
def test_steps_without_pixels(name, prec):
    sizes = BATCHES[name]
    codec, _ = make_codec((3, 32, 1, 5), prec, seed=5, scale=1.5)
    d = [to_dev(i) for i in images(29, sizes)]
    data, offs = codec.compress(d, 0, N.NLC_LAYOUT_ROW)
    for px, ctas in ((1, 0), (1, 7), (4, 0)):
        N.nlc_set_tuning(codec.ctx, px, ctas)
        for _ in range(5):
            outs = codec.decompress(data, offs, sizes, 0, N.NLC_LAYOUT_ROW)
            for o, i in zip(outs, d):
                assert torch.equal(o, i), (px, ctas)
        ref = codec.sample(sizes, 0, 3)
        again = codec.sample(sizes, 0, 3, N.NLC_SCHED_RASTER)
        assert all(torch.equal(a, b) for a, b in zip(ref, again))
