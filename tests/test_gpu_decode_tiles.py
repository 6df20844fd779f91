"""The decoder's tile shapes: every number of pixels per CTA and step at which
the network's split over warps, the coding groups or the number of tiles
changes, against the encoder (whose tables come from the all-pixels pipeline)
and, for the sampler, against one pixel per CTA.

n one-row images give a front of exactly n pixels per step, all on one CTA.
Equality is exact: a wrong table or network output anywhere desynchronises the
streams.
"""
import numpy as np
import pytest
import torch

import oracle as O
from paper_2201_05213_gb300 import nlc as N

from gpu_util import images, make_codec, to_dev

pytestmark = pytest.mark.gpu

CFGS = [(3, 64, 2, 10), (2, 48, 1, 16), (1, 32, 0, 5), (1, 16, 1, 1), (2, 64, 3, 8)]
COUNTS = [1, 2, 3, 4, 5, 8, 9, 15, 16, 17, 31, 32, 33, 48, 63, 64, 65, 81, 97, 127, 128, 129, 200]


@pytest.mark.parametrize("prec", [N.NLC_FP32, N.NLC_BF16, N.NLC_BF16_SHEARED])
@pytest.mark.parametrize("cfg", CFGS)
def test_every_tile_shape_decodes_the_encoders_streams(cfg, prec):
    codec, _ = make_codec(cfg, prec, seed=3, scale=1.5)
    pool = torch.cat([to_dev(i).reshape(-1, 3) for i in images(17, [(40, 60)])])
    for n in COUNTS:
        dimgs = [pool[11 * k:11 * k + 7 + k % 3].reshape(1, -1, 3).contiguous() for k in range(n)]
        sizes = [tuple(i.shape[:2]) for i in dimgs]
        N.nlc_set_tuning(codec.ctx, 1, 1)
        data, offs = codec.compress(dimgs, 0, N.NLC_LAYOUT_ROW)
        for sched in (N.NLC_SCHED_WAVEFRONT, N.NLC_SCHED_RASTER):
            outs = codec.decompress(data, offs, sizes, 0, N.NLC_LAYOUT_ROW, sched)
            for k in range(n):
                assert torch.equal(outs[k], dimgs[k]), (n, sched, k)
        if n in (3, 16, 17, 64, 81, 128):
            one = codec.sample(sizes, 0, 7)
            N.nlc_set_tuning(codec.ctx, 1, 0)
            many = codec.sample(sizes, 0, 7)
            assert all(torch.equal(a, b) for a, b in zip(one, many)), n


@pytest.mark.parametrize("prec", [N.NLC_FP32, N.NLC_BF16, N.NLC_BF16_SHEARED])
def test_rows_of_many_units_share_a_tile(prec):
    # fronts of several rows per unit: window pieces, halo rows and units that
    # end inside a tile
    codec, _ = make_codec((2, 32, 1, 10), prec, seed=4, scale=1.5)
    sizes = [(9, 5), (1, 1), (30, 14), (2, 40), (17, 3), (64, 64)]
    imgs = images(19, sizes)
    d = [to_dev(i) for i in imgs]
    for patch in (0, 13):
        data, offs = codec.compress(d, patch, N.NLC_LAYOUT_ROW)
        for ctas in (1, 3):
            N.nlc_set_tuning(codec.ctx, 1, ctas)
            outs = codec.decompress(data, offs, sizes, patch, N.NLC_LAYOUT_ROW)
            for o, i in zip(outs, imgs):
                assert np.array_equal(o.cpu().numpy(), i), (patch, ctas)


@pytest.mark.parametrize("K", [12, 13, 16])
def test_wide_heads_match_the_oracle(K):
    # 10 K outputs up to 160: the head's accumulator and the tensor-memory
    # operand beside it must not overlap
    cfg = (2, 48, 1, K)
    codec, w = make_codec(cfg, N.NLC_BF16, seed=6)
    img = images(5, [(20, 33)])[0]
    P, _ = codec.forward([to_dev(img)], 0)
    ref = O.forward_image(cfg, w, img).reshape(-1, 10 * K)
    assert np.abs(P.cpu().numpy().astype(np.float64) - ref).max() <= 2e-2


def test_a_small_plan_leaves_an_earlier_large_one_usable():
    # the kernels' shared-memory limit is set per function: a later plan of a
    # small batch must not lower it below an earlier plan's need
    codec, _ = make_codec((1, 32, 1, 5), N.NLC_BF16, seed=3)
    d = torch.cat([to_dev(i).reshape(-1, 3) for i in images(23, [(64, 64)])])
    many = [d[5 * k:5 * k + 9].reshape(1, 9, 3).contiguous() for k in range(700)]
    data, offs = codec.compress(many, 0, N.NLC_LAYOUT_ROW)
    large = codec.plan([(1, 9)] * 700, 0, N.NLC_LAYOUT_ROW)
    small = codec.plan([(1, 9)], 0, N.NLC_LAYOUT_ROW)
    large.run(data, offs)
    codec.check()
    assert all(torch.equal(a, b) for a, b in zip(large.outs, many))
    small.close()
    large.close()
