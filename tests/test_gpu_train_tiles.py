"""The FP32 trainer's tile shapes (channels, components, blocks, small tiles of
models whose weights leave no room for 32 pixels, ragged last tiles) against
the oracle's FP64 gradient, and bitwise determinism.

Tolerance: every gradient element is an FP32 sum over the pixels of products
of FP32 activations, each with a relative error of a few 2^-24 per layer, so
1e-4 of the largest element bounds it as in test_gpu_train.py.
"""
import numpy as np
import pytest
import torch

import oracle as O
from paper_2201_05213_gb300 import nlc as N
from paper_2201_05213_gb300 import synth

from gpu_util import DEV, ensure_built, make_codec

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    ensure_built()


@pytest.mark.parametrize("cfg,shape", [((1, 16, 0, 1), (1, 1, 1)), ((2, 48, 1, 7), (2, 5, 7)),
                                       ((1, 32, 2, 16), (1, 3, 11)), ((3, 64, 0, 13), (3, 9, 8)),
                                       ((1, 64, 3, 2), (2, 6, 9)), ((3, 64, 2, 5), (1, 33, 1))])
def test_fp32_gradient_every_tile_shape(cfg, shape):
    codec, w = make_codec(cfg, N.NLC_FP32, seed=8, scale=1.3)
    n, H, W = shape
    batch = np.stack([synth.make_image(9, 40, 40, index=k)[:H, :W] for k in range(n)])
    d = torch.from_numpy(batch).to(DEV)
    loss, grad = codec.loss_grad(d)
    ref_loss, ref = O.nll_grad(cfg, w.astype(np.float64), batch)
    assert abs(float(loss) - ref_loss) <= 1e-5 * ref_loss
    g = grad.cpu().numpy().astype(np.float64)
    assert np.abs(g - ref).max() <= 1e-4 * np.abs(ref).max()
    again, grad2 = codec.loss_grad(d)
    assert torch.equal(loss, again) and torch.equal(grad, grad2)


def test_fp32_gradient_many_tiles_per_cta_is_deterministic():
    # several tiles per CTA: the slots' reductions keep their order
    codec, _ = make_codec((2, 32, 1, 10), N.NLC_FP32, seed=8)
    d = torch.from_numpy(synth.random_crops(3, 24, size=32, source=64)).to(DEV)
    loss, grad = codec.loss_grad(d)
    for _ in range(5):
        l2, g2 = codec.loss_grad(d)
        assert torch.equal(loss, l2) and torch.equal(grad, g2)


@pytest.mark.parametrize("cfg,shape", [((2, 48, 1, 16), (2, 16, 16)), ((3, 64, 2, 13), (1, 9, 31)),
                                       ((1, 16, 0, 1), (1, 3, 5)), ((3, 64, 2, 10), (3, 20, 20)),
                                       ((1, 32, 2, 6), (5, 11, 13))])
def test_bf16_gradient_every_plan(cfg, shape):
    # BF16 operands: the tolerance of test_gpu_train.py (relative L2 error
    # 3e-2, every element within 5e-2 of the largest, loss within 0.03 bits)
    codec, w = make_codec(cfg, N.NLC_BF16, seed=8)
    n, H, W = shape
    batch = np.stack([synth.make_image(9, 40, 40, index=k)[:H, :W] for k in range(n)])
    d = torch.from_numpy(batch).to(DEV)
    loss, grad = codec.loss_grad(d)
    ref_loss, ref = O.nll_grad(cfg, w.astype(np.float64), batch)
    assert abs(float(loss) - ref_loss) <= 0.03
    g = grad.cpu().numpy().astype(np.float64)
    assert np.linalg.norm(g - ref) <= 3e-2 * np.linalg.norm(ref)
    assert np.abs(g - ref).max() <= 5e-2 * np.abs(ref).max()
    again, grad2 = codec.loss_grad(d)
    assert torch.equal(loss, again) and torch.equal(grad, grad2)
