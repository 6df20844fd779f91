"""Tiles that the batch does not fill: the pixels past its end add nothing to the
gradient, whatever the likelihood of a made-up pixel under the model would be.

All pixels are white and every location lies at 1e36 with the smallest scale, so
that the model gives white probability 1 (loss and gradient are exactly 0) and
any other value probability 0.
"""
import numpy as np
import pytest
import torch

from paper_2201_05213_gb300 import codec as CD
from paper_2201_05213_gb300 import nlc as N

from gpu_util import DEV

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", [N.NLC_FP32, N.NLC_BF16])
@pytest.mark.parametrize("shape", [(1, 1, 1), (1, 3, 5), (2, 7, 9), (1, 4, 32)])
def test_pixels_past_the_batch(shape, prec):
    h, C, R, K = 1, 16, 0, 1
    w = np.zeros(N.nlc_num_weights(h, C, R, K, prec), dtype=np.float32)
    w[-9 * K:-6 * K] = 1e36   # locations
    w[-6 * K:-3 * K] = -8.0   # log-scales (clamped at -7)
    codec = CD.Codec(h, C, R, K, prec, w)
    batch = torch.full((*shape, 3), 255, dtype=torch.uint8, device=DEV)
    loss, grad = codec.loss_grad(batch)
    assert float(loss) == 0.0
    assert bool((grad == 0).all())
