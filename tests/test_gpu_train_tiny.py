"""Weight gradients below the smallest normal float: upstream gradients that are
integers times a power of two, on a network whose head input is exactly 1, so
that every sum of the head's weight and bias gradients is exact in FP32 and the
result has to be the integer sum times that power, bit for bit."""
import numpy as np
import pytest
import torch

from paper_2201_05213_gb300 import codec as CD
from paper_2201_05213_gb300 import nlc as N

from gpu_util import DEV

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec,exps", [(N.NLC_FP32, (0, -100, -120, -130, -149)),
                                       (N.NLC_BF16, (0, -100, -120, -130, -133))])
@pytest.mark.parametrize("shape", [(1, 3, 5), (3, 128, 128)])
def test_head_gradient_is_exact_at_any_scale(shape, prec, exps):
    h, C, R, K = 1, 16, 0, 5
    w = np.zeros(N.nlc_num_weights(h, C, R, K, prec), dtype=np.float32)
    F = 6 * h * (h + 1)
    w[C * F:C * F + C] = 1.0  # b0: the head's input is ELU(1) = 1
    codec = CD.Codec(h, C, R, K, prec, w)
    rng = np.random.default_rng(4)
    batch = torch.from_numpy(rng.integers(0, 256, (*shape, 3), dtype=np.uint8)).to(DEV)
    d = rng.integers(-1, 2, (int(np.prod(shape)), 10 * K)).astype(np.float64)
    d[:, 3] = 0.0
    for e in exps:
        up = torch.from_numpy(np.ldexp(d, e).astype(np.float32)).to(DEV)
        g = codec.backward(batch, up).cpu().numpy().astype(np.float64)
        want = np.ldexp(d.sum(axis=0), e)
        gw = g[C * F + C:C * F + C + 10 * K * C].reshape(10 * K, C)
        assert np.array_equal(g[-10 * K:], want), e
        assert np.array_equal(gw, np.repeat(want[:, None], C, axis=1)), e
