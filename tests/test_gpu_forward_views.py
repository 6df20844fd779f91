"""nlc_forward writes its outputs to any array of floats: views that start at
every float of a 16-byte line give the bits of an aligned buffer and leave the
floats around them alone."""
import pytest
import torch

from paper_2201_05213_gb300 import nlc as N

from gpu_util import DEV, images, make_codec, to_dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", [N.NLC_FP32, N.NLC_BF16, N.NLC_BF16_SHEARED])
@pytest.mark.parametrize("cfg", [(3, 64, 2, 10), (1, 16, 0, 1)])
def test_outputs_at_any_float(cfg, prec):
    codec, _ = make_codec(cfg, prec, seed=2)
    d = [to_dev(i) for i in images(31, [(5, 7), (3, 4)])]
    n = 47
    P0, B0 = codec.forward(d, 0, bits=True)
    for off in (1, 2, 3):
        P = torch.full((n * 10 * cfg[3] + 8,), -77.0, device=DEV)
        B = torch.full((n + 8,), -77.0, device=DEV)
        end = off + n * 10 * cfg[3]
        N.nlc_forward(codec.ctx, d, 0, P[off:end], B[off:off + n])
        codec.check()
        assert torch.equal(P[off:end].view(n, -1), P0)
        assert torch.equal(B[off:off + n], B0)
        assert bool((P[:off] == -77).all()) and bool((P[end:] == -77).all())
        assert bool((B[:off] == -77).all()) and bool((B[off + n:] == -77).all())
