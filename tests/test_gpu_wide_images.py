"""Two rows of more than 2^31 / 3 pixels: the row's stride in bytes does not fit
in 31 bits.  The code length of pixels next to the right end equals that of a
crop (the context is local), and the containers decode to the image."""
import pytest
import torch

from paper_2201_05213_gb300 import nlc as N

from gpu_util import DEV, make_codec

pytestmark = pytest.mark.gpu

W = (1 << 31) // 3 + 1000


@pytest.fixture(scope="module")
def wide():
    if torch.cuda.get_device_properties(0).total_memory < 100 << 30:
        pytest.skip("takes 45 GB")
    g = torch.Generator(device=DEV)
    g.manual_seed(3)
    img = torch.empty((2, W, 3), dtype=torch.uint8, device=DEV)
    img.random_(0, 256, generator=g)
    yield img
    del img
    torch.cuda.empty_cache()


@pytest.mark.parametrize("prec", [N.NLC_FP32, N.NLC_BF16, N.NLC_BF16_SHEARED])
def test_code_length_at_the_end_of_a_wide_row(wide, prec):
    codec, _ = make_codec((1, 16, 0, 1), prec, seed=2)
    _, bits = codec.forward([wide], 0, params=False, bits=True)
    bits = bits.view(2, W)
    for x0 in (W - 300, (1 << 31) // 3 - 200):
        _, crop = codec.forward([wide[:, x0:x0 + 300].contiguous()], 0, params=False, bits=True)
        crop = crop.view(2, 300)
        n = 300 if x0 + 300 == W else 290
        assert torch.equal(bits[:, x0 + 8:x0 + n], crop[:, 8:n])
    codec.close()
    torch.cuda.empty_cache()


def test_round_trip_of_a_wide_image(wide):
    codec, _ = make_codec((1, 16, 0, 1), N.NLC_BF16, seed=2)
    data, offs = codec.compress([wide], 1 << 16)
    out = codec.decompress(data, offs, [(2, W)], 1 << 16)[0]
    assert torch.equal(out, wide)
    codec.close()
    torch.cuda.empty_cache()
