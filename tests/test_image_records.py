"""The image records passed to the C ABI: pointer (8 bytes), H, W (4 bytes
each) per image, the same for a list of tensors and for a batch tensor, and
the tensors they point into kept alive with them."""
import struct

import pytest
import torch

from paper_2201_05213_gb300 import codec as CD
from paper_2201_05213_gb300 import nlc as N


@pytest.mark.parametrize("shape", [(1, 1, 1, 3), (5, 7, 9, 3), (3, 1, 40, 3)])
def test_batch_and_list_give_the_same_records(shape):
    b = torch.zeros(shape, dtype=torch.uint8)
    one, many = N._batch(b), N._images(list(b))
    assert one.data == many.data and one.n == many.n == shape[0]
    assert one.pixels == many.pixels == shape[0] * shape[1] * shape[2]
    assert CD._batch_images(b).data == many.data
    p, H, W = struct.unpack_from("=Qii", one.data, 16 * (shape[0] - 1))
    assert p == b[-1].data_ptr() and (H, W) == shape[1:3]
    assert one.tensors is b and len(many.tensors) == shape[0]


def test_views_and_empty_lists():
    b = torch.zeros((4, 6, 6, 3), dtype=torch.uint8)[::2]  # not contiguous as a whole
    rec = CD._batch_images(b)
    assert rec.data == N._images([b[0], b[1]]).data and rec.n == 2
    none = N._images([])
    assert none.n == 0 and none.pixels == 0 and len(none.data) == 16
