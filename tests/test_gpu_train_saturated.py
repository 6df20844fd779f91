"""FP32 training gradients that pass through saturated units (ELU' = e^x far
below zero) against the oracle's FP64 gradient, row by row.

Tolerance: the derivative's relative error is the pre-activation's absolute
error, a sum of at most 72 products and a bias of magnitude below 32 in all,
hence below 74 * 2^-24 * 32 = 1.4e-4; the gradient that reaches the unit adds
its own error (1e-4 of the largest element, as in test_gpu_train.py) over sums
of a few hundred pixels.  1e-3 of the row's norm bounds both.  A derivative
taken as ELU + 1 keeps 2^-24 / e^x of its bits: 1e-2 at x = -12, none at -18.
"""
import numpy as np
import pytest
import torch

import oracle as O
from paper_2201_05213_gb300 import codec as CD
from paper_2201_05213_gb300 import nlc as N
from paper_2201_05213_gb300 import synth

from gpu_util import DEV

pytestmark = pytest.mark.gpu


def _check_rows(g, ref):
    assert g.shape == ref.shape
    norm = np.linalg.norm(ref, axis=1)
    assert norm.min() > 0
    assert (np.linalg.norm(g - ref, axis=1) <= 1e-3 * norm).all(), \
        (np.linalg.norm(g - ref, axis=1) / norm).max()


@pytest.mark.parametrize("cfg", [(3, 64, 0, 10), (1, 16, 0, 1), (2, 48, 1, 7), (3, 64, 2, 5),
                                 (1, 64, 3, 2)])
def test_rows_of_saturated_units(cfg):
    h, C, R, K = cfg
    F = 6 * h * (h + 1)
    w = synth.xavier_weights(h, C, R, K, seed=12).astype(np.float32)
    # every second unit of one layer at about -11 .. -25: the first layer without
    # residual blocks, else the hidden layer of the last block
    rows = np.arange(0, C, 2)
    if R == 0:
        w0, b0, cols = 0, C * F, F
    else:
        w0 = C * F + C + (R - 1) * 2 * (C * C + C)
        b0, cols = w0 + C * C, C
    w[b0 + rows] = -11.0 - 14.0 * rows / C
    batch = np.stack([synth.make_image(9, 40, 40, index=k)[:7, :11] for k in range(3)])
    codec = CD.Codec(h, C, R, K, N.NLC_FP32, w)
    _, grad = codec.loss_grad(torch.from_numpy(batch).to(DEV))
    _, ref = O.nll_grad(cfg, w.astype(np.float64), batch)
    g = grad.cpu().numpy().astype(np.float64)
    _check_rows(g[w0:w0 + C * cols].reshape(C, cols)[rows], ref[w0:w0 + C * cols].reshape(C, cols)[rows])
    _check_rows(g[b0:b0 + C][rows, None], ref[b0:b0 + C][rows, None])
