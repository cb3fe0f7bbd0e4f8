"""The LNCC loss where tiles, D chunks and the two input paths meet their edges, against the FP64 oracle.

The loss is the mean over the windows of 1 - a correlation in [-1, 1], which divides window sums of variances: in
windows of little variance about the tile's shift the FP32 rounding of the sums is worth up to 3e-4 of a term. The
same sums in FP32 on the host (the shift, products and box sums of the kernel, added one after the other) put the
mean of these volumes within 3.4e-6 of the FP64 value; the gate is 2e-5, six times that. A lost or doubled window among
the at most 2,600 of a volume is worth the loss divided by their number, 4e-5 or more.
"""
import numpy as np
import pytest
import torch

import oracle
import paper_2412_14671_gb300 as m
from paper_2412_14671_gb300 import phantom

pytestmark = pytest.mark.gpu


def _offset(x, n):
    """x on the GPU, starting n floats past an aligned address."""
    buf = torch.empty(x.size + n, device="cuda")
    buf[n:] = torch.from_numpy(np.ascontiguousarray(x)).cuda().reshape(-1)
    return buf[n:].view(x.shape)


@pytest.mark.parametrize("w", [3, 5, 7, 9, 11])
def test_loss_counts_every_window_once(w):
    shapes = [(w, w, w), (w + 1, w + 2, w + 31), (w, w + 15, 32 + w), (w + 2, w + 16, w + 32), (w + 17, w + 7, 20), (w + 33, w + 3, w + 5)]
    for i, shape in enumerate(shapes):
        assert np.prod([a - w + 1 for a in shape]) <= 2600
        F, W = phantom.blob_series(shape, 2, seed=120 + i, n_blobs=6)["images"]
        so, _ = oracle.similarity(F, W, w, m.LNCC, 1e-6, grad=True)
        for off in (0, 1):  # the staged path where the width allows it, and the unstaged one
            s = m.op_similarity(_offset(F, off), _offset(W, off), w, m.LNCC, grad=False)
            assert abs(s - so) <= 2e-5, (shape, off, s, so)
