"""The windowed similarity and its adjoint where the 32 x 16 tiles, their D chunks and the two input
paths meet their edges, against the FP64 oracle: volumes of exactly one window, one tile of windows,
one more and one less, several D chunks, widths that are and are not multiples of 4, and buffers
that do not start on a 16-byte boundary (which take the unstaged path, with the same results).

Tolerances as everywhere: relative gradient (global L2) 1e-3, and relative loss 1e-5 for SiLNCC. (The
LNCC loss is 1 minus a correlation: on volumes of a few hundred windows, as here, the rounding of
the FP32 window sums is worth up to 1.4e-5 of it; it is gated on larger volumes elsewhere.)
"""
import numpy as np
import pytest
import torch

import oracle
import paper_2412_14671_gb300 as m
from paper_2412_14671_gb300 import phantom

pytestmark = pytest.mark.gpu

LOSS_RTOL = 1e-5
GRAD_RTOL = 1e-3


def _shapes(w):
    return [(w, w, w), (w + 1, 15 + w, 31 + w), (9, 16 + w, 32 + w), (w, 14 + w, 36), (35, 17, 40), (18, 33, 41)]


def _offset(x, n):
    """x on the GPU, starting n floats past an aligned address."""
    buf = torch.empty(x.size + n, device="cuda")
    buf[n:] = torch.from_numpy(np.ascontiguousarray(x)).cuda().reshape(-1)
    return buf[n:].view(x.shape)


@pytest.mark.parametrize("kind", [m.SILNCC, m.LNCC])
@pytest.mark.parametrize("w", [3, 5, 7, 9, 11])
def test_tile_and_chunk_edges(w, kind):
    for i, shape in enumerate(_shapes(w)):
        F, W = phantom.blob_series(shape, 2, seed=70 + i, n_blobs=6)["images"]
        s, g = m.op_similarity(_offset(F, 0), _offset(W, 0), w, kind)
        so, go = oracle.similarity(F, W, w, kind, 1e-6, grad=True)
        g = g.cpu().numpy()
        assert kind == m.LNCC or abs(s - so) <= LOSS_RTOL * max(abs(so), 1e-3), (shape, s, so)
        assert np.linalg.norm(g - go) <= GRAD_RTOL * np.linalg.norm(go), shape
        # the unstaged path: same sums, so the same values up to the re-sum's order along D
        s1, g1 = m.op_similarity(_offset(F, 1), _offset(W, 1), w, kind)
        assert kind == m.LNCC or abs(s1 - so) <= LOSS_RTOL * max(abs(so), 1e-3), (shape, s1, so)
        assert np.linalg.norm(g1.cpu().numpy() - go) <= GRAD_RTOL * np.linalg.norm(go), shape
