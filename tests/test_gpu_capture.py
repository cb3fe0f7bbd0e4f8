"""The similarity calls that return nothing to the host, captured into a CUDA graph through the C ABI: a replay
reads the buffers it was captured with and nothing of the capturing call's stack, which has gone by then."""
import ctypes

import pytest
import torch

from paper_2412_14671_gb300 import _native, phantom

pytestmark = pytest.mark.gpu


def _grad(fn, F, W, w, kind, g):
    D, H, Wd = F.shape
    s = ctypes.c_void_p(torch.cuda.current_stream().cuda_stream or None)
    rc = fn(F.data_ptr(), W.data_ptr(), D, H, Wd, w, kind, ctypes.c_float(1e-6), None, g.data_ptr(), s)
    assert rc == _native.OK, _native.lib().muster_ops_last_error()


@pytest.mark.parametrize("name", ["muster_op_similarity", "muster_op_similarity_noalloc"])
@pytest.mark.parametrize("kind", [_native.SILNCC, _native.LNCC])
@pytest.mark.parametrize("shape", [(24, 30, 36), (19, 33, 41)])  # staged and unstaged widths
def test_captured_gradient_replays(name, kind, shape):
    fn = getattr(_native.lib(), name)
    F, W = (torch.from_numpy(x).cuda() for x in phantom.blob_series(shape, 2, seed=90, n_blobs=6)["images"])
    out, ref = torch.empty_like(W), torch.empty_like(W)
    s = torch.cuda.Stream()
    s.wait_stream(torch.cuda.default_stream())
    with torch.cuda.stream(s):
        _grad(fn, F, W, 5, kind, ref)  # the first call of a device is not captured
        s.synchronize()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=s):
            _grad(fn, F, W, 5, kind, out)
        for k in (1.0, 0.75):
            W.copy_(W * k + 0.125 * (1 - k) * F)
            out.zero_()
            graph.replay()
            s.synchronize()
            _grad(fn, F, W, 5, kind, ref)
            s.synchronize()
            assert float(ref.abs().max()) > 0 and torch.equal(out, ref), k
