"""Evaluations of one context issued one after the other without waiting, with exact sums: every kernel of the chain
(overlapping and plain launches, memsets and table copies between them, several pair batches) gives bit for bit what
it gives alone."""
import pytest
import torch

import paper_2412_14671_gb300 as m
from paper_2412_14671_gb300 import _native, phantom

pytestmark = pytest.mark.gpu


def _eval(reg, v, grad):
    """loss not asked for, so the call returns before the GPU has run it"""
    assert _native.lib().muster_eval(reg._ctx, v.data_ptr(), 0, None, grad.data_ptr()) == _native.OK


@pytest.mark.parametrize("own", [False, True])
@pytest.mark.parametrize("shape,window,kind,extra", [
    ((24, 20, 28), 3, m.SILNCC, {}),
    ((33, 48, 37), 7, m.SILNCC, dict(pair_batch=5, rigid=1)),
    ((40, 24, 64), 5, m.LNCC, dict(pair_batch=3, smooth_omega=0.1)),
    ((33, 20, 64), 11, m.LNCC, dict(pair_batch=7, recompute_squaring=1)),
])
def test_evaluations_in_flight_keep_their_order(shape, window, kind, extra, own):
    N = 4
    nf = [(a + 1) // 2 for a in shape]
    imgs = torch.from_numpy(phantom.blob_series(shape, N, seed=95)["images"]).cuda()
    gen = torch.Generator(device="cuda").manual_seed(5)
    vs = [0.4 * torch.randn([N - 1, 3] + nf, generator=gen, device="cuda") for _ in range(6)]
    stream = torch.cuda.Stream() if own else torch.cuda.default_stream()
    torch.cuda.synchronize()
    with m.Muster(shape, N, n_levels=1, steps_per_level=[1], n_squarings=5, window=window, similarity=kind,
                  deterministic=1, **extra) as reg, torch.cuda.stream(stream):
        reg.set_stream(stream.cuda_stream)
        reg.set_images(imgs)
        alone = []
        for v in vs:
            alone.append(torch.zeros_like(v))
            _eval(reg, v, alone[-1])
            torch.cuda.synchronize()
        flight = [torch.zeros_like(v) for v in vs]
        for v, g in zip(vs, flight):
            _eval(reg, v, g)
        torch.cuda.synchronize()
    for a, b in zip(alone, flight):
        assert float(a.abs().max()) > 0 and torch.equal(a, b)
