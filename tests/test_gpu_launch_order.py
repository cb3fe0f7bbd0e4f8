"""Kernels whose CTAs start before their predecessor has finished: results in stream order and under capture."""
import pytest
import torch

import paper_2412_14671_gb300 as m

pytestmark = pytest.mark.gpu


def chain(phi):
    return m.op_jacobian_det(m.op_exp(phi, 6))


# one CTA to several waves per kernel; the legacy default stream and a stream of the caller
@pytest.mark.parametrize("shape", [(4, 5, 6), (24, 24, 24), (70, 65, 64)])
@pytest.mark.parametrize("own", [False, True])
def test_calls_in_flight_keep_their_order(shape, own):
    """Chains of dependent kernels issued without waiting, over reused scratch and with other kernels
    between them, give bit for bit what each gives alone."""
    phis = [torch.randn((3,) + shape, device="cuda") for _ in range(12)]
    alone = []
    for p in phis:
        alone.append(chain(p).clone())
        torch.cuda.synchronize()
    with torch.cuda.stream(torch.cuda.Stream() if own else torch.cuda.default_stream()):
        torch.cuda.current_stream().wait_stream(torch.cuda.default_stream())
        flight = [chain(p * 2 / 2) + 0 for p in phis]
        torch.cuda.current_stream().synchronize()
    for a, b in zip(alone, flight):
        assert torch.equal(a, b)


def test_captured_calls_match_plain_ones():
    phi = torch.randn((3, 20, 24, 28), device="cuda")
    ref = chain(phi)
    s = torch.cuda.Stream()
    s.wait_stream(torch.cuda.default_stream())
    with torch.cuda.stream(s):
        chain(phi)
        s.synchronize()
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=s):
            out = chain(phi)
        for k in (1.0, -0.5):
            phi.copy_(phi * k)
            g.replay()
            s.synchronize()
            assert torch.equal(out, chain(phi)), k
    assert ref.shape == out.shape
