"""Flow-grid smoothing and the Jacobian determinant at the edges of their runs and layouts."""
import numpy as np
import pytest
import torch

import oracle
import paper_2412_14671_gb300 as m

pytestmark = pytest.mark.gpu


# Flow axes of 1 to 9 nodes (less, equal and more than one run of 8 outputs), rows on both sides of the
# longest staged row (256 nodes), a last group of rows that is not full; few taps and the whole circle.
# Each axis adds at most its length in products whose weights sum to about 1: (m0 + m1 + m2) half ulps
# of the largest velocity.
@pytest.mark.parametrize("shape", [(2, 6, 16), (16, 18, 14), (14, 2, 66), (4, 6, 512), (4, 6, 514), (5, 70, 600)])
@pytest.mark.parametrize("omega", [0.15, 0.02])
def test_smoothing_runs(shape, omega):
    nf = tuple((a + 1) // 2 for a in shape)
    theta = np.random.default_rng(4).normal(size=(1, 3) + nf).astype(np.float32)
    with m.Muster(shape, 2, n_squarings=2, window=3, smooth_omega=omega) as reg:
        reg.set_images(torch.rand((2,) + shape, device="cuda"))
        reg.set_level(0)
        reg.set_velocity(theta)
        v = reg.get_field(m.VELOCITY, 0, level=0, device=False)
    vo = np.stack([oracle.smooth(theta[0, c].astype(np.float64), omega, (2.0, 2.0, 2.0)) for c in range(3)])
    assert np.abs(v - vo).max() <= (sum(nf) + 3) * 2.0**-24 * np.abs(theta).max()


# Rows of 1, 2 and 33 runs of 4 voxels, of runs of 2 and single voxels of two rows (an odd number of rows, one
# row), lanes at both ends of a warp, and fields that start 4 or 8 bytes off a 16-byte boundary;
# tolerance of the determinant's 12 products of values up to about 3.
@pytest.mark.parametrize("shape", [(3, 2, 4), (1, 1, 8), (5, 3, 132), (70, 9, 12), (3, 5, 2), (6, 7, 66), (4, 1, 35), (9, 5, 97)])
@pytest.mark.parametrize("shift", [0, 1, 2])
def test_jacobian_runs(shape, shift):
    n = 3 * int(np.prod(shape))
    flat = torch.zeros(n + 4, device="cuda")
    u = flat[shift:shift + n].view((3,) + shape)
    u.copy_(torch.from_numpy(np.random.default_rng(6).normal(scale=0.4, size=(3,) + shape)))
    ref = oracle.jacobian_det(u.cpu().numpy())
    assert np.abs(m.op_jacobian_det(u).cpu().numpy() - ref).max() <= 2e-5 * max(1.0, np.abs(ref).max())
