"""The forward warp where its cells, its node walk and its 32 x 16 voxel tiles meet the volume's
edges: axes of 1 to 3 voxels, odd extents, one voxel more and less than a tile, and displacements
that leave the volume on either side (coordinates clamped to the grid, derivative 0 there).

Constant velocities displace every voxel by exactly 2 c image voxels, so the warped image is scipy's
linear interpolation with replicated edges. Sample points are rounded to a few 1e-6 voxel and the
images stay below 1.2 with differences below 1 between neighbours: 1e-5 absolute.
"""
import numpy as np
import pytest
import scipy.ndimage as ndi
import torch

import oracle
import paper_2412_14671_gb300 as m
from paper_2412_14671_gb300 import phantom

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape", [(1, 5, 33), (2, 2, 2), (3, 1, 64), (7, 16, 32), (9, 17, 35), (34, 15, 31), (70, 18, 65)])
def test_warped_image_at_and_beyond_the_edges(shape):
    rng = np.random.default_rng(5)
    imgs = rng.uniform(0.1, 1.0, size=(2,) + shape).astype(np.float32)
    nf = tuple((a + 1) // 2 for a in shape)
    grid = np.stack(np.meshgrid(*[np.arange(a, dtype=np.float64) for a in shape], indexing="ij"))
    with m.Muster(shape, 2, n_squarings=2, window=3) as reg:
        reg.set_images(torch.from_numpy(imgs).cuda())
        reg.set_level(0)
        for c in ([0.0, 0.0, 0.0], [0.25, -0.5, 0.125], [-0.75, 3.25, -1.5], [40.0, -40.0, 0.375], [-40.0, 0.5, 40.0]):
            v = np.broadcast_to(np.array(c, dtype=np.float32).reshape(1, 3, 1, 1, 1), (1, 3) + nf)
            reg.set_velocity(np.ascontiguousarray(v))
            for j, i, sign in ((1, 0, 1.0), (0, 1, -1.0)):
                got = reg.get_field(m.WARPED, i, j, level=0, device=False)
                q = grid + 2 * sign * np.array(c).reshape(3, 1, 1, 1)
                ref = ndi.map_coordinates(imgs[j].astype(np.float64), q, order=1, mode="nearest")
                assert np.abs(got - ref).max() < 1e-5, (c, j, i)


@pytest.mark.parametrize("shape", [(12, 14, 36), (11, 19, 33), (5, 34, 30)])
def test_gradient_with_samples_outside(shape):
    """Loss and gradient when part of the samples leave the volume (their derivative is 0)."""
    imgs = phantom.blob_series(shape, 2, seed=81, n_blobs=8)["images"]
    nf = tuple((a + 1) // 2 for a in shape)
    phi = phantom.smooth_velocity(nf, 1, seed=81, sigma=2.0, rms=0.6) + np.float32(1.3)
    g = torch.empty((1, 3) + nf, device="cuda")
    with m.Muster(shape, 2, n_squarings=5, window=3, alpha_ss=0.1, alpha_l2=0.01) as reg:
        reg.set_images(torch.from_numpy(imgs).cuda())
        loss = reg.eval(torch.from_numpy(phi).cuda(), 0, g)
    p = oracle.params(K=5, window=3, alpha_ss=0.1, alpha_l2=0.01, alpha_ts=0.0)
    lo, _, go = oracle.loss_grad(imgs, phi, p)
    assert abs(loss - lo) <= 1e-5 * abs(lo)
    assert np.linalg.norm(g.cpu().numpy() - go) <= 1e-3 * np.linalg.norm(go)
