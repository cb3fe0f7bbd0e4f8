"""Contexts without the cells of their images (plain_images, or a device that refuses the cells' block): the forward
warp samples the images themselves, with the same results bit for bit, and everything that needs the warp runs."""
import numpy as np
import pytest
import torch

import paper_2412_14671_gb300 as m
from paper_2412_14671_gb300 import _native, phantom

pytestmark = pytest.mark.gpu


def _results(shape, N, allocator=None, **kw):
    """gradient and loss of an evaluation with displacements that leave the volume, a registration's
    velocities and a warped image"""
    imgs = torch.from_numpy(phantom.blob_series(shape, N, seed=17)["images"]).cuda()
    nf = [(a + 1) // 2 for a in shape]
    v = 2.0 * torch.randn([N - 1, 3] + nf, generator=torch.Generator(device="cuda").manual_seed(3), device="cuda")
    with m.Muster(shape, N, allocator=allocator, n_levels=1, steps_per_level=[4], n_squarings=4, window=3, deterministic=1,
                  **kw) as reg:
        reg.set_images(imgs)
        g = torch.zeros_like(v)
        loss = reg.eval(v, 0, g)
        reg.run()
        return [torch.tensor(loss), g, reg.velocities(0), reg.get_field(m.WARPED, 0, N - 1, level=0)]


@pytest.mark.parametrize("rigid", [0, 1])
@pytest.mark.parametrize("shape,N", [((16, 20, 24), 3), ((13, 9, 35), 4), ((1, 12, 33), 3), ((5, 1, 64), 2)])
def test_same_bits_without_cells(shape, N, rigid):
    for a, b in zip(_results(shape, N, rigid=rigid), _results(shape, N, rigid=rigid, plain_images=1)):
        assert torch.equal(a, b)


def test_a_refused_block_of_cells_leaves_a_working_context():
    shape, N = (13, 9, 35), 4
    cells = 8 * N * (shape[0] + 2) * (shape[1] + 2) * (shape[2] + 1)
    stream, live, refused = torch.cuda.default_stream(), set(), []

    def alloc(nbytes, user):
        if abs(int(nbytes) - cells) < 256:
            refused.append(int(nbytes))
            return None
        p = torch.cuda.caching_allocator_alloc(int(nbytes), torch.cuda.current_device(), stream)
        live.add(p)
        return p

    def release(ptr, user):
        live.discard(ptr)
        torch.cuda.caching_allocator_delete(ptr)

    fns = (_native.ALLOC_FN(alloc), _native.FREE_FN(release))
    for a, b in zip(_results(shape, N), _results(shape, N, allocator=fns)):
        assert torch.equal(a, b)
    assert len(refused) == 2 and not live  # refused, and refused again after the pool was given back


def test_memory_without_cells():
    shape, N = (96, 112, 96), 6
    kw = dict(n_levels=1, steps_per_level=[1], window=7)
    cells = 8 * N * (shape[0] + 2) * (shape[1] + 2) * (shape[2] + 1)
    assert 0 <= m.footprint(shape, N, **kw) - m.footprint(shape, N, plain_images=1, **kw) - cells < 256
    need = m.footprint(shape, N, plain_images=1, **kw)
    torch.cuda.synchronize()
    free = torch.cuda.mem_get_info()[0]
    with m.Muster(shape, N, plain_images=1, **kw):
        took = free - torch.cuda.mem_get_info()[0]
    assert need <= took <= need * 1.02 + 64 * 2**20, (need, took)


@pytest.mark.parametrize("plain", [0, 1])
@pytest.mark.parametrize("at", [(0, 0, 0, 0), (2, 12, 8, 34), (1, 0, 8, 33), (0, 12, 0, 1), (2, 6, 4, 17)])
@pytest.mark.parametrize("value", [np.nan, np.inf, -np.inf])
def test_non_finite_images_are_refused(plain, at, value):
    """the first and last voxel of the series, edges and the middle; the context takes good images afterwards"""
    shape, N = (13, 9, 35), 3
    imgs = phantom.blob_series(shape, N, seed=18)["images"]
    bad = imgs.copy()
    bad[at] = value
    with m.Muster(shape, N, n_levels=2, steps_per_level=[1, 1], window=3, plain_images=plain) as reg:
        with pytest.raises(m.MusterError) as e:
            reg.set_images(torch.from_numpy(bad).cuda())
        assert e.value.code == _native.EINVAL
        with pytest.raises(m.MusterError):
            reg.run()
        reg.set_images(torch.from_numpy(imgs).cuda())
        assert np.isfinite(reg.run())


def test_large_cells_leave_room_on_a_nearly_full_device():
    """with room for the cells but little more, a context leaves them out, with the same results"""
    shape, N = (128, 128, 128), 6
    kw = dict(n_levels=1, steps_per_level=[1], n_squarings=4, window=3, deterministic=1, pair_batch=4)
    lean, full = m.footprint(shape, N, plain_images=1, **kw), m.footprint(shape, N, **kw)
    assert full - lean > 64 * 2**20
    imgs = torch.rand((N,) + shape, generator=torch.Generator(device="cuda").manual_seed(4), device="cuda")
    v = torch.randn([N - 1, 3, 64, 64, 64], generator=torch.Generator(device="cuda").manual_seed(5), device="cuda")
    grads = []
    for fill in (False, True):
        torch.cuda.synchronize()
        torch.cuda.empty_cache()
        free = torch.cuda.mem_get_info()[0]
        filler = torch.empty(free - full - (384 << 20), dtype=torch.uint8, device="cuda") if fill else None  # never touched
        free = torch.cuda.mem_get_info()[0]
        with m.Muster(shape, N, **kw) as reg:
            took = free - torch.cuda.mem_get_info()[0]
            assert (took < lean + (full - lean) // 2) == fill, (took, lean, full)
            reg.set_images(imgs)
            grads.append(torch.zeros_like(v))
            reg.eval(v, 0, grads[-1])
        del filler
        torch.cuda.empty_cache()
    assert torch.equal(*grads)
