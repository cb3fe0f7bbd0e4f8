"""The scratch that the stateless calls keep goes back to the device when a context's allocator refuses a block, and
the block is asked for once more."""
import numpy as np
import pytest
import torch

import paper_2412_14671_gb300 as m
from paper_2412_14671_gb300 import _native, phantom

pytestmark = pytest.mark.gpu

SHAPE, N = (24, 20, 28), 3


@pytest.mark.parametrize("refused", [0, 7])  # which request is refused the first time
def test_a_refused_block_is_asked_for_again_with_the_pool_given_back(refused):
    m.op_exp(torch.zeros((3, 128, 128, 128), device="cuda"), 2)  # leaves 8 * 128^3 floats (64 MiB) in the pool
    torch.cuda.synchronize()
    asked, free, live = [], [], set()
    stream = torch.cuda.default_stream()

    def alloc(nbytes, user):
        asked.append(int(nbytes))
        if len(asked) - 1 == refused or len(asked) - 2 == refused:
            free.append(torch.cuda.mem_get_info()[0])
        if len(asked) - 1 == refused:
            return None
        p = torch.cuda.caching_allocator_alloc(int(nbytes), torch.cuda.current_device(), stream)
        live.add(p)
        return p

    def release(ptr, user):
        live.discard(ptr)
        torch.cuda.caching_allocator_delete(ptr)

    fns = (_native.ALLOC_FN(alloc), _native.FREE_FN(release))
    with m.Muster(SHAPE, N, allocator=fns, n_levels=1, steps_per_level=[2], window=3) as reg:
        assert asked[refused] == asked[refused + 1]
        assert free[1] - free[0] >= 64 * 2**20  # both queries without a block in between
        reg.set_images(torch.from_numpy(np.ascontiguousarray(phantom.blob_series(SHAPE, N, seed=3)["images"])).cuda())
        assert np.isfinite(reg.run())
    assert not live
