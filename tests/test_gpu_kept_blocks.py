"""The context's kept device blocks: the cost of an allocation beside many kept blocks, streams that are left,
refusals under capture and beside other contexts."""
import time

import numpy as np
import pytest
import torch

from paper_1908_06972_gb300 import synth

pytestmark = pytest.mark.gpu

SEED = (0x5EED, 21, 22, 23)


def words(pf, ctx, level):
    info = pf.pft_ctx_info(ctx)
    return torch.from_numpy(synth.residues(1, info["primes"][:level], info["N"], polys=2).view(np.int64)).cuda()


def test_many_kept_blocks_cost_nothing(gpu):
    """New handles of a size that no kept block has (each is a look at the kept blocks and a request to the
    allocator) take as long beside 40000 kept blocks as beside none; a walk over them would take ten times as long."""
    pf = gpu
    ctx = pf.pft_ctx_create(4, 6, 1, 1, 60, 40, 60, 2.0 ** 40, SEED, flags=pf.PFT_ALLOW_INSECURE, allocator=None)
    w = words(pf, ctx, 6)
    handles = []

    def create(level, n):
        t0 = time.perf_counter()
        for _ in range(n):
            h = pf.pft_ct_create(ctx)
            pf.pft_ct_reduce_sum(ctx, w.data_ptr(), level, 2.0 ** 40, 1, h)
            handles.append(h)
        return (time.perf_counter() - t0) / n

    def fastest():
        out = []
        for _ in range(8):
            out.append(create(6, 50))
            torch.cuda.synchronize()
        return min(out)

    create(6, 50)
    before = fastest()
    torch.cuda.synchronize()
    n = len(handles)
    create(2, 40000)
    torch.cuda.synchronize()
    for h in handles[n:]:
        pf.pft_ct_destroy(h)
    del handles[n:]
    after = fastest()
    assert after < 3 * before, (before, after)
    for h in handles:
        pf.pft_ct_destroy(h)
    pf.pft_ctx_destroy(ctx)
