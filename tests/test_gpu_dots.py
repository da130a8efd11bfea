"""Sums of HMULPLAIN products (pft_dot_plain_batch) against exact integers, at the edges of the kernel's groups of
terms (4 loads, 8 products per reduction, 64 pointers per chunk), with residues at their maximum and
60-bit, 50-bit and 20-bit primes."""
import numpy as np
import pytest
import torch

from .pairs import Pair

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("logn,bits", [(4, (60, 50, 60)), (6, (60, 60, 60)), (12, (60, 40, 60)), (4, (20, 20, 21))])
@pytest.mark.parametrize("K,n_out,shared", [(1, 1, True), (3, 2, True), (4, 1, False), (5, 3, True), (8, 2, False),
                                            (9, 2, True), (64, 1, True), (65, 2, False), (131, 2, True)])
def test_dot_plain(gpu, logn, bits, K, n_out, shared):
    p = Pair(gpu, logn, 3, 1, 1, first_bits=bits[0], mid_bits=bits[1], special_bits=bits[2], gpu_keys=False,
             rot_steps=(), relin=False)
    try:
        pf, ctx, L = p.pft, p.ctx, 3
        q = pf.pft_ctx_info(ctx)["primes"][:L]
        rng = np.random.default_rng(K * 100 + n_out)
        # evaluation-form words go in through the integer sum of one term; plaintexts through their
        # coefficient form of one coefficient (a constant polynomial has the same value everywhere)
        words = np.stack([rng.integers(0, qi, (n_out * K, 2, p.N), dtype=np.uint64) for qi in q], axis=2)
        words[: max(1, K // 2)] = np.array([qi - 1 for qi in q], np.uint64)[None, None, :, None]
        consts = np.stack([rng.integers(0, qi, K if shared else n_out * K, dtype=np.uint64) for qi in q], axis=1)
        consts[: max(1, K // 2)] = np.array([qi - 1 for qi in q], np.uint64)
        cts, pts = [], []
        for w in words:
            h = p.empty()
            d = torch.from_numpy(np.ascontiguousarray(w).view(np.int64)).cuda()
            pf.pft_ct_reduce_sum(ctx, d.data_ptr(), L, 1.0, 1, h)
            cts.append(h)
        for c in consts:
            m = np.zeros((L, p.N), np.uint64)
            m[:, 0] = c
            h = pf.pft_pt_import(ctx, m, 1.0)
            p.handles.append(("pt", h))
            pts.append(h)
        outs = [p.empty() for _ in range(n_out)]
        pf.pft_dot_plain_batch(ctx, cts, pts, K, outs, pts_shared=shared)
        for o, h in enumerate(outs):
            got = torch.empty((2, L, p.N), dtype=torch.int64, device="cuda")
            pf.pft_ct_copy_out(ctx, h, got.data_ptr())
            got = got.cpu().numpy().view(np.uint64)
            for r, qi in enumerate(q):
                x = words[o * K:(o + 1) * K, :, r].astype(object)
                c = consts[:K, r] if shared else consts[o * K:(o + 1) * K, r]
                want = (x * c.astype(object)[:, None, None]).sum(axis=0) % int(qi)
                assert np.array_equal(got[:, r].astype(object), want), (o, r)
    finally:
        p.close()
