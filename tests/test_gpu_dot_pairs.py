"""Sums of HMULPLAIN products whose outputs fill the GPU (both polynomials of an output per thread) against exact
integers at some coefficients: the edges of the groups of terms (4 loads, 8 products per reduction, 64 pointers
per chunk), plaintexts shared by the outputs and of their own, maximal residues, 60-bit and 24-bit primes."""
import numpy as np
import pytest
import torch

from .pairs import Pair

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("logn,n_out", [(16, 1), (15, 2), (14, 5)])
@pytest.mark.parametrize("bits", [(60, 60, 60), (60, 40, 60), (24, 24, 25)])
def test_dot_pairs(gpu, logn, n_out, bits):
    L = 3
    assert n_out * ((1 << logn) // 256) * L >= 5 * 152  # the rule for the paired form
    if logn == 16 and bits[0] == 24:
        bits = (30, 30, 31)
    p = Pair(gpu, logn, L, 1, 1, first_bits=bits[0], mid_bits=bits[1], special_bits=bits[2], gpu_keys=False, rot_steps=(),
             relin=False)
    try:
        pf, ctx = p.pft, p.ctx
        q = pf.pft_ctx_info(ctx)["primes"][:L]
        rng = np.random.default_rng(logn)
        n_ct, n_pt = 6, 23
        words = np.stack([rng.integers(0, qi, (n_ct, 2, p.N), dtype=np.uint64) for qi in q], axis=2)
        words[0] = np.array([qi - 1 for qi in q], np.uint64)[None, :, None]
        consts = np.stack([rng.integers(0, qi, n_pt, dtype=np.uint64) for qi in q], axis=1)
        consts[0] = [qi - 1 for qi in q]
        cts, pts = [], []
        for w in words:
            h = p.empty()
            d = torch.from_numpy(np.ascontiguousarray(w).view(np.int64)).cuda()
            pf.pft_ct_reduce_sum(ctx, d.data_ptr(), L, 1.0, 1, h)
            torch.cuda.synchronize()
            cts.append(h)
        for c in consts:  # a constant polynomial has the same value everywhere
            m = np.zeros((L, p.N), np.uint64)
            m[:, 0] = c
            h = pf.pft_pt_import(ctx, m, 1.0)
            p.handles.append(("pt", h))
            pts.append(h)
        idx = np.r_[0:4, 254:260, p.N // 2 - 2:p.N // 2 + 2, p.N - 4:p.N]
        outs = [p.empty() for _ in range(n_out)]
        for K in (9, 11, 12, 13, 16, 63, 64, 65, 72, 131):
            for shared in (True, False):
                a = rng.integers(0, n_ct, n_out * K)
                b = rng.integers(0, n_pt, K if shared else n_out * K)
                a[: K // 2] = 0  # maximal products first
                b[: K // 2] = 0
                pf.pft_dot_plain_batch(ctx, [cts[i] for i in a], [pts[i] for i in b], K, outs, pts_shared=shared)
                for o, h in enumerate(outs):
                    got = torch.empty((2, L, p.N), dtype=torch.int64, device="cuda")
                    pf.pft_ct_copy_out(ctx, h, got.data_ptr())
                    got = got.cpu().numpy().view(np.uint64)
                    for r, qi in enumerate(q):
                        x = words[a[o * K:(o + 1) * K]][:, :, r, idx].astype(object)
                        c = consts[b if shared else b[o * K:(o + 1) * K], r].astype(object)
                        want = (x * c[:, None, None]).sum(axis=0) % int(qi)
                        assert np.array_equal(got[:, r, idx].astype(object), want), (K, shared, o, r)
    finally:
        p.close()
