"""Two-pass transforms (columns of 2^(logn-8) points, rows of 256) of the rings N = 2^12..2^15: the
values against the oracle's evaluations, against the one-pass / staged kernels of the same ring
(transform variant 3), and the fused ModDown and rescale passes through HMUL, RESCALE and ROTATE."""
import numpy as np
import pytest

from oracle import _lib as OC
from oracle import params as OP
from paper_1908_06972_gb300 import synth
from .pairs import Pair

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("logn", [12, 13, 14, 15])
@pytest.mark.parametrize("bits", [(60, 40, 60), (57, 57, 58), (50, 50, 60), (24, 24, 25)])
def test_values_and_variants(gpu, logn, bits):
    import torch

    first, mid, special = bits
    p = Pair(gpu, logn, 3, 1, 1, first_bits=first, mid_bits=mid, special_bits=special, gpu_keys=False, rot_steps=(),
             relin=False)
    try:
        primes = gpu.pft_ctx_info(p.ctx)["primes"]
        n = 1 << logn
        x = synth.residues(5 + logn, primes, n, polys=3)
        for r, q in enumerate(primes):
            x[0, r, :] = q - 1
            x[1, r, :] = np.where(np.arange(n) % 3 == 0, 0, q - 1)
        idx = np.r_[0:17, 250:262, n // 2 - 3:n // 2 + 3, n - 17:n]
        got = {}
        for variant in (0, 1, 3):
            gpu.pft_set_transform_variant(p.ctx, variant)
            t = torch.from_numpy(x.view(np.int64).copy()).cuda()
            gpu.pft_ntt(p.ctx, t.data_ptr(), 3, len(primes), 0)
            got[variant] = t.cpu().numpy().view(np.uint64)
            gpu.pft_ntt(p.ctx, t.data_ptr(), 3, len(primes), 1)
            assert np.array_equal(t.cpu().numpy().view(np.uint64), x), (variant, "round trip")
        assert np.array_equal(got[0], got[3]) and np.array_equal(got[1], got[3])
        for poly in range(3):
            for r, q in enumerate(primes):
                want = OC.eval_at(x[poly, r], OP.root_2n(q, logn), q, logn, idx)
                assert np.array_equal(got[0][poly, r][idx], want), (poly, r)
    finally:
        p.close()


@pytest.mark.parametrize("logn", [12, 13, 14])
@pytest.mark.parametrize("variant", [0, 3])
def test_operations_bit_exact(gpu, logn, variant):
    p = Pair(gpu, logn, 3, 1, 2, rot_steps=[1, -5])
    try:
        o, pf, ctx = p.orc, p.pft, p.ctx
        pf.pft_set_transform_variant(ctx, variant)
        a = o.encrypt_sk(o.encode(synth.slots(3, 64)), 1)
        b = o.encrypt_sk(o.encode(synth.slots(4, 64)), 2)
        m = p.empty()
        pf.pft_mul_relin(ctx, p.ct(a), p.ct(b), m)
        want = o.mul_relin(a, b)
        p.assert_equal(m, want, "mul_relin")
        pf.pft_rescale(ctx, m, m)
        want = o.rescale(want)
        p.assert_equal(m, want, "rescale")
        r = p.empty()
        for step in (1, -5):
            pf.pft_rotate(ctx, m, step, r)
            p.assert_equal(r, o.rotate(want, step), "rotate %d" % step)
    finally:
        p.close()


@pytest.mark.parametrize("logn,variant", [(11, 0), (12, 0), (13, 3), (13, 0), (14, 0), (15, 0), (15, 1), (16, 0), (16, 3)])
def test_rescale_batch_mixed_levels(gpu, logn, variant):
    """One call over ciphertexts of several levels (one in place), 60-bit and 40-bit dropped primes, and
    the allocation-free form."""
    import torch

    p = Pair(gpu, logn, 4, 1, 4, mid_bits=40, rot_steps=(), relin=False)
    try:
        o, pf, ctx = p.orc, p.pft, p.ctx
        pf.pft_set_transform_variant(ctx, variant)
        levels = [4, 2, 3, 4, 2]
        x = [o.encrypt_sk(o.encode(synth.slots(70 + i, 16), level=l), 80 + i) for i, l in enumerate(levels)]
        x[0].c[:, -1, :3] = [0, o.q[3] - 1, o.q[3] // 2]  # the ends of the rounding
        h = [p.ct(c) for c in x]
        outs = [p.empty(), h[1]] + [p.empty() for _ in levels[2:]]
        raw = torch.empty((2, 3, p.N), dtype=torch.int64, device="cuda")
        pf.pft_rescale_noalloc(ctx, pf.pft_ct_data(h[0]), 4, raw.data_ptr())
        pf.pft_rescale_batch(ctx, h, outs)
        for i, (g, c) in enumerate(zip(outs, x)):
            p.assert_equal(g, o.rescale(c), "ciphertext %d at level %d" % (i, levels[i]))
        got = torch.empty_like(raw)
        pf.pft_ct_copy_out(ctx, outs[0], got.data_ptr())
        assert torch.equal(raw, got)
    finally:
        p.close()
