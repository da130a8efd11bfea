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
