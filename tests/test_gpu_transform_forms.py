"""The two-pass transforms' forms for launches that do not fit the GPU at once.  A launch of few limbs takes
the form with every twiddle in registers; the forms bounded for 640 and for 1024 resident threads per SM (variants 0 and
1) read shared-memory and lane-major copies instead, and only larger launches reach them: values on extreme
inputs, and the unscaled, fused, permuted and broadcast passes through the operations, on both sides
of that line, against the staged kernels (variant 3) and the oracle."""
import numpy as np
import pytest
import torch

from oracle import _lib as OC
from oracle import params as OP
from paper_1908_06972_gb300 import synth
from .pairs import Pair

pytestmark = pytest.mark.gpu


def line(logn):
    """The most limbs of a launch that takes the small form: 512 threads on each of 152 SMs, 16 points per thread."""
    return 152 * 512 // (16 << (logn - 8))


def variants(logn):
    return (0, 1) if logn >= 15 else (0,)


@pytest.mark.parametrize("logn", [12, 13, 14, 15, 16])
@pytest.mark.parametrize("bits", [(59, 57, 60), (57, 57, 58), (50, 50, 60), (24, 24, 25)])
@pytest.mark.parametrize("above", [0, 1])
def test_values(gpu, logn, bits, above):
    if logn == 16 and bits[0] == 24:
        bits = (30, 30, 31)
    first, mid, special = bits
    p = Pair(gpu, logn, 3, 1, 1, first_bits=first, mid_bits=mid, special_bits=special, gpu_keys=False, rot_steps=(),
             relin=False)
    try:
        primes = gpu.pft_ctx_info(p.ctx)["primes"]
        n = 1 << logn
        polys = line(logn) // len(primes) + above
        x = synth.residues(9 + logn, primes, n, polys=5)
        for r, q in enumerate(primes):
            x[0, r, :] = q - 1
            x[1, r, :] = np.where(np.arange(n) % 2 == 0, 0, q - 1)
            x[2, r, :] = np.where(np.arange(n) % 3 == 0, 0, q - 1)
        big = torch.from_numpy(x.view(np.int64)).cuda()[torch.arange(polys) % 5].contiguous()
        idx = np.r_[0:17, 250:262, n // 2 - 3:n // 2 + 3, n - 17:n]
        got = {}
        for v in variants(logn) + (3,):
            gpu.pft_set_transform_variant(p.ctx, v)
            t = big.clone()
            gpu.pft_ntt(p.ctx, t.data_ptr(), polys, len(primes), 0)
            got[v] = t.clone()
            gpu.pft_ntt(p.ctx, t.data_ptr(), polys, len(primes), 1)
            assert torch.equal(t, big), (v, "round trip")
            assert torch.equal(got[v], got[variants(logn)[0]]), v
        y = got[0][:5].cpu().numpy().view(np.uint64)
        for poly in range(min(5, polys)):
            for r, q in enumerate(primes):
                want = OC.eval_at(x[poly, r], OP.root_2n(q, logn), q, logn, idx)
                assert np.array_equal(y[poly, r][idx], want), (poly, r)
    finally:
        p.close()


@pytest.mark.parametrize("logn", [12, 13, 14, 15, 16])
def test_operations(gpu, logn):
    """HMUL, RESCALE of two levels in one call and ROTATE over a batch whose every launch is above the line (the
    narrowest transforms one limb of each polynomial), then hoisted rotations of one ciphertext."""
    B = line(logn) // 2 + 1
    n_hoist = line(logn) // 6 + 1
    p = Pair(gpu, logn, 3, 1, 2, rot_steps=[1], gpu_keys=False)
    try:
        o, pf, ctx = p.orc, p.pft, p.ctx
        pf.pft_keygen(ctx, list(range(1, n_hoist + 1)), True)
        x = [(o.encrypt_sk(o.encode(synth.slots(3 + l, 64), level=l), 10 + l),
              o.encrypt_sk(o.encode(synth.slots(5 + l, 64), level=l), 20 + l)) for l in (3, 2)]
        ga, gb = [p.ct(a) for a, _ in x], [p.ct(b) for _, b in x]
        kind = [0 if i % 3 else 1 for i in range(B)]
        outs = [p.empty() for _ in range(B)]
        hoisted = [p.empty() for _ in range(n_hoist)]

        def words(h):
            d = torch.empty((2, pf.pft_ct_level(h), p.N), dtype=torch.int64, device="cuda")
            pf.pft_ct_copy_out(ctx, h, d.data_ptr())
            return d

        def run():
            steps = []
            pf.pft_mul_relin_batch(ctx, [ga[k] for k in kind], [gb[k] for k in kind], outs)
            steps.append([words(h) for h in outs])
            pf.pft_rotate_batch(ctx, outs, 1, outs)
            steps.append([words(h) for h in outs])
            pf.pft_rescale_batch(ctx, outs, outs)
            steps.append([words(h) for h in outs])
            pf.pft_rotate_hoisted(ctx, ga[0], list(range(1, n_hoist + 1)), hoisted)
            steps.append([words(h) for h in hoisted])
            return steps

        pf.pft_set_transform_variant(ctx, 3)
        want = run()
        for i in range(3):  # every ciphertext of a kind is the same
            for k, w in zip(kind, want[i]):
                assert torch.equal(w, want[i][kind.index(k)])
        if logn <= 14:
            for k, (a, b) in enumerate(x):
                p.assert_equal(outs[kind.index(k)], o.rescale(o.rotate(o.mul_relin(a, b), 1)), "oracle")
        for v in variants(logn):
            pf.pft_set_transform_variant(ctx, v)
            for step, (got, ref) in enumerate(zip(run(), want)):
                for i, (g, w) in enumerate(zip(got, ref)):
                    assert torch.equal(g, w), (v, step, i)
    finally:
        p.close()
