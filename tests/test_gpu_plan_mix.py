"""Batches whose launches have plans of different kinds: the plan of a launch goes by its size, and a
batch of more than 256 polynomials is several launches.  The words must not depend on the plans."""
import ctypes
import subprocess

import pytest
import torch

from paper_1908_06972_gb300 import _build, synth

pytestmark = pytest.mark.gpu

SHIM = """
#include "evaluator.h"
extern "C" int set_bucket_plan(pft_ctx* c, int bucket, int plan) {
    pft::DevTables::Plan cand[16];
    if (plan < 0 || plan >= pft::ntt_candidates(c->logn, cand, nullptr, 16)) return 1;
    c->tabs.plan[bucket] = cand[plan];
    return 0;
}
"""
STAGED, TWO_PASS = 0, 5  # indices into the plan list of N = 2^15


@pytest.fixture(scope="module")
def shim(gpu, tmp_path_factory):
    """The plan search can leave such a mixture; this sets one launch-size bucket's plan."""
    gpu.lib()
    d = tmp_path_factory.mktemp("shim")
    src, so = str(d / "shim.cu"), str(d / "shim.so")
    with open(src, "w") as f:
        f.write(SHIM)
    subprocess.run([_build.nvcc(), "-std=c++17", "-shared", "-Xcompiler", "-fPIC", "-I" + _build.CSRC, src, _build.SO, "-o", so],
                   check=True)
    return ctypes.CDLL(so)


def words(pf, ctx, level, seed):
    info = pf.pft_ctx_info(ctx)
    w = torch.from_numpy(synth.residues(seed, info["primes"][:level], info["N"], polys=2).view("int64")).cuda()
    h = pf.pft_ct_create(ctx)
    pf.pft_ct_reduce_sum(ctx, w.data_ptr(), level, 2.0 ** 40, 1, h)
    torch.cuda.synchronize()
    return h


@pytest.mark.parametrize("plans", [(STAGED, TWO_PASS, TWO_PASS), (TWO_PASS, STAGED, TWO_PASS)])
def test_mixed_plans(gpu, shim, plans):
    """131 ciphertexts at level 2: ModDown and RESCALE are launches of 256 polynomials (256 or 512 limbs: the
    second bucket) and of six (the first)."""
    pf, B, level = gpu, 131, 2
    ctx = pf.pft_ctx_create(15, level, 1, 1, 60, 40, 60, 2.0 ** 40, (3, 1, 4, 1), flags=pf.PFT_ALLOW_INSECURE)
    pf.pft_keygen(ctx, [1], True)
    a, b = [words(pf, ctx, level, 7 + i) for i in range(2)]
    outs = [pf.pft_ct_create(ctx) for _ in range(B)]

    def run():
        pf.pft_mul_relin_batch(ctx, [a] * B, [b] * B, outs)
        pf.pft_rotate_batch(ctx, outs, 1, outs)
        got = [pf.pft_ct_export(ctx, h) for h in (outs[0], outs[B - 1])]
        pf.pft_rescale_batch(ctx, outs, outs)
        return got + [pf.pft_ct_export(ctx, h) for h in (outs[0], outs[B - 1])]

    pf.pft_set_transform_plan(ctx, STAGED)
    want = run()
    for bucket, plan in enumerate(plans):
        assert shim.set_bucket_plan(ctx, bucket, plan) == 0
    for g, w in zip(run(), want):
        assert (g == w).all()
    for h in [a, b] + outs:
        pf.pft_ct_destroy(h)
    pf.pft_ctx_destroy(ctx)
