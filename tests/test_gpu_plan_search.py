"""The plan search times launches that its plans run differently: launches that fit the GPU at once take the same
kernels under both two-pass plans."""
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("logn,L,k", [(15, 2, 1), (15, 18, 2), (15, 21, 1), (15, 30, 4), (16, 15, 3), (16, 16, 2)])
def test_representative_launches(gpu, logn, L, k):
    pf = gpu
    ctx = pf.pft_ctx_create(logn, L, k, k, 60, 40, 60, 2.0 ** 40, (1, 2, 3, 4), flags=pf.PFT_ALLOW_INSECURE)
    pf.pft_autotune(ctx)
    limbs = [b["limbs"] for b in pf.pft_autotune_report(ctx)["buckets"]]
    assert 152 * 512 < limbs[0] * (16 << (logn - 8)) and limbs[0] <= 64 < limbs[1] <= 512 < limbs[2]
    pf.pft_ctx_destroy(ctx)
