"""The context's kept device blocks: repeated calls stop asking the caller's allocator, the kept bytes are bounded and
given back on a stream change, on a refusal and with the context, and results do not change."""
import numpy as np
import pytest
import torch

from paper_1908_06972_gb300 import synth
from .test_gpu_faults import CappedAllocator

pytestmark = pytest.mark.gpu

SEED = (0x5EED, 11, 22, 33)


def make(gpu, logn, L, alloc):
    ctx = gpu.pft_ctx_create(logn, L, 1, 2, 60, 40, 60, 2.0 ** 40, SEED, flags=gpu.PFT_ALLOW_INSECURE,
                             allocator=alloc.struct)
    gpu.pft_keygen(ctx, [1], True)
    return ctx


class Counted(dict):
    """An allocator's live blocks; counts how often one was added."""
    added = 0

    def __setitem__(self, k, v):
        self.added += 1
        super().__setitem__(k, v)


def words(pf, ctx, level, seed):
    info = pf.pft_ctx_info(ctx)
    w = torch.from_numpy(synth.residues(seed, info["primes"][:level], info["N"], polys=2).view(np.int64)).cuda()
    h = pf.pft_ct_create(ctx)
    pf.pft_ct_reduce_sum(ctx, w.data_ptr(), level, 2.0 ** 40, 1, h)
    torch.cuda.synchronize()  # the words are read before torch takes their memory back
    return h


def test_reuse_and_release(gpu):
    pf = gpu
    alloc = CappedAllocator(pf, torch)
    alloc.live = Counted()
    ctx = make(pf, 12, 4, alloc)
    handles = [words(pf, ctx, 4, 1), words(pf, ctx, 4, 2), pf.pft_ct_create(ctx)]
    a, b, c = handles

    def step():
        pf.pft_mul_relin(ctx, a, b, c)
        pf.pft_rescale(ctx, c, c)
        pf.pft_rotate(ctx, c, 1, c)
        return pf.pft_ct_export(ctx, c)

    first = step()
    step()
    n = alloc.live.added
    for _ in range(3):
        assert np.array_equal(step(), first)
    assert alloc.live.added == n, "a repeated call asked the allocator"
    torch.cuda.synchronize()
    # the kept blocks go back when the stream changes, and when the allocator refuses
    held = alloc.in_use()
    side = torch.cuda.Stream()
    pf.pft_set_stream(ctx, side.cuda_stream)
    assert alloc.in_use() < held
    assert np.array_equal(step(), first)
    step()
    side.synchronize()
    held = alloc.in_use()
    alloc.cap = held
    big = pf.pft_ct_create(ctx)
    handles.append(big)
    with pytest.raises(pf.PftError) as e:
        pf.pft_mul_relin_batch(ctx, [a] * 64, [b] * 64, [big] + [c] * 63)
    assert e.value.code == pf.PFT_ERR_OOM and alloc.in_use() < held
    alloc.cap = None
    for h in handles:
        pf.pft_ct_destroy(h)
    pf.pft_ctx_destroy(ctx)
    torch.cuda.synchronize()
    assert alloc.in_use() == 0


def test_kept_bytes_are_bounded(gpu):
    pf = gpu
    alloc = CappedAllocator(pf, torch)
    ctx = make(pf, 16, 12, alloc)
    torch.cuda.synchronize()
    base = alloc.in_use()
    hs = [words(pf, ctx, 12, 1) for i in range(120)]  # 12 MiB each
    torch.cuda.synchronize()
    assert alloc.in_use() >= base + 100 * (12 << 20) - (1 << 30)
    for h in hs:
        pf.pft_ct_destroy(h)
    assert alloc.in_use() <= base + (1 << 30)
    pf.pft_ctx_destroy(ctx)
    assert alloc.in_use() == 0


def test_graph_capture_keeps_its_own_memory(gpu):
    """A captured call replays correctly after eager calls have used and freed the kept blocks."""
    pf = gpu
    st = torch.cuda.Stream()
    ctx = pf.pft_ctx_create(12, 4, 1, 2, 60, 40, 60, 2.0 ** 40, SEED, flags=pf.PFT_ALLOW_INSECURE, allocator=None,
                            stream=st.cuda_stream)
    pf.pft_keygen(ctx, [1], True)
    a, b, c, d = words(pf, ctx, 4, 1), words(pf, ctx, 4, 2), pf.pft_ct_create(ctx), pf.pft_ct_create(ctx)
    torch.cuda.synchronize()
    pf.pft_mul_relin(ctx, a, b, c)
    want = pf.pft_ct_export(ctx, c)
    pf.pft_graph_begin(ctx)
    pf.pft_mul_relin(ctx, a, b, c)
    g = pf.pft_graph_end(ctx)
    for _ in range(3):
        pf.pft_mul_relin(ctx, b, b, d)
        pf.pft_rotate(ctx, a, 1, c)
        pf.pft_graph_launch(ctx, g)
        pf.pft_rotate(ctx, b, 1, d)
        assert np.array_equal(pf.pft_ct_export(ctx, c), want)
    pf.pft_graph_destroy(g)
    for h in (a, b, c, d):
        pf.pft_ct_destroy(h)
    pf.pft_ctx_destroy(ctx)
