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


class Labelled:
    """torch's caching allocator; records the stream that each free names."""

    def __init__(self, pf):
        self.live, self.freed_on = set(), []

        def alloc(nbytes, stream, user):
            p = torch.cuda.caching_allocator_alloc(int(nbytes), 0, int(stream or 0))
            self.live.add(p)
            return p

        def free(ptr, stream, user):
            if ptr:
                self.live.remove(ptr)
                self.freed_on.append(int(stream or 0))
                torch.cuda.caching_allocator_delete(ptr)

        self.struct = pf.pft_allocator(pf.ALLOC_FN(alloc), pf.FREE_FN(free), None)


def make(pf, alloc, stream, logn=12):
    ctx = pf.pft_ctx_create(logn, 4, 1, 2, 60, 40, 60, 2.0 ** 40, SEED, flags=pf.PFT_ALLOW_INSECURE, allocator=alloc,
                            stream=stream.cuda_stream)
    pf.pft_keygen(ctx, [1], True)
    return ctx


def fresh(pf, ctx, level=4):
    w = words(pf, ctx, level)
    h = pf.pft_ct_create(ctx)
    torch.cuda.synchronize()
    pf.pft_ct_reduce_sum(ctx, w.data_ptr(), level, 2.0 ** 40, 1, h)
    torch.cuda.synchronize()
    return h


@pytest.mark.parametrize("idle", [True, False])
def test_a_stream_that_is_left_is_not_used_again(gpu, idle):
    """The caller may have destroyed it: what was kept on it is freed elsewhere, after the work queued there."""
    pf, alloc = gpu, Labelled(gpu)
    left, other = torch.cuda.Stream(), torch.cuda.Stream()
    ctx = make(pf, alloc.struct, left)
    a, c, d = fresh(pf, ctx), pf.pft_ct_create(ctx), pf.pft_ct_create(ctx)
    for _ in range(2):
        pf.pft_mul_relin(ctx, a, a, c)
    want = pf.pft_ct_export(ctx, c)
    pf.pft_mul_relin(ctx, a, a, c)
    pf.pft_ct_destroy(c)  # kept outside any call that does work
    if idle:
        torch.cuda.synchronize()
    held, alloc.freed_on[:] = len(alloc.live), []
    pf.pft_set_stream(ctx, other.cuda_stream)
    assert len(alloc.live) < held, "the kept blocks are given back"
    if not idle:
        torch.cuda.synchronize()
    pf.pft_mul_relin(ctx, a, a, d)
    assert np.array_equal(pf.pft_ct_export(ctx, d), want)
    pf.pft_ct_destroy(a)
    pf.pft_ct_destroy(d)
    pf.pft_ctx_destroy(ctx)
    assert alloc.freed_on and left.cuda_stream not in alloc.freed_on
    assert not alloc.live


def test_streams_in_turn(gpu):
    """Independent work on two streams through one context, nothing waited for between them."""
    pf = gpu
    s = [torch.cuda.Stream(), torch.cuda.Stream()]
    ctx = make(pf, None, s[0], logn=14)
    a = fresh(pf, ctx)
    one = pf.pft_ct_create(ctx)
    pf.pft_mul_relin(ctx, a, a, one)
    want = pf.pft_ct_export(ctx, one)
    outs = [pf.pft_ct_create(ctx) for _ in range(40)]
    for i, h in enumerate(outs):
        pf.pft_set_stream(ctx, s[i % 2].cuda_stream)
        pf.pft_mul_relin(ctx, a, a, h)
    torch.cuda.synchronize()
    for h in outs:
        assert np.array_equal(pf.pft_ct_export(ctx, h), want)
    for h in outs + [a, one]:
        pf.pft_ct_destroy(h)
    pf.pft_ctx_destroy(ctx)


@pytest.mark.filterwarnings("ignore")
def test_refusal_under_capture_keeps_the_blocks(gpu):
    """Blocks that were kept before a capture are not freed into it: the call fails, and they serve the next one."""
    from .test_gpu_faults import CappedAllocator

    pf, alloc, st = gpu, CappedAllocator(gpu, torch), torch.cuda.Stream()
    ctx = make(pf, alloc.struct, st)
    a, c = fresh(pf, ctx), pf.pft_ct_create(ctx)
    pf.pft_mul_relin(ctx, a, a, c)
    want = pf.pft_ct_export(ctx, c)
    pf.pft_mul_relin(ctx, a, a, c)
    torch.cuda.synchronize()
    held = set(alloc.live)
    graph = torch.cuda.CUDAGraph()
    alloc.cap = 0
    with torch.cuda.stream(st):
        graph.capture_begin(capture_error_mode="relaxed")
        try:
            with pytest.raises(pf.PftError) as e:
                pf.pft_mul_relin(ctx, a, a, c)
        finally:
            graph.capture_end()
    assert e.value.code == pf.PFT_ERR_OOM
    assert set(alloc.live) == held
    pf.pft_mul_relin(ctx, a, a, c)  # nothing new is needed
    assert np.array_equal(pf.pft_ct_export(ctx, c), want)
    alloc.cap = None
    pf.pft_ct_destroy(a)
    pf.pft_ct_destroy(c)
    pf.pft_ctx_destroy(ctx)
    assert alloc.in_use() == 0


@pytest.mark.parametrize("own_streams", [False, True])
def test_another_contexts_blocks_are_given_back(gpu, own_streams):
    """Two contexts with one allocator: what one keeps does not refuse the other a request."""
    from .test_gpu_faults import CappedAllocator

    pf, alloc = gpu, CappedAllocator(gpu, torch)
    st = [torch.cuda.Stream() if own_streams else torch.cuda.default_stream() for _ in range(2)]
    one, two = [make(pf, alloc.struct, s) for s in st]
    a, b = fresh(pf, one), fresh(pf, two)
    c, d = pf.pft_ct_create(one), pf.pft_ct_create(two)
    pf.pft_mul_relin(two, b, b, d)
    want = pf.pft_ct_export(two, d)
    pf.pft_ct_destroy(d)
    torch.cuda.synchronize()
    alloc.cap = 0
    big = [pf.pft_ct_create(two) for _ in range(64)]
    with pytest.raises(pf.PftError):  # the second context's kept blocks go back (and the first one's)
        pf.pft_mul_relin_batch(two, [b] * 64, [b] * 64, big)
    alloc.cap = None
    pf.pft_mul_relin(one, a, a, c)
    torch.cuda.synchronize()
    alloc.cap = alloc.in_use() + 2 * 4 * 8 * 4096 + 4096  # the product; its working space is kept by the first
    pf.pft_mul_relin(two, b, b, big[0])
    assert np.array_equal(pf.pft_ct_export(two, big[0]), want)
    alloc.cap = None
    pf.pft_mul_relin(one, a, a, c)
    for h in [a, b, c] + big:
        pf.pft_ct_destroy(h)
    pf.pft_ctx_destroy(one)
    pf.pft_ctx_destroy(two)
    assert alloc.in_use() == 0


def test_torch_allocator_is_one(gpu):
    assert gpu.torch_allocator() is gpu.torch_allocator()


def test_what_a_context_keeps_is_small(gpu):
    """Freed handles: at most 256 MiB stay with the context."""
    from .test_gpu_faults import CappedAllocator

    pf, alloc = gpu, CappedAllocator(gpu, torch)
    ctx = make(pf, alloc.struct, torch.cuda.default_stream(), logn=16)
    w = words(pf, ctx, 4)
    torch.cuda.synchronize()
    base = alloc.in_use()
    hs = [pf.pft_ct_create(ctx) for _ in range(100)]  # 4 MiB each
    for h in hs:
        pf.pft_ct_reduce_sum(ctx, w.data_ptr(), 4, 2.0 ** 40, 1, h)
    for h in hs:
        pf.pft_ct_destroy(h)
    torch.cuda.synchronize()
    assert alloc.in_use() <= base + (256 << 20)
    pf.pft_ctx_destroy(ctx)
    assert alloc.in_use() == 0


def test_many_sizes(gpu):
    """More different sizes than a context keeps blocks of (one handle's words each): results, and everything given back."""
    from .test_gpu_faults import CappedAllocator

    pf, alloc, n = gpu, CappedAllocator(gpu, torch), 1300
    ctx = pf.pft_ctx_create(4, 1, 1, 1, 60, 40, 60, 2.0 ** 40, SEED, flags=pf.PFT_ALLOW_INSECURE, allocator=alloc.struct)
    q = pf.pft_ctx_info(ctx)["primes"][0]
    w = torch.arange(n * 16, dtype=torch.int64, device="cuda")
    a = [pf.pft_ct_create(ctx) for _ in range(n)]
    v = torch.cat([w, w]).contiguous()
    for h in a:
        pf.pft_ct_reduce_sum(ctx, v.data_ptr(), 1, 2.0 ** 40, 1, h)
    pt = pf.pft_pt_import(ctx, np.eye(1, 16, dtype=np.uint64), 1.0)  # the constant 1
    out = pf.pft_ct_create(ctx)
    for k in list(range(1, n + 1)) * 2:  # pointer tables of k and 2 k words
        pf.pft_dot_plain_batch(ctx, a[:k], [pt] * k, k, [out], pts_shared=True)
    got = torch.empty((2, 1, 16), dtype=torch.int64, device="cuda")
    pf.pft_ct_copy_out(ctx, out, got.data_ptr())
    want = v[:32].cpu().numpy().astype(object) * n % q
    assert np.array_equal(got.cpu().numpy().reshape(-1).astype(object), want)
    for h in a + [out]:
        pf.pft_ct_destroy(h)
    pf.pft_pt_destroy(pt)
    pf.pft_ctx_destroy(ctx)
    assert alloc.in_use() == 0
