"""Batched calls behind an allocator with little left: a batch that does not fit as a whole runs in
smaller parts (what runs one at a time fits), and a refused call leaves its outputs as they were."""
import numpy as np
import pytest
import torch

from paper_1908_06972_gb300 import synth

from .test_gpu_faults import CappedAllocator

pytestmark = pytest.mark.gpu

LOGN, L = 12, 6
N = 1 << LOGN
LIMB = 8 * N
SPEC = 1  # special primes; one prime per digit, so a ciphertext at level l has l digits
COLS, CLASSES = 8, 4


class Ring:
    def __init__(self, pf):
        self.pf, self.alloc = pf, CappedAllocator(pf, torch)
        self.ctx = pf.pft_ctx_create(LOGN, L, SPEC, 1, 60, 40, 60, 2.0 ** 40, (2, 7, 1, 8), flags=pf.PFT_ALLOW_INSECURE,
                                     allocator=self.alloc.struct)
        steps = list(range(1, COLS)) + [1 << i for i in range(LOGN - 1)]
        pf.pft_keygen(self.ctx, steps, True)
        self.handles = []

    def ct(self, level, seed):
        pf, h = self.pf, self.empty()
        w = synth.residues(seed, pf.pft_ctx_info(self.ctx)["primes"][:level], N, polys=2)
        w = torch.from_numpy(w.view(np.int64)).cuda()
        pf.pft_ct_reduce_sum(self.ctx, w.data_ptr(), level, 2.0 ** 40, 1, h)
        torch.cuda.synchronize()
        return h

    def empty(self):
        h = self.pf.pft_ct_create(self.ctx)
        self.handles.append(h)
        return h

    def words(self, hs):
        return [self.pf.pft_ct_export(self.ctx, h) for h in hs]

    def settle(self):
        """The allocator's bytes that are not kept for reuse: a refused request gives the kept ones back."""
        torch.cuda.synchronize()
        self.alloc.cap = 0
        a, out = [self.handles[0]] * 256, [self.handles[-1]] * 256
        with pytest.raises(self.pf.PftError):  # the tensors' block is too large to be a kept one
            self.pf.pft_mul_relin_batch(self.ctx, a, a, out)
        self.alloc.cap = None
        return self.alloc.in_use()

    def close(self):
        for h in self.handles:
            self.pf.pft_ct_destroy(h)
        self.pf.pft_ctx_destroy(self.ctx)


@pytest.fixture
def ring(gpu):
    r = Ring(gpu)
    yield r
    r.close()


def one_hoisted(l):
    """Working limbs of one ciphertext's hoisted rotations, step by step: coefficient form, extended digits and their
    permuted copy, the products, the conversions, the permuted c0."""
    E = l + SPEC
    return l + 2 * l * E + 2 * E + 2 * l + l


# levels of the documents, and the limbs that inference takes one document (and one level) at a time: the
# accumulators, the rotated copies of a level's documents and one document's working space.  The rotations after
# that take (2 l) + (l + l E + 2 E + 2 l) limbs per document beside the accumulators
@pytest.mark.parametrize("levels,limbs", [([6] * 6, 6 * 12 + 6 * 7 * 12 + one_hoisted(6)),
                                          ([6, 4, 6, 4, 4, 6], 3 * (12 + 8) + 3 * 86 + 3 * 50)])
def test_diagonal_inference(ring, levels, limbs):
    pf, ctx = ring.pf, ring.ctx
    H, O = synth.fasttext_weights(5, N // 2, COLS, CLASSES)
    model = pf.pft_ft_model_create_diag(ctx, H, O, L)
    docs = [ring.ct(l, 20 + i) for i, l in enumerate(levels)]
    scores = [ring.empty() for _ in docs]
    pf.pft_fasttext_infer_batch(ctx, model, docs, 1, scores)
    want = ring.words(scores)
    ring.alloc.cap = ring.settle() + (limbs + 16) * LIMB
    pf.pft_fasttext_infer_batch(ctx, model, docs, 1, scores)
    ring.alloc.cap = None
    for g, w in zip(ring.words(scores), want):
        assert np.array_equal(g, w)
    pf.pft_ft_model_destroy(model)


@pytest.mark.parametrize("spare", [0, 3 * 12 + 8])  # nothing; the outputs but not the working space
def test_refused_hoisted_rotation_leaves_outputs(ring, spare):
    pf, ctx = ring.pf, ring.ctx
    a = ring.ct(6, 1)
    outs = [ring.ct(2, 10 + i) for i in range(3)]
    want = ring.words(outs)
    base = ring.settle()
    ring.alloc.cap = base + spare * LIMB
    with pytest.raises(pf.PftError) as e:
        pf.pft_rotate_hoisted(ctx, a, [1, 2, 3], outs)
    assert e.value.code == pf.PFT_ERR_OOM
    ring.alloc.cap = None
    assert [pf.pft_ct_level(h) for h in outs] == [2] * 3
    for g, w in zip(ring.words(outs), want):
        assert np.array_equal(g, w)
    pf.pft_rotate_hoisted(ctx, a, [1, 2, 3], outs)
    pf.pft_device_status(ctx)


def test_rescale_of_mixed_levels(ring):
    """Room for the outputs and the working space of the largest level alone; one call in place."""
    pf, ctx = ring.pf, ring.ctx
    levels = [6, 2, 5, 3, 4, 6, 2, 5, 3, 4]
    a = [ring.ct(l, 40 + i) for i, l in enumerate(levels)]
    outs = [ring.empty() for _ in levels]
    pf.pft_rescale_batch(ctx, a, outs)
    want = ring.words(outs)
    ring.alloc.cap = ring.settle() + (2 * 10 + 2 * 12 + 4) * LIMB
    pf.pft_rescale_batch(ctx, a, a)
    ring.alloc.cap = None
    for g, w, l in zip(ring.words(a), want, levels):
        assert np.array_equal(g, w) and len(g[0]) == l - 1


def test_rescale_working_space_shrinks(ring):
    """All of one level: the outputs and one ciphertext's working space; then too little for the outputs."""
    pf, ctx = ring.pf, ring.ctx
    a = [ring.ct(5, 60 + i) for i in range(6)]
    outs = [ring.empty() for _ in a]
    pf.pft_rescale_batch(ctx, a, outs)
    want = ring.words(outs)
    base = ring.settle()
    ring.alloc.cap = base + (6 * 8 + 10 + 4) * LIMB
    pf.pft_rescale_batch(ctx, a, outs)
    ring.alloc.cap = base + 5 * 8 * LIMB
    with pytest.raises(pf.PftError) as e:
        pf.pft_rescale_batch(ctx, a, a)
    assert e.value.code == pf.PFT_ERR_OOM
    ring.alloc.cap = None
    assert [pf.pft_ct_level(h) for h in a] == [5] * 6
    pf.pft_rescale_batch(ctx, a, a)
    for g, h, w in zip(ring.words(a), ring.words(outs), want):
        assert np.array_equal(g, w) and np.array_equal(h, w)


def test_rescale_repeated_output(ring):
    """A handle given for several inputs ends with the result of the highest level, then of the last of that level."""
    pf, ctx = ring.pf, ring.ctx
    a = [ring.ct(l, 80 + i) for i, l in enumerate([3, 5, 5, 4])]
    want, out = ring.empty(), ring.empty()
    pf.pft_rescale(ctx, a[2], want)
    pf.pft_rescale_batch(ctx, a, [out] * 4)
    assert np.array_equal(pf.pft_ct_export(ctx, out), pf.pft_ct_export(ctx, want))
