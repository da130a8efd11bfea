"""The measured work of the CKKS evaluator: what a server built on it asks of it.

A case names a ring (one of the repository's parameter sets), an operation through the public C
entry points, a batch size and the range its ciphertext levels are drawn from.  Ciphertext words
are uniform residues, as every ciphertext's are, so inputs are drawn on the GPU and need no
encryption.  Contexts, switching keys and model weights are what a server keeps between requests:
they are made once per ring and kept here.  All outputs are whole words, equal bit for bit from
run to run; a ciphertext is returned as its device buffer [2][level][N].
"""
import math
import random

import numpy as np
import torch

import paper_1908_06972_gb300 as pft
from paper_1908_06972_gb300 import synth

# name: (log2 N, limbs, special primes, primes per digit, bits of q_0, of q_1.., of the special
# primes, scale, flags)
RINGS = {
    # the core smoke chain and its twin at 128-bit security
    "n12": (12, 3, 1, 1, 60, 40, 60, 2.0 ** 40, pft.PFT_ALLOW_INSECURE),
    "n13": (13, 3, 1, 1, 60, 40, 60, 2.0 ** 40, 0),
    # the smaller serving ring
    "n15": (15, 18, 2, 2, 60, 40, 60, 2.0 ** 40, 0),
    # the batched key-switching benchmark's chain (50-bit limbs)
    "n16w50": (16, 30, 4, 4, 60, 50, 60, 2.0 ** 50, 0),
    # the same with seeded compressed switching keys (half the key memory)
    "n16w50c": (16, 30, 4, 4, 60, 50, 60, 2.0 ** 50, pft.PFT_COMPRESSED_KEYS),
    # the inference, serving and training chain (40-bit limbs)
    "n16w40": (16, 30, 4, 4, 60, 40, 60, 2.0 ** 40, 0),
}
SEED = (0x5EED0001, 0x5EED0002, 0x5EED0003, 0x5EED0004)
VOCAB, DIM, CLASSES = 32768, 64, 14  # the inference model
TR_DIM, TR_CLASSES, TR_VOCAB, TR_LIFT, TR_ETA = 32, 4, 8192, 10, 0.25  # the training model

_ctx, _steps, _models, _weights = {}, {}, {}, {}


def context(ring, steps=(), relin=True):
    """The ring's context with (at least) the asked rotation keys."""
    if ring not in _ctx:
        logn, limbs, special, alpha, first, mid, sp, scale, flags = RINGS[ring]
        c = pft.pft_ctx_create(logn, limbs, special, alpha, first, mid, sp, scale, SEED, flags=flags)
        pft.pft_keygen(c, [], relin)
        _ctx[ring], _steps[ring] = c, set()
    new = [s for s in steps if s not in _steps[ring]]
    if new:
        pft.pft_add_rotation_keys(_ctx[ring], new)
        _steps[ring] |= set(new)
    return _ctx[ring]


def primes(ring):
    return pft.pft_ctx_info(context(ring))["primes"]


class Words:
    """Device memory of a handle, for torch."""

    def __init__(self, ptr, shape):
        self.__cuda_array_interface__ = {"shape": shape, "typestr": "<i8", "data": (ptr, False), "version": 2}


class State:
    """Handles of one set of inputs and outputs; they are destroyed with it."""

    def __init__(self, case, seed):
        self.case, self.ring = case, case["ring"]
        self.n = 1 << RINGS[self.ring][0]
        self.handles, self.views = [], {}
        self.gen = torch.Generator(device="cuda")
        self.gen.manual_seed(seed)

    def words(self, shape_limbs, count):
        """[count][limbs][N] uniform canonical residues."""
        q = torch.tensor(primes(self.ring)[:shape_limbs], dtype=torch.int64, device="cuda")
        w = torch.randint(0, 1 << 62, (count, shape_limbs, self.n), generator=self.gen, dtype=torch.int64, device="cuda")
        return w.remainder_(q[None, :, None])

    def ct(self, level, scale=None):
        """A ciphertext of uniform words."""
        c, h = context(self.ring), self.empty()
        w = self.words(level, 2)
        pft.pft_ct_reduce_sum(c, w.data_ptr(), level, scale or RINGS[self.ring][7], 1, h)
        return h

    def empty(self):
        h = pft.pft_ct_create(context(self.ring))
        self.handles.append(h)
        return h

    def view(self, h):
        """The ciphertext's words as a tensor on its own buffer."""
        key = (pft.pft_ct_data(h), pft.pft_ct_level(h))
        if key not in self.views:
            self.views[key] = torch.as_tensor(Words(key[0], (2, key[1], self.n)), device="cuda")
        return self.views[key]

    def __del__(self):
        for h in self.handles:
            pft.pft_ct_destroy(h)


def levels_of(case):
    r = random.Random(case.get("mix", 0))
    return [r.randint(case["lo"], case["hi"]) for _ in range(case["batch"])]


# ---- the cases -----------------------------------------------------------------------------------
def listed():
    return [
        # the core smoke test's eight ciphertexts through every homomorphic operation: the smallest ring
        dict(name="ops_n12_b8", op="ops", ring="n12", batch=8, lo=3, hi=3, mix=0, step=1),
        # one product of a client's small ring, as it arrives: launches and latency count
        dict(name="relin_n13_one", op="relin", ring="n13", batch=1, lo=3, hi=3, mix=0, rescale=True),
        # one rotation at the top level, the latency of one key switch
        dict(name="rotate_n16_one", op="rotate", ring="n16w50", batch=1, lo=30, hi=30, mix=0, step=1),
        # the headline workload: a batch at uneven levels through HMUL + relinearisation and rotations
        dict(name="relin_rotate_n16_b32", op="relin_rotate", ring="n16w50", batch=32, lo=5, hi=30, mix=1, rotations=4),
        # products and rescales of the smaller serving ring, an odd batch at uneven levels
        dict(name="relin_n15_b31", op="relin", ring="n15", batch=31, lo=12, hi=18, mix=2, rescale=True),
        # rescales between products, over all levels down to the last one that has one
        dict(name="rescale_n16_b13", op="rescale", ring="n16w40", batch=13, lo=2, hi=30, mix=3),
        # the transforms by themselves, both directions, as the kernel-level entry gives them
        dict(name="ntt_n16_16x30", op="ntt", ring="n16w50", batch=16, lo=30, hi=30, mix=0),
        # a column of HMULPLAIN sums: one encrypted vector per term against plaintext weights
        dict(name="dot_n16_k48", op="dot", ring="n16w40", batch=2, lo=12, hi=12, mix=0, terms=48),
        # the paper's inference sequence, one document
        dict(name="infer_columns_one", op="infer", ring="n16w40", batch=1, lo=3, hi=3, mix=0, columns=True),
        # inference with few rotations, a full batch of documents
        dict(name="infer_diag_b32", op="infer", ring="n16w40", batch=32, lo=3, hi=3, mix=0, columns=False),
        # the serving mix on the smaller ring (vocabulary in two ciphertexts), requests at uneven levels
        dict(name="infer_diag_n15_b4", op="infer", ring="n15", batch=4, lo=12, hi=18, mix=4, columns=False),
        # an encrypted training step: forward, adjoint and update
        dict(name="train_n16_b4", op="train", ring="n16w40", batch=4, lo=16, hi=16, mix=0),
    ]


def _log_int(rng, lo, hi):
    return min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi + 0.5)))))))


def draw(rng):
    case = _draw(rng)
    most = max(work(c)["flops"] for c in listed())
    while case["batch"] > 1 and work(case)["flops"] > most:
        case["batch"] -= 1
    return case


def _draw(rng):
    op = rng.choice(["ops", "relin", "relin", "rotate", "relin_rotate", "rescale", "ntt", "dot", "hoisted", "infer",
                     "infer", "train"])
    mix = rng.randint(1, 1 << 20)
    if op == "ops":
        ring = rng.choice(["n12", "n13"])
        return dict(op=op, ring=ring, batch=_log_int(rng, 1, 20), lo=2, hi=3, mix=mix, step=rng.choice([1, -1, 2, 64]))
    if op == "train":
        return dict(op=op, ring="n16w40", batch=rng.randint(2, 4), lo=(l := rng.randint(10, 16)), hi=l, mix=mix)
    if op == "infer":
        columns = rng.random() < 0.3
        ring = "n16w40" if columns else rng.choice(["n15", "n16w40"])
        lo = rng.randint(3, 6) if columns else _log_int(rng, 3, 18)
        hi = lo if columns else min(18, lo + rng.choice([0, 1, 3]))
        return dict(op=op, ring=ring, batch=1 if columns else _log_int(rng, 1, 32), lo=lo, hi=hi, mix=mix,
                    columns=columns)
    ring = rng.choice(["n13", "n15", "n15", "n16w40", "n16w50", "n16w50", "n16w50c"])
    if op == "dot" and ring == "n16w50c":
        ring = "n16w50"
    top = RINGS[ring][1]
    a, b = sorted(rng.randint(2, top) for _ in range(2))
    most = 32 if RINGS[ring][0] >= 16 else 48
    case = dict(op=op, ring=ring, batch=_log_int(rng, 1, most), lo=a, hi=b, mix=mix)
    if op == "relin":
        case["rescale"] = rng.random() < 0.5
    elif op == "rotate":
        case["step"] = rng.choice([1, -1, 2, 64, 1024])
    elif op == "relin_rotate":
        case["rotations"] = rng.randint(1, 4)
    elif op == "ntt":
        case["lo"] = case["hi"]
    elif op == "hoisted":
        case.update(batch=1, lo=case["hi"], rotations=_log_int(rng, 2, 24))
    elif op == "dot":
        case.update(batch=rng.randint(1, 4), lo=min(a, 16), hi=min(a, 16), terms=_log_int(rng, 2, 64))
    return case


ROTATIONS = [1, 2, 4, 8]


def _model(ring, columns):
    """The served model, encoded once for every level."""
    key = (ring, columns)
    if key not in _models:
        H, O = synth.fasttext_weights(77, VOCAB, DIM, CLASSES)
        top = RINGS[ring][1]
        make = pft.pft_ft_model_create if columns else pft.pft_ft_model_create_diag
        _models[key] = make(context(ring), H, O, top)
    return _models[key]


def _infer_steps(ring, columns):
    t = 1 << (RINGS[ring][0] - 1)
    steps = [1 << i for i in range(t.bit_length() - 1)]
    return steps if columns else steps + list(range(3, DIM))


def _plaintexts(ring, level, count):
    """Weights encoded once."""
    key = (ring, level)
    have = _weights.setdefault(key, [])
    slots = 1 << (RINGS[ring][0] - 1)
    while len(have) < count:
        z = synth.slots(900 + len(have), min(slots, 256))
        have.append(pft.pft_encode(context(ring), z, 2.0 ** 20, level))
    return have[:count]


def prepare(case, seed):
    ring, op = case["ring"], case["op"]
    if op in ("ops", "rotate"):
        context(ring, [case["step"]])
    elif op == "relin_rotate":
        context(ring, ROTATIONS[:case["rotations"]])
    elif op == "hoisted":
        context(ring, list(range(1, case["rotations"] + 1)))
    elif op == "infer":
        context(ring, _infer_steps(ring, case["columns"]))
    elif op == "train":
        t = 1 << (RINGS[ring][0] - 1)
        n = TR_DIM
        context(ring, list(range(1, n)) + [n << i for i in range((t // n).bit_length() - 1)]
                + [1 << i for i in range(n.bit_length() - 1)] + [-(1 << i) for i in range(n.bit_length() - 1)])
    s = State(case, seed)
    if op in ("ops", "relin", "relin_rotate", "rotate", "rescale"):
        s.a = [s.ct(l) for l in levels_of(case)]
        s.c = [s.empty() for _ in s.a]
        if op not in ("rotate", "rescale"):
            s.b = [s.ct(l) for l in levels_of(case)]
        if op == "ops":
            s.sum, s.prod = [s.empty() for _ in s.a], [s.empty() for _ in s.a]
            s.p = [_plaintexts(ring, pft.pft_ct_level(h), 1)[0] for h in s.a]
    elif op == "ntt":
        s.fwd, s.inv = s.words(case["hi"], case["batch"]), s.words(case["hi"], case["batch"])
    elif op == "dot":
        s.cts = [s.ct(case["hi"]) for _ in range(case["batch"] * case["terms"])]
        s.pts = _plaintexts(ring, case["hi"], case["terms"])
        s.c = [s.empty() for _ in range(case["batch"])]
    elif op == "hoisted":
        s.a = [s.ct(case["hi"])]
        s.c = [s.empty() for _ in range(case["rotations"])]
    elif op == "infer":
        s.chunks = -(-VOCAB // (s.n // 2))
        s.model = _model(ring, case["columns"])
        scale = 2.0 ** 40 if case["columns"] else 2.0 ** 50
        s.v = [s.ct(l, scale) for l in levels_of(case) for _ in range(s.chunks)]
        s.c = [s.empty() for _ in range(case["batch"])]
    elif op == "train":
        c, l0, sc = context(ring), case["hi"], RINGS[ring][7]
        s.D = [s.ct(l0) for _ in range(TR_DIM)]
        s.P = s.ct(l0 - 1)
        if "mask" not in _weights:
            z = np.zeros(s.n // 2)
            z[:TR_DIM * TR_CLASSES:TR_DIM] = 1.0
            _weights["mask"] = pft.pft_encode(c, z, 2.0 ** (40 - TR_LIFT), RINGS[ring][1])
        s.mask = _weights["mask"]
        m = pft.pft_ft_enc_model_create_diag(c, s.D, s.P, s.mask, TR_VOCAB, TR_DIM, TR_CLASSES, TR_LIFT)
        dl, ll, ls = pft.pft_fasttext_train_spec(c, m, sc)
        pft.pft_ft_enc_model_destroy(m)
        s.docs = [s.ct(dl) for _ in range(case["batch"])]
        s.labels = [s.ct(ll, ls) for _ in range(case["batch"])]
        s.gD, s.gP = [s.empty() for _ in range(TR_DIM)], [s.empty()]
    return s


def run(s):
    case, op, c = s.case, s.case["op"], context(s.ring)
    if op == "ntt":
        pft.pft_ntt(c, s.fwd.data_ptr(), case["batch"], case["hi"], False)
        pft.pft_ntt(c, s.inv.data_ptr(), case["batch"], case["hi"], True)
        return [s.fwd, s.inv]
    if op == "ops":
        pft.pft_add_batch(c, s.a, s.b, s.sum)
        pft.pft_mul_plain_batch(c, s.sum, s.p, s.prod)
        pft.pft_mul_relin_batch(c, s.a, s.b, s.c)
        pft.pft_rescale_batch(c, s.c, s.c)
        pft.pft_rotate_batch(c, s.c, case["step"], s.c)
        return [s.view(h) for h in s.sum + s.prod + s.c]
    if op in ("relin", "relin_rotate"):
        if case["batch"] == 1:
            pft.pft_mul_relin(c, s.a[0], s.b[0], s.c[0])
        else:
            pft.pft_mul_relin_batch(c, s.a, s.b, s.c)
        if op == "relin" and case["rescale"]:
            pft.pft_rescale_batch(c, s.c, s.c)
        for k in range(case.get("rotations", 0)):
            pft.pft_rotate_batch(c, s.c, ROTATIONS[k], s.c)
    elif op == "rotate":
        if case["batch"] == 1:
            pft.pft_rotate(c, s.a[0], case["step"], s.c[0])
        else:
            pft.pft_rotate_batch(c, s.a, case["step"], s.c)
    elif op == "rescale":
        pft.pft_rescale_batch(c, s.a, s.c)
    elif op == "hoisted":
        pft.pft_rotate_hoisted(c, s.a[0], list(range(1, case["rotations"] + 1)), s.c)
    elif op == "dot":
        pft.pft_dot_plain_batch(c, s.cts, s.pts, case["terms"], s.c, pts_shared=True)
    elif op == "infer":
        if case["batch"] == 1:
            pft.pft_fasttext_infer(c, s.model, s.v, s.c[0])
        else:
            pft.pft_fasttext_infer_batch(c, s.model, s.v, s.chunks, s.c)
    elif op == "train":
        # the step consumes levels of its model, so each pass trains a model of its own
        m = pft.pft_ft_enc_model_create_diag(c, s.D, s.P, s.mask, TR_VOCAB, TR_DIM, TR_CLASSES, TR_LIFT)
        pft.pft_fasttext_train_step(c, m, s.docs, s.labels, TR_ETA, s.gD, s.gP)
        pft.pft_ft_enc_model_destroy(m)
        return [s.view(h) for h in s.gD + s.gP]
    return [s.view(h) for h in s.c]


# ---- the work of a pass ----------------------------------------------------------------------------
def _limb(ring):
    return (1 << RINGS[ring][0]) * 8


def _transform_muls(ring):
    return (1 << (RINGS[ring][0] - 1)) * RINGS[ring][0]


def _keyswitch(ring, l, key=True, modup=True):
    """(modular multiplications, bytes of the key) of one key switch at level l."""
    logn, _, k, alpha = RINGS[ring][:4]
    n, e, beta = 1 << logn, l + k, -(-l // alpha)
    muls = (2 * k + 2 * l) * _transform_muls(ring) + (2 * k * l + 2 * beta * e + 2 * l) * n
    if modup:
        muls += beta * e * _transform_muls(ring)
        muls += sum((e - d) * d for d in [min(alpha, l - j * alpha) for j in range(beta)]) * n
    rows = 1 if RINGS[ring][8] & pft.PFT_COMPRESSED_KEYS else 2
    return muls, (rows * beta * e * _limb(ring) if key else 0)


def _rescale(ring, l):
    return 2 * l * _transform_muls(ring) + 2 * l * (1 << RINGS[ring][0])


def work(case):
    """Modular multiply-adds count as two operations; bytes are the inputs, keys and plaintexts
    read once and the outputs written once (a key once per call, for the highest level)."""
    ring, op = case["ring"], case["op"]
    limb, n = _limb(ring), 1 << RINGS[ring][0]
    lv = levels_of(case) if op not in ("ntt", "dot", "hoisted", "train") else [case["hi"]] * case["batch"]
    top, muls, nbytes = max(lv), 0.0, 0.0
    if op == "ntt":
        limbs = 2 * sum(lv)
        return {"bytes": 2.0 * limbs * limb, "flops": 2.0 * limbs * _transform_muls(ring)}
    if op == "dot":
        l, k = case["hi"], case["terms"]
        return {"bytes": float((case["batch"] * 2 * (k + 1) + k) * l * limb),
                "flops": 2.0 * case["batch"] * 2 * k * l * n}
    if op in ("ops", "relin", "relin_rotate"):
        rots = 1 if op == "ops" else case.get("rotations", 0)
        rescaled = op == "ops" or case.get("rescale", False)
        nbytes += _keyswitch(ring, top)[1] + rots * _keyswitch(ring, top - rescaled)[1]
        for l in lv:
            muls += _keyswitch(ring, l)[0] + 4 * l * n + (_rescale(ring, l) if rescaled else 0)
            muls += rots * _keyswitch(ring, l - rescaled)[0] + (2 * l * n if op == "ops" else 0)
            nbytes += 2 * (2 * l + l - rescaled) * limb + (3 * l * limb if op == "ops" else 0)
    elif op == "rotate":
        nbytes += _keyswitch(ring, top)[1] + sum(4 * l * limb for l in lv)
        muls += sum(_keyswitch(ring, l)[0] for l in lv)
    elif op == "rescale":
        nbytes += sum(2 * (2 * l - 1) * limb for l in lv)
        muls += sum(_rescale(ring, l) for l in lv)
    elif op == "hoisted":
        l, r = case["hi"], case["rotations"]
        first, one = _keyswitch(ring, l), _keyswitch(ring, l, modup=False)
        muls += first[0] + (r - 1) * one[0]
        nbytes += r * one[1] + 2 * (1 + r) * l * limb
    elif op == "infer":
        chunks = -(-VOCAB // (n // 2))
        slot_bits = RINGS[ring][0] - 1
        dim_bits = DIM.bit_length() - 1
        for l in lv:
            if case["columns"]:
                muls += DIM * (slot_bits * _keyswitch(ring, l)[0] + 2 * chunks * l * n + _rescale(ring, l) + 2 * l * n)
            else:
                muls += chunks * (_keyswitch(ring, l)[0] + (DIM - 2) * _keyswitch(ring, l, modup=False)[0])
                muls += 2 * chunks * DIM * l * n + (slot_bits - dim_bits) * _keyswitch(ring, l)[0]
                muls += _rescale(ring, l) + dim_bits * _keyswitch(ring, l - 1)[0] + 2 * l * n
            muls += _rescale(ring, l - 1)
            nbytes += 2 * (chunks * l + l - 2) * limb
        nbytes += (DIM * chunks * top + (DIM if case["columns"] else 1) * (top - 1)) * limb
        rots = slot_bits if case["columns"] else (DIM - 1) + slot_bits
        nbytes += rots * _keyswitch(ring, top)[1]
    elif op == "train":
        l, b, d = case["hi"], case["batch"], TR_DIM
        slot_bits = RINGS[ring][0] - 1
        dim_bits = d.bit_length() - 1
        per_doc = _keyswitch(ring, l)[0] + (d - 2) * _keyswitch(ring, l, modup=False)[0]  # rotated documents
        per_doc += (2 * (slot_bits - dim_bits) + 2 * dim_bits + 4) * _keyswitch(ring, l - 3)[0] + 8 * d * l * n
        muls += b * per_doc + d * (_keyswitch(ring, l - 5)[0] + 2 * _rescale(ring, l - 5))
        nbytes += 2 * ((d + b) * l + d * (l - 6) + d * (l - 7)) * limb
        nbytes += (d - 1 + slot_bits + dim_bits + 1) * _keyswitch(ring, l)[1]
    return {"bytes": float(nbytes), "flops": 2.0 * muls}


def exact(case, seed):
    """Outputs are whole words: they are equal or they are wrong."""
    return None
