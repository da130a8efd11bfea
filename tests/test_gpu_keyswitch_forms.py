"""The streamed key inner product over its range of digit counts (1..16, the generic kernel above),
inputs per stage and levels in one batch, and its permuted form through hoisted rotations: bit for bit
against the oracle."""
import pytest

from paper_1908_06972_gb300 import synth
from .pairs import Pair

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def p18(gpu):
    """One prime per digit: a ciphertext at level l has l digits."""
    p = Pair(gpu, 12, 18, 1, 1, rot_steps=[1, -3, 64])
    yield p
    p.close()


@pytest.fixture(scope="module")
def p8(gpu):
    p = Pair(gpu, 13, 8, 2, 2, rot_steps=[1, 5])
    yield p
    p.close()


def enc(p, i, level):
    o = p.orc
    return o.encrypt_sk(o.encode(synth.slots(50 + i, 32), level=level), 60 + i)


@pytest.mark.parametrize("levels", [[18], [16], [17, 1, 3], [9, 1, 2, 8, 16, 5, 9], [2] * 7, [1] * 19, [8, 4, 4, 3],
                                    [9, 9, 4], [10, 1, 9], [12, 8, 11, 9]])
def test_digit_counts(p18, levels):
    p, o, pf = p18, p18.orc, p18.pft
    distinct = {l: (enc(p, 2 * l, l), enc(p, 2 * l + 1, l)) for l in set(levels)}
    want = {l: o.rotate(o.mul_relin(a, b), -3) for l, (a, b) in distinct.items()}
    outs = [p.empty() for _ in levels]
    pf.pft_mul_relin_batch(p.ctx, [p.ct(distinct[l][0]) for l in levels], [p.ct(distinct[l][1]) for l in levels], outs)
    pf.pft_rotate_batch(p.ctx, outs, -3, outs)
    for i, (h, l) in enumerate(zip(outs, levels)):
        p.assert_equal(h, want[l], "input %d at level %d" % (i, l))


@pytest.mark.parametrize("level", [1, 2, 3, 8, 9, 10, 12, 16, 18])
def test_hoisted_digit_counts(p18, level):
    p, o, pf = p18, p18.orc, p18.pft
    a = enc(p, 7, level)
    steps = [1, 0, -3, 64]
    outs = [p.empty() for _ in steps]
    pf.pft_rotate_hoisted(p.ctx, p.ct(a), steps, outs)
    want = o.rotate_hoisted(a, [1, -3, 64])
    for h, w, st in zip(outs, [want[0], a, want[1], want[2]], steps):
        p.assert_equal(h, w, "hoisted rotate %d at level %d" % (st, level))


def test_hoisted_repeated_output(p8):
    """A handle given for several steps ends with the last one's rotation."""
    p, o, pf = p8, p8.orc, p8.pft
    a = enc(p, 9, 7)
    x, y = p.empty(), p.empty()
    pf.pft_rotate_hoisted(p.ctx, p.ct(a), [1, 5, 1, 0], [x, y, y, x])
    w = o.rotate_hoisted(a, [1])
    p.assert_equal(y, w[0], "last step of a repeated output")
    p.assert_equal(x, a, "identity as the last step")
