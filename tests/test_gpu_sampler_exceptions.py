"""The sampler's running sums where most values of a step of 32 leave the prefix
sum of integers (ties, values above the sum's binade, steps out of it): the rest
is then added one after the other, in blocks and over blocks, with the same samples."""
import math
from fractions import Fraction

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def sv():
    from paper_2605_15098_gb300 import build as B
    B.build()
    from paper_2605_15098_gb300 import sv as mod
    return mod


def exceptions(p):
    """Per step of 32 values of the first block: values that take an addition of their own."""
    out, run = [], 0.0
    for i, x in enumerate(p[:1024].tolist()):
        if i % 32 == 0:
            out.append(0)
        nxt = run + x
        if x:
            tie = run > 0.0 and 2 * abs(Fraction(run) + Fraction(x) - Fraction(nxt)) == Fraction(math.ulp(run))
            out[-1] += tie or math.frexp(run)[1] != math.frexp(nxt)[1]
        run = nxt
    return out


@pytest.mark.parametrize("kind,n", [(k, n) for k in ("ties", "doubling", "doubling_from_the_middle") for n in (6, 10, 11)] +
                         [("block_ties", 18), ("block_ties", 20)])
def test_samples_with_many_exceptions(sv, orc, kind, n):
    size = 1 << n
    i = np.arange(size)
    step = 1024 if kind == "block_ties" else 1
    tie = 2 if step == 1 else step
    if kind in ("ties", "block_ties"):  # two values, then only (block sums of) half the last place of their sum
        a = np.zeros(size, np.complex128)
        a[::step] = 2.0 ** -27
        a[:2] = math.sqrt(1.0 - 2.0 ** -20), 0.0
    else:
        start = 0 if kind == "doubling" else min(size // 2, 300)
        a = np.ldexp(1.0, np.minimum(np.maximum(i - start, 0), 400)).astype(np.complex128)
        a /= np.linalg.norm(a)
    mask = size - 1
    with sv.State(n, sv.SV_C128) as s:
        sv.sv_copy_in(s.h, a)
        p = s.probabilities(mask)
        for _ in range(8):  # the ties want a total of exactly 1
            if "ties" not in kind or p[tie] == 2.0 ** -54:
                break
            a[1] = math.sqrt(max(0.0, abs(a[1]) ** 2 + 1.0 - 2.0 ** -54 / p[tie]))
            sv.sv_copy_in(s.h, a)
            p = s.probabilities(mask)
        c = np.cumsum(p)
        at = c[::max(1, size // 256)] / c[-1]
        u = np.concatenate([np.random.default_rng(n).random(300), at, np.nextafter(at, 0.0)])
        u = np.minimum(u, np.nextafter(1.0, 0.0))
        got = s.sample(mask, u)
    assert max(exceptions(p if step == 1 else p.reshape(-1, step).sum(1))) > 16
    want, _ = orc.sample(p, u)
    assert np.array_equal(got, want)
