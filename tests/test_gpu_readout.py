"""Read-outs at the sizes where their kernels change: few and many outcomes,
with and without physical bit 0, fewer than 32 amplitudes per outcome, one and
many thread blocks, blocks of the CDF and its steps; probabilities against the
oracle, samples equal to the oracle's on the same probabilities."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def sv():
    from paper_2605_15098_gb300 import build as B
    B.build()
    from paper_2605_15098_gb300 import sv as mod
    return mod


MASKS = [
    (1, [0]), (2, [1]), (5, [0, 1, 2, 3, 4]), (9, [3]), (9, [0]), (11, [0, 10]), (11, list(range(7))),
    (14, [1, 2, 3, 4, 5, 6, 7, 8, 9, 10, 11, 12, 13]),   # no bit 0, one amplitude pair per outcome
    (14, list(range(14))), (16, [2, 9, 15]), (16, [0, 3, 9, 15]), (18, list(range(2, 13))),
    (20, [19]), (20, [0]), (20, list(range(0, 20, 2))), (20, list(range(1, 20))), (21, list(range(21))),
    (22, [21, 7]), (22, list(range(0, 18))), (22, list(range(4, 22))),
]


@pytest.mark.parametrize("dt", ["c64", "c128"])
@pytest.mark.parametrize("n,qubits", MASKS)
def test_probabilities_argmax_samples(sv, orc, dt, n, qubits):
    rng = np.random.default_rng(100 * n + len(qubits))
    psi = rng.normal(size=1 << n) + 1j * rng.normal(size=1 << n)
    psi = (psi / np.linalg.norm(psi)).astype(np.complex64 if dt == "c64" else np.complex128)
    mask = sum(1 << q for q in qubits)
    ref = orc.marginal(n, psi.astype(np.complex128), mask)
    u = rng.random(700)
    u[:2] = [0.0, np.nextafter(1.0, 0.0)]
    with sv.State(n, sv.SV_C64 if dt == "c64" else sv.SV_C128) as s:
        sv.sv_copy_in(s.h, psi)
        p = s.probabilities(mask)
        again = s.probabilities(mask)
        idx, pmax = s.argmax(mask)
        got = s.sample(mask, u)
    # FP64 sums of up to 2^21 terms (complex64: squares to 2^-44)
    assert np.max(np.abs(p - ref)) <= 2e-13 * np.max(ref)
    assert np.array_equal(p, again)
    assert idx == int(np.argmax(ref)) and abs(pmax - ref[idx]) <= 2e-13 * ref[idx]
    want, _ = orc.sample(p, u)
    assert np.array_equal(got, want)


def test_ties_take_the_lowest_index(sv):
    from paper_2605_15098_gb300 import circuits as C
    for n, mask in ((6, 0b111000), (12, 0xFFF), (20, 0xFFFF0), (20, 0b11)):
        with sv.State(n, sv.SV_C64) as s:
            s.apply(C.gates([C.h(q) for q in range(n)]))
            idx, p = s.argmax(mask)
        assert idx == 0 and p == 2.0 ** -bin(mask).count("1")


@pytest.mark.parametrize("n", [5, 10, 12, 15, 21])
@pytest.mark.parametrize("kind", ["uniform", "sparse", "binades", "dyadic", "growing", "tiny"])
def test_samples_follow_the_running_sums(sv, orc, n, kind):
    """Running sums with ties, steps out of the binade at many places, zeros, and
    values above the sum so far: samples equal the oracle's, also at the CDF's own values."""
    rng = np.random.default_rng(n)
    size = 1 << n
    a = {"uniform": lambda: np.ones(size),
         "sparse": lambda: (rng.random(size) < 0.01) * rng.random(size),
         "binades": lambda: np.ldexp(rng.random(size), rng.integers(-60, 60, size)),
         "dyadic": lambda: np.ldexp(1.0, rng.integers(0, 12, size)),
         "growing": lambda: np.ldexp(1.0 + rng.random(size), np.arange(size) * 200 // size),
         "tiny": lambda: np.where(np.arange(size) < size // 2, 1e-160, 1.0)}[kind]()
    a[-1] = max(a[-1], 1e-3)
    psi = (a / np.linalg.norm(a)).astype(np.complex128)
    mask = size - 1
    with sv.State(n, sv.SV_C128) as s:
        sv.sv_copy_in(s.h, psi)
        p = s.probabilities(mask)
        c = np.cumsum(p)
        at = c[rng.integers(0, size, 200)] / c[-1]
        u = np.minimum(np.concatenate([rng.random(300), at, np.nextafter(at, 0.0)]), np.nextafter(1.0, 0.0))
        got = s.sample(mask, u)
    want, _ = orc.sample(p, u)
    assert np.array_equal(got, want)
