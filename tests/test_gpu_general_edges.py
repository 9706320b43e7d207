"""General gates where their sweeps change form: qubit 0 and others (one or two
amplitudes per vector), the smallest states, many controls, measurements of
both outcomes; against the oracle, in both dtypes."""
import numpy as np
import pytest

from paper_2605_15098_gb300 import circuits as C

pytestmark = pytest.mark.gpu

TOL = {"c64": 2e-5, "c128": 1e-12}


@pytest.fixture(scope="module")
def sv():
    from paper_2605_15098_gb300 import build as B
    B.build()
    from paper_2605_15098_gb300 import sv as mod
    return mod


def haar(rng, k):
    z = rng.normal(size=(k, k)) + 1j * rng.normal(size=(k, k))
    q, r = np.linalg.qr(z)
    return q * (np.diag(r) / np.abs(np.diag(r)))


@pytest.mark.parametrize("dt", ["c64", "c128"])
@pytest.mark.parametrize("n", [1, 2, 3, 5, 12, 19])
def test_against_oracle(sv, orc, dt, n):
    rng = np.random.default_rng(n)
    psi = rng.normal(size=1 << n) + 1j * rng.normal(size=1 << n)
    psi /= np.linalg.norm(psi)
    top = n - 1
    recs = []
    if n >= 2:
        recs += C.u2q(0, top, haar(rng, 4)) + C.u2q(top, 0, haar(rng, 4))
        recs += [C.mcu([0], top, haar(rng, 2)), C.mcu([top], 0, haar(rng, 2))]
    if n >= 3:
        recs += C.u2q(1, top, haar(rng, 4))
        recs += [C.mcu([1], top, haar(rng, 2)), C.mcu(list(range(n - 1)), top, haar(rng, 2)),
                 C.mcu(list(range(1, n)), 0, haar(rng, 2))]
    for q in sorted({0, min(1, top), n // 2, top}):
        # the input's own p0 after the gates so far, and a u well inside an outcome
        cur = orc.apply_measured(n, (v := psi.copy()), C.gates(recs)) if recs else None
        v = psi if cur is None else v
        p0 = float(np.sum(np.abs(v[((np.arange(1 << n) >> q) & 1) == 0]) ** 2))
        recs.append(C.measure(q, 0.5 * p0 if q % 2 == 0 else min(0.999, 0.5 * (1 + p0))))
        if p0 < 0.01 or p0 > 0.99:
            recs.pop()
    g = C.gates(recs) if recs else C.gates([C.measure(0, 0.3)])
    ref = psi.copy()
    bits = orc.apply_measured(n, ref, g)
    with sv.State(n, sv.SV_C64 if dt == "c64" else sv.SV_C128) as s:
        sv.sv_copy_in(s.h, psi)
        s.apply(g, sv.make_config(sv.SV_MODE_PERGATE))
        assert np.array_equal(s.measurements(), bits)
        got = s.amplitudes()
    assert np.max(np.abs(got - ref)) <= TOL[dt] * max(1.0, np.max(np.abs(ref)))
