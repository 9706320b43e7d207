"""Rotations in the register-stage kernels: angles around the switch between
the cosine and the sine form (complex128), quarter and half turns, repeated
rotations of one qubit, runs of rotations on every tile bit, and phases of
large angles; against the oracle in both dtypes, from a generated and from a
stored state."""
import numpy as np
import pytest

from paper_2605_15098_gb300 import circuits as C

pytestmark = pytest.mark.gpu

# FP64 on both sides; FP32 storage, at most 200 gates (tests/test_gpu_parity.py)
TOL = {"c64": 2e-5, "c128": 1e-12}
EPS = np.finfo(np.float64).eps


@pytest.fixture(scope="module")
def sv():
    from paper_2605_15098_gb300 import build as B
    B.build()
    from paper_2605_15098_gb300 import sv as mod
    return mod


ANGLES = [0.0, np.pi / 2, np.pi / 2 * (1 + 4 * EPS), np.pi / 2 * (1 - 4 * EPS), np.pi, -np.pi / 2, 3 * np.pi / 2,
          2 * np.pi, 1e-9, np.pi - 1e-9, 5.0, -2.2]


@pytest.mark.parametrize("dt", ["c64", "c128"])
@pytest.mark.parametrize("stored", [False, True])
def test_rotation_forms(sv, orc, dt, stored):
    n = 14
    rng = np.random.default_rng(3)
    psi = rng.normal(size=1 << n) + 1j * rng.normal(size=1 << n)
    psi /= np.linalg.norm(psi)
    recs = []
    for i, th in enumerate(ANGLES):  # every angle on several tile bits, in runs and repeated
        for q in (i % n, (5 * i + 1) % n, (7 * i + 2) % n, 0):
            recs.append(C.u3(q, th, *rng.uniform(0, 2 * np.pi, 2)))
        recs.append(C.u3(i % n, th, 0.0, 0.0))
        recs.append(C.cz(i % n, (i + 3) % n))
    for q in range(n):  # a run over all bits
        recs.append(C.u3(q, float(rng.uniform(0, 7)), 0.0, 0.0))
    for q in range(0, n, 3):
        recs.append(C.p(q, float(10.0 ** rng.integers(0, 9) * rng.uniform(-1, 1))))
    g = C.gates(recs)
    start = psi.copy() if stored else orc.init(n)
    ref = orc.apply(n, start, g)
    with sv.State(n, sv.SV_C64 if dt == "c64" else sv.SV_C128) as s:
        if stored:
            sv.sv_copy_in(s.h, psi)
        s.apply(g, sv.make_config(sv.SV_MODE_PARTITIONED))
        got = s.amplitudes()
    # a phase p is known to an ulp of p: up to 1e8 * eps here, on top of TOL
    assert np.max(np.abs(got - ref)) <= TOL[dt] + 1e8 * EPS * np.max(np.abs(ref)) * len([r for r in recs if r[0] == C.P])
