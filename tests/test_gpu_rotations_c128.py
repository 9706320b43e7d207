"""The complex128 rotation forms and large phases at FP64 accuracy: angles
around the switch between the cosine and the sine form, quarter and half
turns, runs and repeats.  The difference to the oracle is bounded in 2-norm,
where each gate's rounding adds at most 4 eps on either side and the oracle's
rounded phi + lambda (below 4 pi) another 8 eps: 16 eps a gate."""
import numpy as np
import pytest

from paper_2605_15098_gb300 import circuits as C
from test_gpu_rotations import ANGLES, EPS

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def sv():
    from paper_2605_15098_gb300 import build as B
    B.build()
    from paper_2605_15098_gb300 import sv as mod
    return mod


def check(sv, orc, n, g, stored, per_gate):
    rng = np.random.default_rng(n)
    psi = rng.normal(size=1 << n) + 1j * rng.normal(size=1 << n)
    psi /= np.linalg.norm(psi)
    ref = orc.apply(n, psi.copy() if stored else orc.init(n), g)
    with sv.State(n, sv.SV_C128) as s:
        if stored:
            sv.sv_copy_in(s.h, psi)
        s.apply(g, sv.make_config(sv.SV_MODE_PARTITIONED))
        got = s.amplitudes()
    assert np.linalg.norm(got - ref) <= per_gate * EPS * len(g)


@pytest.mark.parametrize("stored", [False, True])
@pytest.mark.parametrize("phases", [False, True])
@pytest.mark.parametrize("n", [14, 16])
def test_rotation_forms(sv, orc, n, phases, stored):
    rng = np.random.default_rng(3)
    recs = []
    for i, th in enumerate(ANGLES):
        for q in (i % n, (5 * i + 1) % n, (7 * i + 2) % n, 0):
            recs.append(C.u3(q, th, *(rng.uniform(0, 2 * np.pi, 2) if phases else (0.0, 0.0))))
        recs.append(C.cz(i % n, (i + 3) % n))
    for q in range(n):
        recs.append(C.u3(q, float(rng.uniform(0, 7)), 0.0, 0.0))
    check(sv, orc, n, C.gates(recs), stored, 16)


@pytest.mark.parametrize("stored", [False, True])
def test_large_phases(sv, orc, stored):
    """Both sides take the angle's double as exact, whatever its size."""
    n, rng = 14, np.random.default_rng(8)
    recs = [C.u3(q, 1.3, 0.0, 0.0) for q in range(n)]
    for q in range(n):
        recs.append(C.p(q, float(10.0 ** rng.integers(0, 11) * rng.uniform(-1, 1))))
        recs.append(C.cp(q, (q + 5) % n, float(10.0 ** rng.integers(0, 11) * rng.uniform(-1, 1))))
    check(sv, orc, n, C.gates(recs), stored, 8)
