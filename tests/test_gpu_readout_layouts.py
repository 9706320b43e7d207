"""Marginals without physical bit 0 at the lines between their layouts: a warp,
two lanes or a thread per outcome, loads of one or two amplitudes (complex64
from n = 20), fewer than five bits summed over; both ends of the state's
qubits, and outcome bits out of order.  Tolerances as tests/test_gpu_readout.py."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def sv():
    from paper_2605_15098_gb300 import build as B
    B.build()
    from paper_2605_15098_gb300 import sv as mod
    return mod


def spread(n, m, low):
    """m qubits from `low` up, the rest drawn."""
    rng = np.random.default_rng(97 * n + m)
    return [low] + sorted(int(q) for q in rng.choice(np.arange(low + 1, n), size=m - 1, replace=False))


CASES = [(n, spread(n, m, low)) for n, m in ((19, 13), (19, 14), (20, 14), (20, 15), (21, 15), (21, 16), (22, 15), (22, 18))
         for low in (1, 2, 3)]
CASES += [(20, list(range(5, 20))), (20, list(range(4, 20))), (22, list(range(7, 22))), (22, list(range(5, 22))),
          (23, list(range(5, 23))), (24, list(range(5, 24))), (24, [1] + list(range(6, 24))),
          (24, list(range(9, 24))), (25, list(range(10, 25))), (25, [1] + list(range(11, 25))),
          (26, list(range(1, 17)))]  # complex128: a warp's lanes far apart


@pytest.mark.parametrize("dt", ["c64", "c128"])
@pytest.mark.parametrize("n,qubits", CASES)
def test_against_oracle(sv, orc, dt, n, qubits):
    rng = np.random.default_rng(n + len(qubits))
    psi = rng.normal(size=1 << n) + 1j * rng.normal(size=1 << n)
    psi = (psi / np.linalg.norm(psi)).astype(np.complex64 if dt == "c64" else np.complex128)
    mask = sum(1 << q for q in qubits)
    ref = orc.marginal(n, psi.astype(np.complex128), mask)
    with sv.State(n, sv.SV_C64 if dt == "c64" else sv.SV_C128) as s:
        sv.sv_copy_in(s.h, psi)
        p = s.probabilities(mask)
        idx, pmax = s.argmax(mask)
        again = s.probabilities(mask)
    assert np.max(np.abs(p - ref)) <= 2e-13 * np.max(ref)
    assert np.array_equal(p, again)
    assert idx == int(np.argmax(ref)) and abs(pmax - ref[idx]) <= 2e-13 * ref[idx]


@pytest.mark.parametrize("dt", ["c64", "c128"])
@pytest.mark.parametrize("n,low,m", [(20, 1, 15), (20, 2, 15), (22, 3, 18), (23, 4, 19)])
def test_permuted_qubits(sv, orc, dt, n, low, m):
    """The same after SWAPs, which only change the qubit map: outcome bits then
    lie in another order than their physical bits."""
    from paper_2605_15098_gb300 import circuits as C

    rng = np.random.default_rng(m)
    psi = rng.normal(size=1 << n) + 1j * rng.normal(size=1 << n)
    psi = (psi / np.linalg.norm(psi)).astype(np.complex64 if dt == "c64" else np.complex128)
    g = C.gates([C.swap(low, n - 1), C.swap(low + 3, n - 2), C.swap(low + 1, n - 4)])
    ref_psi = orc.apply(n, psi.astype(np.complex128), g)
    mask = ((1 << m) - 1) << low
    ref = orc.marginal(n, ref_psi, mask)
    with sv.State(n, sv.SV_C64 if dt == "c64" else sv.SV_C128) as s:
        sv.sv_copy_in(s.h, psi)
        s.apply(g, sv.make_config(sv.SV_MODE_PARTITIONED))
        p = s.probabilities(mask)
        idx, _ = s.argmax(mask)
    assert np.max(np.abs(p - ref)) <= 2e-13 * np.max(ref)
    assert idx == int(np.argmax(ref))
