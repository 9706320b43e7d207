"""Measurements of complex64 states far from unit norm, and of a half far
smaller than the other: FP32 squares of such amplitudes vanish, lose their
remainders or overflow, the FP64 sums of the contract do not.  Against the
oracle on the same FP32 amplitudes; the tolerance is tests/test_gpu_parity.py's
for FP32 storage."""
import numpy as np
import pytest

from paper_2605_15098_gb300 import circuits as C

pytestmark = pytest.mark.gpu

TOL = 2e-5


@pytest.fixture(scope="module")
def sv():
    from paper_2605_15098_gb300 import build as B
    B.build()
    from paper_2605_15098_gb300 import sv as mod
    return mod


def check(sv, orc, n, psi, q, u):
    g = C.gates([C.measure(q, u)])
    psi = psi.astype(np.complex64).astype(np.complex128)
    ref = psi.copy()
    bits = orc.apply_measured(n, ref, g)
    with sv.State(n, sv.SV_C64) as s:
        sv.sv_copy_in(s.h, psi)
        s.apply(g, sv.make_config(sv.SV_MODE_PERGATE))
        assert np.array_equal(s.measurements(), bits)
        got = s.amplitudes()
    assert abs(np.linalg.norm(ref) - 1.0) < 1e-9  # the oracle renormalised a half
    assert np.max(np.abs(got - ref)) <= TOL * np.max(np.abs(ref))


@pytest.mark.parametrize("scale", [1e-30, 1e-23, 1e-20, 1.0, 1e15, 1e25])
@pytest.mark.parametrize("n", [1, 2, 5, 12, 19])
def test_scaled_states(sv, orc, n, scale):
    rng = np.random.default_rng(n)
    psi = rng.normal(size=1 << n) + 1j * rng.normal(size=1 << n)
    psi *= scale / np.linalg.norm(psi)
    for q in sorted({0, n // 2, n - 1}):
        for u in (0.001, 0.999):  # both outcomes, far from p0
            check(sv, orc, n, psi, q, u)


@pytest.mark.parametrize("small", [1e-12, 1e-20, 1e-23, 1e-30, 0.0])
@pytest.mark.parametrize("n,q", [(2, 0), (5, 4), (16, 0), (16, 9), (16, 15)])
def test_a_small_half(sv, orc, n, q, small):
    """u = 0 picks outcome 0 whenever p0 > 0, however small (and 1 when it is 0)."""
    rng = np.random.default_rng(100 * n + q)
    psi = rng.normal(size=1 << n) + 1j * rng.normal(size=1 << n)
    psi /= np.linalg.norm(psi)
    psi[((np.arange(1 << n) >> q) & 1) == 0] *= small
    check(sv, orc, n, psi, q, 0.0)


@pytest.mark.parametrize("n,q,q0", [(3, 1, 0), (5, 4, 0), (14, 0, 5), (14, 6, 0), (17, 9, 16), (17, 9, 9)])
@pytest.mark.parametrize("scale", [1e-30, 1.0])
def test_zeros_of_both_signs(sv, orc, n, q, q0, scale):
    """A qubit q0 cleared by an earlier measurement, its zeros of either sign, and
    few amplitudes left in the other half: zeros add nothing, the rest counts."""
    rng = np.random.default_rng(n + q)
    psi = (rng.normal(size=1 << n) + 1j * rng.normal(size=1 << n)) * scale
    i = np.arange(1 << n)
    psi[(((i >> q0) & 1) == 1) | (rng.random(1 << n) < 0.7)] = 0.0
    psi[i[psi == 0][::2]] = complex(-0.0, -0.0)
    psi[0] = scale
    for u in (0.0, 0.999):
        check(sv, orc, n, psi, q, u)
