"""The most likely outcome of states with NaN amplitudes, of either sign: a NaN
never wins, so the index is the largest other entry's, or 2^64 - 1 where there
is none; the probability is NaN."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

NONE = 2 ** 64 - 1


@pytest.fixture(scope="module")
def sv():
    from paper_2605_15098_gb300 import build as B
    B.build()
    from paper_2605_15098_gb300 import sv as mod
    return mod


@pytest.mark.parametrize("bits", [0x7FF8000000000000, 0xFFF8000000000000])
@pytest.mark.parametrize("dt", ["c64", "c128"])
@pytest.mark.parametrize("n", [4, 18])
def test_nan(sv, n, dt, bits):
    nan = np.array([bits], dtype=np.uint64).view(np.float64)[0]
    some = np.full((1 << n, 2), 0.1)
    some[5] = 0.3
    some[9] = nan
    for psi, want in ((np.full((1 << n, 2), nan), (NONE, NONE, NONE)), (some, (5, 5, 2))):
        for mask, idx in zip(((1 << n) - 1, 7, 6), want):
            with sv.State(n, sv.SV_C64 if dt == "c64" else sv.SV_C128) as s:
                sv.sv_copy_in(s.h, psi.view(np.complex128).reshape(-1))
                got, p = s.argmax(mask)
            assert got == idx and np.isnan(p)
