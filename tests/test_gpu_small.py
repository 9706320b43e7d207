"""SV_MODE_AUTO on small states (the resident kernel): bit-identical to the
per-gate kernels, at the sizes where its layout changes (one CTA, clusters of
2, 4 and 8, the largest slice), with lists longer than one launch holds, with
general gates in between, from a recorded and from a stored state."""
import numpy as np
import pytest

from gen import general_circuit, mixed_circuit
from paper_2605_15098_gb300 import circuits as C

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def sv():
    from paper_2605_15098_gb300 import build as B
    B.build()
    from paper_2605_15098_gb300 import sv as mod
    return mod


@pytest.mark.parametrize("dt", ["c64", "c128"])
@pytest.mark.parametrize("n", [1, 2, 3, 4, 7, 8, 10, 11, 12, 13, 14, 15])
def test_same_bits_as_per_gate(sv, dt, n):
    dtype = sv.SV_C64 if dt == "c64" else sv.SV_C128
    rng = np.random.default_rng(n)
    psi = rng.normal(size=1 << n) + 1j * rng.normal(size=1 << n)
    psi /= np.linalg.norm(psi)
    for m, make in ((60, mixed_circuit), (1100, mixed_circuit), (40, general_circuit if n > 1 else mixed_circuit)):
        g = make(n, m, 17 * n + m)
        for start in (None, psi):
            got = []
            for cfg in (None, sv.make_config(sv.SV_MODE_PERGATE)):
                with sv.State(n, dtype) as s:
                    if start is not None:
                        sv.sv_copy_in(s.h, start)
                    s.apply(g, cfg)
                    got.append(s.amplitudes())
            assert np.array_equal(got[0], got[1])


def test_launches(sv):
    """One launch for a list that fits one, whatever its length up to that."""
    g = C.random_circuit(15, 20)
    with sv.State(15, sv.SV_C64) as s:
        s.apply(g)
        st = s.stats()
    assert st["gates"] == 440 and st["kernels"] == 1 and st["passes"] == 1
