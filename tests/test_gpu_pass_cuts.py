"""Complex128 passes cut to the length of a register-stage programme, against
the oracle; from |0...0> (a generated first piece) and from a stored state."""
import numpy as np
import pytest

from paper_2605_15098_gb300 import circuits as C
from test_pass_cuts import layers

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def sv():
    from paper_2605_15098_gb300 import build as B
    B.build()
    from paper_2605_15098_gb300 import sv as mod
    return mod


@pytest.mark.parametrize("stored", [False, True])
@pytest.mark.parametrize("n,k,count,cz", [(13, 13, 12, True), (14, 10, 10, False), (16, 16, 20, False),
                                          (18, 18, 12, True)])
def test_against_oracle(sv, orc, n, k, count, cz, stored):
    g = C.gates(([C.h(q) for q in range(0, n, 3)] if not stored else []) + list(layers(range(k), count, n, cz)))
    with sv.State(n, sv.SV_C128) as s:
        if stored:
            rng = np.random.default_rng(n)
            psi = rng.normal(size=1 << n) + 1j * rng.normal(size=1 << n)
            psi /= np.linalg.norm(psi)
            sv.sv_copy_in(s.h, psi)
            orc.apply(n, psi, g)
        else:
            psi = orc.run(n, g)
        s.apply(g, sv.make_config(sv.SV_MODE_PARTITIONED))
        got = s.amplitudes()
    assert np.max(np.abs(got - psi)) <= 1e-12  # FP64 on both sides (tests/test_gpu_parity.py)
