"""Diagonal runs whose register-bit factors are signs (CZ, CP by a half turn):
within a tile, across tiles, with and without phases beside them, and next to
phases that are not signs; against the oracle in both dtypes, from a generated
and from a stored state."""
import numpy as np
import pytest

from paper_2605_15098_gb300 import circuits as C

pytestmark = pytest.mark.gpu

# FP64 on both sides; FP32 storage, at most 200 gates (tests/test_gpu_parity.py)
TOL = {"c64": 2e-5, "c128": 1e-12}


@pytest.fixture(scope="module")
def sv():
    from paper_2605_15098_gb300 import build as B
    B.build()
    from paper_2605_15098_gb300 import sv as mod
    return mod


def layers(n, seed, phases, other):
    rng = np.random.default_rng(seed)
    recs = []
    for d in range(3):
        for q in range(n):
            recs.append(C.u3(q, *rng.uniform(0, 6, 3)) if phases else C.u3(q, float(rng.uniform(0, 6)), 0.0, 0.0))
        for _ in range(n):
            a, b = (int(x) for x in rng.choice(n, 2, replace=False))
            recs.append(C.cz(a, b))
        recs.append(C.cp(0, n - 1, np.pi))
        if other:
            a, b = (int(x) for x in rng.choice(n, 2, replace=False))
            recs.append(C.cp(a, b, 0.7))
            recs.append(C.cp(a, b, -np.pi))
            recs.append(C.p(a, 1.1))
    return C.gates(recs)


@pytest.mark.parametrize("dt", ["c64", "c128"])
@pytest.mark.parametrize("n,tile", [(6, 0), (13, 0), (15, 0), (17, 0), (16, 14)])
@pytest.mark.parametrize("phases", [False, True])
@pytest.mark.parametrize("other", [False, True])
def test_sign_factors(sv, orc, dt, n, tile, phases, other):
    if tile and dt == "c128":
        tile = 0
    g = layers(n, n + tile, phases, other)
    rng = np.random.default_rng(9)
    psi = rng.normal(size=1 << n) + 1j * rng.normal(size=1 << n)
    psi /= np.linalg.norm(psi)
    cfg = sv.make_config(sv.SV_MODE_PARTITIONED, **({"tile_qubits": tile} if tile else {}))
    for stored in (False, True):
        ref = orc.apply(n, psi.copy() if stored else orc.init(n), g)
        with sv.State(n, sv.SV_C64 if dt == "c64" else sv.SV_C128) as s:
            if stored:
                sv.sv_copy_in(s.h, psi)
            s.apply(g, cfg)
            got = s.amplitudes()
        assert np.max(np.abs(got - ref)) <= TOL[dt]
