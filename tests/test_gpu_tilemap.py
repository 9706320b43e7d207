"""The tensor copies that gather a register-stage pass's tiles, at the shapes
where their description changes: scattered local qubits (more runs than the
tensor's dimensions, so several copies per tile), one run of 13 bits (wider
than a box dimension), a wide gap, 2^14 tiles, and both dtypes; from a state
that is in the buffer, so that every pass reads its tiles."""
import numpy as np
import pytest

from paper_2605_15098_gb300 import circuits as C

pytestmark = pytest.mark.gpu

# FP64 on both sides / FP32 storage with at most 60 gates (tests/test_gpu_parity.py)
TOL = {"c64": 2e-5, "c128": 1e-12}


@pytest.fixture(scope="module")
def sv():
    from paper_2605_15098_gb300 import build as B
    B.build()
    from paper_2605_15098_gb300 import sv as mod
    return mod


CASES = [
    (20, [5, 7, 9, 11, 13, 15, 17, 19], 13, 4, 0),    # every high local bit a run of its own
    (19, [4, 6, 8, 9, 11, 13, 14, 16, 18], 13, 4, 0),
    (20, [12, 13, 14, 15, 16, 17, 18, 19], 13, 5, 0),  # a gap above the chunk, then one run
    (15, [5, 6, 7, 8, 9, 10, 11, 12], 13, 5, 0),       # one run of 13 bits
    (20, [4, 6, 8, 10, 12, 14, 16, 18, 19], 14, 5, 0),  # wide tiles
    (18, [13, 15, 17, 2], 13, 13, 2),                  # contiguous blocks after remaps
    (13, [0, 5, 12], 13, 5, 0),                        # the tile is the state
]


@pytest.mark.parametrize("dt", ["c64", "c128"])
@pytest.mark.parametrize("n,targets,k,c,flags", CASES)
def test_gather(sv, orc, dt, n, targets, k, c, flags):
    if dt == "c128" and k == 14:
        k = 13
    rng = np.random.default_rng(1000 * n + len(targets) + k + c)
    psi = rng.normal(size=1 << n) + 1j * rng.normal(size=1 << n)
    psi /= np.linalg.norm(psi)
    recs = []
    for q in targets + targets[::-1]:
        recs.append(C.u3(q, *rng.uniform(0, 2 * np.pi, 3)))
        recs.append(C.cp(q, int((q + 1 + rng.integers(0, n - 1)) % n), float(rng.uniform(-3, 3))))
    g = C.gates(recs)
    ref = orc.apply(n, psi.copy(), g)
    cfg = sv.make_config(sv.SV_MODE_PARTITIONED, tile_qubits=k, chunk_qubits=c, flags=flags)
    with sv.State(n, sv.SV_C64 if dt == "c64" else sv.SV_C128) as s:
        sv.sv_copy_in(s.h, psi)
        s.apply(g, cfg)
        got = s.amplitudes()
    assert np.max(np.abs(got - ref)) <= TOL[dt]
