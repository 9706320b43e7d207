"""Batches made and destroyed in turn, so that one batch's tensor maps lie where
another's lay: instances of the same sizes on qubits numbered upwards or
downwards, whose later passes read tiles at other physical bits.  Every
outcome equals the closed form."""
import numpy as np
import pytest

from paper_2605_15098_gb300 import circuits as C

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def sv():
    from paper_2605_15098_gb300 import build as B
    B.build()
    from paper_2605_15098_gb300 import sv as mod
    return mod


def instance(n, seed, down):
    """A QPE instance (n, gates, mask, outcome); `down`: qubit q is n - 1 - q."""
    g, _, info = C.qpe(n, seed)
    if not down:
        return n, g, info["mask"], info["y"]
    g = g.copy()
    two = g["control"] >= 0
    g["target"] = n - 1 - g["target"]
    g["control"][two] = n - 1 - g["control"][two]
    t = info["t"]
    y = sum(((info["y"] >> j) & 1) << (t - 1 - j) for j in range(t))
    return n, g, info["mask"] << (n - t), y


@pytest.mark.parametrize("split", [0, 14])
def test_alternating_batches(sv, split):
    cfg = sv.make_config(sv.SV_MODE_PARTITIONED, batch_split=split)
    sizes = [14, 15, 16, 17, 18] * 8
    for turn in range(8):
        work = [instance(n, 1000 * turn + i, turn & 1) for i, n in enumerate(sizes)]
        b = sv.sv_batch_create([(n, g, m) for n, g, m, _ in work], cfg)
        try:
            assert sv.sv_batch_info(b)["passes"] > len(work)  # passes that read their tiles
            for _ in range(2):
                idx, p, _ = sv.sv_batch_run(b, len(work))
                assert [int(v) for v in idx] == [w[3] for w in work], turn
                assert np.max(np.abs(p - 1.0)) <= 1e-5  # as tests/test_gpu_parity.py
        finally:
            sv.sv_batch_destroy(b)
