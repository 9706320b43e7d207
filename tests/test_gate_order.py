"""The stage compiler orders the gates between two diagonal runs: gates on one
qubit keep their order, controlled gates keep their place, and a layer over
all tile qubits takes fewer stages.  The exported programme runs in the NumPy
executor against the oracle."""
import numpy as np
import pytest

import planemu
from paper_2605_15098_gb300 import build as B
from paper_2605_15098_gb300 import circuits as C


@pytest.fixture(scope="module")
def sv():
    B.build()
    from paper_2605_15098_gb300 import sv as mod
    return mod


def sequence(n, seed, controlled):
    """Non-commuting gates in repeated and shuffled order, with and without
    controlled ones and diagonals between them."""
    rng = np.random.default_rng(seed)
    recs = []
    for _ in range(6 * n):
        q, c = (int(x) for x in rng.choice(n, 2, replace=False))
        u = rng.uniform()
        if controlled and u < 0.25:
            recs.append(C.cu(c, q, np.array([[0, 1], [1, 0]])))
        elif u < 0.35:
            recs.append(C.cz(c, q))
        elif u < 0.5:
            recs.append(C.h(q))
        elif u < 0.6:
            recs.append(C.x(q))
        else:
            recs.append(C.u3(q, *rng.uniform(0, 6, 3)))
    return C.gates(recs)


@pytest.mark.parametrize("controlled", [False, True])
@pytest.mark.parametrize("dtype,n,seed", [(0, 5, 1), (0, 10, 2), (0, 13, 3), (0, 15, 4), (1, 13, 5), (1, 15, 6)])
def test_ordered_gates(sv, orc, controlled, dtype, n, seed):
    g = sequence(n, seed, controlled)
    ref = orc.run(n, g)
    plan = sv.sv_plan_export(n, dtype, g, sv.make_config(sv.SV_MODE_PARTITIONED))
    for use_gen in (True, False):
        got = planemu.run_plan(n, plan, use_gen=use_gen)
        # FP32 matrices and 32-bit phases / FP64 (tests/test_planner_host.py)
        assert np.max(np.abs(got - ref)) <= (1e-12 if dtype else 2e-5)


def test_layers_share_stages(sv):
    """Layers of rotations over 13 tile qubits, a diagonal run between each:
    the register bits of one layer's last stage start the next layer."""
    n, depth = 13, 6
    recs = []
    for d in range(depth):
        recs += [C.u3(q, 0.3 + q, 1.1 + d, 2.2) for q in range(n)]
        recs += [C.cz(q, q + 1) for q in range(d % 2, n - 1, 2)]
    plan = sv.sv_plan_export(n, 0, C.gates(recs), sv.make_config(sv.SV_MODE_PARTITIONED))
    stages = [i for i in plan["passes"][0]["t2"]["ins"] if i["op"] == 0]
    assert len(stages) <= 2 * depth + 2
