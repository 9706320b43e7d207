"""The learned planner in complex128: its plans run on the FP64 register-stage
kernel where the greedy rule's do, and the greedy prediction is that plan's."""
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


@pytest.fixture(scope="module")
def model(sv):
    import os
    import paper_2605_15098_gb300 as pkg
    m = sv.sv_cost_model_load(os.path.join(os.path.dirname(pkg.__file__), "data", "costmodel_gb300.svcm"))
    yield m
    sv.sv_cost_model_destroy(m)


def kinds_of(sv, s, g, cfg):
    sv.sv_profile(s.h, True)
    s.reset()
    s.apply(g, cfg)
    recs = sv.sv_profile_read(s.h)
    sv.sv_profile(s.h, False)
    return [r["gate_kind"] for r in recs if r["kind"] == sv.SV_KERNEL_TILE]


@pytest.mark.parametrize("n,make", [(20, lambda n: C.random_circuit(n, 8, 3)), (20, lambda n: C.qpe(n)[0]),
                                    (18, lambda n: layers(range(n), 12, 1, False)),  # cut passes
                                    (20, lambda n: layers(range(10), 10, 1, True))])
def test_register_stage_plans(sv, orc, model, n, make):
    g = make(n)
    greedy = sv.make_config(sv.SV_MODE_PARTITIONED)
    with sv.State(n, sv.SV_C128) as s:
        sv.sv_set_cost_model(s.h, model)
        choice = sv.sv_learned_plan(s.h, g, greedy)
        assert 0 < choice["predicted_ms"] <= choice["greedy_predicted_ms"]
        learned = kinds_of(sv, s, g, sv.make_config(sv.SV_MODE_PARTITIONED, planner=sv.SV_PLANNER_LEARNED))
        assert s.stats()["planner"] == sv.SV_PLANNER_LEARNED
        got = s.amplitudes()
        # -2: the register-stage kernel
        assert set(learned) == {-2} == set(kinds_of(sv, s, g, greedy))
        assert len(learned) == choice["passes"]
    assert np.max(np.abs(got - orc.run(n, g))) <= 1e-12


def test_same_structure_other_angles(sv, orc, model):
    """The choice is kept by the circuit's structure; angles of 0 (phases that
    vanish) change how its passes are cut, not whether they run."""
    n = 16
    g = layers(range(n), 12, 1, True)
    z = g.copy()
    z["p"][z["kind"] == C.U3, 1:] = 0.0
    cfg = sv.make_config(sv.SV_MODE_PARTITIONED, planner=sv.SV_PLANNER_LEARNED)
    for first, second in ((g, z), (z, g)):
        with sv.State(n, sv.SV_C128) as s:
            sv.sv_set_cost_model(s.h, model)
            for lst in (first, second):
                s.reset()
                s.apply(lst, cfg)
                assert s.stats()["planner"] == sv.SV_PLANNER_LEARNED
                assert np.max(np.abs(s.amplitudes() - orc.run(n, lst))) <= 1e-12
