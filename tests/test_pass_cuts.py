"""Complex128 passes longer than a register-stage programme are cut in two:
no exported pass falls back to the generic tile kernel, gate counts stay, and
the cut plans' steps give the oracle's amplitudes (NumPy, complex128)."""
import numpy as np
import pytest

import planemu
from paper_2605_15098_gb300 import circuits as C
from paper_2605_15098_gb300 import sv


def layers(qubits, count, seed, cz):
    """`count` layers of U3 on the given qubits, with CZ on a matching."""
    rng = np.random.default_rng(seed)
    recs = []
    for _ in range(count):
        recs += [C.u3(q, *(float(v) for v in rng.uniform(0, 2 * np.pi, 3))) for q in qubits]
        perm = [int(q) for q in rng.permutation(qubits)]
        recs += [C.cz(a, b) for a, b in zip(perm[0::2], perm[1::2]) if cz]
    return C.gates(recs)


LONG = [(20, list(range(10)), 10, False), (20, list(range(10)), 10, True), (20, list(range(13)), 12, True),
        (16, list(range(16)), 40, False), (18, list(range(18)), 20, False), (14, list(range(14)), 12, True)]


@pytest.mark.parametrize("n,qubits,count,cz", LONG)
def test_no_pass_on_the_generic_kernel(n, qubits, count, cz):
    g = layers(qubits, count, n, cz)
    plan = sv.sv_plan_export(n, sv.SV_C128, g, sv.make_config(sv.SV_MODE_PARTITIONED))
    assert [p["kernel"] for p in plan["passes"] if p["ops"]].count("t2d") == len(plan["passes"]) > 1
    assert sum(p["ngates"] for p in plan["passes"]) == len(g)


def test_cut_plan_matches_oracle(orc):
    n, qubits, count, cz = LONG[-1]
    g = layers(qubits, count, n, cz)
    plan = sv.sv_plan_export(n, sv.SV_C128, g, sv.make_config(sv.SV_MODE_PARTITIONED))
    got = planemu.run_plan(n, plan, use_gen=False)
    # FP64 on both sides; 304 gates
    assert np.max(np.abs(got - orc.run(n, g))) <= 1e-12


def test_swaps_in_the_tile_keep_u3_whole():
    """A pass with an in-tile SWAP runs on the generic kernel, where a split U3
    costs the same arithmetic and diagonal runs besides."""
    n = 16
    whole = [C.swap(0, 9)]
    for r in layers(range(n), 2, 1, True):  # U3 as the general 2x2, which is never split
        t, (th, ph, la) = int(r["target"]), (float(v) for v in r["p"][:3])
        whole.append(r if r["kind"] != C.U3 else C.u(t, [
            [np.cos(th / 2), -np.exp(1j * la) * np.sin(th / 2)],
            [np.exp(1j * ph) * np.sin(th / 2), np.exp(1j * (ph + la)) * np.cos(th / 2)]]))
    cfg = sv.make_config(sv.SV_MODE_PARTITIONED, flags=sv.SV_FLAG_NO_RELABEL)
    steps = [[[op["type"] for op in p["ops"]] for p in sv.sv_plan_export(n, sv.SV_C128, C.gates(g), cfg)["passes"]]
             for g in ([C.swap(0, 9)] + list(layers(range(n), 2, 1, True)), whole)]
    assert any(planemu.TOP_SWAP in p for p in steps[1])
    assert steps[0] == steps[1]
