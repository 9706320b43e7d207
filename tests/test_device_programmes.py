"""The device form of register-stage programmes (tileprog.h), which the kernels
run, executed step by step in NumPy (complex128) from the library's export and
compared with the oracle: grouped rotations, rotations divided by their cosine
or sine, sign steps, tables and factors with their records in the step, phased
butterflies, the closing scale, and stage changes marked to stay within the
warps, which must not move an amplitude to another warp."""
import numpy as np
import pytest

import planemu
from gen import fold_leading, mixed_circuit
from paper_2605_15098_gb300 import circuits as C
from paper_2605_15098_gb300 import sv
from test_pass_cuts import layers

# handler codes (tileprog.h); gates: 16 + 8 kind + register bit (7: controlled)
STAGE, SCALE, ROTS, TABLE, FACTOR, ROTS4, SIGNS = 1, 2, 4, 5, 6, 7, 8
TOL = {"c64": 2e-5, "c128": 1e-12}  # as tests/test_gpu_parity.py


def run_pass(state, p, t2, wide, start=None):
    """One pass; `start` = (basis index, Hadamard mask): its generated form."""
    k, rb, seen = p["k"], t2["rb"], set()
    loc = np.arange(1 << k)
    mats = np.asarray(t2["dev_mats"], dtype=np.float64).reshape(-1, 8)
    rows = np.asarray(t2["statc"], dtype=np.float64).reshape(-1, t2["threads"], 2)
    rows = rows[:, :, 0] + 1j * rows[:, :, 1]
    turn = 2.0 ** (64 if wide else 32)

    def table(m0):
        fl, x = mats[m0:m0 + 8].reshape(-1), np.arange(32)
        if wide:
            return fl[2 * x] + 1j * fl[2 * x + 1]
        return fl[4 * (x >> 1) + (x & 1)] + 1j * fl[4 * (x >> 1) + 2 + (x & 1)]

    for tile in range(state.size >> k):
        base = planemu.pdep(tile, p["gmask"])
        idx = planemu.tile_index(p, base)
        t = state[idx].copy()
        if start is not None:
            basis, hq = start
            lead = sum(1 << q for s, q in enumerate(p["slot_phys"]) if (t2["gen_hmask"] >> s) & 1)
            # the leading Hadamards, unnormalised, on H^hq|basis>
            t = planemu.product_state(int(np.log2(state.size)), basis, hq ^ lead)[idx]
            both = bin(lead & hq).count("1")
            v = 2.0 ** (0.5 * bin(hq ^ lead).count("1") + 0.5 * (both - (bin(hq).count("1") - both)))
            t = t * v * t2["dev_gen_scale"]
        slots = []
        for terms in t2["slot_terms"]:
            u = sum(th for g0, g1, th in terms if (base >> g0) & 1 and (g1 < 0 or (base >> g1) & 1))
            slots.append(np.exp(2j * np.pi * ((u % int(turn)) / turn)))
        tid = warp = None
        for ins in t2["dev"]:
            hd = ins["hd"]
            seen.add(hd if hd < 16 else 16 + 8 * ((hd - 16) // 8))
            if hd == STAGE:
                st = t2["stages"][ins["aux"]]
                nw = t2["threads"].bit_length() - 6
                reg, thread = st[:rb], st[5:10 + nw]
                tid = sum(((loc >> b) & 1) << i for i, b in enumerate(thread))
                if ins["cidx"] & 1:
                    seen.add("local")
                    assert np.array_equal(warp, tid >> 5)
                warp = tid >> 5
                xreg = sum(((loc >> b) & 1) << j for j, b in enumerate(reg))
            elif hd == SCALE:
                t *= ins["scale"]
            elif hd in (ROTS, ROTS4):
                for n, j in enumerate((1, 2, 3, 4, 0)):
                    if not (ins["cidx"] >> j) & 1:
                        continue
                    m = mats[ins["aux"] + (n if hd == ROTS4 else (ins["e0"] >> (3 * j)) & 7)]
                    if wide and (ins["idx"] >> j) & 1:
                        u = [[m[2], -1], [1, m[2]]]
                    elif wide:
                        u = [[1, -m[2]], [m[2], 1]]
                    else:
                        assert m[0] == m[1] and m[2] == m[3]
                        a, b = np.array([[1, m[0]], [0, 1]]), np.array([[1, 0], [m[2], 1]])
                        u = a @ b @ a
                    planemu.apply_pairs(t, reg[j], np.asarray(u, dtype=complex))
            elif hd == TABLE:
                on = ((tid >> (ins["cidx"] - 1)) & 1) == 1 if ins["cidx"] else True
                t *= np.where(on, table(ins["aux"])[xreg], 1.0)
            elif hd == FACTOR:
                f = rows[ins["e0"]][tid] if ins["e0"] >= 0 else np.ones(t.size, dtype=complex)
                if ins["cidx"] >= 0:
                    f = f * slots[ins["cidx"]]
                dyn = [b for b in range(9) if (ins["aux"] >> b) & 1]
                for i, b in enumerate(dyn):
                    f = np.where((tid >> b) & 1, f * slots[ins["e1"] + i], f)
                t *= np.where((xreg >> (ins["idx"] - 1)) & 1, f, 1.0) if ins["idx"] else f
            elif hd == SIGNS:
                for j in range(rb):
                    if not (ins["cidx"] >> j) & 1:
                        continue
                    m, sl = ins["words"][j] & 0xFFFF, ins["words"][j] >> 16
                    neg = np.array([bin(v & m).count("1") & 1 for v in range(t2["threads"])])[tid]
                    if sl >= 0:
                        assert abs(abs(slots[sl].real) - 1) < 1e-9
                        neg = neg ^ int(slots[sl].real < 0)
                    t *= np.where(neg & (xreg >> j), -1.0, 1.0)
            else:
                kind, j = (hd - 16) // 8, ins["idx"]
                assert kind in (0, 1, 2, 4, 5), hd
                if kind == 5:  # phased butterfly
                    trec, row = (ins["aux"] & 0xFFFF) - 1, ((ins["aux"] >> 16) & 0xFFFF) - 1
                    f = table(trec)[xreg] if trec >= 0 else np.ones(t.size, dtype=complex)
                    if row >= 0:
                        f = f * rows[row][tid]
                    if ins["cidx"] >= 0:
                        f = f * slots[ins["cidx"]]
                    t *= np.where((xreg >> j) & 1, f, 1.0)
                cond = None
                if kind != 5 and ins["ccls"] == planemu.C_GLOBAL:
                    if not (base >> ins["cidx"]) & 1:
                        continue
                elif kind != 5 and ins["ccls"] in (planemu.C_REG, planemu.C_THREAD):
                    cond = ((xreg if ins["ccls"] == planemu.C_REG else tid) >> ins["cidx"]) & 1 == 1
                u = ([[1, 1], [1, -1]] if kind in (0, 5) else [[0, 1], [1, 0]] if kind == 1 else
                     planemu.mat_of(mats[ins["aux"]]))
                planemu.apply_pairs(t, reg[j], np.asarray(u, dtype=complex), cond)
        state[idx] = t
    return seen


CIRCUITS = {
    "random": (15, lambda n: C.random_circuit(n, 6, 5)),
    "layers": (14, lambda n: layers(range(n), 14, 3, False)),  # cut passes in complex128
    "mixed": (15, lambda n: mixed_circuit(n, 160, 11)),
    "qpe": (16, lambda n: C.qpe(n, 9)[0]),
    "angles": (14, lambda n: C.gates([C.u3(q, th, 0.3, 1.1) for i, th in enumerate(
        (0.0, np.pi / 2, np.pi, -np.pi / 2, 3 * np.pi, 1e-9, 5.0, -2.2)) for q in (i, 13 - i, 0)])),
}


@pytest.mark.parametrize("dt", ["c64", "c128"])
@pytest.mark.parametrize("name", list(CIRCUITS))
def test_against_oracle(orc, name, dt):
    n, make = CIRCUITS[name]
    wide = dt == "c128"
    basis, hq, g = fold_leading(make(n))
    plan = sv.sv_plan_export(n, sv.SV_C128 if wide else sv.SV_C64, g, sv.make_config(sv.SV_MODE_PARTITIONED))
    key = "t2d" if wide else "t2"
    seen = set()
    for generated in (False, True):
        state = planemu.product_state(n, basis, hq)
        for i, p in enumerate(plan["passes"]):
            if not p["ops"]:
                continue
            first = generated and i == 0
            if p.get("remap_before"):
                state = planemu.remap(state, p["remap_before"])
            if p["kernel"] == "generic":  # longer than a programme holds (complex64)
                planemu.run_generic_pass(state, p)
                continue
            seen |= run_pass(state, p, p[("t2dgen" if wide else "t2gen") if first else key], wide,
                             (basis, hq) if first else None)
        x = np.arange(1 << n)
        phys = sum(((x >> q) & 1) << plan["phys"][q] for q in range(n))
        assert np.max(np.abs(state[phys] - orc.run(n, make(n)))) <= TOL[dt]
    want = {"random": {TABLE, SIGNS, STAGE, SCALE, "local"} | ({ROTS} if wide else {ROTS4}), "mixed": {FACTOR, TABLE, 48},
            "layers": {ROTS, FACTOR} if wide else set(), "qpe": {16 + 40, SCALE}, "angles": {ROTS}}[name]
    if not wide:
        want = want - {SCALE} if name == "random" else want  # rotations keep the norm there
    assert want <= seen
