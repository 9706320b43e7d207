"""The phase of P gates as a fraction of a turn in units of 2^-64: against
p / (2 pi) mod 1 in exact rational arithmetic.  The two parts of the product
are each rounded to one unit (half a unit of error each), and the rest of the
reduction is below 2^-4 of a unit for |p| < 2^40."""
from fractions import Fraction
import math
import random

import pytest

from paper_2605_15098_gb300 import circuits as C
from paper_2605_15098_gb300 import sv

TERM_L, TERM_G = 0, 2


def pi_fraction(bits=400):
    """pi by Machin's formula, 16 atan(1/5) - 4 atan(1/239), in fixed point."""
    one = 1 << (bits + 20)

    def atan_inv(x):
        t, s, k = one // x, 0, 0
        while t:
            s += t // (2 * k + 1) * (-1 if k & 1 else 1)
            t //= x * x
            k += 1
        return s

    return Fraction(16 * atan_inv(5) - 4 * atan_inv(239), one)


PI = pi_fraction()
r = random.Random(5)
ANGLES = {
    "small": [r.uniform(-1e-9, 1e-9) for _ in range(16)],
    "one turn": [r.uniform(-math.pi, math.pi) for _ in range(16)],
    "third quarter": [r.uniform(-3.1, -1.6) for _ in range(16)],
    "several turns": [r.uniform(-40.0, 40.0) for _ in range(16)],
    "large": [r.uniform(-1, 1) * 2.0 ** r.uniform(6, 39) for _ in range(16)],
    "ends": [math.pi, -math.pi, math.pi / 2, -math.pi / 2, 2 * math.pi, -2 * math.pi, 3 * math.pi, 0.0, -0.0,
             math.nextafter(math.pi, 0), math.nextafter(-math.pi, -4), 1.0, -1.0, math.pi / 4, -math.pi / 4, 1e-300],
}


@pytest.mark.parametrize("dtype", [sv.SV_C64, sv.SV_C128])
@pytest.mark.parametrize("name", list(ANGLES))
def test_turns(name, dtype):
    n, angles = 16, ANGLES[name]
    plan = sv.sv_plan_export(n, dtype, C.gates([C.p(q, a) for q, a in enumerate(angles)]),
                             sv.make_config(sv.SV_MODE_PARTITIONED))
    got = [0] * n
    for p in plan["passes"]:
        for kind, a, _, theta in p["terms"]:
            got[p["slot_phys"][a] if kind == TERM_L else a] += theta
            assert kind in (TERM_L, TERM_G)
    for a, t in zip(angles, got):
        want = Fraction(a) / (2 * PI) * (1 << 64)
        d = (Fraction(t) - want) % (1 << 64)
        assert min(d, (1 << 64) - d) <= Fraction(9, 8), (a, t)
