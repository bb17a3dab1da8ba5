"""Groups of moduli of the 16-bit-digit reconstruct (float formats): for every
frozen configuration the greedy consecutive groups keep the bounds that the
kernel relies on, and the grouped sum equals the CRT sum."""
import math
import random

import pytest

import paper_2609_37693_gb300 as oz


def groups_of(moduli):
    """Consecutive moduli while (size) M < 2^30, as the planner takes them."""
    out, q = [], 0
    while q < len(moduli):
        e, M = q, 1
        while e < len(moduli) and (e - q + 1) * M * moduli[e] < 2**30:
            M *= moduli[e]
            e += 1
        assert e > q
        out.append((q, e, M))
        q = e
    return out


@pytest.mark.parametrize("fmt", sorted(oz.FORMATS))
@pytest.mark.parametrize("k", [8192, 16384, 40000])
def test_digit16_groups_are_exact(fmt, k):
    m = oz.PlanFP(fmt, k).moduli
    P, groups = math.prod(m), groups_of(m)
    assert len(groups) <= 8 and P.bit_length() <= 125 and len(m) <= 31
    assert sum((e - q) * M for q, e, M in groups) < 2**32        # 64-bit limb accumulators
    rng = random.Random(k)
    for case in range(200):
        y = [x - 1 for x in m] if case == 0 else [rng.randrange(x) for x in m]
        S, f = 0, 0.0
        for q, e, M in groups:
            t = sum(y[i] * (M // m[i]) for i in range(q, e))
            assert t < 2**32
            S += t * (P // M)
            f += t / M
        assert S == sum(yi * (P // mi) for yi, mi in zip(y, m)) and S < 32 * P
        assert abs(f - S / P) < 2**-10
