"""The groups of moduli that the planner itself forms for the 16-bit-digit
reconstruct: for every frozen base configuration they cover the moduli in order,
keep the bounds of the kernel's 32- and 64-bit sums, and have sizes that the kernel
is compiled for, so that no configuration falls back to pairs unseen."""
import math
import pathlib
import re

import pytest

import paper_2609_37693_gb300 as oz

# the sizes that oz_reconstruct.cu compiles the kernel for
SHAPES = {(2, 2, 4, 5, 6, 1), (2, 2, 2, 3, 5, 5), (3, 3, 3, 5, 5), (3, 3, 3, 4, 5), (3, 3, 3, 3, 6), (3, 4, 4, 4, 6)}
CONFIGS = [(fmt, k) for fmt in sorted(oz.FORMATS) for k in (1, 4096, 8192, 8193, 16384, 16385, 40000, 65536)]


def _plan(fmt, k):
    try:
        return oz.PlanFP(fmt, k)
    except oz.OzError as e:
        assert e.status == oz.OZ_ERR_K_TOO_LARGE
        pytest.skip("no configuration holds this many terms")


@pytest.mark.parametrize("fmt,k", CONFIGS)
def test_every_base_configuration_takes_the_grouped_kernel(fmt, k):
    plan = _plan(fmt, k)
    st, starts, compiled = oz.oz_selftest_digit16_groups(plan.handle)
    assert st == oz.OZ_OK and compiled
    m = plan.moduli
    assert starts[0] == 0 and starts[-1] == len(m)
    sizes = tuple(b - a for a, b in zip(starts, starts[1:]))
    assert sizes in SHAPES and min(sizes) >= 1 and len(sizes) <= 8
    sums = [(b - a) * math.prod(m[a:b]) for a, b in zip(starts, starts[1:])]
    assert max(sums) < 2**30 and sum(sums) < 2**32
    assert math.prod(m).bit_length() <= 125 and len(m) < 32
    for g, (a, b) in enumerate(zip(starts, starts[1:])):       # greedy: the next modulus would not have fitted
        if b < len(m):
            assert (b - a + 1) * math.prod(m[a:b + 1]) >= 2**30, (g, sizes)


def test_all_compiled_shapes_are_in_use():
    seen = set()
    for fmt in sorted(oz.FORMATS):
        for k in (8192, 16384, 40000):
            _, starts, _ = oz.oz_selftest_digit16_groups(oz.PlanFP(fmt, k).handle)
            seen.add(tuple(b - a for a, b in zip(starts, starts[1:])))
    assert seen == SHAPES


def test_widened_and_integer_plans():
    """Widened configurations (P past 2^125) have no groups; INT8 plans are refused."""
    plan = oz.PlanFP("E4M3", 16384, 69)
    assert oz.oz_selftest_digit16_groups(plan.handle) == (oz.OZ_OK, [0], False)
    assert oz.oz_selftest_digit16_groups(oz.Plan(16, 0, 64).handle)[0] == oz.OZ_ERR_INVALID_ARG


def test_code_tables_fit_the_row_split():
    """The split's table (a word per balanced residue) and the kernel's own shared
    memory stay within the 48 KB of a launch that asks for no more, at the
    limit that the launcher allows and for every base configuration."""
    src = (pathlib.Path(oz.__file__).parent / "csrc" / "oz_fp.cu").read_text()
    limit = int(re.search(r"kFpTableMax = (\d+) \* 1024;", src).group(1)) * 1024
    own = 8 * 8 + 4                                       # red[8], s_sh
    assert limit + own <= 48 * 1024 - 256
    for fmt, k in CONFIGS:
        try:
            moduli = oz.PlanFP(fmt, k).moduli
        except oz.OzError:
            continue
        assert sum(2 * (m // 2) + 1 for m in moduli) * 4 <= limit
