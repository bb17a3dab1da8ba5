"""The reconstruct phase on integers that take each of its paths, fed as CRT
digits: every length from one bit to the window's (a magnitude is moved up by
none to three 32-bit limbs, or from the fifth), exact zeros, ties of the final
rounding and the same decided by the lowest bit, the window's edges (quotients
next to a tie, corrected by the general path), subnormal and overflowing results,
and the largest digit sums; neighbours in a row take different paths. Byte digits
for every group shape of the INT8 plans, 16-bit digits for every group shape of
the float formats, with rows that the grouped kernels take (a pitch that is a
multiple of 8 or 4) and rows that they leave to the general kernel. Results are
exact integers rounded once, so every comparison is of bits."""
import numpy as np
import pytest

import oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("needs a CUDA device", allow_module_level=True)

import paper_2609_37693_gb300 as oz  # noqa: E402

DEV = torch.device("cuda:0")
EXPS = [0, -1, 5, -1074, -1100, -1200, 1000, 900, 1023, -1022, -30, -120]
# one plan for each shape of the groups of 16-bit digits
FP_PLANS = [("E2M1", 8192), ("E4M3", 8192), ("E4M3", 40000), ("E3M2", 8192), ("E3M2", 16384), ("E3M2", 40000)]


def _integers(P, moduli, rng):
    half = P // 2
    xs = [0, 1, -1, half - 1, -half, half - 2**40, -half + 3, 0]
    for length in list(range(1, 160, 7)) + [25, 26, 27, 32, 33, 53, 54, 64, 65, 96, 97, 124, 125, 126,
                                             128, 129, 156]:
        x = (1 << (length - 1)) | (int(rng.integers(0, 2**62)) % (1 << (length - 1)) if length > 1 else 0)
        xs += [x, -x]
        if length > 54:                       # a tie, and one unit of the lowest bit either side
            tie = ((2**52 + int(rng.integers(0, 2**52))) << (length - 53)) + (1 << (length - 54))
            xs += [tie, -tie, tie + 1, -tie - 1, tie - 1, -tie + 1]
            xs += [(1 << length) - 1, -(1 << length) + 1]      # rounds up to a power of two
    for digits in ([m - 1 for m in moduli], [int(rng.integers(0, m)) for m in moduli]):
        x = sum(d * (P // m) for d, m in zip(digits, moduli)) % P
        xs.append(x - P if x >= P - half else x)
    xs = [x for x in xs if -half <= x < P - half]
    return [xs[i] for i in rng.permutation(len(xs))]


def _check(plan, dtype, multiple, seed):
    moduli = plan.moduli
    P = oracle.modulus_product(moduli)
    rng = np.random.default_rng(seed)
    xs = _integers(P, moduli, rng)
    while (len(xs) % multiple != 0) if multiple > 1 else (len(xs) % 2 == 0):
        xs.append(int(rng.integers(-2**40, 2**40)))
    m, n = len(EXPS), len(xs)
    digits = np.zeros((len(moduli), m, n), dtype=dtype)
    for q, mq in enumerate(moduli):
        inv = pow((P // mq) % mq, -1, mq)
        digits[q] = np.array([((x % mq) * inv) % mq for x in xs], dtype=dtype)
    Y = torch.from_numpy(digits.view(np.uint8)).to(DEV)
    s = torch.tensor([-e for e in EXPS], dtype=torch.int32, device=DEV)
    t = torch.zeros(n, dtype=torch.int32, device=DEV)
    C = torch.zeros((m, n), dtype=torch.float64, device=DEV)
    assert oz.oz_reconstruct(plan.handle, m, n, Y.data_ptr(), s.data_ptr(), t.data_ptr(), C.data_ptr(), n,
                             oz._stream_handle()) == oz.OZ_OK
    torch.cuda.synchronize()
    want = np.array([oracle.round_scaled(xs, [e] * n) for e in EXPS])
    got = C.cpu().numpy()
    bad = np.argwhere(got.view(np.uint64) != want.view(np.uint64))
    assert bad.size == 0, [(xs[j], EXPS[i], got[i, j], want[i, j]) for i, j in bad[:4]]


@pytest.mark.parametrize("q", range(9, 21))
@pytest.mark.parametrize("multiple", [8, 4, 1])
def test_byte_digits(q, multiple):
    _check(oz.Plan(q, 0, 4, oz.OZ_ENGINE_IMMA), np.uint8, multiple, q)


@pytest.mark.parametrize("fmt,k", FP_PLANS)
@pytest.mark.parametrize("multiple", [4, 1])
def test_16_bit_digits(fmt, k, multiple):
    _check(oz.PlanFP(fmt, k), np.uint16, multiple, k)


@pytest.mark.parametrize("zero_rows", [False, True])
@pytest.mark.parametrize("q", [9, 16])
def test_zero_products_are_plus_zero(q, zero_rows):
    m, n, k = 70, 130, 90
    g = torch.Generator(device=DEV).manual_seed(q)
    A = torch.randn(m, k, generator=g, device=DEV, dtype=torch.float64)
    B = torch.randn(k, n, generator=g, device=DEV, dtype=torch.float64)
    if zero_rows:
        A[::3] = -0.0
    else:
        A.zero_()
    C = oz.dgemm(A, B, oz.Plan(q, 0, k))
    torch.cuda.synchronize()
    zeros = C[::3] if zero_rows else C
    assert not zeros.view(torch.int64).any()
