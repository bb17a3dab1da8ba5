"""oz_dgemm's split of both operands (TC engines): rows, strips of columns
split by clusters (k_pad up to 1024) and column maxima plus tiles (longer), in
one launch for small products and in several for large ones. Every route gives
the oracle's bits, reports a non-finite entry of either operand and recovers,
and dependent launches keep their order: products whose operand is the result
of the product before, on one workspace, equal the same products run one at a
time. Results are exact integers rounded once, so every comparison is of bits."""
import numpy as np
import pytest

import synth
from tests.oracle_check import assert_oracle_bits

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("needs a CUDA device", allow_module_level=True)

import paper_2609_37693_gb300 as oz  # noqa: E402

DEV = torch.device("cuda:0")


def _dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).to(DEV)


def _operands(m, n, k, ta, tb, seed):
    A, B = synth.phi_pair(m, n, k, 1.0, seed=seed)
    return A, B, _dev(A.T if ta else A), _dev(B.T if tb else B)


# one tile of a strip, a strip over several blocks, the last strip length and
# the first tiled one; small (one launch) and large (several) products; few
# and many columns
SHAPES = [(1, 1, 1), (40, 33, 64), (65, 257, 65), (300, 31, 513), (129, 300, 1024), (129, 300, 1025), (3000, 50, 700),
          (50, 3000, 700), (1100, 2300, 2050)]


@pytest.mark.parametrize("ta,tb", [(0, 0), (1, 0), (0, 1), (1, 1)])
@pytest.mark.parametrize("m,n,k", SHAPES)
def test_split_routes_match_oracle(m, n, k, ta, tb):
    plan = oz.Plan(16, 0, k)
    A, B, Ad, Bd = _operands(m, n, k, ta, tb, m + n + k)
    C = oz.dgemm(Ad, Bd, plan, trans_a=bool(ta), trans_b=bool(tb))
    torch.cuda.synchronize()
    assert_oracle_bits(C, A, B, plan.moduli, plan.bits, what=f"{m}x{n}x{k} ta={ta} tb={tb}", count=600)


# either side of the most strided entries that are split together, and of the
# largest output whose kernels are launched dependent
@pytest.mark.parametrize("m,n,k,ta,tb", [(16300, 40, 256, 0, 0), (16300, 40, 256, 1, 0), (40, 16300, 256, 0, 0),
                                         (40, 16300, 256, 0, 1), (8200, 8200, 250, 1, 1), (4095, 2048, 64, 0, 0),
                                         (4096, 2048, 64, 0, 0), (2559, 2048, 64, 0, 0), (2560, 2048, 64, 0, 0)])
def test_routes_of_large_products_of_short_vectors(m, n, k, ta, tb):
    plan = oz.Plan(16, 0, k)
    A, B, Ad, Bd = _operands(m, n, k, ta, tb, m + k)
    C = oz.dgemm(Ad, Bd, plan, trans_a=bool(ta), trans_b=bool(tb))
    torch.cuda.synchronize()
    assert_oracle_bits(C, A, B, plan.moduli, plan.bits, what=f"{m}x{n}x{k} ta={ta} tb={tb}", count=600)


@pytest.mark.parametrize("q,bits", [(14, 0), (18, 62), (20, 70), (19, 66)])
@pytest.mark.parametrize("k", [200, 1500])
def test_split_routes_of_every_piece_count(q, bits, k):
    m, n = 70, 90
    plan = oz.Plan(q, bits, k)
    A, B, Ad, Bd = _operands(m, n, k, 0, 0, q + k)
    C = oz.dgemm(Ad, Bd, plan)
    torch.cuda.synchronize()
    assert_oracle_bits(C, A, B, plan.moduli, plan.bits, what=f"q={q} bits={bits} k={k}", count=m * n)


@pytest.mark.parametrize("engine", [oz.OZ_ENGINE_TC, oz.OZ_ENGINE_TC1])
@pytest.mark.parametrize("ta,tb", [(0, 0), (1, 0), (0, 1)])
@pytest.mark.parametrize("k", [130, 1200])
@pytest.mark.parametrize("side", ["A", "B"])
def test_nonfinite_is_reported_then_clear(engine, ta, tb, k, side):
    m, n = 300, 280
    plan = oz.Plan(16, 0, k, engine)
    A, B, Ad, Bd = _operands(m, n, k, ta, tb, 5)
    ws = oz.workspace(plan, m, n, k, DEV)
    X = Ad if side == "A" else Bd
    i, j = X.shape[0] - 1, X.shape[1] - 3
    good = X[i, j].item()
    for bad in (float("nan"), float("-inf")):
        X[i, j] = bad
        oz.dgemm(Ad, Bd, plan, trans_a=bool(ta), trans_b=bool(tb), ws=ws)
        assert oz.query_status(ws) == oz.OZ_ERR_NONFINITE
    X[i, j] = good
    C = oz.dgemm(Ad, Bd, plan, trans_a=bool(ta), trans_b=bool(tb), ws=ws)
    assert oz.query_status(ws) == oz.OZ_OK
    assert_oracle_bits(C, A, B, plan.moduli, plan.bits, what="after a non-finite run", count=400)


@pytest.mark.parametrize("n", [96, 600, 1300])
@pytest.mark.parametrize("graph", [False, True])
def test_chained_products_keep_their_order(n, graph):
    plan = oz.Plan(16, 0, n)
    g = torch.Generator(device=DEV).manual_seed(n)
    X0 = torch.randn(n, n, generator=g, device=DEV, dtype=torch.float64)
    M = torch.randn(n, n, generator=g, device=DEV, dtype=torch.float64) / n
    ws = oz.workspace(plan, n, n, n, DEV)
    bufs = [torch.empty_like(X0) for _ in range(2)]

    def chain(wait):
        X = X0
        for i in range(8):
            out = bufs[i & 1]
            if i % 3 == 2:
                oz.dgemm(M, X, plan, trans_b=True, out=out, ws=ws)
            else:
                oz.dgemm(X, M, plan, trans_a=bool(i % 2), out=out, ws=ws)
            X = out
            if wait:
                torch.cuda.synchronize()
        return X

    want = chain(True).clone()
    if graph:
        G = torch.cuda.CUDAGraph()
        with torch.cuda.graph(G):
            got = chain(False)
        for b in bufs:
            b.zero_()
        for _ in range(3):
            G.replay()
    else:
        for _ in range(3):
            got = chain(False)
    torch.cuda.synchronize()
    assert torch.equal(got.view(torch.int64), want.view(torch.int64))
