"""What a workspace holds before a call does not reach its result. Plane rows past
the operands and digits past the last column are not written by the products, so
they are whatever the memory held, and the reconstruct reads such digits with the
row's last ones: every product here runs on workspaces filled with bytes that
make the largest digits (0xFF, as planes NaN), large finite planes (0x7F) or
small ones (0x01), and gives the oracle's bits. And products that are split in one
launch with column maxima and tiles (inner dimensions past 1024) keep their order
when they are launched dependent on one another, plain and from a graph."""
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


@pytest.fixture(params=[0xFF, 0x7F, 0x01], ids=hex)
def filled(request, monkeypatch):
    """Every byte tensor that the library allocates (its workspaces) starts with this byte."""
    empty = torch.empty

    def poisoned(*args, **kwargs):
        t = empty(*args, **kwargs)
        return t.fill_(request.param) if t.dtype == torch.uint8 else t

    monkeypatch.setattr(torch, "empty", poisoned)
    return request.param


# few columns past a tile, a digit word, a 16-byte run; splits of the inner dimension; one slab and several
SHAPES = [(70, 1, 200), (130, 33, 64), (257, 75, 1100), (300, 301, 700), (40, 523, 2100), (64, 90, 6000)]


@pytest.mark.parametrize("engine", [oz.OZ_ENGINE_TC, oz.OZ_ENGINE_TC1, oz.OZ_ENGINE_IMMA])
@pytest.mark.parametrize("q", [9, 16, 20])
@pytest.mark.parametrize("m,n,k", SHAPES)
def test_integer_products(filled, engine, q, m, n, k):
    plan = oz.Plan(q, 0, k, engine)
    A, B = synth.phi_pair(m, n, k, 1.0, seed=q + n)
    C = oz.dgemm(_dev(A), _dev(B), plan)
    torch.cuda.synchronize()
    assert_oracle_bits(C, A, B, plan.moduli, plan.bits, what=f"q={q} {m}x{n}x{k}")


@pytest.mark.parametrize("fmt", ["E4M3", "E3M2", "E2M1"])
@pytest.mark.parametrize("m,n,k", SHAPES[:5])
def test_float_products(filled, fmt, m, n, k):
    plan = oz.PlanFP(fmt, k)
    A, B = synth.phi_pair(m, n, k, 1.0, seed=n)
    C = oz.dgemm(_dev(A), _dev(B), plan)
    torch.cuda.synchronize()
    assert_oracle_bits(C, A, B, plan.moduli, plan.bits, what=f"{fmt} {m}x{n}x{k}")


@pytest.mark.parametrize("slab", [300, 1100])
def test_blocked_products(filled, slab):
    m, n, k = 130, 75, 2500
    for plan in (oz.Plan(16, 53, k), oz.PlanFP("E4M3", k)):
        A, B = synth.phi_pair(m, n, k, 1.0, seed=slab)
        C = oz.dgemm_blocked(_dev(A), _dev(B), plan, slab)
        torch.cuda.synchronize()
        assert_oracle_bits(C, A, B, plan.moduli, plan.bits, what=f"blocked {slab}")


@pytest.mark.parametrize("kind", ["grouped", "batched"])
def test_many_products(filled, kind):
    rng = np.random.default_rng(4)
    ops = [synth.phi_pair(m, n, k, 1.0, seed=int(rng.integers(1000))) for m, n, k in SHAPES]
    As, Bs = [_dev(a) for a, _ in ops], [_dev(b) for _, b in ops]
    Cs = [torch.zeros(m, n, dtype=torch.float64, device=DEV) for m, n, _ in SHAPES]
    if kind == "grouped":
        batch = oz.GroupedGemm(As, Bs, Cs)
        batch.run()
    else:
        batch = oz.BatchedGemm(SHAPES, nstreams=2)
        batch.run(As, Bs, Cs)
    torch.cuda.synchronize()
    for (A, B), C, p in zip(ops, Cs, batch.plans):
        assert_oracle_bits(C, A, B, p.moduli, p.bits, what=kind)


def test_host_products(filled):
    m, n, k = 300, 290, 500
    plan = oz.Plan(16, 0, k)
    A, B = synth.phi_pair(m, n, k, 1.0, seed=1)
    C = torch.zeros(m, n, dtype=torch.float64).pin_memory()
    h = oz.HostGemm(plan, m, n, k, 256, cols_per_chunk=256)
    h(torch.from_numpy(np.ascontiguousarray(A)).pin_memory(), torch.from_numpy(np.ascontiguousarray(B)).pin_memory(), C)
    torch.cuda.synchronize()
    assert_oracle_bits(C, A, B, plan.moduli, plan.bits, what="host")


@pytest.mark.parametrize("graph", [False, True])
@pytest.mark.parametrize("n", [1030, 1100])
def test_chain_of_products_split_in_tiles(n, graph):
    plan = oz.Plan(16, 0, n)
    g = torch.Generator(device=DEV).manual_seed(n)
    X0 = torch.randn(n, n, generator=g, device=DEV, dtype=torch.float64)
    M = torch.randn(n, n, generator=g, device=DEV, dtype=torch.float64) / n
    ws = oz.workspace(plan, n, n, n, DEV)
    bufs = [torch.empty_like(X0) for _ in range(2)]

    def chain(wait):
        X = X0
        for i in range(8):                        # rows and tiles, tiles on both sides, rows on both
            out = bufs[i & 1]
            oz.dgemm(X, M, plan, trans_a=i % 4 in (1, 2), trans_b=i % 4 >= 2, out=out, ws=ws)
            X = out
            if wait:
                torch.cuda.synchronize()
        return X

    want = chain(True).clone()
    if graph:
        G = torch.cuda.CUDAGraph()
        with torch.cuda.graph(G):
            got = chain(False)
        for _ in range(3):
            for b in bufs:
                b.zero_()
            G.replay()
    else:
        for _ in range(3):
            got = chain(False)
    torch.cuda.synchronize()
    assert torch.equal(got.view(torch.int64), want.view(torch.int64))
