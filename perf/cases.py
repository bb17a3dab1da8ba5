"""The workloads this library's speed is judged by: what a user's program has
in hand before a product (``prepare``), one pass through the public entry
points (``run``), what a pass cannot do without (``work``) and the same result
in plain float64 (``exact``).

A case is a dict of plain values. ``kind`` picks the entry point:

* ``dgemm``     oz.dgemm on a kept plan and workspace: m, n, k, the transposes,
                the modulus count q (bits: the widest the window allows);
* ``autograd``  oz.EmuMatmul forward and backward: C, dA, dB;
* ``grouped``   oz.GroupedGemm, captured once and replayed: many uneven
                products in one launch per phase;
* ``batched``   oz.BatchedGemm: many uneven products over several streams;
* ``blocked``   oz.dgemm_blocked: a long inner dimension in slabs;
* ``fp``        oz.dgemm on a float-format plan (fmt);
* ``host``      oz.HostGemm on pinned host matrices.

Operands are (U(-0.5, 0.5)) exp(phi N(0, 1)); upstream gradients N(0, 1).
"""
import math

import numpy as np
import torch

import paper_2609_37693_gb300 as oz


def listed():
    return [
        # One small product, the size a solver calls in an inner loop: launches and latency count.
        {"name": "dgemm_256", "kind": "dgemm", "m": 256, "n": 256, "k": 256, "ta": False, "tb": False, "q": 14, "phi": 0.5},
        # A middling product whose sizes fit no tile, both operands stored transposed.
        {"name": "dgemm_ragged_tt", "kind": "dgemm", "m": 1000, "n": 777, "k": 1531, "ta": True, "tb": True, "q": 16, "phi": 2.0},
        # The most moduli (70 bits kept): operands of a wide exponent spread, where accuracy is what the caller pays for.
        {"name": "dgemm_2048_q20", "kind": "dgemm", "m": 2048, "n": 2048, "k": 2048, "ta": False, "tb": False, "q": 20, "phi": 4.0},
        # The headline product.
        {"name": "dgemm_8192", "kind": "dgemm", "m": 8192, "n": 8192, "k": 8192, "ta": False, "tb": False, "q": 16, "phi": 0.5},
        # The largest size of the square sweep.
        {"name": "dgemm_16384", "kind": "dgemm", "m": 16384, "n": 16384, "k": 16384, "ta": False, "tb": False, "q": 16, "phi": 1.0},
        # A square layer trained in emulated FP64: one forward and one backward.
        {"name": "autograd_4096", "kind": "autograd", "m": 4096, "n": 4096, "k": 4096, "phi": 1.0},
        # A tall and skinny layer: bound by memory, and dB has a long inner dimension over few tiles.
        {"name": "autograd_tall", "kind": "autograd", "m": 65536, "n": 256, "k": 256, "phi": 1.0},
        # 256 uneven products, each dimension log-uniform on [64, 4096], as one captured graph.
        {"name": "grouped_256", "kind": "grouped", "count": 256, "hi": 4096, "shapes": 0, "phi": 1.0},
        # A few uneven products whose operands change from call to call, spread over streams without a graph.
        {"name": "batched_24", "kind": "batched", "count": 24, "hi": 2048, "shapes": 7, "streams": 4, "phi": 1.0},
        # A long inner dimension in slabs: the workspace holds one slab's planes.
        {"name": "blocked_32768", "kind": "blocked", "m": 8192, "n": 8192, "k": 32768, "slab": 8192, "phi": 0.5},
        # The FP8 variant.
        {"name": "fp_e4m3_4096", "kind": "fp", "fmt": "E4M3", "m": 4096, "n": 4096, "k": 4096, "phi": 0.5},
        # Operands and result in host memory, the copies part of the product.
        {"name": "host_8192", "kind": "host", "m": 8192, "n": 8192, "k": 8192, "phi": 0.5},
    ]


def _log_uniform(rng, lo, hi):
    x = int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))
    return min(max(x, lo), hi)


def draw(rng):
    kind = rng.choice(["dgemm", "dgemm", "dgemm", "dgemm", "autograd", "grouped", "batched", "blocked", "fp", "host"])
    phi = rng.choice([0.5, 1.0, 2.0, 4.0])
    if kind == "grouped":
        return {"kind": kind, "count": _log_uniform(rng, 8, 192), "hi": _log_uniform(rng, 512, 4096),
                "shapes": rng.randrange(1, 1 << 20), "phi": phi}
    if kind == "batched":
        return {"kind": kind, "count": _log_uniform(rng, 4, 48), "hi": _log_uniform(rng, 256, 3000),
                "shapes": rng.randrange(1, 1 << 20), "streams": rng.choice([1, 2, 4, 8]), "phi": phi}
    if kind == "blocked":
        return {"kind": kind, "m": _log_uniform(rng, 256, 6000), "n": _log_uniform(rng, 256, 6000),
                "k": _log_uniform(rng, 12000, 60000), "slab": rng.choice([4096, 8192, 16384]), "phi": phi}
    if kind == "fp":
        return {"kind": kind, "fmt": rng.choice(["E4M3", "E5M2", "E2M3", "E3M2", "E2M1"]),
                "m": _log_uniform(rng, 256, 8192), "n": _log_uniform(rng, 256, 8192), "k": _log_uniform(rng, 256, 8192),
                "phi": phi}
    if kind == "host":
        return {"kind": kind, "m": _log_uniform(rng, 1024, 8192), "n": _log_uniform(rng, 1024, 8192),
                "k": _log_uniform(rng, 1024, 8192), "phi": phi}
    if kind == "autograd":
        if rng.random() < 0.5:
            return {"kind": kind, "m": _log_uniform(rng, 4096, 65536), "n": _log_uniform(rng, 64, 512),
                    "k": _log_uniform(rng, 64, 512), "phi": phi}
        return {"kind": kind, "m": _log_uniform(rng, 256, 4096), "n": _log_uniform(rng, 256, 4096),
                "k": _log_uniform(rng, 256, 4096), "phi": phi}
    return {"kind": "dgemm", "m": _log_uniform(rng, 64, 12000), "n": _log_uniform(rng, 64, 12000),
            "k": _log_uniform(rng, 64, 12000), "ta": rng.random() < 0.25, "tb": rng.random() < 0.25,
            "q": rng.choice([14, 15, 16, 16, 16, 18, 20]), "phi": phi}


def _shapes(case):
    rng = np.random.default_rng(case["shapes"])
    x = np.exp(rng.uniform(math.log(64), math.log(case["hi"]), size=(case["count"], 3)))
    return [tuple(int(v) for v in row) for row in np.clip(np.rint(x), 64, case["hi"])]


def _matrix(gen, rows, cols, phi):
    x = torch.rand(rows, cols, generator=gen, device="cuda", dtype=torch.float64).sub_(0.5)
    return x.mul_(torch.randn(rows, cols, generator=gen, device="cuda", dtype=torch.float64).mul_(phi).exp_())


def _inputs(case, seed):
    """The operands alone, from the seed."""
    gen = torch.Generator(device="cuda").manual_seed(seed)
    phi = case["phi"]
    if case["kind"] in ("grouped", "batched"):
        shapes = _shapes(case)
        return [(_matrix(gen, m, k, phi), _matrix(gen, k, n, phi)) for m, n, k in shapes]
    m, n, k = case["m"], case["n"], case["k"]
    A = _matrix(gen, k, m, phi) if case.get("ta") else _matrix(gen, m, k, phi)
    B = _matrix(gen, n, k, phi) if case.get("tb") else _matrix(gen, k, n, phi)
    if case["kind"] == "autograd":
        return A, B, torch.randn(m, n, generator=gen, device="cuda", dtype=torch.float64)
    return A, B


def _outputs(shapes):
    """One buffer for the results of many products, each result on a 256-byte boundary."""
    begin, total = [], 0
    for m, n, _ in shapes:
        begin.append(total)
        total += (m * n + 31) // 32 * 32
    flat = torch.zeros(total, dtype=torch.float64, device="cuda")
    return flat, [flat[b:b + m * n].view(m, n) for b, (m, n, _) in zip(begin, shapes)]


def prepare(case, seed):
    kind = case["kind"]
    state = {"kind": kind, "case": case}
    if kind in ("grouped", "batched"):
        shapes = _shapes(case)
        pairs = _inputs(case, seed)
        As, Bs = [a for a, _ in pairs], [b for _, b in pairs]
        flat, Cs = _outputs(shapes)
        state.update(flat=flat, As=As, Bs=Bs, Cs=Cs)
        if kind == "grouped":
            state["runner"] = oz.GroupedGemm(As, Bs, Cs)
            state["runner"].capture()
        else:
            state["runner"] = oz.BatchedGemm(shapes, nstreams=case["streams"])
        return state
    m, n, k = case["m"], case["n"], case["k"]
    if kind == "autograd":
        A, B, dC = _inputs(case, seed)
        state.update(A=A.requires_grad_(), B=B.requires_grad_(), dC=dC)
        return state
    A, B = _inputs(case, seed)
    if kind == "host":
        state.update(A=A.cpu().pin_memory(), B=B.cpu().pin_memory(),
                     C=torch.zeros(m, n, dtype=torch.float64).pin_memory(),
                     runner=oz.HostGemm(oz.Plan(16, 0, k), m, n, k))
        return state
    state.update(A=A, B=B)
    if kind == "blocked":
        plan = oz.Plan(0, 53, k)
        state["ws"] = torch.empty(oz.oz_blocked_workspace_bytes(plan.handle, m, n, min(case["slab"], k)),
                                  dtype=torch.uint8, device="cuda")
    else:
        plan = oz.PlanFP(case["fmt"], k) if kind == "fp" else oz.Plan(case["q"], 0, k)
        state["ws"] = oz.workspace(plan, m, n, k)
    state["plan"] = plan
    return state


def run(state):
    kind, case = state["kind"], state["case"]
    if kind == "grouped":
        state["runner"].replay()
        return state["flat"]
    if kind == "batched":
        state["runner"].run(state["As"], state["Bs"], state["Cs"])
        return state["flat"]
    if kind == "autograd":
        C = oz.EmuMatmul.apply(state["A"], state["B"])
        dA, dB = torch.autograd.grad(C, (state["A"], state["B"]), state["dC"])
        return {"C": C.detach(), "dA": dA, "dB": dB}
    if kind == "host":
        return state["runner"](state["A"], state["B"], state["C"])
    if kind == "blocked":
        return oz.dgemm_blocked(state["A"], state["B"], state["plan"], case["slab"], ws=state["ws"])
    return oz.dgemm(state["A"], state["B"], state["plan"], trans_a=case.get("ta", False), trans_b=case.get("tb", False),
                    ws=state["ws"])


def _exact_gemms(bits, k):
    """The fewest exact 16-bit tensor-core products an emulated product of
    `bits`-bit integers needs: the result takes 2 bits + 1 + log2 k bits, and a
    plane of bf16 integers (magnitude at most 2^8, all that its significand
    holds) fixes at most 9 of them."""
    return math.ceil((2 * bits + 1 + math.log2(k)) / 9)


def _product_work(m, n, k, gemms):
    return 8 * (m * k + k * n + m * n), 2 * m * n * k * gemms


def work(case):
    kind = case["kind"]
    if kind in ("grouped", "batched"):
        parts = [_product_work(m, n, k, _exact_gemms(53, k)) for m, n, k in _shapes(case)]
        return {"bytes": sum(b for b, _ in parts), "flops": sum(f for _, f in parts)}
    m, n, k = case["m"], case["n"], case["k"]
    if kind == "autograd":
        flops = sum(2 * m * n * k * _exact_gemms(oz.Plan(16, 0, x).bits, x) for x in (k, n, m))
        return {"bytes": 8 * 2 * (m * k + k * n + m * n), "flops": flops}
    if kind == "fp":
        gemms = oz.PlanFP(case["fmt"], k).q            # the format's own configuration
    elif kind == "blocked":
        gemms = _exact_gemms(53, k)
    else:
        gemms = _exact_gemms(oz.Plan(case.get("q", 16), 0, k).bits, k)
    b, f = _product_work(m, n, k, gemms)
    return {"bytes": b, "flops": f}


def exact(case, seed):
    kind = case["kind"]
    if kind in ("grouped", "batched"):
        flat, Cs = _outputs(_shapes(case))
        for (A, B), C in zip(_inputs(case, seed), Cs):
            C.copy_(A @ B)
        return flat
    if kind == "autograd":
        A, B, dC = _inputs(case, seed)
        return {"C": A @ B, "dA": dC @ B.t(), "dB": A.t() @ dC}
    A, B = _inputs(case, seed)
    C = (A.t() if case.get("ta") else A) @ (B.t() if case.get("tb") else B)
    return C.cpu() if kind == "host" else C
