"""Performance cases: the calls a user of the library makes, over the sizes they make them at.

Every case runs one pass through the public binding (``paper_2605_29752_gb300.rg``) on inputs made from
a seed.  The context, the plans, the grouped-GEMM object and the server are made once per process, as a
program that serves GEMMs keeps them.  A single GEMM runs through a plan autotuned for its cell of the
128-step grid (one sweep of that cell).  Mixed traffic runs through a plan over the whole grid, whose table
is modelled in place of the minutes-long sweep of 32,768 cells.
"""
from __future__ import annotations

import random

import numpy as np
import torch

from paper_2605_29752_gb300 import rg

STEP, COUNT = 128, 32          # the plan grid: {128, 256, ..., 4096}^3
BLOCK = 128                    # FP8 scale block edge
BF16_BYTES, F32_BYTES = 2, 4


def _up(x: int, m: int) -> int:
    return (x + m - 1) // m * m


# ---------------------------------------------------------------- cases

def listed() -> list[dict]:
    return [
        # the smallest cell of the small sweep ({128..512}^3, the fixed 128x128 tile): launch latency
        {"name": "plain_128", "kind": "plain", "m": 128, "n": 128, "k": 128},
        # its largest cell but one step in K: a few tiles, still latency
        {"name": "plain_512", "kind": "plain", "m": 512, "n": 512, "k": 384},
        # an odd shape through the plan: no extent is a multiple of a tile, a K block or a vector
        {"name": "plan_ragged", "kind": "plan", "m": 1001, "n": 1095, "k": 1303},
        # few rows against a large weight matrix, as in token-by-token decoding: bytes and split-K
        {"name": "plan_skinny", "kind": "plan", "m": 72, "n": 4096, "k": 4096},
        # the middle of the landscape (the cross-tile sweep at M = K = 2048)
        {"name": "plan_mid", "kind": "plan", "m": 2048, "n": 2432, "k": 2048},
        # the landscape's last cell: tensor throughput
        {"name": "plan_large", "kind": "plan", "m": 4096, "n": 4096, "k": 4096},
        # many small and middling problems in one grouped call, each with its planned variant
        {"name": "grouped_mixed", "kind": "grouped", "count": 48, "lo": 128, "hi": 1536, "shapes": 11},
        # a burst of mixed requests to a running server, until the last result is there
        {"name": "serve_burst", "kind": "serve", "count": 24, "lo": 128, "hi": 4096, "shapes": 5},
        # operands in pinned host memory, result back in host memory: the end-to-end call
        {"name": "host_2048", "kind": "host", "m": 2048, "n": 2048, "k": 2048},
        # activations or weights to e4m3 codes and block scales
        {"name": "fp8_quantize", "kind": "quantize", "m": 4096, "n": 4096},
        # a middling FP8 cell, with odd rows: few tiles, so split-K or idle SMs
        {"name": "fp8_small", "kind": "fp8", "m": 500, "n": 1536, "k": 2048},
        # the FP8 subgrid's last cell: FP8 throughput with per-block promotion
        {"name": "fp8_large", "kind": "fp8", "m": 4096, "n": 4096, "k": 4096},
    ]


def _size(rng, lo: int, hi: int) -> int:
    """A size spread over the logarithm of [lo, hi]: half of them multiples of 128, a quarter of 8, the
    rest as they come."""
    x = int(round(lo * (hi / lo) ** rng.random()))
    x = max(lo, min(hi, x))
    r = rng.random()
    if r < 0.5 and x >= 96:
        return max(128, min(hi, int(round(x / 128)) * 128))
    return min(hi, _up(x, 8)) if r < 0.75 else x


def draw(rng) -> dict:
    kind = rng.choice(["plain", "plan", "plan", "skinny", "grouped", "serve", "host", "quantize", "fp8", "fp8"])
    if kind == "plain":
        return {"kind": "plain", "m": _size(rng, 64, 512), "n": _size(rng, 64, 512), "k": _size(rng, 64, 512)}
    if kind == "plan":
        return {"kind": "plan", "m": _size(rng, 128, 4096), "n": _size(rng, 128, 4096), "k": _size(rng, 128, 4096)}
    if kind == "skinny":
        return {"kind": "plan", "m": _size(rng, 1, 128), "n": _size(rng, 1024, 4096), "k": _size(rng, 1024, 4096)}
    if kind == "grouped":
        return {"kind": "grouped", "count": rng.randint(8, 60), "lo": 64, "hi": _size(rng, 512, 1536),
                "shapes": rng.randrange(1 << 16)}
    if kind == "serve":
        return {"kind": "serve", "count": rng.randint(4, 28), "lo": 64, "hi": _size(rng, 1024, 4096),
                "shapes": rng.randrange(1 << 16)}
    if kind == "host":
        return {"kind": "host", "m": _size(rng, 256, 3072), "n": _size(rng, 256, 3072), "k": _size(rng, 256, 3072)}
    if kind == "quantize":
        return {"kind": "quantize", "m": _size(rng, 64, 4096), "n": _size(rng, 64, 4096)}
    return {"kind": "fp8", "m": _size(rng, 128, 4096), "n": _size(rng, 256, 4096), "k": _size(rng, 256, 4096)}


def _shapes(case: dict) -> list[tuple[int, int, int]]:
    rng = random.Random(case["shapes"])
    return [tuple(_size(rng, case["lo"], case["hi"]) for _ in range(3)) for _ in range(case["count"])]


# ---------------------------------------------------------------- what a program keeps

# Modelled ns per 64-deep K block of a unit (a CTA's tile, or a pair's)
_CTA_NS = {(128, 64): 190, (128, 128): 195, (128, 192): 236, (128, 256): 255, (256, 64): 300, (256, 128): 350,
           (256, 192): 365, (256, 256): 500}
_PAIR_NS = {(256, 128): 195, (256, 192): 250, (256, 256): 250}


def _modelled_table():
    """BF16 variant ids and their modelled times (ns) over the grid: a fixed cost, waves of units, the last
    tile's store and, for split-K, the sum of the partials."""
    ax = STEP * np.arange(1, COUNT + 1, dtype=np.float64)
    m, n, k = ax.reshape(-1, 1, 1), ax.reshape(1, -1, 1), ax.reshape(1, 1, -1)
    ids, rows = [], []

    def add(variant, bm, bn, cta_rows, ns, slots, split=1):
        units, kblocks = np.ceil(m / bm) * np.ceil(n / bn), np.ceil(k / 64)
        store = cta_rows * bn * F32_BYTES / 64.0
        t = 4000.0 + np.ceil(units * split / slots) * np.ceil(kblocks / split) * ns + store
        if split > 1:
            t = np.where((units < slots) & (kblocks >= 2 * split), t + 1500.0 + 0.35 * split * store, 1e12)
        ids.append(variant)
        rows.append(np.broadcast_to(np.round(t), (COUNT,) * 3).astype(np.int64))

    for tile, (bm, bn) in enumerate(rg.TILES):
        for split in rg.SPLITS:
            add(rg.variant(tile, split), bm, bn, bm, _CTA_NS[bm, bn], 152, split)
    for tile in rg.PAIR_TILES:
        bm, bn = rg.TILES[tile]
        add(rg.variant(tile, rg.TWO_SM), bm, bn, 128, _PAIR_NS[bm, bn], 76)
    return np.stack(rows).reshape(len(ids), -1), ids


_kept: dict = {}


def _keep(name, make):
    if name not in _kept:
        _kept[name] = make()
    return _kept[name]


def _ctx():
    return _keep("ctx", lambda: rg.rg_init(0))


def _grid_plan():
    """The whole grid's plan, from the modelled table."""
    def make():
        table, ids = _modelled_table()
        return rg.rg_plan_build(rg.make_grid((STEP, STEP, COUNT)), table, ids)
    return _keep("grid plan", make)


def _cell_plan(m: int, n: int, k: int, fp8: bool = False):
    """The plan of one grid cell, autotuned over all variants."""
    m, n, k = _up(m, STEP), _up(n, STEP), _up(k, STEP)

    def make():
        grid = rg.make_grid((m, m, 1), (n, n, 1), (k, k, 1))
        opts = rg.rg_sweep_opts_default()
        opts.reps = 10
        g = _gen(0)
        c = torch.empty(m * n, device="cuda")
        if fp8:
            ids = [rg.fp8_variant(t, s) for t in range(rg.RG_FP8_NUM_TILES) for s in rg.SPLITS]
            (qa, sa), (qb, sb) = _quantized(_normal(m, k, g)), _quantized(_normal(k, n, g))
            times = rg.rg_sweep_fp8(_ctx(), grid, qa, sa, qb, sb, c, opts, variant_ids=ids)
        else:
            ids = list(range(rg.RG_NUM_VARIANTS))
            times = rg.rg_sweep(_ctx(), grid, ids, _bf16(m, k, g), _bf16(k, n, g), c, opts)
        return rg.rg_plan_build(grid, times, ids)
    return _keep(("cell plan", m, n, k, fp8), make)


def _group():
    return _keep("group", lambda: rg.rg_group_create(_ctx(), 1, 64, 256 << 20))


def _server():
    def make():
        o = rg.rg_serve_opts_default()
        o.hbm_budget_bytes = 8 << 30
        return rg.rg_serve_start(_ctx(), _grid_plan(), o)
    return _keep("server", make)


# ---------------------------------------------------------------- inputs

def _gen(seed: int) -> torch.Generator:
    return torch.Generator(device="cuda").manual_seed(seed)


def _bf16(rows: int, cols: int, g) -> torch.Tensor:
    """U[-1, 1) in BF16, in a buffer whose leading dimension is a multiple of 8 elements."""
    buf = torch.zeros((rows, _up(cols, 8)), dtype=torch.bfloat16, device="cuda")
    buf[:, :cols] = torch.rand((rows, cols), generator=g, device="cuda") * 2 - 1
    return buf[:, :cols]


def _out(rows: int, cols: int) -> torch.Tensor:
    return torch.empty((rows, _up(cols, 4)), dtype=torch.float32, device="cuda")[:, :cols]


def _operands(case, seed):
    g = _gen(seed)
    return _bf16(case["m"], case["k"], g), _bf16(case["k"], case["n"], g)


def _many(case, seed):
    g = _gen(seed)
    return [(_bf16(m, k, g), _bf16(k, n, g)) for m, n, k in _shapes(case)]


def _normal(rows: int, cols: int, g) -> torch.Tensor:
    return torch.randn((rows, cols), generator=g, device="cuda")


def _quantized(x: torch.Tensor):
    rows, cols = x.shape
    q = torch.zeros((rows, _up(cols, 16)), dtype=torch.uint8, device="cuda")
    s = torch.empty((_up(rows, BLOCK) // BLOCK, _up(cols, BLOCK) // BLOCK), device="cuda")
    rg.rg_fp8_quantize(_ctx(), x, rows, cols, cols, q, q.stride(0), s)
    return q, s


def _pinned(t: torch.Tensor) -> torch.Tensor:
    return t.contiguous().cpu().pin_memory()


def _grouped_problems(ops, outs):
    """Each problem with the variant its plan cell chose (one leaf per problem; a cell the plan splits
    runs the first leaf's variant over the whole problem)."""
    plan, items = _grid_plan(), []
    for (a, b), c in zip(ops, outs):
        (m, k), n = a.shape, b.shape[1]
        leaf = rg.rg_plan_lookup(plan, m, n, k)[0][0]
        items.append((m, n, k, a, a.stride(0), b, b.stride(0), c, c.stride(0), 0, 0, 0, 0, leaf[0]))
    return rg.group_problems(items)


def prepare(case: dict, seed: int):
    kind = case["kind"]
    if kind in ("plain", "plan"):
        a, b = _operands(case, seed)
        plan = _cell_plan(case["m"], case["n"], case["k"]) if kind == "plan" else None
        return {"kind": kind, "ctx": _ctx(), "plan": plan, "a": a, "b": b, "c": _out(case["m"], case["n"])}
    if kind == "grouped":
        ops = _many(case, seed)
        outs = [_out(a.shape[0], b.shape[1]) for a, b in ops]
        return {"kind": kind, "group": _group(), "ops": ops, "outs": outs, "problems": _grouped_problems(ops, outs)}
    if kind == "serve":
        ops = _many(case, seed)
        return {"kind": kind, "server": _server(), "ops": ops, "outs": [_out(a.shape[0], b.shape[1]) for a, b in ops]}
    if kind == "host":
        a, b = (_pinned(x) for x in _operands(case, seed))
        c = torch.empty((case["m"], case["n"]), dtype=torch.float32).pin_memory()
        return {"kind": kind, "ctx": _ctx(), "plan": _cell_plan(case["m"], case["n"], case["k"]), "a": a, "b": b, "c": c}
    if kind == "quantize":
        m, n = case["m"], case["n"]
        x = _normal(m, n, _gen(seed))
        q = torch.empty((m, n), dtype=torch.uint8, device="cuda")
        s = torch.empty((_up(m, BLOCK) // BLOCK, _up(n, BLOCK) // BLOCK), device="cuda")
        return {"kind": kind, "ctx": _ctx(), "x": x, "q": q, "s": s}
    m, n, k = case["m"], case["n"], case["k"]
    g = _gen(seed)
    qa, sa = _quantized(_normal(m, k, g))
    qb, sb = _quantized(_normal(k, n, g))
    return {"kind": kind, "ctx": _ctx(), "plan": _cell_plan(m, n, k, fp8=True), "mnk": (m, n, k), "qa": qa, "sa": sa,
            "qb": qb, "sb": sb, "c": _out(m, n)}


# ---------------------------------------------------------------- one pass

def run(s):
    kind = s["kind"]
    if kind in ("plain", "plan", "host"):
        a, b, c = s["a"], s["b"], s["c"]
        (m, k), n = a.shape, b.shape[1]
        lda, ldb, ldc = a.stride(0), b.stride(0), c.stride(0)
        if kind == "plain":
            rg.rg_gemm(s["ctx"], m, n, k, a, lda, b, ldb, c, ldc, rg.variant(1, 1))
        elif kind == "plan":
            rg.rg_gemm_plan(s["ctx"], s["plan"], m, n, k, a, lda, b, ldb, c, ldc)
        else:
            rg.rg_gemm_plan_host(s["ctx"], s["plan"], m, n, k, a, lda, b, ldb, c, ldc)
        return c
    if kind == "grouped":
        rg.rg_gemm_grouped(s["group"], s["problems"], len(s["outs"]))
        return s["outs"]
    if kind == "serve":
        ids = [rg.rg_serve_submit(s["server"], a.shape[0], b.shape[1], a.shape[1], a, a.stride(0), b, b.stride(0), c,
                                  c.stride(0)) for (a, b), c in zip(s["ops"], s["outs"])]
        for i in ids:
            if rg.rg_serve_wait(s["server"], i)["status"] != rg.RG_OK:
                raise RuntimeError("a request failed")
        return s["outs"]
    if kind == "quantize":
        (m, n), q = s["x"].shape, s["q"]
        rg.rg_fp8_quantize(s["ctx"], s["x"], m, n, s["x"].stride(0), q, q.stride(0), s["s"])
        return {"codes": q, "scales": s["s"]}
    m, n, k = s["mnk"]
    qa, sa, qb, sb, c = s["qa"], s["sa"], s["qb"], s["sb"], s["c"]
    rg.rg_gemm_fp8_plan(s["ctx"], s["plan"], m, n, k, qa, qa.stride(0), sa, sa.stride(0), qb, qb.stride(0), sb,
                        sb.stride(0), c, c.stride(0))
    return c


# ---------------------------------------------------------------- work and exact values

def _gemm_work(m, n, k, operand=BF16_BYTES):
    return operand * (m * k + k * n) + F32_BYTES * m * n, 2 * m * n * k


def work(case: dict) -> dict:
    kind = case["kind"]
    if kind in ("grouped", "serve"):
        each = [_gemm_work(*s) for s in _shapes(case)]
        return {"bytes": sum(b for b, _ in each), "flops": sum(f for _, f in each)}
    if kind == "quantize":
        m, n = case["m"], case["n"]
        blocks = _up(m, BLOCK) // BLOCK * (_up(n, BLOCK) // BLOCK)
        return {"bytes": 5 * m * n + F32_BYTES * blocks, "flops": 2 * m * n}
    m, n, k = case["m"], case["n"], case["k"]
    if kind == "fp8":
        b, f = _gemm_work(m, n, k, 1)
        blocks = _up(k, BLOCK) // BLOCK * (_up(m, BLOCK) // BLOCK + _up(n, BLOCK) // BLOCK)
        return {"bytes": b + F32_BYTES * blocks, "flops": f}
    b, f = _gemm_work(m, n, k)
    return {"bytes": b, "flops": f}


def _blocks(x: torch.Tensor) -> torch.Tensor:
    """x, zero-padded to whole scale blocks, as [block row, row, block column, column]."""
    r, c = x.shape
    x = torch.nn.functional.pad(x, (0, _up(c, BLOCK) - c, 0, _up(r, BLOCK) - r))
    return x.reshape(x.shape[0] // BLOCK, BLOCK, x.shape[1] // BLOCK, BLOCK)


def _dequantized(x: torch.Tensor) -> torch.Tensor:
    """x through e4m3 codes with one FP32 scale per 128 x 128 block, in 64 bits."""
    v = _blocks(x)
    amax = v.abs().amax(dim=(1, 3), keepdim=True)
    # a tensor divisor: a division proper, where torch turns one by a number into a product
    s = torch.where(amax > 0, amax / torch.full_like(amax, 448.0), torch.ones_like(amax))
    q = (v / s).to(torch.float8_e4m3fn).to(torch.float64) * s.to(torch.float64)
    return q.reshape(q.shape[0] * BLOCK, -1)[: x.shape[0], : x.shape[1]]


def exact(case: dict, seed: int):
    kind = case["kind"]
    if kind in ("plain", "plan", "host"):
        a, b = _operands(case, seed)
        return a.double() @ b.double()
    if kind in ("grouped", "serve"):
        return [a.double() @ b.double() for a, b in _many(case, seed)]
    if kind == "quantize":
        amax = _blocks(_normal(case["m"], case["n"], _gen(seed))).abs().amax(dim=(1, 3)).double()
        return {"codes": None, "scales": torch.where(amax > 0, amax / 448.0, torch.ones_like(amax))}
    g = _gen(seed)
    a = _dequantized(_normal(case["m"], case["k"], g))
    b = _dequantized(_normal(case["k"], case["n"], g))
    return a @ b
