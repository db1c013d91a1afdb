"""Performance cases of the dispatch runtime: what a program does with it
through its public entry points, over the range of its configurations.

Five kinds of work, by entry point:
  trace    lk_init, lk_run_trace (closed loop, one submitter thread per
           cluster), dispose: latency-bound dispatch of many small items
  batch    lk_init, lk_submit_batch with the next batch posted while one
           runs, dispose
  serve    lk_init, lk_serve through the device queue, dispose
  finite   lk_run_finite: a fixed list of descriptors in one launch
  launch   lk_launch_noalloc: one ordinary launch per body on the caller's
           stream, without waiting

A context's CTAs hold their SMs while it runs (a device-wide synchronise
would wait for them), so a pass opens its context and disposes it, as the
steps of the repository's benchmark do.

Values follow the repository's configurations: int32 uniform on
[-2^20, 2^20], uniform bytes (or bytes of a clipped normal, as image data
has), float32 N(0,1).  Inputs are slices of pools larger than L2, so that
items read from HBM.  Outputs of different items never overlap.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2310_01212_gb300 import lk

MIB = 1 << 20
OPS = ("add", "copy", "hist", "sum", "gemm")
CODE = {"add": lk.LK_OP_ADD_I32, "copy": lk.LK_OP_COPY_I32, "hist": lk.LK_OP_HIST_U8, "sum": lk.LK_OP_SUM_F32,
        "gemm": lk.LK_OP_GEMM64_F32}
IN_BYTES = {"add": 8, "copy": 4, "hist": 1, "sum": 4, "gemm": 32768}     # per element (byte, tile)
OUT_BYTES = {"add": 4, "copy": 4, "hist": 0, "sum": 0, "gemm": 16384}
FIXED_OUT = {"add": 0, "copy": 0, "hist": 1024, "sum": 4, "gemm": 0}
FLOPS = {"add": 1, "copy": 0, "hist": 1, "sum": 1, "gemm": 2 * 64 ** 3}


def listed():
    return [
        # the small configuration: 4 SMs as 2 x 2, closed-loop adds of 4,096
        dict(name="dispatch_small_add", kind="trace", sizes="2,2", threads=256, items=4000, add=4096, hist=0, sum=0,
             gemm=0),
        # the full-chip mixed workload: 4 x 37 SMs, the four bodies in equal shares
        dict(name="dispatch_mixed", kind="trace", sizes="37,37,37,37", threads=256, items=4000, add=65536,
             hist=1 << 20, sum=65536, gemm=1),
        # a real-time loop that cannot allocate: each body once, ragged, tens of MB
        dict(name="launch_each_body", kind="launch", ctas=152, threads=256, add=3_000_001, hist=33_554_393,
             sum=7_999_999, gemm=1000),
        # the batching stream: sums and adds of 1,024 .. 16.7M elements, 4 MiB units
        dict(name="batch_stream", kind="batch", sizes="152", threads=256, posts=2, items=400, ops=2, lo=8192,
             hi=128 * MIB, part=4 * MIB),
        # small requests coalesced into batch posts: four bodies, 4 KB .. 4 MB, 256 KiB units
        dict(name="batch_coalesced", kind="batch", sizes="148", threads=256, posts=6, items=1000, ops=4, lo=4096,
             hi=4 * MIB, part=256 << 10),
        # the serving configuration at its top rate: 4 KB .. 256 MB requests through the device queue
        dict(name="serve_queue", kind="serve", sizes="37,37,37,37", threads=256, items=500, rate=200_000, lo=4096,
             hi=256 * MIB),
        # the largest streams: add, copy and sum over one cluster of every SM
        dict(name="finite_streams", kind="finite", sizes="152", per_sm=1, threads=256, ffma=False, reps=2,
             data="uniform", add=(1 << 27) + 5, copy=(1 << 27) + 3, hist=0, sum=(1 << 28) + 1, gemm=0),
        # the largest histograms
        dict(name="finite_hist", kind="finite", sizes="152", per_sm=1, threads=256, ffma=False, reps=3,
             data="uniform", add=0, copy=0, hist=(1 << 30) - 7, sum=0, gemm=0),
        # the largest GEMM lists, whole tiles (tensor cores by default)
        dict(name="finite_gemm", kind="finite", sizes="152", per_sm=1, threads=256, ffma=False, reps=2,
             data="uniform", add=0, copy=0, hist=0, sum=0, gemm=40_000),
        # the same tiles for a program that asks for bit-reproducible FFMA
        dict(name="finite_gemm_ffma", kind="finite", sizes="152", per_sm=1, threads=256, ffma=True, reps=1,
             data="uniform", add=0, copy=0, hist=0, sum=0, gemm=40_000),
        # ordinary work in between: four clusters, ragged descriptors of a few MB
        dict(name="finite_ragged", kind="finite", sizes="38,38,38,38", per_sm=1, threads=256, ffma=False, reps=12,
             data="uniform", add=700_001, copy=900_007, hist=5_000_011, sum=1_500_003, gemm=151),
        # two CTAs per SM: two clusters that each span every SM
        dict(name="finite_coresident", kind="finite", sizes="152,152", per_sm=2, threads=256, ffma=False, reps=2,
             data="uniform", add=20_000_003, copy=30_000_001, hist=200_000_003, sum=40_000_001, gemm=3001),
    ]


def _log_int(rng, lo, hi):
    return max(lo, min(hi, int(math.exp(rng.uniform(math.log(lo), math.log(hi))))))


def draw(rng):
    kind = rng.choice(("trace", "launch", "batch", "serve", "finite", "finite", "finite"))
    if kind == "trace":
        if rng.random() < 0.5:
            k = rng.randint(1, 4)
            return dict(kind=kind, sizes=",".join([str(k)] * 2), threads=256, items=rng.randint(1000, 4000),
                        add=_log_int(rng, 1024, 16384), hist=0, sum=0, gemm=0)
        s = rng.randint(16, 37)
        return dict(kind=kind, sizes=",".join([str(s)] * 4), threads=256, items=rng.randint(1000, 4000),
                    add=_log_int(rng, 16384, 131072), hist=_log_int(rng, 65536, 1 << 20),
                    sum=_log_int(rng, 16384, 131072), gemm=rng.randint(1, 3))
    if kind == "launch":
        return dict(kind=kind, ctas=rng.choice((37, 76, 152)), threads=rng.choice((128, 256, 512)),
                    add=_log_int(rng, 1 << 18, 1 << 24), hist=_log_int(rng, 1 << 20, 1 << 27),
                    sum=_log_int(rng, 1 << 18, 1 << 25), gemm=_log_int(rng, 152, 4000))
    if kind == "batch":
        if rng.random() < 0.5:
            return dict(kind=kind, sizes=str(rng.choice((148, 152))), threads=256, posts=rng.randint(1, 3),
                        items=rng.randint(100, 400), ops=2, lo=8192, hi=128 * MIB, part=4 * MIB)
        return dict(kind=kind, sizes=str(rng.randint(100, 152)), threads=256, posts=rng.randint(2, 6),
                    items=rng.randint(300, 1000), ops=4, lo=4096, hi=_log_int(rng, MIB, 4 * MIB),
                    part=256 << 10)
    if kind == "serve":
        return dict(kind=kind, sizes="37,37,37,37", threads=256, items=rng.randint(200, 500),
                    rate=rng.choice((100_000, 200_000)), lo=4096, hi=_log_int(rng, 32 * MIB, 256 * MIB))
    c = dict(kind=kind, sizes="152", per_sm=1, threads=256, ffma=False, reps=rng.randint(1, 2), data="uniform",
             add=0, copy=0, hist=0, sum=0, gemm=0)
    what = rng.choice(("stream", "hist", "gemm", "ffma", "mix", "two"))
    if what == "stream":
        c.update(add=_log_int(rng, 1 << 22, 1 << 27), copy=_log_int(rng, 1 << 22, 1 << 27),
                 sum=_log_int(rng, 1 << 22, 1 << 28))
    elif what == "hist":
        c.update(hist=_log_int(rng, 1 << 24, 1 << 30), threads=rng.choice((128, 256, 512)),
                 data=rng.choice(("uniform", "skewed")))
    elif what in ("gemm", "ffma"):
        c.update(gemm=_log_int(rng, 2000, 40_000), ffma=what == "ffma")
    else:
        c.update(reps=rng.randint(2, 12), add=_log_int(rng, 1 << 17, 1 << 21), copy=_log_int(rng, 1 << 17, 1 << 21),
                 hist=_log_int(rng, 1 << 19, 1 << 24), sum=_log_int(rng, 1 << 17, 1 << 22),
                 gemm=_log_int(rng, 16, 1000), data=rng.choice(("uniform", "skewed")))
        if what == "mix":
            k = rng.choice((1, 2, 4))
            c.update(sizes=",".join([str(152 // k)] * k))
        else:
            k = rng.choice((2, 4))
            c.update(sizes=",".join([str(304 // k)] * k), per_sm=2)
    return c


# ---- the items of a case: (op, n) each, from the case and the seed ---------
def _sizes(case):
    return [int(x) for x in case["sizes"].split(",")]


def _sized(op, nbytes):
    """Elements of an item of about `nbytes` input bytes."""
    if op == "gemm":
        return max(1, nbytes // 49152)
    return max(1, nbytes // IN_BYTES[op])


def _items(case):
    """The work list, the same for every seed: (op, n)."""
    kind = case["kind"]
    if kind in ("trace", "launch"):
        present = [op for op in OPS if case.get(op)]
        count = case["items"] if kind == "trace" else len(present)
        ops = [present[i % len(present)] for i in range(count)]
        if kind == "trace":
            ops = [ops[i] for i in np.random.RandomState(1).permutation(count)]
        return [(op, case[op]) for op in ops]
    if kind == "finite":
        # descriptors shrink a little and unevenly, so that their shares are ragged
        return [(op, max(1, case[op] - (case[op] // 50) * r // case["reps"] - r))
                for r in range(case["reps"] * len(_sizes(case)))
                for op in OPS if case[op]]
    count = case["items"] * case.get("posts", 1)
    names = ("add", "sum") if case.get("ops") == 2 else ("add", "hist", "sum", "gemm")
    r = np.random.RandomState(2)
    size = np.exp(r.uniform(math.log(case["lo"]), math.log(case["hi"]), count)).astype(np.int64)
    # as many items of each body in every post: a post splits at most 256 histograms
    return [(names[i % len(names)], int(_sized(names[i % len(names)], int(size[i])))) for i in range(count)]


def work(case):
    items = _items(case)
    return {"bytes": float(sum((IN_BYTES[op] + OUT_BYTES[op]) * n + FIXED_OUT[op] for op, n in items)),
            "flops": float(sum(FLOPS[op] * n for op, n in items))}


# ---- inputs ----------------------------------------------------------------
def _round(n, k):
    return -(-n // k) * k


def _inputs(case, seed):
    """Pools, every item's input offsets (elements of its pool) and output slot."""
    items = _items(case)
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    r = np.random.RandomState(seed & 0x7FFFFFFF)
    most = {op: max([n for o, n in items if o == op], default=0) for op in OPS}
    need = {"i32": 2 * max(most["add"], most["copy"]), "u8": most["hist"], "f32": max(most["sum"], 2 * 4096 * most["gemm"])}
    least = {"i32": 64 * MIB, "u8": 256 * MIB, "f32": 64 * MIB}      # elements: 256 MiB each, larger than L2
    size = {k: _round(max(need[k] + 4096, least[k]), 4096) if need[k] else 0 for k in need}
    pool = {"i32": torch.randint(-(1 << 20), (1 << 20) + 1, (size["i32"],), dtype=torch.int32, device="cuda", generator=g),
            "f32": torch.randn(size["f32"], device="cuda", generator=g)}
    if case.get("data") == "skewed":
        pool["u8"] = torch.empty(size["u8"], dtype=torch.uint8, device="cuda")
        for a in range(0, size["u8"], 1 << 28):
            b = min(size["u8"], a + (1 << 28))
            pool["u8"][a:b] = (torch.randn(b - a, device="cuda", generator=g) * 24 + 128).clamp_(0, 255).to(torch.uint8)
    else:
        pool["u8"] = torch.randint(0, 256, (size["u8"],), dtype=torch.uint8, device="cuda", generator=g)
    of = {"add": "i32", "copy": "i32", "hist": "u8", "sum": "f32", "gemm": "f32"}
    off0, off1, slot, used = [], [], [], dict.fromkeys(OPS, 0)
    for op, n in items:
        span = n * (4096 if op == "gemm" else 1)
        align = 16 if op == "hist" else 4
        room = (size[of[op]] - span) // align
        off0.append(int(r.randint(0, room + 1)) * align)
        off1.append(int(r.randint(0, room + 1)) * align if op in ("add", "gemm") else 0)
        slot.append(used[op])
        used[op] += 1 if op in ("hist", "sum") else _round(span, 4)
    return items, pool, of, off0, off1, slot, used


def prepare(case, seed):
    items, pool, of, off0, off1, slot, used = _inputs(case, seed)
    out = {"add": torch.zeros(used["add"], dtype=torch.int32, device="cuda"),
           "copy": torch.zeros(used["copy"], dtype=torch.int32, device="cuda"),
           "hist": torch.zeros((used["hist"], 256), dtype=torch.int32, device="cuda"),
           "sum": torch.zeros((used["sum"], 4), device="cuda"),        # one 16-byte slot each
           "gemm": torch.zeros(used["gemm"], device="cuda")}
    base = {k: t.data_ptr() for k, t in pool.items()}
    width = {"i32": 4, "u8": 1, "f32": 4}
    step = {"add": 4, "copy": 4, "hist": 1024, "sum": 16, "gemm": 4}
    op_of = [op for op, _ in items]
    in0 = [base[of[op]] + width[of[op]] * a for op, a in zip(op_of, off0)]
    in1 = [base[of[op]] + width[of[op]] * a if op in ("add", "gemm") else 0 for op, a in zip(op_of, off1)]
    dst = [out[op].data_ptr() + step[op] * s for op, s in zip(op_of, slot)]
    st = {"case": case, "pool": pool, "out": out, "sizes": _sizes(case) if "sizes" in case else None}
    kind = case["kind"]
    if kind == "trace":
        it = np.zeros(len(items), dtype=lk.TRACE_ITEM_DTYPE)
        it["cluster"] = np.arange(len(items)) % len(st["sizes"])
    elif kind == "batch":
        it = np.zeros(len(items), dtype=lk.BATCH_ITEM_DTYPE)
    elif kind == "serve":
        it = np.zeros(len(items), dtype=lk.REQUEST_DTYPE)
        gaps = np.random.RandomState(3).exponential(1e9 / case["rate"], len(items))
        it["t_arrival_ns"] = np.cumsum(gaps).astype(np.uint64)
        it["producer"] = np.arange(len(items)) % 8
        st["arena_bytes"] = lk.lk_serve_queue_state_bytes() + MIB
        st["arena"] = torch.zeros(st["arena_bytes"], dtype=torch.uint8, device="cuda")
    else:
        st["items"] = [(CODE[op], n) for op, n in items]
        st["in0"], st["in1"], st["dst"] = in0, in1, dst
        st["ins"] = [(a, b) if op in ("add", "gemm") else (a,) for op, a, b in zip(op_of, in0, in1)]
        return st
    it["op"] = [CODE[op] for op in op_of]
    it["n"] = [n for _, n in items]
    it["in0"], it["in1"], it["out"] = in0, in1, dst
    if kind == "batch":
        k = case["items"]
        st["posts"] = [it[i * k:(i + 1) * k] for i in range(case["posts"])]
    st["it"] = it
    return st


def _check(rc):
    if rc != lk.LK_OK:
        raise RuntimeError(lk.lk_strerror(rc))


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "trace":
        with lk.lk_init(state["sizes"], threads_per_cta=case["threads"]) as c:
            rc, _ = lk.lk_run_trace(c, state["it"], len(state["sizes"]), closed_loop=True, pin_cpu_base=2)
        _check(rc)
    elif kind == "batch":
        with lk.lk_init(state["sizes"], threads_per_cta=case["threads"]) as c:
            flying = []
            for post in state["posts"]:
                while (h := lk.lk_submit_batch(c, 0, post, part_bytes=case["part"])) is None:
                    _check(lk.lk_wait(c, flying.pop(0)))
                flying.append(h)
            for h in flying:
                _check(lk.lk_wait(c, h))
    elif kind == "serve":
        with lk.lk_init(state["sizes"], threads_per_cta=case["threads"]) as c:
            rc, _ = lk.lk_serve(c, state["it"], 8, 64 << 30, state["arena"], state["arena_bytes"],
                                mode=lk.LK_SERVE_QUEUE)
        _check(rc)
    elif kind == "finite":
        n = len(state["sizes"])
        lk.lk_run_finite(state["sizes"], state["items"], [i % n for i in range(len(state["items"]))],
                         in0=state["in0"], in1=state["in1"], out=state["dst"], threads_per_cta=case["threads"],
                         ctas_per_sm=case["per_sm"], flags=lk.LK_INIT_GEMM_FFMA if case["ffma"] else 0)
    else:
        stream = torch.cuda.current_stream().cuda_stream
        for (op, n), ins, dst in zip(state["items"], state["ins"], state["dst"]):
            _check(lk.lk_launch_noalloc(op, n, ins, dst, ctas=case["ctas"], threads=case["threads"], stream=stream))
    out = state["out"]
    return {"add": out["add"], "copy": out["copy"], "hist": out["hist"], "sum": out["sum"][:, 0], "gemm": out["gemm"]}


def exact(case, seed):
    """Sums and GEMM tiles in 64 bits; whole-number outputs have no error to measure."""
    items, pool, _, off0, off1, slot, used = _inputs(case, seed)
    x = pool["f32"]
    sums = torch.zeros(used["sum"], dtype=torch.float64, device="cuda")
    tiles = torch.zeros(used["gemm"], dtype=torch.float64, device="cuda")
    for (op, n), a, b, s in zip(items, off0, off1, slot):
        if op == "sum":
            sums[s] = sum(x[a + i:a + min(n, i + (1 << 26))].double().sum() for i in range(0, n, 1 << 26))
        elif op == "gemm":
            for t in range(0, n, 8192):
                k = 4096 * min(8192, n - t)
                t *= 4096
                p, q = (x[o + t:o + t + k].view(-1, 64, 64).double() for o in (a, b))
                tiles[s + t:s + t + k] = (p @ q).view(-1)
    return {"add": None, "copy": None, "hist": None, "sum": sums, "gemm": tiles}
