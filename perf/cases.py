"""Performance cases of the streaming-load library.

Each case is one use of a public entry point on one payload: what a program
that verifies, sums or sweeps device buffers calls.  ``prepare`` makes the
payload (and, for batches, the captured graph) that such a program holds;
``run`` makes the call.  ``exact`` recomputes every result with torch in 64
bits.

A case is a flat dict:

  call     the entry point ("run", "noalloc", "enqueue", "steps", "sweep",
           "batch", "host")
  dtype    payload type: "u32", "f32", "bf16", "fp8" ("mixed": a batch whose
           buffers take the four types in turn)
  bytes    payload bytes (a multiple of 16; of each buffer for "steps", the
           batch's total for "batch")
  mech, k, cta, order, copies, stage_bytes, stages, ring, passes
           the launch configuration, as in ``config``
  steps    passes enqueued by one "steps" call
  n, lo, hi  buffers of a batch and the bounds of their sizes
"""
from __future__ import annotations

import math
import random

import numpy as np
import torch

import paper_2608_15764_gb300 as sl
from paper_2608_15764_gb300 import workloads

KIB, MIB, GIB = 1 << 10, 1 << 20, 1 << 30
ELEM = {"u32": 4, "f32": 4, "bf16": 2, "fp8": 1}
MIXED = ("u32", "f32", "bf16", "fp8")
ORDER64 = (("xor_u64", 0), ("issued_loads", 1))  # 64-bit words of a device sl_result
SWEEP_K = (1, 2, 4, 8)


def listed():
    return [
        # A synchronous integrity check of one small message with the default
        # configuration: latency only.
        dict(name="run_64k_u32", call="run", dtype="u32", bytes=64 * KIB, mech="ldg", k=2, cta=256, order="asc"),
        # A small tensor checked inside a latency-critical loop that may not
        # allocate; the last tile is ragged.
        dict(name="noalloc_1m_f32", call="noalloc", dtype="f32", bytes=MIB + 16 * 37, mech="ldg", k=4, cta=256,
             order="asc"),
        # One layer's bfloat16 weights, the benchmark's fastest bfloat16 point.
        dict(name="enqueue_48m_bf16_cpasync", call="enqueue", dtype="bf16", bytes=48 * MIB + 16 * 1237,
             mech="cpasync", k=2, copies=8, cta=256, order="dyn"),
        # FP8 weights through the TMA ring (one ring per CTA), ragged.
        dict(name="enqueue_96m_fp8_tma", call="enqueue", dtype="fp8", bytes=96 * MIB + 16 * 5, mech="tma", cta=256,
             stage_bytes=16384, stages=4, ring="cta", order="asc"),
        # The 256 MiB parity configuration with 32-byte loads.
        dict(name="enqueue_256m_u32_ldg32", call="enqueue", dtype="u32", bytes=256 * MIB, mech="ldg32", k=2, cta=256,
             order="dyn"),
        # A gigabyte of float32 parameters, the benchmark's fastest float point.
        dict(name="enqueue_1g_f32", call="enqueue", dtype="f32", bytes=GIB, mech="ldg", k=8, cta=256, order="dyn"),
        # The L2-targeted backend: a buffer below the L2 size read many times.
        dict(name="enqueue_l2_32m_u32", call="enqueue", dtype="u32", bytes=32 * MIB, mech="ldg", k=4, cta=256,
             order="asc", passes=16),
        # The benchmark's timed form: back-to-back passes over two resident
        # copies of a 4 GiB buffer.
        dict(name="steps_4g_u32", call="steps", dtype="u32", bytes=4 * GIB, mech="ldg", k=4, cta=512, order="dyn",
             steps=8),
        # One allocation of the K sweep (fixed work at every K), the paper's
        # own use: a timed launch and a warm-up per cell.
        dict(name="sweep_512m_u32", call="sweep", dtype="u32", bytes=512 * MIB, mech="ldg", cta=256, order="asc"),
        # A small model's tensors of four types in one graph launch.
        dict(name="batch_64_mixed", call="batch", dtype="mixed", bytes=16 * MIB, n=64, lo=4 * KIB, hi=MIB),
        # The batched configuration: 1,024 uneven buffers, 16 GiB.
        dict(name="batch_1024_16g_bf16", call="batch", dtype="bf16", bytes=16 * GIB, n=1024, lo=64 * KIB,
             hi=256 * MIB),
        # A payload that arrives in pinned host memory (staged copies).
        dict(name="host_64m_u32", call="host", dtype="u32", bytes=64 * MIB, mech="ldg", k=4, cta=512, order="dyn"),
    ]


def _log_bytes(rng: random.Random, lo: int, hi: int, unit: int = 16) -> int:
    return max(unit, int(math.exp(rng.uniform(math.log(lo), math.log(hi)))) // unit * unit)


def _point(rng: random.Random, dtype: str) -> dict:
    """A mechanism, its concurrency and its traversal."""
    mech = rng.choice(("ldg", "ldg", "ldg32", "cpasync", "tma"))
    if mech == "ldg":
        return dict(mech=mech, k=rng.choice((2, 3, 4, 6, 8, 12)), cta=rng.choice((128, 256, 512)),
                    order=rng.choice(("asc", "desc", "dyn", "dyn")))
    if mech == "ldg32":
        return dict(mech=mech, k=rng.choice((1, 2, 3, 4)), cta=rng.choice((128, 256, 512)),
                    order=rng.choice(("asc", "dyn")))
    if mech == "cpasync":
        k, g = rng.choice(((4, 1), (6, 1), (2, 2), (2, 4), (1, 8), (2, 8)))
        return dict(mech=mech, k=k, copies=g, cta=rng.choice((128, 256)), order=rng.choice(("asc", "dyn")))
    if rng.random() < 0.5:
        sb, st = rng.choice(((16384, 2), (16384, 4), (65536, 2)))
        return dict(mech=mech, cta=256, stage_bytes=sb, stages=st, ring="cta", order=rng.choice(("asc", "desc")))
    sb, st, cta = rng.choice(((4096, 6, 192), (4096, 8, 256), (16384, 7, 224), (16384, 6, 192)))
    return dict(mech=mech, cta=cta, stage_bytes=sb, stages=st, ring="warp", order="asc")


def draw(rng: random.Random) -> dict:
    call = rng.choice(("run", "noalloc", "enqueue", "enqueue", "enqueue", "l2", "steps", "sweep", "batch", "batch",
                       "host"))
    dtype = rng.choice(("u32", "u32", "f32", "bf16", "fp8"))
    if call == "run":
        return dict(call=call, dtype=dtype, bytes=_log_bytes(rng, KIB, 16 * MIB), **_point(rng, dtype))
    if call == "noalloc":
        return dict(call=call, dtype=dtype, bytes=_log_bytes(rng, KIB, 16 * MIB), mech="ldg",
                    k=rng.choice((1, 2, 4, 8)), cta=rng.choice((128, 256, 512)), order=rng.choice(("asc", "desc")))
    if call == "enqueue":
        return dict(call=call, dtype=dtype, bytes=_log_bytes(rng, 4 * MIB, 4 * GIB), **_point(rng, dtype))
    if call == "l2":
        return dict(call="enqueue", dtype="u32", bytes=_log_bytes(rng, 16 * MIB, 64 * MIB), mech="ldg",
                    k=rng.choice((1, 2, 4, 8)), cta=rng.choice((256, 512)), order=rng.choice(("asc", "desc")),
                    passes=rng.choice((8, 16, 32)))
    if call == "steps":
        return dict(call=call, dtype="u32", bytes=_log_bytes(rng, 64 * MIB, 4 * GIB), mech="ldg",
                    k=rng.choice((2, 4, 8)), cta=rng.choice((256, 512)), order=rng.choice(("asc", "dyn", "dyn")),
                    steps=rng.choice((4, 8)))
    if call == "sweep":
        return dict(call=call, dtype="u32", bytes=_log_bytes(rng, 64 * MIB, 2 * GIB), mech="ldg",
                    cta=rng.choice((256, 512, 1024)), order=rng.choice(("asc", "desc")))
    if call == "batch":
        n = rng.choice((16, 64, 256, 1024))
        lo = rng.choice((4 * KIB, 64 * KIB))
        hi = rng.choice((MIB, 16 * MIB, 256 * MIB))
        total = _log_bytes(rng, max(2 * n * lo, 2 * MIB), min(16 * GIB, max(4 * n * lo, n * hi // 4)), 4096)
        return dict(call=call, dtype=rng.choice(("mixed", "u32", "f32", "bf16", "fp8")), bytes=total, n=n, lo=lo,
                    hi=hi)
    return dict(call="host", dtype=dtype, bytes=_log_bytes(rng, 256 * KIB, 512 * MIB), mech="ldg",
                k=rng.choice((2, 4, 8)), cta=rng.choice((256, 512)), order=rng.choice(("asc", "dyn")))


# ---- payloads ---------------------------------------------------------------

def _payload(dtype: str, nbytes: int, gen: torch.Generator) -> torch.Tensor:
    """nbytes of payload on the GPU, as bytes: random words, or N(0,1) values
    (FP8: eight times that)."""
    if dtype == "u32":
        t = torch.empty(nbytes // 8, dtype=torch.int64, device="cuda").random_(-2 ** 63, None, generator=gen)
        return t.view(torch.uint8)
    n = nbytes // ELEM[dtype]
    if dtype != "fp8":
        t = torch.empty(n, dtype=torch.float32 if dtype == "f32" else torch.bfloat16, device="cuda")
        return t.normal_(generator=gen).view(torch.uint8)
    out = torch.empty(n, dtype=torch.uint8, device="cuda")
    for s in range(0, n, 256 * MIB):
        e = min(n, s + 256 * MIB)
        x = torch.empty(e - s, dtype=torch.float32, device="cuda").normal_(generator=gen).mul_(8.0)
        out[s:e] = x.to(torch.float8_e4m3fn).view(torch.uint8)
    return out


def _generator(seed: int) -> torch.Generator:
    return torch.Generator(device="cuda").manual_seed(seed)


def _buffers(case: dict, seed: int):
    """The payload tensors of a case, as (bytes tensor, dtype) pairs."""
    gen = _generator(seed)
    if case["call"] == "batch":
        sizes = workloads.batch_sizes(case["n"], case["bytes"], case["lo"], case["hi"])
        kinds = [case["dtype"] if case["dtype"] != "mixed" else MIXED[i % 4] for i in range(case["n"])]
        if case["dtype"] != "mixed":  # one arena, buffers back to back
            arena, bufs, off = _payload(case["dtype"], case["bytes"], gen), [], 0
            for s in sizes:
                bufs.append(arena[off:off + s])
                off += s
        else:
            bufs = [_payload(k, s, gen) for k, s in zip(kinds, sizes)]
        return list(zip(bufs, kinds))
    count = 2 if case["call"] == "steps" else 1
    return [(_payload(case["dtype"], case["bytes"], gen), case["dtype"]) for _ in range(count)]


def _config(case: dict, **over):
    kw = {k: case[k] for k in ("k", "cta", "order", "copies", "stage_bytes", "stages", "ring", "passes") if k in case}
    kw.update(over)
    return sl.config(case["mech"], **kw)


def _table():
    """A tuning table as the autotuner writes it for this range of sizes."""
    return [sl.tune_entry(0, MIB - 1, sl.config("ldg", k=8, cta=256)),
            sl.tune_entry(MIB, 16 * MIB - 1, sl.config("ldg", k=8, cta=128)),
            sl.tune_entry(16 * MIB, 1 << 62, sl.config("tma", cta=256, stage_bytes=16384, stages=2))]


def prepare(case: dict, seed: int) -> dict:
    bufs = _buffers(case, seed)
    call = case["call"]
    st = {"case": case, "bufs": [b for b, _ in bufs]}
    if call == "batch":
        st["batch"] = sl.sl_batch_create([(b, b.numel(), dt) for b, dt in bufs], _table())
    elif call == "sweep":
        st["cells"] = [_config(case, k=k) for k in SWEEP_K]
    else:
        st["cfg"] = _config(case)
    if call == "host":
        st["bufs"] = [bufs[0][0].cpu().pin_memory()]
    if call in ("noalloc", "enqueue", "steps"):
        n = case.get("steps", 1)
        st["out"] = torch.zeros(n * sl.RESULT_BYTES, dtype=torch.uint8, device="cuda")
        w = st["out"].view(torch.int64).view(n, sl.RESULT_BYTES // 8)
        st["views"] = {name: w[:, i] for name, i in ORDER64}
        st["views"]["fsum"] = w.view(torch.float64)[:, 4]
        st["views"]["sum_u32"] = st["out"].view(torch.int32).view(n, sl.RESULT_BYTES // 4)[:, 12]
    torch.cuda.synchronize()
    return st


# ---- the call -----------------------------------------------------------------

_FIELDS = np.dtype({"names": ["xor_u64", "issued_loads", "fsum", "sum_u32"],
                    "formats": ["<i8", "<i8", "<f8", "<i4"], "offsets": [0, 8, 32, 48], "itemsize": sl.RESULT_BYTES})


def _host_results(results) -> dict:
    a = np.frombuffer(b"".join(results), dtype=_FIELDS)
    return {name: a[name] for name in _FIELDS.names}


def run(state: dict):
    case, call = state["case"], state["case"]["call"]
    buf = state["bufs"][0]
    if call == "run":
        return _host_results([sl.sl_run(buf, dtype=case["dtype"], cfg=state["cfg"])])
    if call == "host":
        return _host_results([sl.sl_run_host(buf, dtype=case["dtype"], cfg=state["cfg"])])
    if call == "sweep":
        rows = sl.sl_sweep(buf, state["cells"], dtype=sl.SL_U32, repeats=1, warmup=1)
        return _host_results([r[0] for r in rows])
    if call == "batch":
        return _host_results(sl.sl_batch_run(state["batch"])[0])
    if call == "steps":
        sl.sl_enqueue_steps(state["bufs"], state["out"], case["steps"], dtype=case["dtype"], cfg=state["cfg"])
    elif call == "noalloc":
        sl.sl_run_noalloc(buf, state["out"], dtype=case["dtype"], cfg=state["cfg"])
    else:
        sl.sl_enqueue(buf, state["out"], dtype=case["dtype"], cfg=state["cfg"])
    return state["views"]


def work(case: dict) -> dict:
    """Bytes read once per call (a buffer read in several passes, steps or
    cells is read that often) plus the results; operations: one addition per
    element."""
    reps = {"steps": case.get("steps", 1), "sweep": 2 * len(SWEEP_K)}.get(case["call"], case.get("passes", 1))
    outs = {"steps": case.get("steps", 1), "sweep": len(SWEEP_K), "batch": case.get("n", 1)}.get(case["call"], 1)
    elem = ELEM.get(case["dtype"], 4)
    return {"bytes": case["bytes"] * reps + outs * sl.RESULT_BYTES, "flops": case["bytes"] * reps / elem}


# ---- the same results in 64 bits ----------------------------------------------

def _xor(x: torch.Tensor) -> int:
    while x.numel() > 1:
        h = x.numel() // 2
        y = x[:h] ^ x[h:2 * h]
        if x.numel() & 1:
            y[0] ^= x[-1]
        x = y
    return int(x.item()) if x.numel() else 0


def _signed32(v: int) -> int:
    v &= 0xFFFFFFFF
    return v - (1 << 32) if v >> 31 else v


def _exact_one(t: torch.Tensor, dtype: str, passes: int, width: int):
    words = int(t.view(torch.int32).sum(dtype=torch.int64).item())
    f = 0.0
    if dtype == "fp8":
        for s in range(0, t.numel(), 256 * MIB):
            f += float(t[s:s + 256 * MIB].view(torch.float8_e4m3fn).to(torch.float32).sum(dtype=torch.float64).item())
    elif dtype != "u32":
        v = t.view(torch.float32 if dtype == "f32" else torch.bfloat16)
        f = float(v.sum(dtype=torch.float64).item())
    return (_xor(t.view(torch.int64)) if passes & 1 else 0, passes * (-(-t.numel() // width)), f * passes,
            _signed32(words * passes))


def exact(case: dict, seed: int):
    width = 32 if case.get("mech") == "ldg32" else 16
    rows = [_exact_one(b, dt, case.get("passes", 1), width) for b, dt in _buffers(case, seed)]
    reps = {"steps": case.get("steps", 1), "sweep": len(SWEEP_K)}.get(case["call"], len(rows))
    rows = [rows[i % len(rows)] for i in range(reps)]
    cols = list(zip(*rows))
    return {"xor_u64": np.array(cols[0], dtype=np.int64), "issued_loads": np.array(cols[1], dtype=np.int64),
            "fsum": np.array(cols[2], dtype=np.float64), "sum_u32": np.array(cols[3], dtype=np.int32)}
