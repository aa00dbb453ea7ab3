"""The work that programs give this library, as cases to be timed.

A case is a set of GEMMs with its inputs on the device, planned once, and
handed over in one of the ways that include/goldy.h offers:

* ``exec``   a prepared run (``goldy_exec_create`` once, ``goldy_exec_launch``
             per pass), the way a serving or training loop repeats a step;
* ``run``    ``goldy_run`` on each pass: pointers marshalled, tensor maps
             encoded and kernels launched every time, the way a program whose
             buffers change calls the library;
* ``graph``  a CUDA graph captured once, launched per pass;
* ``noalloc`` one GEMM of a caller that may not allocate device memory;
* ``corun``  a GEMM next to an element-wise add (``goldy_corun_run``).

The sizes are those of this repository's benchmark configurations and of the
ranges its randomized, batched and co-run sets are drawn from (M in
[16, 4096]; N and K in [256, 8192]; 2 to 16 GEMMs per set; sequences of 128
to 2048 with 16 or 32 heads of dimension 128).  All passes go out on one set
of streams, the first of which is the program's own.
"""
from __future__ import annotations

import math
import random

import torch

from paper_2409_02227_gb300 import goldy as G

# Drawn cases do at most three quarters of the largest listed one's arithmetic
# (two GEMMs of 4096 x 8192 x 8192): they cost no more than it does.
_MAX_FLOPS = 3 * 4096 * 8192 * 8192


def listed():
    return [
        # The smallest call: two small GEMMs of an idle program, planned once
        # and called with goldy_run; launch and host time count.
        {"name": "pair_256", "family": "equal", "n": 2, "M": 256, "N": 256, "K": 512,
         "out": "f32", "entry": "run", "ready": False, "layers": 1},
        # Gate GEMMs of a recurrent network at small batch, four cells one
        # after another: weights stream from memory, and the state that each
        # step reads was written by the step before (inputs not ready).
        {"name": "lstm_gates", "family": "equal", "n": 8, "M": 32, "N": 4096, "K": 1024,
         "out": "f32", "entry": "exec", "ready": False, "layers": 4},
        # Tensor-sliced feed-forward layers at low batch, four layers.
        {"name": "ffn_slices", "family": "equal", "n": 4, "M": 128, "N": 1024, "K": 4096,
         "out": "bf16", "entry": "exec", "ready": True, "layers": 4},
        # Two models on one GPU, a large GEMM among small ones: bench.py's set.
        {"name": "hetero_pair", "family": "two", "n": 1, "M": 2048, "N": 8192, "K": 2048,
         "n2": 3, "M2": 512, "N2": 1024, "K2": 1024, "out": "f32", "entry": "exec", "ready": True, "layers": 1},
        # Low-batch GEMMs of many models at once: ragged M, mostly bound by memory.
        {"name": "mixed_low_batch", "family": "mixed", "n": 9, "m_max": 512, "nk_max": 8192, "shapes": 1,
         "out": "f32", "entry": "exec", "ready": True, "layers": 1},
        # Many GEMMs of every size, from a few rows to full training batches.
        {"name": "mixed_all", "family": "mixed", "n": 14, "m_max": 4096, "nk_max": 8192, "shapes": 2,
         "out": "f32", "entry": "exec", "ready": True, "layers": 1},
        # A mixed set of medium GEMMs whose buffers change from call to call
        # (goldy_run each time, after the kernels that wrote its inputs).
        {"name": "mixed_medium", "family": "mixed", "n": 6, "m_max": 2048, "nk_max": 4096, "shapes": 3,
         "out": "bf16", "entry": "run", "ready": False, "layers": 1},
        # Attention over sequences of different lengths: scores (Q K^T) and
        # outputs (P V) of four requests as strided-batched GEMMs.
        {"name": "attention", "family": "attention", "n": 4, "l_max": 2048, "shapes": 3,
         "out": "bf16", "entry": "exec", "ready": False, "layers": 1},
        # A GEMM next to an element-wise add over its output's size.
        {"name": "gemm_and_add", "family": "corun", "n": 1, "M": 1024, "N": 4096, "K": 1024,
         "out": "bf16", "entry": "corun", "ready": False, "layers": 1},
        # One GEMM of odd sizes (rows padded to 16 bytes) for a caller that
        # cannot allocate.
        {"name": "odd_noalloc", "family": "odd", "n": 1, "M": 777, "N": 1501, "K": 1003,
         "out": "f32", "entry": "noalloc", "ready": False, "layers": 1},
        # Odd sizes in a set, called with goldy_run.
        {"name": "odd_set", "family": "odd", "n": 5, "M": 333, "N": 2051, "K": 1499,
         "out": "bf16", "entry": "run", "ready": False, "layers": 1},
        # The largest: two training-size GEMMs on the CD streams, captured in a graph.
        {"name": "large_graph", "family": "equal", "n": 2, "M": 4096, "N": 8192, "K": 8192,
         "out": "bf16", "entry": "graph", "ready": False, "layers": 1},
    ]


def _log_uniform(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def draw(rng):
    while True:
        case = _draw(rng)
        if work(case)["flops"] <= _MAX_FLOPS:
            return case


def _draw(rng):
    family = rng.choice(["equal", "two", "mixed", "mixed", "mixed", "attention", "corun", "odd"])
    case = {"family": family, "n": 1, "out": rng.choice(["f32", "bf16"]), "entry": "exec",
            "ready": rng.random() < 0.5, "layers": 1}
    if family in ("equal", "two", "corun"):
        case["M"] = int(round(_log_uniform(rng, 16, 4096)))
        case["N"] = 64 * int(round(_log_uniform(rng, 256, 8192) / 64))
        case["K"] = 64 * int(round(_log_uniform(rng, 256, 8192) / 64))
    if family == "equal":
        case["n"] = rng.choice([2, 3, 4, 8])
        case["entry"] = rng.choice(["exec", "exec", "run", "graph"])
        case["layers"] = rng.choice([1, 4]) if case["entry"] == "exec" else 1
    elif family == "two":
        case["n2"] = rng.randint(1, 4)
        case["M2"] = int(round(_log_uniform(rng, 16, 1024)))
        case["N2"] = 64 * int(round(_log_uniform(rng, 256, 2048) / 64))
        case["K2"] = 64 * int(round(_log_uniform(rng, 256, 2048) / 64))
    elif family == "mixed":
        case["n"] = rng.randint(3, 16)
        case["m_max"] = rng.choice([512, 2048, 4096])
        case["nk_max"] = rng.choice([4096, 8192])
        case["shapes"] = rng.randrange(1 << 20)
        case["entry"] = rng.choice(["exec", "exec", "run"])
    elif family == "attention":
        case["n"] = rng.choice([2, 4])
        case["l_max"] = rng.choice([512, 1024, 2048])
        case["shapes"] = rng.randrange(1 << 20)
    elif family == "corun":
        case["entry"] = "corun"
    else:
        case["n"] = rng.choice([1, 2, 3, 5])
        case["M"] = int(round(_log_uniform(rng, 17, 2047))) | 1
        case["N"] = int(round(_log_uniform(rng, 257, 4095))) | 1
        case["K"] = int(round(_log_uniform(rng, 257, 4095))) | 1
        case["entry"] = "noalloc" if case["n"] == 1 else "run"
    if case["entry"] in ("run", "graph", "noalloc", "corun"):
        case["ready"] = False
    return case


def _shapes(case):
    """(M, N, K, batch) of the case's GEMMs."""
    n, family = case["n"], case["family"]
    if family in ("equal", "corun"):
        return [(case["M"], case["N"], case["K"], 1)] * n
    if family == "two":
        return [(case["M2"], case["N2"], case["K2"], 1)] * case["n2"] + [(case["M"], case["N"], case["K"], 1)] * n
    if family == "odd":
        return [(case["M"] + 16 * i, max(257, case["N"] - 128 * i), case["K"] + 2 * i, 1) for i in range(n)]
    rng = random.Random(case["shapes"])
    if family == "mixed":
        return [(int(round(_log_uniform(rng, 16, case["m_max"]))),
                 64 * int(round(_log_uniform(rng, 256, case["nk_max"]) / 64)),
                 64 * int(round(_log_uniform(rng, 256, case["nk_max"]) / 64)), 1) for _ in range(n)]
    lengths = [l for l in (128, 256, 512, 1024, 2048) if l <= case["l_max"]]
    out = []
    for i in range(n):
        L, heads = rng.choice(lengths), rng.choice([16, 32])
        out.append((L, L, 128, heads) if i % 2 == 0 else (L, 128, L, heads))
    return out


def _pad8(x):
    return (x + 7) // 8 * 8


def _inputs(case, seed):
    """Per layer and GEMM, A and B on the GPU with rows padded to 16 bytes:
    activations N(0, 1), weights N(0, 1 / sqrt(K)), bf16; and the operands of
    the add, if the case has one."""
    gen = torch.Generator(device="cuda")
    gen.manual_seed(int(seed))

    def normal(batch, rows, cols, scale):
        x = torch.randn((batch, rows, _pad8(cols)), generator=gen, device="cuda", dtype=torch.float32)
        return (x * scale).to(torch.bfloat16)

    ab = [[(normal(b, M, K, 1.0), normal(b, K, N, 1.0 / math.sqrt(K))) for M, N, K, b in _shapes(case)]
          for _ in range(case["layers"])]
    xy = None
    if case["family"] == "corun":
        dt = torch.bfloat16 if case["out"] == "bf16" else torch.float32
        xy = [torch.randn((case["M"], case["N"]), generator=gen, device="cuda").to(dt) for _ in range(2)]
    return ab, xy


_streams = []          # the program's streams, the first one its own
_tables = {}           # lookup table and predictor, loaded once per program


def _program():
    if not _streams:
        _streams.extend(torch.cuda.Stream() for _ in range(G.GOLDY_MAX_STREAMS))
        _tables["lut"] = G.goldy_lut_load()
    return [s.cuda_stream for s in _streams], _tables["lut"]


def _descs(case):
    dt = G.GOLDY_BF16 if case["out"] == "bf16" else G.GOLDY_F32
    return [G.desc(M, N, K, dt, lda=_pad8(K), ldb=_pad8(N), ldc=N, batch=b) for M, N, K, b in _shapes(case)]


def prepare(case, seed):
    streams, lut = _program()
    ab, xy = _inputs(case, seed)
    out = torch.bfloat16 if case["out"] == "bf16" else torch.float32
    shapes = _shapes(case)
    C = [[torch.empty((M, N) if b == 1 else (b, M, N), dtype=out, device="cuda") for M, N, K, b in shapes]
         for _ in ab]
    descs = _descs(case)
    state = {"entry": case["entry"], "C": C, "keep": (ab, xy), "descs": descs}
    ptrs = [([a.data_ptr() for a, _ in layer], [b.data_ptr() for _, b in layer], [c.data_ptr() for c in cs])
            for layer, cs in zip(ab, C)]
    state["ptrs"] = ptrs
    if case["entry"] == "noalloc":
        # the table's kernel for a GEMM that runs alone
        _, variants = G.goldy_lut_lookup(lut, descs[0])
        state["variant"], state["streams"] = variants[0], streams[:1]
    elif case["entry"] == "corun":
        plan = G.goldy_corun_plan(descs[0], case["M"] * case["N"], G.GOLDY_BF16 if case["out"] == "bf16" else G.GOLDY_F32,
                                  lut)
        concurrent, _, _, ws_bytes = G.goldy_corun_query(plan)
        ws = torch.zeros(max(ws_bytes, 256), dtype=torch.uint8, device="cuda")
        Z = torch.empty_like(xy[0])
        state.update(plan=plan, ws=ws, ws_bytes=ws_bytes, Z=Z, xyz=(xy[0].data_ptr(), xy[1].data_ptr(), Z.data_ptr()),
                     streams=streams[:2 if concurrent else 1])
    else:
        fused = 0 if case["entry"] == "graph" else G.GOLDY_PLAN_FUSED
        plan = G.goldy_plan(descs, lut, G.GOLDY_PLAN_AUTO | fused)
        _, _, n_streams, ws_bytes = G.goldy_schedule_query(plan)
        ws = torch.zeros(max(ws_bytes, 256), dtype=torch.uint8, device="cuda")
        state.update(plan=plan, ws=ws, ws_bytes=ws_bytes, streams=streams[:n_streams])
        # inputs and workspace are complete before anything of the library is enqueued
        torch.cuda.synchronize()
        if case["entry"] == "exec":
            state["execs"] = [G.goldy_exec_create(plan, A, B, Cp, ws.data_ptr(), ws_bytes, state["streams"],
                                                  inputs_ready=bool(case["ready"])) for A, B, Cp in ptrs]
        elif case["entry"] == "graph":
            state["graph"] = G.goldy_graph_create(plan, *ptrs[0], ws.data_ptr(), ws_bytes, state["streams"])
    torch.cuda.synchronize()
    return state


def run(state):
    entry = state["entry"]
    if entry == "exec":
        for e in state["execs"]:
            G.goldy_exec_launch(e)
    elif entry == "run":
        for A, B, C in state["ptrs"]:
            G.goldy_run(state["plan"], A, B, C, state["ws"].data_ptr(), state["ws_bytes"], state["streams"])
    elif entry == "graph":
        G.goldy_graph_launch(state["graph"], state["streams"][0])
    elif entry == "noalloc":
        A, B, C = state["ptrs"][0]
        G.goldy_gemm_noalloc(state["descs"][0], state["variant"], A[0], B[0], C[0], state["streams"][0])
    else:
        A, B, C = state["ptrs"][0]
        G.goldy_corun_run(state["plan"], A[0], B[0], C[0], state["ws"].data_ptr(), state["ws_bytes"], *state["xyz"],
                          state["streams"])
        return [state["C"], state["Z"]]
    return [state["C"]]


def work(case):
    s = 2 if case["out"] == "bf16" else 4
    nbytes = flops = 0
    for M, N, K, b in _shapes(case):
        flops += 2 * b * M * N * K
        nbytes += b * (2 * M * K + 2 * K * N + s * M * N)
    if case["family"] == "corun":
        flops += case["M"] * case["N"]
        nbytes += 3 * s * case["M"] * case["N"]
    return {"bytes": case["layers"] * nbytes, "flops": case["layers"] * flops}


def exact(case, seed):
    ab, xy = _inputs(case, seed)
    C = []
    for layer in ab:
        row = []
        for (a, b), (M, N, K, batch) in zip(layer, _shapes(case)):
            c = torch.matmul(a[:, :, :K].double(), b[:, :, :N].double())
            row.append(c[0] if batch == 1 else c)
        C.append(row)
    if xy is not None:
        return [C, xy[0].double() + xy[1].double()]
    return [C]
