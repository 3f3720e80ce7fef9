"""Performance cases of the GPU manager and of its task kernels.

A case is a dict of plain values. ``prepare`` makes what a program has in hand
before the call (operands on the device or in page-locked host memory, the
manager with its ranks attached, the task arrays), ``run`` is one pass through
the public entry points and returns the results whole, ``exact`` gives the same
results in binary64 by plain torch, ``work`` the bytes and operations that a
pass cannot do without.

Kinds:

``step``   SPMD steps through a barrier-mode manager with operands resident on
           the device: every rank submits its batch, the request barrier
           opens, every rank collects its batch. ``driver`` is "calls" (one
           thread makes the calls itself) or "threads" (``Manager.spmd_run``,
           one native thread per rank, ``steps`` steps on the same buffers, as
           an iterative SPMD program runs).
``host``   the same with page-locked host buffers, two steps in flight per rank
           (``Manager.spmd_run_overlapped``), copies in and out included.
``sgemm``, ``vadd``, ``vmul``  one task's kernel alone on device buffers.

Batches (``mix``): "vadd" and "sgemm" (equal tasks), "grouped" (SGEMMs with m,
n, k independent multiples of 64 in 128 .. 2048), "serving" (half vector adds
of 2^16 .. 2^24 elements, half square SGEMMs of 256 .. 2048), "stress" (70%
vector adds, 30% square SGEMMs, lognormal sizes, so mostly odd). Their sizes
follow from ``recipe``; operands follow from the seed.
"""
import math
import random

import torch

import paper_1511_07658_gb300 as g

VADD, SGEMM = g.GVM_TASK_VADD, g.GVM_TASK_SGEMM


def listed():
    return [
        # 4 ranks x 8 vector adds of 65536 floats, one step by plain calls: the
        # smallest use of the manager, all latency.
        {"name": "step_vadd_4x8_64k", "kind": "step", "driver": "calls", "mix": "vadd", "ranks": 4, "per_rank": 8,
         "n": 65536, "path": "split3", "steps": 1, "recipe": 0},
        # Input/output-bound ranks whose vector adds fill HBM.
        {"name": "step_vadd_16x4_4m", "kind": "step", "driver": "threads", "mix": "vadd", "ranks": 16, "per_rank": 4,
         "n": 1 << 22, "path": "split3", "steps": 4, "recipe": 0},
        # The headline workload: 16 ranks x 64 SGEMM 512^3 on the default path.
        {"name": "step_sgemm512_16x64", "kind": "step", "driver": "threads", "mix": "sgemm", "ranks": 16,
         "per_rank": 64, "m": 512, "n": 512, "k": 512, "path": "split3", "steps": 4, "recipe": 0},
        # The same tasks in plain FP32 arithmetic (the plain form's path).
        {"name": "step_sgemm512_fma_16x16", "kind": "step", "driver": "threads", "mix": "sgemm", "ranks": 16,
         "per_rank": 16, "m": 512, "n": 512, "k": 512, "path": "fma", "steps": 2, "recipe": 0},
        # Batched mixed shapes in one launch, in the tile form tuned for them.
        {"name": "step_grouped_16x24", "kind": "step", "driver": "threads", "mix": "grouped", "ranks": 16,
         "per_rank": 24, "path": "split3_wide", "steps": 2, "recipe": 11},
        # Uneven ranks: vector adds and SGEMMs of odd sizes side by side.
        {"name": "step_stress_16x12", "kind": "step", "driver": "threads", "mix": "stress", "ranks": 16,
         "per_rank": 12, "path": "split3", "steps": 2, "recipe": 5},
        # End to end from and to host memory, two steps in flight.
        {"name": "host_sgemm512_16x4", "kind": "host", "mix": "sgemm", "ranks": 16, "per_rank": 4, "m": 512, "n": 512,
         "k": 512, "path": "split3", "steps": 4, "recipe": 0},
        # One task's kernel alone: a small product, the 2048^2 one (the paper's
        # MM), a ragged one with odd row lengths.
        {"name": "sgemm_512", "kind": "sgemm", "m": 512, "n": 512, "k": 512, "path": "split3"},
        {"name": "sgemm_2048", "kind": "sgemm", "m": 2048, "n": 2048, "k": 2048, "path": "split3"},
        {"name": "sgemm_1530x1027x2001", "kind": "sgemm", "m": 1530, "n": 1027, "k": 2001, "path": "split3"},
        # The paper's VecMul (16M floats, 15 products) and VecAdd (50M floats).
        {"name": "vmul_16m", "kind": "vmul", "n": 1 << 24, "iters": 15},
        {"name": "vadd_50m", "kind": "vadd", "n": 50_000_000},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _ragged(rng, v):
    """Half of the sizes as multiples of 64, half as they come."""
    return max(64, v // 64 * 64) if rng.random() < 0.5 else v


def draw(rng):
    kind = rng.choice(["step", "step", "step", "step", "sgemm", "sgemm", "sgemm", "vec", "host"])
    if kind == "vec":
        n = _log_int(rng, 1 << 16, 1 << 26)
        return {"kind": "vadd", "n": n} if rng.random() < 0.5 else {"kind": "vmul", "n": n, "iters": rng.randint(1, 24)}
    if kind == "sgemm":
        path = rng.choice(["split3", "split3", "split3_fused", "split3_wide", "fma"])
        hi = 2048 if path == "fma" else 4096
        m, n, k = (_ragged(rng, _log_int(rng, 64, hi)) for _ in range(3))
        return {"kind": "sgemm", "m": m, "n": n, "k": k, "path": path}
    if kind == "host":
        m, n, k = (_ragged(rng, _log_int(rng, 128, 768)) for _ in range(3))
        return {"kind": "host", "mix": "sgemm", "ranks": rng.choice([4, 8, 16]), "per_rank": rng.randint(2, 6),
                "m": m, "n": n, "k": k, "path": "split3", "steps": 4, "recipe": 0}
    c = {"kind": "step", "driver": rng.choice(["calls", "threads", "threads"]),
         "mix": rng.choice(["vadd", "sgemm", "sgemm", "grouped", "serving", "stress"]), "ranks": rng.choice([4, 8, 16]),
         "per_rank": rng.randint(4, 24), "path": rng.choice(["split3", "split3", "split3_wide"]), "steps": 2,
         "recipe": rng.randrange(1 << 20)}
    if c["mix"] == "vadd":
        c["n"] = _log_int(rng, 1 << 14, min(1 << 22, (1 << 28) // (c["ranks"] * c["per_rank"])))
    elif c["mix"] == "sgemm":
        c["m"], c["n"], c["k"] = (_ragged(rng, _log_int(rng, 64, 1024)) for _ in range(3))
        if rng.random() < 0.2:
            c["path"] = "fma"
    else:
        c["per_rank"] = rng.randint(4, 8)
    return c


def _batches(case):
    """Per rank, its tasks in order: (type, m, n, k) with n the length of a vector add."""
    R, P, mix = case["ranks"], case["per_rank"], case["mix"]
    rng = random.Random(case["recipe"])
    out = []
    for _ in range(R):
        tasks = []
        for _ in range(P):
            if mix == "vadd":
                tasks.append((VADD, 0, case["n"], 0))
            elif mix == "sgemm":
                tasks.append((SGEMM, case["m"], case["n"], case["k"]))
            elif mix == "grouped":
                tasks.append((SGEMM, *(64 * rng.randint(2, 32) for _ in range(3))))
            elif mix == "serving":
                if rng.random() < 0.5:
                    tasks.append((VADD, 0, int(2.0 ** rng.uniform(16, 24)), 0))
                else:
                    s = rng.choice([256, 512, 1024, 2048])
                    tasks.append((SGEMM, s, s, s))
            elif rng.random() < 0.7:
                tasks.append((VADD, 0, min(max(round(2.0 ** 20 * math.exp(1.5 * rng.gauss(0, 1))), 1 << 10), 1 << 24), 0))
            else:
                s = min(max(round(768 * math.exp(0.7 * rng.gauss(0, 1))), 64), 2560)
                tasks.append((SGEMM, s, s, s))
        out.append(tasks)
    return out


def _sizes(t):
    """Elements of a task's a, b and c."""
    typ, m, n, k = t
    return (n, n, n) if typ == VADD else (m * k, k * n, m * n)


def _pad(n):
    return (n + 63) // 64 * 64  # operands start on 256-byte boundaries


def _layout(tasks):
    """Offsets (elements) of a batch's operands in one block, inputs first, and the offset where outputs begin."""
    at, offs = 0, []
    for t in tasks:
        a, b, _ = _sizes(t)
        offs.append([at, at + _pad(a)])
        at += _pad(a) + _pad(b)
    first = at
    for o, t in zip(offs, tasks):
        o.append(at)
        at += _pad(_sizes(t)[2])
    return offs, first, at


def _fill_inputs(block, tasks, offs, gen):
    """Standard-normal matrices, uniform [-1, 1) vectors."""
    for t, (oa, ob, _) in zip(tasks, offs):
        a, b, _ = _sizes(t)
        for o, n in ((oa, a), (ob, b)):
            if t[0] == VADD:
                block[o:o + n].uniform_(-1.0, 1.0, generator=gen)
            else:
                block[o:o + n].normal_(generator=gen)


def _generator(seed):
    return torch.Generator(device="cuda").manual_seed(seed * 7919 + 17)


def _pow2(n):
    return 1 << max(1, (n - 1).bit_length())


class _State:
    """What a program keeps; its manager stops with it."""

    def __init__(self, case):
        self.case = case
        self.mgr = None

    def __del__(self):
        if self.mgr is not None:
            self.mgr.shutdown()


def _task(t):
    x = g.GvmTask()
    x.type, x.m, x.n, x.k = t
    return x


def _prepare_step(case, seed):
    batches = _batches(case)
    layouts = [_layout(t) for t in batches]
    resident = max(4 * size for _, _, size in layouts)
    s = _State(case)
    s.mgr = g.Manager(case["ranks"], ring_depth=_pow2(case["per_rank"]), mode="barrier", sgemm_path=case["path"],
                      slice_bytes=(resident + (1 << 20)) // 256 * 256, resident_bytes=resident)
    s.ranks = [s.mgr.attach(r) for r in range(case["ranks"])]
    s.arrays, s.out = [], []
    gen = _generator(seed)
    for rank, tasks, (offs, first, size) in zip(s.ranks, batches, layouts):
        block = rank.resident_view(0, (size,))
        _fill_inputs(block, tasks, offs, gen)
        block[first:].zero_()
        arr = (g.GvmTask * len(tasks))()
        for i, (t, (oa, ob, oc)) in enumerate(zip(tasks, offs)):
            arr[i] = _task(t)
            arr[i].flags = g.GVM_TASK_RESIDENT
            arr[i].a_off, arr[i].b_off, arr[i].c_off = 4 * oa, 4 * ob, 4 * oc
        s.arrays.append(arr)
        s.out.append(block[first:])
    return s


def _prepare_host(case, seed):
    batches = _batches(case)
    layouts = [_layout(t) for t in batches]
    staging = max(4 * size for _, _, size in layouts)
    s = _State(case)
    s.mgr = g.Manager(case["ranks"], ring_depth=_pow2(2 * case["per_rank"]), mode="barrier", sgemm_path=case["path"],
                      slice_bytes=2 * staging + (1 << 20))
    s.ranks = [s.mgr.attach(r) for r in range(case["ranks"])]
    s.even, s.odd, s.keep, s.out = [], [], [], []
    gen = _generator(seed)
    for tasks, (offs, first, size) in zip(batches, layouts):
        dev = torch.empty(first, device="cuda")
        _fill_inputs(dev, tasks, offs, gen)
        inp = torch.zeros(first, pin_memory=True)
        inp.copy_(dev)
        outs = [torch.zeros(size - first, pin_memory=True) for _ in range(2)]
        for arrays, out in ((s.even, outs[0]), (s.odd, outs[1])):
            arr = (g.GvmTask * len(tasks))()
            for i, (t, (oa, ob, oc)) in enumerate(zip(tasks, offs)):
                arr[i] = _task(t)
                arr[i].a, arr[i].b = inp.data_ptr() + 4 * oa, inp.data_ptr() + 4 * ob
                arr[i].c = out.data_ptr() + 4 * (oc - first)
            arrays.append(arr)
        s.keep.append(inp)
        s.out.extend(outs)
    return s


def _alone_inputs(case, seed):
    gen = _generator(seed)
    if case["kind"] == "sgemm":
        m, n, k = case["m"], case["n"], case["k"]
        return torch.randn(m, k, device="cuda", generator=gen), torch.randn(k, n, device="cuda", generator=gen)
    a = torch.empty(case["n"], device="cuda").uniform_(-1.0, 1.0, generator=gen)
    lo, hi = (0.75, 1.25) if case["kind"] == "vmul" else (-1.0, 1.0)
    return a, torch.empty(case["n"], device="cuda").uniform_(lo, hi, generator=gen)


def prepare(case, seed):
    if case["kind"] == "step":
        return _prepare_step(case, seed)
    if case["kind"] == "host":
        return _prepare_host(case, seed)
    s = _State(case)
    s.a, s.b = _alone_inputs(case, seed)
    s.scratch = None
    if case["kind"] == "sgemm":
        s.c = torch.empty(case["m"], case["n"], device="cuda")
        if case["path"] == "split3":
            s.scratch = torch.empty(g.sgemm_scratch_bytes(case["m"], case["n"], case["k"]) + 256, dtype=torch.uint8,
                                    device="cuda")
    else:
        s.c = torch.empty_like(s.a)
    return s


def run(state):
    s, case = state, state.case
    kind = case["kind"]
    if kind == "sgemm":
        g.sgemm_f32(s.a, s.b, s.c, case["path"], s.scratch)
        return s.c
    if kind == "vadd":
        g.vadd_f32(s.a, s.b, s.c)
        return s.c
    if kind == "vmul":
        g.vmul_f32(s.a, s.b, s.c, case["iters"])
        return s.c
    if kind == "host":
        s.mgr.spmd_run_overlapped(s.ranks, s.even, s.odd, case["steps"])
    elif case["driver"] == "threads":
        s.mgr.spmd_run(s.ranks, s.arrays, case["steps"])
    else:
        for _ in range(case["steps"]):
            last = [first + count - 1 for first, count in (r.submit_many(a) for r, a in zip(s.ranks, s.arrays))]
            s.mgr.flush()
            for r, seq in zip(s.ranks, last):
                r.sync(seq)
    return s.out


def work(case):
    if case["kind"] == "sgemm":
        m, n, k = case["m"], case["n"], case["k"]
        return {"bytes": 4 * (m * k + k * n + m * n), "flops": 2 * m * n * k}
    if case["kind"] in ("vadd", "vmul"):
        return {"bytes": 12 * case["n"], "flops": case["n"] * case.get("iters", 1)}
    nbytes = flops = 0
    for tasks in _batches(case):
        for t in tasks:
            nbytes += 4 * sum(_sizes(t))
            flops += t[2] if t[0] == VADD else 2 * t[1] * t[2] * t[3]
    return {"bytes": case["steps"] * nbytes, "flops": case["steps"] * flops}


def exact(case, seed):
    if case["kind"] == "sgemm":
        a, b = _alone_inputs(case, seed)
        return a.double() @ b.double()
    if case["kind"] in ("vadd", "vmul"):
        a, b = (x.double() for x in _alone_inputs(case, seed))
        if case["kind"] == "vadd":
            return a + b
        for _ in range(case["iters"]):
            a = a * b
        return a
    out = []
    gen = _generator(seed)
    for tasks in _batches(case):
        offs, first, size = _layout(tasks)
        block = torch.empty(first, device="cuda")
        _fill_inputs(block, tasks, offs, gen)
        res = torch.zeros(size - first, dtype=torch.float64, device="cuda")
        for t, (oa, ob, oc) in zip(tasks, offs):
            (a, b, c), (_, m, n, k) = _sizes(t), t
            x, y = block[oa:oa + a].double(), block[ob:ob + b].double()
            z = x + y if t[0] == VADD else (x.view(m, k) @ y.view(k, n)).view(-1)
            res[oc - first:oc - first + c] = z
        out.append(res)
    if case["kind"] == "host":  # even and odd steps write a buffer each
        out = [x.cpu() for r in out for x in (r, r)]
    return out
