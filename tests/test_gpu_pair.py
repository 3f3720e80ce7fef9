"""The CTA-pair form of split3, the scheduler's vector chunks and FMA tiles,
and the SPMD harness' kept threads, at the sizes where they can go wrong."""
import numpy as np
import pytest
import torch

import oracle
import synth

pytestmark = pytest.mark.gpu

from sgemm_bounds import check_sgemm, gamma  # noqa: E402


@pytest.fixture(scope="module")
def gvm():
    import __graft_entry__

    __graft_entry__.build()
    import paper_1511_07658_gb300 as g

    torch.cuda.set_device(0)
    return g


def bits(x):
    return np.ascontiguousarray(x).view(np.uint32)


def operand(rows, cols, shift):
    x = torch.empty(rows * cols + shift, device="cuda")
    return x[shift:].view(rows, cols)


# Several tiles a cluster with one to four k-steps each (landings, stages and
# accumulators all wrap); aligned, packed A, packed B, both.
@pytest.mark.parametrize(
    "shape", [(4096, 4096, 32), (4096, 4096, 96), (4095, 4094, 67), (4096, 4090, 64), (4090, 4096, 65)]
)
def test_pair_tiles_in_a_row(gvm, shape):
    m, n, k = shape
    g = torch.Generator(device="cuda").manual_seed(m + n + k)
    A = torch.randn(m, k, device="cuda", generator=g)
    B = torch.randn(k, n, device="cuda", generator=g)
    R = A.double() @ B.double()
    # the bound of sgemm_bounds.check_sgemm, evaluated on the device
    bound = gamma(k) * (A.double().abs() @ B.double().abs()) + k * 2.0 ** -149
    first = None
    for _ in range(4):
        C = torch.full((m, n), float("nan"), device="cuda")
        gvm.sgemm_f32(A, B, C, path="split3")
        torch.cuda.synchronize()
        if first is None:
            first = C
            assert bool(((C.double() - R).abs() <= bound).all())
        else:
            assert torch.equal(C, first)
    from paper_1511_07658_gb300.manager import kernel_status

    assert kernel_status() == 0


# Edges of the tile widths (64, 192, 256 columns) and of a k-step, rows shorter
# than one 16-byte piece, and bases off by 4, 8 and 12 bytes.
@pytest.mark.parametrize(
    "shape,shifts",
    [((2, 5, 3), (0, 0, 0)), ((300, 3, 2), (0, 0, 0)), ((3, 300, 37), (1, 0, 0)), ((259, 261, 35), (0, 0, 0)),
     ((257, 191, 33), (0, 0, 0)), ((255, 193, 31), (0, 0, 1)), ((256, 255, 100), (0, 0, 0)),
     ((131, 66, 1001), (0, 0, 0)), ((300, 520, 256), (1, 0, 0)), ((300, 520, 256), (0, 2, 0)),
     ((256, 256, 64), (3, 1, 1)), ((257, 131, 67), (3, 1, 2)), ((64, 385, 448), (0, 0, 3))],
)
def test_pair_odd_operands(gvm, shape, shifts):
    m, n, k = shape
    A, B = synth.sgemm_inputs(synth.task_seed(m % 100, n), m, n, k)
    tA, tB, tC = operand(m, k, shifts[0]), operand(k, n, shifts[1]), operand(m, n, shifts[2])
    tA.copy_(torch.from_numpy(A))
    tB.copy_(torch.from_numpy(B))
    tC.fill_(float("nan"))
    gvm.sgemm_f32(tA, tB, tC, path="split3")
    torch.cuda.synchronize()
    check_sgemm(tC.cpu().numpy(), A, B)


# Vector tasks around the 4096-value chunks, on 4-byte offsets, between SGEMM
# tasks (landings pass from one kind to the other, and the 64 x 64 FMA tiles
# meet ragged edges); results must be those of the task alone.
@pytest.mark.parametrize("path", ["split3", "fma"])
@pytest.mark.parametrize("mode", ["barrier", "continuous"])
def test_chunks_between_sgemm_tiles(gvm, path, mode):
    vec = [(n, s) for n in (1, 3, 4095, 4096, 4097, 8192, 16384 + 5, 70001) for s in ((0, 0, 0), (1, 1, 1), (0, 1, 3))]
    mats = [(256, 256, 32), (63, 65, 64), (64, 64, 1), (65, 129, 33), (513, 190, 96), (257, 388, 31)]
    with gvm.Manager(1, ring_depth=64, mode=mode, sgemm_path=path, slice_bytes=64 << 20,
                     resident_bytes=48 << 20) as mgr:
        rk = mgr.attach(0)
        at = 0

        def place(x, shift):
            nonlocal at
            off = (at + 255) // 256 * 256 + 4 * shift
            at = off + x.nbytes
            rk.write(off, torch.from_numpy(x))
            return off

        jobs = []
        for i, (n, (sa, sb, sc)) in enumerate(vec):
            a, b = synth.vadd_inputs(synth.task_seed(1, i), n) if i % 2 else synth.vmul_inputs(synth.task_seed(1, i), n)
            c = np.full(n, np.nan, np.float32)
            jobs.append((i % 2, (n,), (a, b), place(a, sa), place(b, sb), place(c, sc)))
            if i % 4 == 3:
                m, n, k = mats[i // 4 % len(mats)]
                A, B = synth.sgemm_inputs(synth.task_seed(2, i), m, n, k)
                C = np.full((m, n), np.nan, np.float32)
                jobs.append((2, (m, n, k), (A, B), place(A, 4), place(B, 0), place(C, 8)))
        for kind, dims, _, oa, ob, oc in jobs:
            if kind == 0:
                seq = rk.submit_vmul_resident(oa, ob, oc, dims[0], 15)
            elif kind == 1:
                seq = rk.submit_vadd_resident(oa, ob, oc, dims[0])
            else:
                seq = rk.submit_sgemm_resident(oa, ob, oc, *dims)
        mgr.flush()
        rk.sync(seq)
        for kind, dims, (x, y), _, _, oc in jobs:
            out = torch.empty(dims[0] if kind < 2 else dims[:2])
            rk.read(oc, out)
            if kind == 2:
                check_sgemm(out.numpy(), x, y)
            else:
                want = oracle.vadd(x, y) if kind else oracle.vmul(x, y, 15)
                assert np.array_equal(bits(out.numpy()), bits(want)), dims
        assert mgr.stats()["device_status"] == 0


# The harness keeps its threads: fewer, then more ranks than the run before,
# every run's results its own (one task a rank, a fresh operand each run).
@pytest.mark.parametrize("counts", [(1, 4, 2, 4)])
def test_spmd_runs_with_other_rank_counts(gvm, counts):
    n = 4096 + 1
    with gvm.Manager(max(counts), ring_depth=4, slice_bytes=8 << 20, resident_bytes=1 << 20) as mgr:
        ranks = [mgr.attach(r) for r in range(max(counts))]
        for run, count in enumerate(counts):
            arrays, want = [], []
            for r in range(count):
                a, b = synth.vadd_inputs(synth.task_seed(r, run), n)
                ranks[r].write(0, torch.from_numpy(a))
                ranks[r].write(1 << 16, torch.from_numpy(b))
                t = (gvm.GvmTask * 1)()
                t[0].type, t[0].flags, t[0].n = gvm.GVM_TASK_VADD, gvm.GVM_TASK_RESIDENT, n
                t[0].a_off, t[0].b_off, t[0].c_off = 0, 1 << 16, 2 << 16
                arrays.append(t)
                want.append(oracle.vadd(a, b))
            mgr.spmd_run(ranks[:count], arrays, 3)
            for r in range(count):
                out = torch.empty(n)
                ranks[r].read(2 << 16, out)
                assert np.array_equal(bits(out.numpy()), bits(want[r])), (run, r)
