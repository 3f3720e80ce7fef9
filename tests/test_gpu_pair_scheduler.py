"""The pair scheduler over a long launch and beside other work."""
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


# One pair of CTAs runs every tile, so that its k-step numbers are taken back
# (after 1536 k-steps) several times in the launch; vector tasks between the
# products set the landings' numbers apart from the k-steps'. The same product
# must give the same bits before and after, on each landing form.
@pytest.mark.parametrize("m,n,k", [(130, 70, 2048), (258, 67, 2047), (3, 64, 992)])
@pytest.mark.parametrize("mode", ["barrier", "continuous"])
def test_kstep_numbers_are_taken_back(gvm, mode, m, n, k):
    count = 5 * 1536 // ((k + 31) // 32)
    A, B = synth.sgemm_inputs(synth.task_seed(3, k), m, n, k)
    x, y = synth.vadd_inputs(synth.task_seed(4, k), 4097)
    out_at, step = 32 << 20, 256 << 10
    with gvm.Manager(1, ring_depth=512, mode=mode, sgemm_path="split3", slice_bytes=128 << 20,
                     resident_bytes=120 << 20, grid_ctas=2) as mgr:
        rk = mgr.attach(0)
        for off, v in ((0, A), (8 << 20, B), (16 << 20, x), (17 << 20, y)):
            rk.write(off, torch.from_numpy(v))
        jobs = []
        for i in range(count):
            c = out_at + step * (i % 300)
            seq = rk.submit_sgemm_resident(0, 8 << 20, c, m, n, k)
            if i % 7 == 0:
                seq = rk.submit_vadd_resident(16 << 20, 17 << 20, 18 << 20, 4097)
            jobs.append(c)
        mgr.flush_if_barrier()
        rk.sync(seq)
        first = None
        for c in jobs:
            got = torch.empty(m, n)
            rk.read(c, got)
            if first is None:
                first = got.numpy()
                check_sgemm(first, A, B)
            assert np.array_equal(bits(got.numpy()), bits(first))
        v = torch.empty(4097)
        rk.read(18 << 20, v)
        assert np.array_equal(bits(v.numpy()), bits(oracle.vadd(x, y)))
        assert mgr.stats()["device_status"] == 0


# The FMA scheduler's vector tiles: 96 threads, groups of four values (16-byte
# aligned operands) or of every 96th value, eleven groups under way. Lengths
# around a part, a step of all threads (384), the groups under way and a tile's
# end; the words around each result must stay as they were.
@pytest.mark.parametrize("shift", [(0, 0, 0), (1, 0, 0), (0, 2, 0), (0, 0, 3), (3, 1, 2)])
@pytest.mark.parametrize("op", ["vadd", "vmul"])
def test_fma_scheduler_vector_groups(gvm, op, shift):
    sizes = [1, 3, 4, 95, 96, 97, 383, 384, 385, 11 * 384 - 1, 11 * 384, 11 * 384 + 1, 12 * 384 + 5, 1024, 1025, 9999]
    with gvm.Manager(1, ring_depth=64, sgemm_path="fma", slice_bytes=16 << 20, resident_bytes=12 << 20,
                     vadd_tile=8192) as mgr:
        rk = mgr.attach(0)
        step = 64 << 10
        jobs = []
        for i, n in enumerate(sizes):
            seed = synth.task_seed(5, n)
            x, y = synth.vadd_inputs(seed, n) if op == "vadd" else synth.vmul_inputs(seed, n)
            offs = [(3 * i + j) * step + 64 + 4 * s for j, s in enumerate(shift)]
            rk.write(offs[0], torch.from_numpy(x))
            rk.write(offs[1], torch.from_numpy(y))
            rk.write(offs[2] - 16, torch.full((n + 8,), 7.0))
            jobs.append((n, x, y, offs))
        for n, _, _, offs in jobs:
            seq = rk.submit_vadd_resident(*offs, n) if op == "vadd" else rk.submit_vmul_resident(*offs, n, 15)
        mgr.flush()
        rk.sync(seq)
        for n, x, y, offs in jobs:
            got = torch.empty(n + 8)
            rk.read(offs[2] - 16, got)
            got = got.numpy()
            want = oracle.vadd(x, y) if op == "vadd" else oracle.vmul(x, y, 15)
            assert np.array_equal(bits(got[4:-4]), bits(want)), n
            assert np.all(got[:4] == 7.0) and np.all(got[-4:] == 7.0), n
        assert mgr.stats()["device_status"] == 0


# What the split3 scheduler's vector landings took for a result that is not
# 16-byte aligned must not be slower than for one that is by more than half.
# (Its stores are 4 bytes a lane; the loads bound it.) The FMA scheduler's
# groups: three times, for four times the requests.
@pytest.mark.parametrize("path,most", [("split3", 1.5), ("fma", 3.0)])
def test_misaligned_vectors_keep_their_rate(gvm, path, most):
    n, per, ranks = 1 << 20, 8, 8
    step = 4 * n + 256
    best = {}
    with gvm.Manager(ranks, ring_depth=8, sgemm_path=path, slice_bytes=3 * per * step + (1 << 20),
                     resident_bytes=3 * per * step) as mgr:
        rks = [mgr.attach(r) for r in range(ranks)]
        for rk in rks:
            rk.resident_view(0, (3 * per * step // 4,)).fill_(1.0)
        torch.cuda.synchronize()
        for shift in (0, 1):
            arrays = []
            for _ in rks:
                a = (gvm.GvmTask * per)()
                for i in range(per):
                    a[i].type, a[i].flags, a[i].n = gvm.GVM_TASK_VADD, gvm.GVM_TASK_RESIDENT, n
                    a[i].a_off, a[i].b_off, a[i].c_off = 3 * i * step, (3 * i + 1) * step, (3 * i + 2) * step + 4 * shift
                arrays.append(a)
            mgr.spmd_run(rks, arrays, 3)
            best[shift] = min(mgr.spmd_run(rks, arrays, 20)[1])
    assert best[1] <= most * best[0], best


# Interior and ragged tiles, rows aligned to 4, 8 and 16 bytes, k below one
# k-step, several tiles a cluster: the standalone kernel against binary64 by the
# bound of sgemm_bounds.check_sgemm, and bit for bit the manager's result, whose
# tiles are 256 (or 192) columns wide where the standalone kernel picks 64 to 256.
@pytest.mark.parametrize(
    "shape",
    [(128, 256, 32), (257, 130, 67), (512, 512, 512), (129, 257, 513), (300, 1001, 77), (130, 260, 100),
     (1000, 520, 2052), (4096, 2048, 96), (2500, 3000, 40), (256, 256, 1), (768, 1024, 512), (1024, 512, 2048),
     (520, 512, 256), (200, 300, 96), (384, 640, 44), (1, 257, 31)],
)
def test_standalone_kernel_equals_the_manager(gvm, shape):
    m, n, k = shape
    A, B = synth.sgemm_inputs(synth.task_seed(13, m % 1000), m, n, k)
    tA, tB = torch.from_numpy(A).cuda(), torch.from_numpy(B).cuda()
    C = torch.full((m, n), float("nan"), device="cuda")
    gvm.sgemm_f32(tA, tB, C, path="split3")
    torch.cuda.synchronize()
    R = tA.double() @ tB.double()
    bound = gamma(k) * (tA.double().abs() @ tB.double().abs()) + k * 2.0 ** -149
    assert bool(((C.double() - R).abs() <= bound).all())
    step = [(4 * x + 255) // 256 * 256 for x in (m * k, k * n, m * n)]
    with gvm.Manager(1, ring_depth=4, sgemm_path="split3", slice_bytes=sum(step) + (1 << 20),
                     resident_bytes=sum(step)) as mgr:
        rk = mgr.attach(0)
        rk.write(0, torch.from_numpy(A))
        rk.write(step[0], torch.from_numpy(B))
        seq = rk.submit_sgemm_resident(0, step[0], step[0] + step[1], m, n, k)
        mgr.flush()
        rk.sync(seq)
        out = torch.empty(m, n)
        rk.read(step[0] + step[1], out)
        assert np.array_equal(bits(out.numpy()), bits(C.cpu().numpy()))
    from paper_1511_07658_gb300.manager import kernel_status

    assert kernel_status() == 0


# A host result buffer off a 4-byte boundary is not one the kernel can store to:
# with direct output it takes the staged path, and the bytes around it stay.
@pytest.mark.parametrize("path", ["split3", "fma"])
@pytest.mark.parametrize("offset", [1, 2, 3, 4])
def test_direct_output_to_any_byte_address(gvm, path, offset):
    n = 5001
    x, y = synth.vadd_inputs(synth.task_seed(6, offset), n)
    a, b = torch.from_numpy(x).pin_memory(), torch.from_numpy(y).pin_memory()
    out = torch.full((4 * n + 16,), 0x5A, dtype=torch.uint8).pin_memory()
    with gvm.Manager(1, ring_depth=4, sgemm_path=path, slice_bytes=8 << 20, direct_output=True) as mgr:
        rk = mgr.attach(0)
        t = gvm.GvmTask()
        t.type, t.n = gvm.GVM_TASK_VADD, n
        t.a, t.b, t.c = a.data_ptr(), b.data_ptr(), out.data_ptr() + offset
        seq = rk.submit(t)
        mgr.flush()
        rk.sync(seq)
        got = out.numpy()
        assert np.array_equal(got[offset:offset + 4 * n].copy().view(np.uint32), bits(oracle.vadd(x, y)))
        assert np.all(got[:offset] == 0x5A) and np.all(got[offset + 4 * n:] == 0x5A)
        assert mgr.stats()["device_status"] == 0
