"""The pair scheduler over a long launch and beside other work."""
import numpy as np
import pytest
import torch

import oracle
import synth

pytestmark = pytest.mark.gpu

from sgemm_bounds import check_sgemm  # noqa: E402


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
