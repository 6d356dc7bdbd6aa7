"""Handles of different lattices used from different host threads at the same time."""
import threading

import pytest

import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def dg():
    import __graft_entry__
    __graft_entry__.build()
    import paper_1808_05506_gb300 as dg
    torch.cuda.set_device(0)
    return dg


def test_tensor_core_sweeps_from_threads(dg):
    """The tiles of the lattices take different amounts of shared memory for
    the same kernel; every launch of any thread gets what it needs."""
    jobs = []
    apply = dg.lib().dirac_apply
    for L in ((8, 2, 2, 2), (2, 2, 2, 4)) * 2:
        D = dg.Dirac("brillouin", L, 16, 0.05, "bf16")
        D.set_links(torch.from_numpy(synth.gauge_links(L, 3, "near_identity", 5).astype("complex64")).cuda())
        D.set_kernel_config(1, 128, 7)
        x = D.pack(torch.from_numpy(synth.spinor(L, 16, 4, 3, 6).astype("complex64")).cuda())
        jobs.append((D, x, D.apply(x)))
    torch.cuda.synchronize()
    failed = []
    start = threading.Barrier(4)

    def run(D, x, want):
        y = D.new_internal()
        start.wait()
        st = [apply(D.h, y.data_ptr(), x.data_ptr(), dg.INTERNAL) for _ in range(5000)]
        torch.cuda.synchronize()
        if any(st):
            failed.append((sum(map(bool, st)), dg.last_error(D.h)))
        elif not torch.equal(y, want):
            failed.append("another result")

    ts = [threading.Thread(target=run, args=j) for j in jobs]
    for t in ts:
        t.start()
    for t in ts:
        t.join()
    for D, _, _ in jobs:
        D.close()
    assert not failed, failed
