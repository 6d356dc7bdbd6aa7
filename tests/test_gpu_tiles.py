"""Sweep kernels at the edges of their tiles, against the FP64 oracle on the
inputs as stored, at the tolerances of the storage types of test_gpu_apply.py."""
import numpy as np
import pytest

import oracle
import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

TOL = {"f64": 1e-13, "f32": 1e-6, "bf16": 3e-2, "f16": 4e-3}
NS = {"staggered": 1, "wilson": 4, "brillouin": 4}


@pytest.fixture(scope="module")
def dg():
    import __graft_entry__
    __graft_entry__.build()
    import paper_1808_05506_gb300 as dg
    torch.cuda.set_device(0)
    return dg


def rel_l2(got, want):
    ax = tuple(i for i in range(got.ndim) if i != 4)
    return float((np.sqrt((np.abs(got - want) ** 2).sum(ax)) / np.sqrt((np.abs(want) ** 2).sum(ax))).max())


# partial tiles in x and y (5 x 3, 6 x 2, 8 x 2 sites), every number of column tiles, two blocks of rhs
@pytest.mark.parametrize("L,Nv", [((10, 7, 3, 3), 4), ((17, 3, 2, 3), 7), ((12, 5, 2, 2), 12), ((16, 6, 2, 3), 16),
                                  ((5, 2, 3, 2), 21)])
@pytest.mark.parametrize("prec", ["bf16", "f16"])
def test_brillouin_tensor_core_tiles(dg, L, Nv, prec):
    V = synth.round_to(synth.gauge_links(L, 3, "near_identity", 51), "f32")
    psi = synth.round_to(synth.spinor(L, Nv, 4, 3, 52), prec)
    D = dg.Dirac("brillouin", L, Nv, 0.05, prec)
    D.set_links(torch.from_numpy(V).cuda())
    D.set_kernel_config(1, 128, 7)
    x = torch.from_numpy(psi.astype(np.complex64)).cuda()
    for order in (0, 2):
        D.set_site_order(order)
        for dag in (False, True):
            got = D.apply(x, dagger=dag).cpu().numpy().astype(np.complex128)
            want = oracle.apply("brillouin", V, psi, 0.05, dagger=dag)
            assert rel_l2(got, want) <= TOL[prec], (order, dag)
    D.close()
