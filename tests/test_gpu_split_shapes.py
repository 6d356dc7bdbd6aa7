"""Solves of 16-bit Brillouin handles that are configured for the tensor cores,
whose inner sweeps on CUDA cores take their own launch shape (one, two and three right-hand
sides per thread, groups of one), certified by an FP64 handle's residual."""
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


@pytest.mark.parametrize("L,Nv", [((4, 4, 4, 4), 1), ((5, 3, 4, 2), 4), ((4, 4, 4, 4), 5), ((8, 8, 8, 8), 16),
                                  ((8, 8, 8, 16), 12)])
@pytest.mark.parametrize("prec", ["bf16", "f16"])
def test_solve_of_a_tensor_core_handle(dg, L, Nv, prec):
    V = torch.from_numpy(synth.gauge_links(L, 3, "near_identity", 31)).cuda()
    b = torch.from_numpy(synth.spinor(L, Nv, 4, 3, 32)).cuda()
    D = dg.Dirac("brillouin", L, Nv, 0.05, prec)
    D.set_links(V)
    D.set_kernel_config(1, 128, 7)
    x, res, st, status = D.solve(b, tol=1e-10)
    assert status == dg.OK and st["split_fields"] == 1
    E = dg.Dirac("brillouin", L, Nv, 0.05, "f64")
    E.set_links(V)
    r = b - E.apply(x)
    ax = (0, 1, 2, 3, 5, 6)
    assert (r.abs().square().sum(ax) / b.abs().square().sum(ax)).sqrt().max().item() <= 1.01e-10
    E.close()
    D.close()
