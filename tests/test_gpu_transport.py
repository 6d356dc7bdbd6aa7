"""The Brillouin link gradient in double-float arithmetic (FP32 and 16-bit
handles) against the FP64 handle's on the same inputs: the only error left is
the rounding of each entry to FP32, at most 2^-24 of it, next to a
double-float chain of a few hundred operations at 2^-48 each."""
import numpy as np
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


# extents 2 (both neighbours are one site), odd, not a multiple of the 128 threads of a block
@pytest.mark.parametrize("L,Nv", [((2, 3, 2, 3), 1), ((4, 3, 5, 2), 3), ((6, 4, 4, 6), 5)])
@pytest.mark.parametrize("prec", ["f32", "bf16", "f16"])
def test_brillouin_force_double_float(dg, L, Nv, prec):
    V = synth.round_to(synth.gauge_links(L, 3, "near_identity", 41), "f32")
    psi = synth.round_to(synth.spinor(L, Nv, 4, 3, 42), prec)
    g = synth.round_to(synth.spinor(L, Nv, 4, 3, 43), prec)
    F = {}
    for p, cdt in (("f64", torch.complex128), (prec, torch.complex64)):
        D = dg.Dirac("brillouin", L, Nv, 0.05, p)
        D.set_links(torch.from_numpy(V).cuda())
        F[p] = D.force(torch.from_numpy(psi).to(cdt).cuda(), torch.from_numpy(g).to(cdt).cuda()).cpu().numpy()
        D.close()
    a, b = F[prec].astype(np.complex128), F["f64"]
    err = np.linalg.norm(a - b) / np.linalg.norm(b)
    assert err <= 2.0 ** -24 + 1e-11, err
