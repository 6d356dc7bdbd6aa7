"""The tensor-core Brillouin sweep of FP16 handles whose link products fall
below FP16's normal numbers, against the CUDA-core sweep of the same stored links."""
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


@pytest.mark.parametrize("scale", [1.0, 2.0 ** -3])
def test_small_links(dg, scale):
    """Without the diagonal (m0 = -15/8).  Both round their result once (2^-11 of it);
    240 products, each off by at most 2^-25 of 4/27 psi, add less than 240 2^-25 4/27 / (scale / 8)
    to that, as the eight one-hop links alone give an eighth of scale psi."""
    L, Nv = (8, 4, 3, 2), 4
    V = torch.from_numpy(scale * synth.gauge_links(L, 3, "near_identity", 61)).cuda()
    D = dg.Dirac("brillouin", L, Nv, -15.0 / 8.0, "f16")
    D.set_links(V)
    x = torch.from_numpy(synth.spinor(L, Nv, 4, 3, 62).astype("complex64")).cuda()
    out = []
    for cfg in ((1, 128, 7), (1, 128, 0)):
        D.set_kernel_config(*cfg)
        out.append(D.apply(x).to(torch.complex128))
    err = ((out[0] - out[1]).norm() / out[1].norm()).item()
    assert err <= 2 * 2.0 ** -11 + 240 * 2.0 ** -25 * 4 / 27 / (scale / 8), err
    D.close()
