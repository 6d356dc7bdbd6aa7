"""What a Brillouin handle keeps in device memory: the links, and the scratch of
the link gradient only once it has taken one."""
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


def _used():
    torch.cuda.synchronize()
    free, total = torch.cuda.mem_get_info()
    return total - free


def test_links_keep_no_scratch(dg):
    L, Nv = (12, 12, 12, 16), 1
    V = torch.from_numpy(synth.gauge_links((4, 4, 4, 4), 3, "near_identity", 3).astype("complex64")).cuda()
    V = V.repeat(4, 3, 3, 3, 1, 1, 1).contiguous()
    sites = 12 * 12 * 12 * 16
    links, scratch = sites * (36 * 16 + 360 * 8), sites * 360 * 16   # FP64 V and FP32 W; the W build
    psi = torch.randn(L[3], L[2], L[1], L[0], Nv, 4, 3, dtype=torch.complex64, device="cuda")
    D = dg.Dirac("brillouin", L, Nv, 0.05, "f32")
    before = _used()
    D.set_links(V)
    held = _used() - before
    assert links <= held < links + scratch // 4
    F, G = (torch.empty_like(V) for _ in range(2))
    D.force(psi, psi, out=F)
    D.set_links(V)
    kept = _used()
    D.force(psi, psi, out=G)
    assert torch.equal(torch.view_as_real(F), torch.view_as_real(G))
    assert _used() == kept   # the gradient's scratch is taken once
    D.close()
