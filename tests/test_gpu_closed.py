"""A closed handle refuses every call, whatever was asked of it before."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def dg():
    import __graft_entry__
    __graft_entry__.build()
    import paper_1808_05506_gb300 as dg
    torch.cuda.set_device(0)
    return dg


def test_closed_handle(dg):
    D = dg.Dirac("staggered", (4, 2, 2, 2), 1, 0.05, "f32")
    x = D.new_internal()
    y = torch.zeros(D.canonical_shape, dtype=torch.complex64, device="cuda")
    D.close()
    for call in (D.new_internal, lambda: D.field_bytes(dg.INTERNAL), lambda: D.apply(x), lambda: D.apply(y),
                 lambda: D.pack(y), lambda: D.unpack(x)):
        with pytest.raises(dg.DiracError):
            call()
