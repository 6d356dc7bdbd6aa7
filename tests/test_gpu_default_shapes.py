"""The launch shapes of handles that were not tuned where they reorder the sites
(a t-slice of more than 25 MB): the same numbers as in lexicographic order, through the internal and
the canonical call, with a last t-chunk shorter than the others; and the order a
shape set by hand starts from."""
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


# x-rows in a warp or not
@pytest.mark.parametrize("L,Nv", [((16, 16, 16, 10), 64), ((12, 14, 14, 9), 112)])
def test_default_site_order(dg, L, Nv):
    gen = torch.Generator(device="cuda").manual_seed(23)

    def rand(*shape):
        return torch.view_as_complex(torch.randn(shape + (2,), generator=gen, device="cuda"))

    D = dg.Dirac("wilson", L, Nv, 0.12, "f32")
    assert D.site_order() == 8
    D.set_links(rand(L[3], L[2], L[1], L[0], 4, 3, 3))
    x = rand(*D.canonical_shape)
    order = {}
    for tc in (D.site_order(), 0):
        D.set_site_order(tc)
        order[tc] = [D.apply(x, dagger=dag) for dag in (False, True)] + [D.unpack(D.apply(D.pack(x)))]
    for a, b in zip(order[8], order[0]):
        assert torch.equal(torch.view_as_real(a), torch.view_as_real(b))
    D.close()


def test_shape_set_by_hand_starts_lexicographic(dg):
    D = dg.Dirac("wilson", (16, 16, 16, 10), 64, 0.12, "f32")
    assert D.site_order() == 8
    D.set_kernel_config(2, 64, 1)
    assert D.site_order() == 0
    D.set_site_order(3)
    D.set_kernel_config(1, 128, 0)
    assert D.site_order() == 3
    D.close()
