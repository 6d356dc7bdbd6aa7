"""Where sums are rounded: properties of the FP64 results that hold bit for bit
when each hop, and each product of the link force, is formed by itself before it joins
the sum, and that a chain of all the products breaks (its error is larger)."""
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


def _same(a, b):
    return torch.equal(torch.view_as_real(a), torch.view_as_real(b))


@pytest.mark.parametrize("L,Nv", [((3, 2, 5, 2), 1), ((4, 6, 2, 3), 5), ((8, 4, 4, 4), 4)])
def test_staggered_f64_sums_the_directions(dg, L, Nv):
    """At m = 0 the sweep over all links is the sum, direction by direction, of
    the sweeps in which only that direction's links are not zero."""
    V = torch.from_numpy(synth.gauge_links(L, 3, "near_identity", 81)).cuda()
    x = torch.from_numpy(synth.spinor(L, Nv, 1, 3, 82)).cuda()
    D = dg.Dirac("staggered", L, Nv, 0.0, "f64")
    for dag in (False, True):
        part = []
        for mu in range(4):
            Vm = torch.zeros_like(V)
            Vm[..., mu, :, :] = V[..., mu, :, :]
            D.set_links(Vm)
            part.append(D.apply(x, dagger=dag))
        D.set_links(V)
        want = ((part[0] + part[1]) + part[2]) + part[3]
        for R, block, variant in ((1, 128, 0), (2, 64, 0), (4, 128, 0), (1, 32, 1), (2, 64, 1)):
            D.set_kernel_config(R, block, variant)
            assert _same(D.apply(x, dagger=dag), want), (dag, R, block, variant)
            assert _same(D.unpack(D.apply(D.pack(x), dagger=dag)), want), (dag, R, block, variant)
    D.close()


def _parity(L):
    Nx, Ny, Nz, Nt = L
    t, z, y, x = torch.meshgrid(*[torch.arange(n) for n in (Nt, Nz, Ny, Nx)], indexing="ij")
    return ((x + y + z + t) % 2).cuda()


# extents are even, so every link joins an even and an odd site
@pytest.mark.parametrize("op,L", [("staggered", (4, 2, 6, 4)), ("staggered", (8, 4, 4, 4)), ("wilson", (4, 2, 6, 4)),
                                  ("wilson", (8, 4, 4, 4))])
def test_force_f64_sums_the_products(dg, op, L):
    """With psi and g cut by the parity of the site (and, for Wilson, into the
    spins that one half-spinor component is made of) the force at the even sites is
    one product in each run; they add up to the whole force in the order of the
    hops, then of the components."""
    ns = 1 if op == "staggered" else 4
    psi = torch.from_numpy(synth.spinor(L, 1, ns, 3, 91)).cuda()
    g = torch.from_numpy(synth.spinor(L, 1, ns, 3, 92)).cuda()
    D = dg.Dirac(op, L, 1, 0.12, "f64")
    D.set_links(torch.from_numpy(synth.gauge_links(L, 3, "near_identity", 93)).cuda())
    whole = D.force(psi, g)
    par = _parity(L)
    even = (par == 0).reshape(par.shape + (1,) * (psi.dim() - 4))
    mus = range(4) if op == "staggered" else (2, 3)   # half spinors of the spins (0, 2) and (1, 3)
    want = None
    for g_side, p_side in ((even, ~even), (~even, even)):   # the hop with g(x), then the one with psi(x)
        for spins in ((slice(None),) if op == "staggered" else ([0, 2], [1, 3])):
            p, q = torch.zeros_like(psi), torch.zeros_like(g)
            if op == "staggered":
                p, q = psi * p_side, g * g_side
            else:
                p[..., spins, :] = (psi * p_side)[..., spins, :]
                q[..., spins, :] = (g * g_side)[..., spins, :]
            F = D.force(p, q)
            want = F if want is None else want + F
    for mu in mus:
        assert _same(whole[..., mu, :, :][par == 0], want[..., mu, :, :][par == 0]), mu
    D.close()
