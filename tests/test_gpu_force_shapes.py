"""The Wilson and staggered link force at the lattice sizes where the number of
links per thread changes, against its defining sums in 64 bits."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

TOL = {"f32": 1e-6, "bf16": 1e-6}   # the inputs are exact in the storage type


@pytest.fixture(scope="module")
def dg():
    import __graft_entry__
    __graft_entry__.build()
    import paper_1808_05506_gb300 as dg
    torch.cuda.set_device(0)
    return dg


def _gammas():
    s = torch.zeros((3, 2, 2), dtype=torch.complex128)
    s[0, 0, 1] = s[0, 1, 0] = 1
    s[1, 0, 1], s[1, 1, 0] = -1j, 1j
    s[2, 0, 0], s[2, 1, 1] = 1, -1
    g = torch.zeros((4, 4, 4), dtype=torch.complex128)
    for k in range(3):
        g[k, :2, 2:], g[k, 2:, :2] = -1j * s[k], 1j * s[k]
    g[3, :2, 2:] = g[3, 2:, :2] = torch.eye(2)
    return g.cuda()


def _force(op, psi, g):
    """canonical F[t, z, y, x, mu, a, b] of Re <g, D psi>"""
    up = [lambda f, m=m: torch.roll(f, -1, dims=3 - m) for m in range(4)]
    Nt, Nz, Ny, Nx = psi.shape[:4]
    F = []
    t, z, y, x = torch.meshgrid(*[torch.arange(n, device="cuda") for n in (Nt, Nz, Ny, Nx)], indexing="ij")
    gam = _gammas()
    one = torch.eye(4, dtype=torch.complex128, device="cuda")
    for mu in range(4):
        pn, gn = up[mu](psi), up[mu](g)
        if op == "staggered":
            eta = (1 - 2 * ((0 * x, x, x + y, x + y + z)[mu] % 2))[..., None, None]
            F.append(0.5 * eta * (torch.einsum("tzyxva,tzyxvb->tzyxab", g, pn.conj())
                                  - torch.einsum("tzyxva,tzyxvb->tzyxab", psi, gn.conj())))
        else:
            gm = torch.einsum("su,tzyxvua->tzyxvsa", one - gam[mu], g)
            gp = torch.einsum("su,tzyxvua->tzyxvsa", one + gam[mu], gn)
            F.append(-0.5 * (torch.einsum("tzyxvsa,tzyxvsb->tzyxab", gm, pn.conj())
                             + torch.einsum("tzyxvsa,tzyxvsb->tzyxab", psi, gp.conj())))
    return torch.stack(F, dim=4)


# 16383 sites and fewer, from 16384 on, 20736 (two blocks of links per thread), 32768, 49152, 200000 and more
@pytest.mark.parametrize("L,Nv", [((7, 9, 5, 52), 2), ((16, 8, 8, 16), 3), ((12, 12, 12, 12), 1), ((12, 12, 12, 12), 2),
                                  ((16, 16, 8, 16), 3), ((16, 16, 16, 12), 2), ((23, 25, 25, 14), 2)])
@pytest.mark.parametrize("op", ["wilson", "staggered"])
@pytest.mark.parametrize("prec", ["f32", "bf16"])
def test_force_links_per_thread(dg, op, prec, L, Nv):
    gen = torch.Generator(device="cuda").manual_seed(17)
    shape = (L[3], L[2], L[1], L[0], Nv) + ((3,) if op == "staggered" else (4, 3))
    st = torch.bfloat16 if prec == "bf16" else torch.float32

    def field():
        f = torch.randn(shape + (2,), generator=gen, device="cuda").to(st).float()
        return torch.view_as_complex(f)

    psi, g = field(), field()
    D = dg.Dirac(op, L, Nv, 0.12, prec)
    D.set_links(torch.eye(3, dtype=torch.complex64, device="cuda").expand(L[3], L[2], L[1], L[0], 4, 3, 3).contiguous())
    got = D.force(psi, g).to(torch.complex128)
    want = _force(op, psi.to(torch.complex128), g.to(torch.complex128))
    err = ((got - want).abs().square().sum((0, 1, 2, 3, 5, 6)) / want.abs().square().sum((0, 1, 2, 3, 5, 6))).sqrt()
    assert err.max().item() <= TOL[prec], err
    D.close()


def test_force_without_links(dg):
    """Wilson and staggered forces do not read the links; the Brillouin gradient
    refuses a handle that has none."""
    L, Nv = (4, 2, 3, 2), 2
    for op in ("wilson", "staggered", "brillouin"):
        D = dg.Dirac(op, L, Nv, 0.12, "f32")
        psi = torch.ones(D.canonical_shape, dtype=torch.complex64, device="cuda")
        if op == "brillouin":
            with pytest.raises(dg.DiracError, match="dirac_set_links"):
                D.force(psi, psi)
        else:
            assert torch.isfinite(torch.view_as_real(D.force(psi, psi))).all()
        D.close()
