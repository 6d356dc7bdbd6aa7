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


# whole and partial warps of sites, partial groups of right-hand sides, one and several blocks
@pytest.mark.parametrize("op", ["wilson", "staggered"])
@pytest.mark.parametrize("prec", ["f32", "f64"])
@pytest.mark.parametrize("L,Nv", [((3, 2, 5, 2), 1), ((7, 5, 3, 3), 5), ((8, 4, 4, 2), 8), ((16, 4, 2, 4), 7)])
def test_canonical_output_is_the_internal_one(dg, op, prec, L, Nv):
    """A sweep that writes a canonical field itself stores the numbers that
    unpacking its internal result gives, in every launch shape, and leaves no
    entry out; backward gives what apply_dagger and force give."""
    cdt = torch.complex128 if prec == "f64" else torch.complex64
    V = torch.from_numpy(synth.gauge_links(L, 3, "near_identity", 61)).to(cdt).cuda()
    x = torch.from_numpy(synth.spinor(L, Nv, NS[op], 3, 62)).to(cdt).cuda()
    g = torch.from_numpy(synth.spinor(L, Nv, NS[op], 3, 63)).to(cdt).cuda()
    D = dg.Dirac(op, L, Nv, 0.12, prec)
    D.set_links(V)
    done = 0
    for R in (1, 2, 4, 6):
        for block in (32, 64, 128, 256):
            for variant in (0, 1, 6):
                if not dg.config_supported(op, prec, R, block, variant, L):
                    continue
                D.set_kernel_config(R, block, variant)
                done += 1
                for dag in (False, True):
                    want = D.unpack(D.apply(D.pack(x), dagger=dag))
                    got = D.new_canonical()
                    got.fill_(complex(float("nan"), float("nan")))
                    D.apply(x, out=got, dagger=dag)
                    assert torch.equal(torch.view_as_real(got), torch.view_as_real(want)), (R, block, variant, dag)
    assert done >= 4
    gpsi, F = D.backward(x, g)
    assert torch.equal(gpsi, D.apply_dagger(g)) and torch.equal(F, D.force(x, g))
    D.close()


# the launch shapes of handles that were not tuned: x-rows in a warp or not, R by Nv, t-chunks or not
@pytest.mark.parametrize("op", ["wilson", "staggered"])
@pytest.mark.parametrize("prec", ["f32", "bf16"])
@pytest.mark.parametrize("L,Nv", [((8, 4, 2, 3), 1), ((8, 4, 2, 3), 5), ((6, 3, 2, 5), 3), ((5, 3, 3, 2), 7),
                                  ((4, 4, 2, 2), 12), ((3, 2, 2, 3), 24)])
def test_default_launch_shape(dg, op, prec, L, Nv):
    V = synth.round_to(synth.gauge_links(L, 3, "near_identity", 71), "f32")
    psi = synth.round_to(synth.spinor(L, Nv, NS[op], 3, 72), prec)
    mass = 0.12
    D = dg.Dirac(op, L, Nv, mass, prec)
    D.set_links(torch.from_numpy(V).cuda())
    Vs = synth.round_to(V, prec)
    x = torch.from_numpy(psi.astype(np.complex64)).cuda()
    m0 = oracle.kappa_to_m0(mass) if op == "wilson" else mass
    for dag in (False, True):
        got = D.apply(x, dagger=dag).cpu().numpy().astype(np.complex128)
        assert rel_l2(got, oracle.apply(op, Vs, psi, m0, dagger=dag)) <= TOL[prec]
    D.close()


# the packed 16-bit Wilson sweeps: whole and partial pairs, x-rows of 4 to 32 sites and none, both link formats
@pytest.mark.parametrize("prec", ["bf16", "f16"])
@pytest.mark.parametrize("L,Nv", [((4, 4, 2, 3), 2), ((32, 2, 2, 2), 3), ((6, 5, 3, 2), 5), ((16, 2, 4, 3), 14)])
def test_wilson_pairs_16bit(dg, prec, L, Nv):
    V = synth.round_to(synth.gauge_links(L, 3, "near_identity", 81), "f32")
    psi = synth.round_to(synth.spinor(L, Nv, 4, 3, 82), prec)
    D = dg.Dirac("wilson", L, Nv, 0.12, prec)
    D.set_links(torch.from_numpy(V).cuda())
    Vs = synth.round_to(V, prec)
    x = torch.from_numpy(psi.astype(np.complex64)).cuda()
    for fmt in (0, 1):
        D.set_link_format(fmt)
        for variant in (1, 6):
            if not dg.config_supported("wilson", prec, 2, 32, variant, L):
                continue
            D.set_kernel_config(2, 32, variant)
            for dag in (False, True):
                got = D.apply(x, dagger=dag).cpu().numpy().astype(np.complex128)
                want = oracle.apply("wilson", Vs, psi, oracle.kappa_to_m0(0.12), dagger=dag)
                assert rel_l2(got, want) <= TOL[prec], (fmt, variant, dag)
    D.close()


# even-odd sweeps of pairs of right-hand sides against those of one: four inner iterations of two columns and of
# each alone.  FP32 rounding through four iterations: 1e-7 x 1e3; the split fields add flips of 16-bit roundings
# (2^-8 (F16: 2^-11) at a rate of 1e-7 / 2^-8, so 2e-5 rms each, a dozen of them, amplified 1e1)
@pytest.mark.parametrize("prec,tol", [("f32", 1e-4), ("bf16", 3e-3), ("f16", 3e-3)])
@pytest.mark.parametrize("L", [(4, 4, 2, 4), (6, 2, 4, 10)])
def test_even_odd_pairs(dg, prec, tol, L):
    V = torch.from_numpy(synth.round_to(synth.gauge_links(L, 3, "near_identity", 91), "f32")).cuda()
    b = synth.spinor(L, 2, 4, 3, 92)
    xs = []
    for cols in ((0, 1), (0,), (1,)):
        D = dg.Dirac("wilson", L, len(cols), 0.12, prec)
        D.set_links(V)
        x, _, st, _ = D.solve(torch.from_numpy(np.ascontiguousarray(b[:, :, :, :, list(cols)])).cuda(), tol=1e-10,
                              max_outer=1, max_inner=4)
        assert st["even_odd"] == 1
        xs.append(x.cpu().numpy())
        D.close()
    for v in (0, 1):
        want = xs[1 + v][:, :, :, :, 0]
        assert np.linalg.norm(want) > 0
        assert np.linalg.norm(xs[0][:, :, :, :, v] - want) <= tol * np.linalg.norm(want)
