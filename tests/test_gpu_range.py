"""The transporters and the link gradient of FP32 and 16-bit Brillouin handles
over the whole range of their FP32 results: sums that leave FP32's range where
the result does not, and results below its normal numbers, against the FP64
handle on the same inputs."""
import math

import numpy as np
import pytest

import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

L, NV = (4, 3, 5, 2), 3


@pytest.fixture(scope="module")
def dg():
    import __graft_entry__
    __graft_entry__.build()
    import paper_1808_05506_gb300 as dg
    torch.cuda.set_device(0)
    return dg


def _force(dg, prec, V, psi, g):
    cdt = torch.complex128 if prec == "f64" else torch.complex64
    D = dg.Dirac("brillouin", L, NV, 0.05, prec)
    D.set_links(torch.from_numpy(V).cuda())
    F = D.force(torch.from_numpy(psi).to(cdt).cuda(), torch.from_numpy(g).to(cdt).cuda()).cpu().numpy()
    D.close()
    return F.astype(np.complex128)


@pytest.mark.parametrize("prec", ["f32", "bf16"])
@pytest.mark.parametrize("top", [127.5, -130.0])
def test_brillouin_force_range(dg, prec, top):
    """psi and g times powers of two that take the largest component of F near the
    largest FP32 number, or below the smallest normal one: the rounding of F is
    still the only error (half a unit in the last place, next to 1e-11 of F)."""
    V = synth.round_to(synth.gauge_links(L, 3, "near_identity", 41), "f32")
    psi = synth.round_to(synth.spinor(L, NV, 4, 3, 42), prec)
    g = synth.round_to(synth.spinor(L, NV, 4, 3, 43), prec)
    F = _force(dg, "f64", V, psi, g).view(np.float64)
    e = math.floor(top - math.log2(np.abs(F).max()))
    e1 = e // 2
    got = _force(dg, prec, V, psi * 2.0 ** e1, g * 2.0 ** (e - e1)).view(np.float64)
    want = F * 2.0 ** e
    assert np.isfinite(got).all()
    half_ulp = np.maximum(np.abs(want) * 2.0 ** -24, 2.0 ** -150)
    assert (np.abs(got - want) <= half_ulp * (1 + 2.0 ** -6) + 1e-11 * np.abs(want).max()).all()


@pytest.mark.parametrize("prec,tol", [("f32", 1e-6), ("bf16", 3e-2)])
def test_brillouin_links_range(dg, prec, tol):
    """W_xy is the average of two products: their sum leaves FP32's range, W_xy does not."""
    V = np.zeros((L[3], L[2], L[1], L[0], 4, 3, 3), np.complex128)
    V[..., 0, :, :] = 2.0 ** 64 * np.eye(3)
    V[..., 1, :, :] = 1.5 * 2.0 ** 63 * np.eye(3)
    psi = synth.round_to(synth.spinor(L, NV, 4, 3, 44), prec) * 2.0 ** -100
    out = {}
    for p, cdt in (("f64", torch.complex128), (prec, torch.complex64)):
        D = dg.Dirac("brillouin", L, NV, 0.05, p)
        D.set_links(torch.from_numpy(V).cuda())
        out[p] = D.apply(torch.from_numpy(psi).to(cdt).cuda()).cpu().numpy().astype(np.complex128)
        D.close()
    err = np.linalg.norm(out[prec] - out["f64"]) / np.linalg.norm(out["f64"])
    assert err <= tol, err
