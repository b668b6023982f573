"""The mixed stage where FP32 numbers of its physics are subnormal (below 1.2e-38): a cold flow whose pressure is, keeps its
high-order fluxes; and a metric so small that det(gamma) is (coordinates in small units, an exact power of two of an
ordinary block) gives the ordinary block's results in those units."""
import numpy as np
import pytest

import oracle as O
from paper_2311_04989_gb300 import grstage as G
from paper_2311_04989_gb300 import inputs as I
from tests import gpu_harness as GH

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("recon", [G.GR_RECON_WENOZ, G.GR_RECON_WENO5])
def test_cold_flow_with_a_subnormal_pressure_keeps_its_order(recon):
    P = GH.mixed_params(O.Params(gamma_ad=2.0, recon=recon, rho_atm=1e-14, p_atm=1e-40, tol=1e-10))
    b = I.random_block(n=(12, 9, 10), g=3, seed=23, rho_range=(1e-4, 1e-3), metric_amp=0.02, u_max=0.3)
    b.B = [np.zeros_like(f) for f in b.B]
    b.W[4] = 1e-39
    dt = 0.2 * min(b.dx)
    out, ref = GH.gpu_stage([b], P, dt, precision=G.GR_PREC_MIXED), GH.oracle_stage([b], P, dt)
    g, r = (GH.H.interior(x[0]["U"], b.n, b.ng) for x in (out, ref))
    d0 = GH.H.interior(GH.H.cons_from_prims(b, P, 2), b.n, b.ng)
    assert np.max(np.abs(r[0] / d0[0] - 1)) > 1e-4                       # the flux divergence moves D
    assert np.max(np.abs(g[0] - r[0]) / r[0]) < GH.MIXED_BOUNDS["random"]["D"]
    for v in (1, 2, 3):
        assert np.max(np.abs(g[v] - r[v]) / (r[0] + np.abs(r[4]))) < GH.MIXED_BOUNDS["random"]["S_x"]


@pytest.mark.parametrize("guess", [G.GR_GUESS_NONE, G.GR_GUESS_FP32])
def test_a_metric_with_a_subnormal_determinant(guess):
    P = GH.mixed_params(O.Params(gamma_ad=2.0, rho_atm=1e-14, tol=1e-10))
    b = I.random_block(n=(10, 8, 9), g=3, seed=29, metric_amp=0.02)
    det = b.metric[4] * b.metric[7] * b.metric[9]
    b.metric[4:10] *= (0.5 / det.max()) ** (1.0 / 3.0)                   # det(gamma) about 0.5
    dt = 0.1 * min(b.dx)
    ref = GH.oracle_stage([b], P, dt)
    # lengths in units of 2^-21: x = 2^21 x', so gamma 2^-42, u^i, beta^i and dx 2^21, sqrt(gamma) 2^-63
    L, sg = 2.0 ** 21, 2.0 ** -63
    s = I.random_block(n=b.n, g=3, seed=29, metric_amp=0.02)
    s.metric, s.W, s.B = b.metric.copy(), b.W.copy(), [f * (sg * L) for f in b.B]
    s.metric[1:4] *= L
    s.metric[4:10] *= L ** -2
    s.W[1:4] *= L
    s.dx = tuple(h * L for h in b.dx)
    U = GH.H.cons_from_prims(b, P, 2) * (sg * np.array([1, 1 / L, 1 / L, 1 / L, 1]))[:, None, None, None]
    assert np.float32(0.5 * L ** -6) < 2.0 ** -126
    out = GH.gpu_stage([s], P, dt, precision=G.GR_PREC_MIXED, U=[U], c2p_guess=guess)
    o = out[0]
    o["U"] = o["U"] / (sg * np.array([1, 1 / L, 1 / L, 1 / L, 1]))[:, None, None, None]
    o["W"][1:4] /= L
    o["B"] = [f / (sg * L) for f in o["B"]]
    # the variables that take one rounding of the flux (u~, p are ill-conditioned in it, and B^2 of an atmosphere cell
    # underflows in FP32 in these units); statuses equal: no cell fails
    bounds = {k: v for k, v in GH.MIXED_BOUNDS["random"].items() if k[0] in "DSB"}
    GH.check_mixed(out, ref, [b], bounds, "subnormal det(gamma)")
