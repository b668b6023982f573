"""gr_con2prim on cells whose metric is not positive definite: the comparisons with a threshold that is not a number, or with a
negative tau floor, give the oracle's status."""
import numpy as np
import pytest

import oracle as O
from paper_2311_04989_gb300 import grstage as G
from paper_2311_04989_gb300 import inputs as I
from tests import gpu_harness as GH

pytestmark = pytest.mark.gpu
H = GH.H


@pytest.mark.parametrize("guess", [G.GR_GUESS_NONE, G.GR_GUESS_FP32])
@pytest.mark.parametrize("sign", [(-1.0, 1.0, 1.0), (-1.0, -1.0, 1.0)])   # det(gamma) < 0; > 0 with B^2 of either sign
def test_status_on_an_indefinite_metric_is_the_oracles(sign, guess):
    import torch
    P = O.Params(gamma_ad=2.0, rho_atm=1e-9, tol=1e-14)
    b = I.random_block(n=(9, 6, 5), g=3, seed=31, rho_range=(1e-6, 1e-3), metric_amp=0.0)
    for c, s in zip((4, 7, 9), sign):
        b.metric[c] *= s
    rng = np.random.default_rng(3)
    U = np.abs(b.W[:5]) * 1.0
    U[0] = b.W[0]
    U[0][rng.random(U[0].shape) < 0.3] *= -1.0                              # negative D
    U[1:4] = 0.01 * b.W[0] * rng.uniform(-1, 1, U[1:4].shape)
    U[4] = b.W[0] * rng.uniform(-1, 1, U[4].shape) * 10.0 ** rng.uniform(-6, 0, U[4].shape)   # tau around B^2 / 2
    pools = GH.Pools([b])
    Ud, Bd, Md = pools.cells([U], 5), pools.faces([b.B]), pools.verts([b.metric])
    Wd = torch.zeros((5, Ud.shape[1]), dtype=torch.float64, device="cuda")
    st = torch.zeros(pools.L.ncell, dtype=torch.uint8, device="cuda")
    mesh = G.gr_mesh_create(GH.ctx(), pools.L.descriptors())
    try:
        G.gr_con2prim(mesh, G.metric_struct(Md), list(Ud), Bd, list(Wd), st, GH.gr_params_from(P, c2p_guess=guess))
        torch.cuda.synchronize()
    finally:
        G.gr_mesh_destroy(mesh)
    n, g = b.n, b.ng
    cm, cb = H.cell_metric(b), H.cell_B(b)
    met = cm[g:g + n[2], g:g + n[1], g:g + n[0]].reshape(-1, 16)
    bd = cb[g:g + n[2], g:g + n[1], g:g + n[0]].reshape(-1, 3)
    _, _, ref, _ = O.con2prim(met, np.moveaxis(H.interior(U, n, g), 0, -1).reshape(-1, 5), bd, P)
    got = H.interior(pools.unpack_cells(st, 1)[0], n, g).reshape(-1) & 0x3F
    assert np.array_equal(got, ref), (np.unique(got[got != ref]), np.unique(ref[got != ref]))
