"""One FP64 sqrt(gamma): the reset of an atmosphere cell in the FP64 stage, its reset in gr_con2prim and the conserved density
gr_prim2con gives the same state at rest are the same bits, D = sqrt(gamma) rho_atm, and the stage with no atmosphere band agrees
with gr_con2prim on which cells lie below a threshold set on that very value."""
import numpy as np
import pytest

import oracle as O
from paper_2311_04989_gb300 import grstage as G
from paper_2311_04989_gb300 import inputs as I
from tests import gpu_harness as GH

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("order", [2, 4])
@pytest.mark.parametrize("n", [(16, 16, 16), (9, 5, 11)])
def test_atmosphere_density_is_the_same_bits_everywhere(order, n):
    import torch
    P = O.Params(gamma_ad=2.0, rho_atm=1.37e-6, tol=1e-14, interp_order=order, atm_band=0.0)
    b = I.random_block(n=n, g=4 if order == 4 else 3, seed=17, metric_amp=0.1)
    b.B = [np.zeros_like(f) for f in b.B]
    b.W[1:4] = 0.0
    b.W[0], b.W[4] = P.rho_atm, 1e-10
    pools = GH.Pools([b])
    Wd, Bd, Md = pools.cells([b.W], 5), pools.faces([b.B]), pools.verts([b.metric])
    metric, gp = G.metric_struct(Md, order=order), GH.gr_params_from(P)
    mesh = G.gr_mesh_create(GH.ctx(), pools.L.descriptors())
    st = torch.zeros(pools.L.ncell, dtype=torch.uint8, device="cuda")

    def inner(t, nv=5):
        return GH.H.interior(pools.unpack_cells(t, nv)[0], n, b.ng)

    def stage(U):
        Uo, Wo, Bo = torch.zeros_like(U), torch.zeros_like(U), [torch.zeros_like(f) for f in Bd]
        G.gr_stage(mesh, metric, G.state_struct(U, U, Bd, Bd, Wd, Uo, Bo, Wo, st), 0.0, gp)
        torch.cuda.synchronize()
        return inner(Uo), inner(st, 1)

    try:
        Up = torch.zeros_like(Wd)
        G.gr_prim2con(mesh, metric, list(Wd), Bd, list(Up), gp)
        low = Up.clone()
        low[0] *= 0.5                                       # below the threshold everywhere
        Uc, Wc = low.clone(), torch.zeros_like(Wd)
        G.gr_con2prim(mesh, metric, list(Uc), Bd, list(Wc), st, gp)
        torch.cuda.synchronize()
        assert (inner(st, 1) == G.GR_ST_ATM_THRESHOLD).all()
        Us, ss = stage(low)
        assert (ss == G.GR_ST_ATM_THRESHOLD).all()
        assert np.array_equal(inner(Uc)[0], inner(Up)[0])   # prim2con and con2prim
        assert np.array_equal(Us[0], inner(Uc)[0])          # the stage and con2prim
        # cells on the threshold and one ulp to either side: the same status by both
        at = Up.clone()
        d = pools.unpack_cells(at, 5)[0][0]
        up, dn = np.nextafter(d, 1.0), np.nextafter(d, 0.0)
        k = np.arange(d.size).reshape(d.shape) % 3
        at[0, :d.size] = torch.from_numpy(np.where(k == 0, d, np.where(k == 1, up, dn)).ravel()).cuda()
        _, ss = stage(at)
        Uc = at.clone()
        G.gr_con2prim(mesh, metric, list(Uc), Bd, list(Wc), st, gp)
        torch.cuda.synchronize()
        assert np.array_equal(ss, inner(st, 1))
    finally:
        G.gr_mesh_destroy(mesh)
