"""gr_con2prim's first pass queues cells on an FP32 bound: cells straddling the atmosphere threshold by factors from 1e-6
to 10, on metrics from flat to strongly non-diagonal and of very different scale, end with the oracle's status and
primitives."""
import numpy as np
import pytest

import oracle as O
from paper_2311_04989_gb300 import grstage as G
from paper_2311_04989_gb300 import inputs as I
from tests import gpu_harness as GH

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("scale", [1.0, 1e-6, 1e9])
@pytest.mark.parametrize("n", [(5, 4, 3), (17, 8, 9)])
def test_cells_around_the_threshold_match_the_oracle(n, scale):
    import torch
    rng = np.random.default_rng(5)
    P = O.Params(gamma_ad=2.0, rho_atm=1e-6, tol=1e-14)
    b = I.random_block(n=n, g=1, seed=9, rho_range=(1e-3, 1e-2), metric_amp=0.0)
    b.metric[4:10] = scale * np.array([1.0, 0.55, 0.2, 1.3, 0.6, 0.9])[:, None, None, None]   # positive definite
    b.B = [np.zeros_like(f) for f in b.B]
    b.W[1:4] = 0.0
    # D from threshold (1 +- small) to factors of ten around it
    f = np.exp(rng.uniform(np.log(0.1), np.log(10.0), b.W[0].shape))
    near = rng.random(f.shape) < 0.5
    f[near] = 1 + rng.choice([-1.0, 1.0], near.sum()) * 10.0 ** rng.uniform(-6, -2, near.sum())
    b.W[0] = P.rho_atm * f
    b.W[4] = 0.1 * b.W[0]
    U = GH.H.cons_from_prims(b, P, P.interp_order)
    pools = GH.Pools([b])
    Ud = pools.cells([U], 5)
    Wd = torch.zeros_like(Ud)
    Bd, Md = pools.faces([b.B]), pools.verts([b.metric])
    st = torch.zeros(pools.L.ncell, dtype=torch.uint8, device="cuda")
    mesh = G.gr_mesh_create(GH.ctx(), pools.L.descriptors())
    try:
        G.gr_con2prim(mesh, G.metric_struct(Md), list(Ud), Bd, list(Wd), st, GH.gr_params_from(P))
        torch.cuda.synchronize()
    finally:
        G.gr_mesh_destroy(mesh)
    sl = tuple(slice(1, 1 + n[a]) for a in (2, 1, 0))
    W, S = pools.unpack_cells(Wd, 5)[0][(slice(None),) + sl], pools.unpack_cells(st, 1)[0][sl]
    atm = f[sl] < 1 + 1e-12
    assert np.array_equal((S & G.GR_ST_ATM_THRESHOLD) != 0, atm) and 0 < atm.sum() < atm.size
    np.testing.assert_allclose(W[0], np.where(atm, P.rho_atm, b.W[0][sl]), rtol=1e-9)
    np.testing.assert_allclose(W[4][~atm], b.W[4][sl][~atm], rtol=1e-7)
