"""What decides con2prim's form in a mixed stage is the parameters alone: a driver step is bitwise the stages it is made of, and
the proposal that gr_autotune picks for GR_GUESS_AUTO is one of two solves that differ in time."""
import pytest

import oracle as O
from paper_2311_04989_gb300 import grstage as G
from paper_2311_04989_gb300 import inputs as I
from tests import gpu_harness as GH

pytestmark = pytest.mark.gpu

RK = {2: [(0.0, 1.0, 1.0), (0.5, 0.5, 0.5)],
      3: [(0.0, 1.0, 1.0), (0.75, 0.25, 0.25), (1.0 / 3.0, 2.0 / 3.0, 2.0 / 3.0)]}


def _pools(blocks, P):
    p = GH.Pools(blocks)
    U = p.cells([GH.H.cons_from_prims(b, P, P.interp_order) for b in blocks], P.nq)
    return p, U, p.cells([b.W for b in blocks], P.nw), p.faces([b.B for b in blocks]), p.verts([b.metric for b in blocks])


@pytest.mark.parametrize("precision", [G.GR_PREC_MIXED, G.GR_PREC_FP64])
@pytest.mark.parametrize("guess", [G.GR_GUESS_NONE, G.GR_GUESS_FP32])
@pytest.mark.parametrize("table,rk", [(False, 3), (False, 2), (True, 3)])
def test_a_driver_step_is_the_stages_it_is_made_of(precision, guess, table, rk):
    import torch
    kw, P = dict(rho_range=(1e-8, 1e-3)), O.Params(gamma_ad=2.0, rho_atm=1e-9, tol=1e-10)
    if table:
        eos = I.SyntheticEOS()
        kw = dict(eos=eos, rho_range=(1e-8, 1e-3), T_range=(1e-3, 5e-2), ye_range=(0.05, 0.5))
        P = O.Params(table=eos.table(), rho_atm=1e-9, T_atm=1e-4, tol=1e-10)
    P = GH.mixed_params(P)
    blocks = [I.random_block(n=(12, 10, 14), g=3, seed=80 + k, u_max=0.5, metric_amp=0.02, **kw) for k in range(4)]
    pools, U, W, B, M = _pools(blocks, P)
    metric = G.metric_struct(M)
    gp = GH.gr_params_from(P, precision, guess)
    mesh = G.gr_mesh_create(GH.ctx(), pools.L.descriptors())
    drv = G.gr_driver_create(mesh, I.block_grid_neighbours((2, 2, 1)))
    try:
        Us, Ws, Bs = U.clone(), W.clone(), [b.clone() for b in B]
        st = torch.zeros(pools.L.ncell, dtype=torch.uint8, device="cuda")
        G.gr_driver_step(drv, metric, list(Us), list(Ws), Bs, st, gp, 0.2, G.GR_DT_GRID, rk)
        torch.cuda.synchronize()
        dt = G.gr_driver_dt(drv)
        G.gr_ghost_fill(drv, list(W), B)
        iU, iW, iB = U, W, B
        for s, (g0, g1, beta) in enumerate(RK[rk]):
            oU, oW, oB = torch.zeros_like(U), torch.zeros_like(W), [torch.zeros_like(b) for b in B]
            so = torch.zeros_like(st)
            gp.rk_g0, gp.rk_g1, gp.rk_beta = g0, g1, beta
            G.gr_stage(mesh, metric, G.state_struct(iU, U, iB, B, iW, oU, oB, oW, so), dt, gp)
            if s + 1 < rk:
                G.gr_ghost_fill(drv, list(oW), oB)
            torch.cuda.synchronize()
            iU, iW, iB = oU, oW, oB
    finally:
        G.gr_driver_destroy(drv)
        G.gr_mesh_destroy(mesh)
    g = slice(3, -3)
    for nv, a, b in ((P.nq, Us, iU), (P.nw, Ws, iW), (1, st, so)):
        for x, y in zip(pools.unpack_cells(a, nv), pools.unpack_cells(b, nv)):
            assert (x[..., g, g, g] == y[..., g, g, g]).all()
    for x, y in zip(pools.unpack_faces(Bs), pools.unpack_faces(iB)):
        for d in range(3):   # the faces of interior cells
            assert (x[d][g, g, g] == y[d][g, g, g]).all()


def test_auto_takes_the_pre_solve_on_a_batch_of_matter():
    """All cells matter: the FP32 pre-solve saves half the FP64 evaluations there, far more than timings scatter."""
    import torch
    blocks = [I.random_block(n=(24, 24, 24), g=3, seed=5, metric_amp=0.02)] * 64
    P = GH.mixed_params(O.Params(gamma_ad=2.0, rho_atm=1e-14, tol=1e-10))
    pools, U, W, B, M = _pools(blocks, P)
    st = torch.zeros(pools.L.ncell, dtype=torch.uint8, device="cuda")
    state = G.state_struct(U, U, B, B, W, torch.zeros_like(U), [torch.zeros_like(b) for b in B], torch.zeros_like(W), st)
    gp = GH.gr_params_from(P, G.GR_PREC_MIXED, G.GR_GUESS_AUTO)
    for _ in range(4):
        mesh = G.gr_mesh_create(GH.ctx(), pools.L.descriptors())
        try:
            G.gr_autotune(mesh, G.metric_struct(M), state, 0.1 * min(blocks[0].dx), gp, 3)
            assert G.gr_mesh_get_guess(mesh, G.GR_PREC_MIXED, 0) == G.GR_GUESS_FP32
        finally:
            G.gr_mesh_destroy(mesh)
