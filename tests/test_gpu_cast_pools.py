"""A mixed stage that converts every pool it can need (table EOS, extrinsic curvature, no FP32 copies from the caller) gives
bitwise what it gives from the caller's own FP32 copies, and leaves its inputs untouched."""
import numpy as np
import pytest

import oracle as O
from paper_2311_04989_gb300 import grstage as G
from paper_2311_04989_gb300 import inputs as I
from tests import gpu_harness as GH

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [(16, 16, 16), (7, 10, 9)])
@pytest.mark.parametrize("table", [False, True])
def test_the_stage_from_its_own_conversions_and_from_copies(n, table):
    import torch
    kw, P = dict(), O.Params(gamma_ad=2.0, rho_atm=1e-14, tol=1e-10)
    if table:
        eos = I.SyntheticEOS()
        kw = dict(eos=eos, rho_range=(1e-8, 1e-3), T_range=(1e-3, 5e-2), ye_range=(0.05, 0.5), u_max=0.6, sigma_range=(1e-3, 1.0))
        P = O.Params(table=eos.table(), rho_atm=1e-12, T_atm=1e-4, tol=1e-10)
    b = I.random_block(n=n, g=3, seed=61, metric_amp=0.02, with_K=True, **kw)
    assert np.abs(b.metric[10:]).max() > 0
    P = GH.mixed_params(P)
    pools = GH.Pools([b])
    Ud = pools.cells([GH.H.cons_from_prims(b, P, P.interp_order)], P.nq)
    Wd, Bd, Md = pools.cells([b.W], P.nw), pools.faces([b.B]), pools.verts([b.metric])
    keep = [t.clone() for t in (Ud, Wd, Md, *Bd)]
    W32, B32, M32 = Wd[:6 if table else 5].float(), [x.float() for x in Bd], Md.float()
    mesh = G.gr_mesh_create(GH.ctx(), pools.L.descriptors())
    got = []
    try:
        for copies in (False, True):
            Uo, Wo, Bo = torch.zeros_like(Ud), torch.zeros_like(Wd), [torch.zeros_like(x) for x in Bd]
            st = torch.zeros(pools.L.ncell, dtype=torch.uint8, device="cuda")
            state = G.state_struct(Ud, Ud, Bd, Bd, Wd, Uo, Bo, Wo, st)
            if copies:
                G.set_fp32_copies(state, W32=W32, B32=B32)
            metric = G.metric_struct(Md, k_zero=False, metric32=M32 if copies else None)
            G.gr_stage(mesh, metric, state, 0.2 * min(b.dx), GH.gr_params_from(P, G.GR_PREC_MIXED))
            torch.cuda.synchronize()
            got.append([Uo, Wo, st, *Bo])
    finally:
        G.gr_mesh_destroy(mesh)
    for a, c in zip([Ud, Wd, Md, *Bd], keep):
        assert torch.equal(a, c)
    for a, c in zip(*got):
        assert torch.equal(a, c)
    assert (got[0][0] != 0).any()
