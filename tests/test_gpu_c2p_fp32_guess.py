"""gr_con2prim with the FP32 pre-solve (ideal gas): statuses and FP64 evaluation counts, which hang on the pre-solve's bracket, are
the recorded ones (tests/golden/c2p_fp32_guess.json: the library's own integers, before any FP32 division of the solve was
replaced) over magnetisations, Lorentz factors, tolerances and iteration caps from mild to extreme."""
import json
import os
import zlib

import numpy as np
import pytest

import oracle as O
from paper_2311_04989_gb300 import grstage as G
from paper_2311_04989_gb300 import inputs as I
from tests import gpu_harness as GH

pytestmark = pytest.mark.gpu
GOLDEN = os.path.join(os.path.dirname(os.path.abspath(__file__)), "golden", "c2p_fp32_guess.json")
CASES = [dict(), dict(tol=1e-14), dict(u_max=30.0, W_max=1e4), dict(sigma=1e4, M_max=1e8, gamma=5.0 / 3.0),
         dict(tol=1e-6, max_iter=3), dict(tol=1e-15, max_iter=5, u_max=3.0), dict(theta=10.0, gamma=4.0 / 3.0)]


def measure(tol=1e-10, max_iter=100, u_max=0.5, W_max=20.0, M_max=1e4, sigma=10.0, theta=0.1, gamma=2.0):
    import torch
    P = O.Params(gamma_ad=gamma, rho_atm=1e-14, tol=tol, max_iter=max_iter, W_max=W_max, M_max=M_max)
    b = I.random_block(n=(16, 15, 14), g=1, seed=53, u_max=u_max, sigma_range=(1e-3, sigma), theta_range=(1e-3, theta), metric_amp=0.02)
    pools = GH.Pools([b])
    Ud = pools.cells([GH.H.cons_from_prims(b, P, 2)], 5)
    Wd, Bd, Md = torch.zeros_like(Ud), pools.faces([b.B]), pools.verts([b.metric])
    st = torch.zeros(pools.L.ncell, dtype=torch.uint8, device="cuda")
    ev = torch.zeros(pools.L.ncell, dtype=torch.int32, device="cuda")
    mesh = G.gr_mesh_create(GH.ctx(), pools.L.descriptors())
    try:
        G.gr_con2prim(mesh, G.metric_struct(Md), list(Ud), Bd, list(Wd), st, GH.gr_params_from(P, c2p_guess=G.GR_GUESS_FP32), evals=ev)
        torch.cuda.synchronize()
    finally:
        G.gr_mesh_destroy(mesh)
    s, e = (np.ascontiguousarray(GH.H.interior(pools.unpack_cells(t, 1)[0], b.n, b.ng)) for t in (st, ev))
    return {"status": {str(k): int(v) for k, v in zip(*np.unique(s, return_counts=True))},
            "evals": {str(k): int(v) for k, v in zip(*np.unique(e, return_counts=True))},
            "crc": zlib.crc32(s.tobytes() + e.astype("<i4").tobytes())}


@pytest.mark.parametrize("k", range(len(CASES)))
def test_statuses_and_evaluations_are_the_recorded_ones(k):
    assert measure(**CASES[k]) == json.load(open(GOLDEN))[k]
