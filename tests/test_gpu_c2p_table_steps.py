"""gr_con2prim with the table: statuses and FP64 evaluation counts are the recorded ones (tests/golden/c2p_table_steps.json: the
library's own integers, before its divisions became integer arithmetic), without a proposal and with the FP32 pre-solve, from
mild states to tight tolerances and iteration caps."""
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
GOLDEN = os.path.join(os.path.dirname(os.path.abspath(__file__)), "golden", "c2p_table_steps.json")
CASES = [dict(guess=g, **kw) for g in (G.GR_GUESS_NONE, G.GR_GUESS_FP32)
         for kw in (dict(), dict(tol=1e-14), dict(u_max=3.0, sigma=1e3), dict(tol=1e-14, max_iter=6), dict(tol=1e-6, max_iter=3, u_max=3.0))]


def measure(guess, tol=1e-10, max_iter=100, u_max=0.5, sigma=10.0):
    import torch
    eos = I.SyntheticEOS()
    P = O.Params(table=eos.table(), rho_atm=1e-12, T_atm=1e-5, tol=tol, max_iter=max_iter)
    b = I.random_block(n=(16, 15, 14), g=1, seed=59, u_max=u_max, sigma_range=(1e-3, sigma), metric_amp=0.02, eos=eos,
                       rho_range=(1e-11, 1e-2), T_range=(1e-4, 5e-2), ye_range=(0.05, 0.5))
    pools = GH.Pools([b])
    Ud = pools.cells([GH.H.cons_from_prims(b, P, 2)], 6)
    Bd, Md = pools.faces([b.B]), pools.verts([b.metric])
    Wd = torch.zeros((7, Ud.shape[1]), dtype=torch.float64, device="cuda")
    st = torch.zeros(pools.L.ncell, dtype=torch.uint8, device="cuda")
    ev = torch.zeros(pools.L.ncell, dtype=torch.int32, device="cuda")
    mesh = G.gr_mesh_create(GH.ctx(), pools.L.descriptors())
    try:
        G.gr_con2prim(mesh, G.metric_struct(Md), list(Ud), Bd, list(Wd), st, GH.gr_params_from(P, c2p_guess=guess), evals=ev)
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
