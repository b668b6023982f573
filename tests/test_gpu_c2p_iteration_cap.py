"""gr_params.max_iter caps the root find of the mixed stage in each of its forms: with one iteration no cell of a batch of
matter converges and every one is reported as failed, as by the oracle; with the default none is."""
import numpy as np
import pytest

import oracle as O
from paper_2311_04989_gb300 import grstage as G
from paper_2311_04989_gb300 import inputs as I
from tests import gpu_harness as GH

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("guess", [G.GR_GUESS_NONE, G.GR_GUESS_FP32])
@pytest.mark.parametrize("max_iter", [1, 100])
@pytest.mark.parametrize("table", [False, True])
def test_the_iteration_cap_holds(guess, max_iter, table):
    kw, P = dict(rho_range=(1e-8, 1e-3)), O.Params(gamma_ad=2.0, rho_atm=1e-14, tol=1e-10, max_iter=max_iter)
    if table:
        eos = I.SyntheticEOS()
        kw = dict(eos=eos, rho_range=(1e-8, 1e-3), T_range=(1e-3, 5e-2), ye_range=(0.05, 0.5))
        P = O.Params(table=eos.table(), rho_atm=1e-12, T_atm=1e-4, tol=1e-10, max_iter=max_iter)
    P = GH.mixed_params(P)
    b = I.random_block(n=(9, 8, 7), g=3, seed=37, u_max=0.5, metric_amp=0.02, sigma_range=(1e-3, 1.0), **kw)
    dt = 0.1 * min(b.dx)
    got, ref = GH.gpu_stage([b], P, dt, precision=G.GR_PREC_MIXED, c2p_guess=guess)[0], GH.oracle_stage([b], P, dt)[0]
    s, r = (GH.H.interior(x["status"], b.n, b.ng) & G.GR_ST_FAILED != 0 for x in (got, ref))
    assert np.array_equal(s, r)
    assert r.all() if max_iter == 1 else not r.any()
