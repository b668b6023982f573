"""The cell preparation cuts its walk along z on a mesh of few tiles: a lone block (cut down to single planes) gives
bitwise the results it has as one of many (not cut), in both precisions, for odd sizes and for more than one tile."""
import numpy as np
import pytest

import oracle as O
from paper_2311_04989_gb300 import grstage as G
from paper_2311_04989_gb300 import inputs as I
from tests import gpu_harness as GH

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", [G.GR_PREC_FP64, G.GR_PREC_MIXED])
@pytest.mark.parametrize("n,copies", [((3, 4, 5), 960), ((30, 7, 6), 480)])
def test_lone_block_matches_the_same_block_in_a_large_mesh(n, copies, precision):
    P = O.Params(gamma_ad=2.0, rho_atm=1e-14, recon=1)
    b = I.random_block(n=n, g=3, seed=77)
    U = GH.H.cons_from_prims(b, P, P.interp_order)
    one = GH.gpu_stage([b], P, dt=0.1 * min(b.dx), precision=precision, U=[U])[0]
    many = GH.gpu_stage([b] * copies, P, dt=0.1 * min(b.dx), precision=precision, U=[U] * copies)
    for k in (0, copies - 1):
        for key in ("U", "W", "status"):
            assert np.array_equal(one[key], many[k][key])
        for d in range(3):
            assert np.array_equal(one["B"][d], many[k]["B"][d])
