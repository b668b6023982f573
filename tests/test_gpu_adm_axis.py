"""The cell-to-vertex transfer of the matter sources in FP64, bit for bit: each axis adds its weighted cells from the low end with
one rounding per addition.  On a flat metric, with the gas cold and at rest and no field, rho_ADM of a cell is rho exactly."""
from fractions import Fraction

import numpy as np
import pytest

import oracle as O
from paper_2311_04989_gb300 import grstage as G
from paper_2311_04989_gb300 import inputs as I
from tests import gpu_harness as GH

pytestmark = pytest.mark.gpu
WEIGHTS = {2: (Fraction(1, 2),) * 2, 4: (Fraction(-1, 16), Fraction(9, 16), Fraction(9, 16), Fraction(-1, 16))}


def _axis(a, axis, w):
    a = np.moveaxis(a, axis, -1)
    out = np.empty(a.shape[:-1] + (a.shape[-1] - len(w) + 1,))
    for i in np.ndindex(out.shape):
        s = 0.0
        for q, wq in enumerate(w):
            s = float(Fraction(s) + wq * Fraction(float(a[i[:-1] + (i[-1] + q,)])))
        out[i] = s
    return np.moveaxis(out, -1, axis)


@pytest.mark.parametrize("vc", [2, 4])
@pytest.mark.parametrize("n", [(5, 4, 6), (9, 3, 4)])
def test_vertex_values_are_the_axis_sums_from_the_low_end(vc, n):
    import torch
    b = I.random_block(n=n, g=3, seed=47, flat=True)
    b.W[:] = 0.0
    b.W[0] = np.exp(np.random.default_rng(2).uniform(-20, 0, b.W[0].shape))
    b.B = [np.zeros_like(f) for f in b.B]
    pools = GH.Pools([b])
    out = torch.zeros((10, pools.L.nvert), dtype=torch.float64, device="cuda")
    Wd, Bd, Md = pools.cells([b.W], 5), pools.faces([b.B]), pools.verts([b.metric])
    mesh = G.gr_mesh_create(GH.ctx(), pools.L.descriptors())
    try:
        G.gr_adm_sources(mesh, G.metric_struct(Md), list(Wd), Bd, GH.gr_params_from(O.Params(gamma_ad=2.0)), vc, list(out))
        torch.cuda.synchronize()
    finally:
        G.gr_mesh_destroy(mesh)
    N = [v + 2 * b.ng + 1 for v in n[::-1]]
    off = int(pools.L.vert_off[0])
    got = out[0].cpu().numpy()[off:off + N[0] * N[1] * N[2]].reshape(N)
    got = got[tuple(slice(b.ng, b.ng + v + 1) for v in n[::-1])]
    r = vc // 2
    a = b.W[0][tuple(slice(b.ng - r, b.ng + v + r) for v in n[::-1])]
    for axis in (2, 1, 0):
        a = _axis(a, axis, WEIGHTS[vc])
    assert np.array_equal(got, a)
