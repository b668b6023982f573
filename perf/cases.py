"""Workloads of the GRMHD stage library as a program runs them, through its public entry points.

Each case is a dict of plain values.  `prepare` makes the seeded inputs on the GPU together with what such a
program keeps (context, mesh, EOS table, driver), `run` is one pass through the library, `exact` is the same pass in
plain torch FP64 without the library, and `work` counts the bytes and operations a pass cannot do without.

kind      entry point               what a pass is
stage     gr_stage                  one Runge-Kutta stage of a batch of MeshBlocks
step      gr_driver_step            one SSP-RK time step of a periodic grid of blocks (ghost exchange included)
con2prim  gr_con2prim               conserved -> primitive of a batch of blocks
prim2con  gr_prim2con               primitive -> conserved (initial data)
adm       gr_adm_sources            matter sources of the spacetime equations at the vertices
"""
from __future__ import annotations

import functools
import math

import numpy as np
import torch

from paper_2311_04989_gb300 import grstage as G
from paper_2311_04989_gb300 import inputs as I

F64 = torch.float64
RECON = {"plm": G.GR_RECON_PLM, "wenoz": G.GR_RECON_WENOZ, "weno5": G.GR_RECON_WENO5, "ppm": G.GR_RECON_PPM}


def _dev():
    return torch.device("cuda" if torch.cuda.is_available() else "cpu")


# ---------------------------------------------------------------------------------------------------------------
# cases
# ---------------------------------------------------------------------------------------------------------------
def _case(kind, **kw):
    c = dict(kind=kind, inputs="random", nb=1, nx=16, ny=16, nz=16, g=3, mix=False, precision="mixed", eos="ideal",
             recon="wenoz", order=2, K=False, copies=False, rk_mid=False, emf="upwind", guess="none", tune=False,
             gamma=2.0, vc_order=2, rk_order=3, gx=1, gy=1, gz=1)
    c.update(kw)
    return c


def listed():
    L = []
    # the smallest call: the magnetised shock tube on one 16^3 block (a convergence test's inner loop; launches count)
    L.append(_case("stage", name="tube_16_mixed", inputs="tube", recon="plm", gamma=5.0 / 3.0))
    # one magnetised star on one 64^3 block, the single-star set-up: too few blocks to fill the GPU
    L.append(_case("stage", name="star_64_mixed", inputs="star", nx=64, ny=64, nz=64, copies=True, tune=True))
    # the headline: two stars on 4096 blocks of 16^3, the steady state of an evolution (FP32 copies chained)
    L.append(_case("stage", name="stars_4096_mixed", inputs="stars", nb=4096, copies=True, tune=True))
    # a batch of uneven blocks at three refinement levels, all matter: con2prim does real work in every cell
    L.append(_case("stage", name="amr_256_mixed", nb=256, mix=True, copies=True, tune=True, guess="fp32",
                   gamma=5.0 / 3.0))
    # the same kind of batch on the plain FP64 path, the accuracy reference of a study
    L.append(_case("stage", name="amr_48_fp64", nb=48, mix=True, precision="fp64", gamma=5.0 / 3.0))
    # a lone ragged block in FP64: a debugging or convergence run
    L.append(_case("stage", name="block_fp64", nx=20, ny=17, nz=24, precision="fp64", recon="weno5"))
    # evolution: a whole RK3 step of a periodic box of 8^3 blocks, ghost exchange and FP32 copies inside
    L.append(_case("step", name="rk3_512_mixed", nb=512, gx=8, gy=8, gz=8))
    # fourth-order metric interpolation with extrinsic curvature: the accurate set-up of a dynamical spacetime
    L.append(_case("stage", name="order4_K_mixed", nb=64, nx=24, ny=24, nz=24, g=4, order=4, K=True, copies=True,
                   guess="fp32"))
    # a nuclear (tabulated) equation of state in a mixed stage
    L.append(_case("stage", name="table_64_mixed", nb=64, nx=24, ny=24, nz=24, eos="table", guess="fp32"))
    # con2prim on its own (after a regrid, or a code that has its own fluxes), ideal gas
    L.append(_case("con2prim", name="c2p_ideal", nb=64, nx=32, ny=32, nz=32, g=1, precision="fp64"))
    # con2prim with the table over wide magnetisation and Lorentz-factor ranges
    L.append(_case("con2prim", name="c2p_table", nb=32, nx=32, ny=32, nz=32, g=1, precision="fp64", eos="table",
                   guess="fp32"))
    # matter sources for the spacetime solver, fourth-order transfer
    L.append(_case("adm", name="adm_512_fp64", nb=512, precision="fp64", vc_order=4))
    return L


def draw(rng):
    kind = rng.choices(["stage", "step", "con2prim", "prim2con", "adm"], [58, 14, 12, 4, 12])[0]

    def log(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    def size():
        return rng.choice([16, 24, 32]) if rng.random() < 0.4 else log(8, 44)

    gamma = rng.choice([2.0, 5.0 / 3.0, 4.0 / 3.0])
    precision = "mixed" if rng.random() < 0.65 else "fp64"
    guess = rng.choice(["none", "fp32"])
    eos = "table" if rng.random() < 0.2 else "ideal"
    n = [size()] * 3 if rng.random() < 0.5 else [size(), size(), size()]
    vol = n[0] * n[1] * n[2]
    if kind == "stage":
        # cells a pass updates at most: below the listed cases' times on either path
        cap = {("mixed", "ideal"): 4_000_000, ("mixed", "table"): 700_000, ("fp64", "ideal"): 450_000,
               ("fp64", "table"): 150_000}[precision, eos]
        cells = log(4096, cap)
        order = 4 if rng.random() < 0.2 else 2
        mixed = precision == "mixed"
        return _case("stage", nb=max(1, cells // vol), nx=n[0], ny=n[1], nz=n[2], g=4 if order == 4 else 3,
                     precision=precision, eos=eos, recon=rng.choices(["wenoz", "plm", "weno5", "ppm"], [55, 20, 15, 10])[0],
                     order=order, K=rng.random() < 0.4, copies=mixed and rng.random() < 0.6, rk_mid=rng.random() < 0.5,
                     emf="mean" if rng.random() < 0.15 else "upwind", guess=guess, gamma=gamma)
    if kind == "step":
        cap = 2_500_000 if precision == "mixed" else 150_000
        m = [rng.randint(1, 6) for _ in range(3)]
        while m[0] * m[1] * m[2] * vol > cap and max(m) > 1:
            m[m.index(max(m))] -= 1
        while vol > cap:
            n = [max(8, v // 2) for v in n]
            vol = n[0] * n[1] * n[2]
        return _case("step", nb=m[0] * m[1] * m[2], gx=m[0], gy=m[1], gz=m[2], nx=n[0], ny=n[1], nz=n[2],
                     precision=precision, recon=rng.choices(["wenoz", "plm"], [75, 25])[0], gamma=gamma,
                     guess=guess, rk_order=rng.choice([2, 3, 3]))
    if kind == "con2prim":
        cells = log(8192, 2_000_000 if eos == "ideal" else 1_000_000)
        return _case("con2prim", nb=max(1, cells // vol), nx=n[0], ny=n[1], nz=n[2], g=1, precision="fp64", eos=eos,
                     guess=guess, gamma=gamma)
    if kind == "prim2con":
        return _case("prim2con", nb=max(1, log(8192, 2_000_000) // vol), nx=n[0], ny=n[1], nz=n[2], g=1,
                     precision="fp64", eos="ideal", gamma=gamma)
    vc = rng.choice([2, 4])
    return _case("adm", nb=max(1, log(8192, 2_000_000) // vol), nx=n[0], ny=n[1], nz=n[2], precision=precision,
                 vc_order=vc, gamma=gamma)


# ---------------------------------------------------------------------------------------------------------------
# geometry: blocks of one shape are consecutive, so a pool of them is one strided view (block, z, y, x)
# ---------------------------------------------------------------------------------------------------------------
class _Blk:
    def __init__(self, n, ng, dx, x0):
        self.n, self.ng, self.dx, self.x0 = tuple(n), ng, tuple(dx), tuple(x0)


def _blocks(case, seed):
    rng = np.random.default_rng(seed * 7919 + 11)
    g, nb = case["g"], case["nb"]
    if case["inputs"] == "stars":
        k = round(nb ** (1 / 3))
        n = case["nx"]
        dx = 64.0 / (k * n)
        return [_Blk((n,) * 3, g, (dx,) * 3, tuple(-32.0 + o * n * dx for o in (b % k, (b // k) % k, b // (k * k))))
                for b in range(k ** 3)]
    n = (case["nx"], case["ny"], case["nz"])
    if case["inputs"] == "star":
        dx = 2 * 10.02 / n[0]
        return [_Blk(n, g, (dx,) * 3, (-10.02,) * 3)]
    if case["inputs"] == "tube":
        dx = 1.0 / n[0]
        return [_Blk(n, g, (dx,) * 3, (-0.5, 0.0, 0.0))]
    if case["kind"] == "step":   # a periodic unit box cut into gx x gy x gz blocks
        m = (case["gx"], case["gy"], case["gz"])
        dx = tuple(1.0 / (m[a] * n[a]) for a in range(3))
        return [_Blk(n, g, dx, (bx * n[0] * dx[0], by * n[1] * dx[1], bz * n[2] * dx[2]))
                for bz in range(m[2]) for by in range(m[1]) for bx in range(m[0])]
    if case["mix"]:
        ns = [16] * (nb - 2 * (nb // 3)) + [24] * (nb // 3) + [32] * (nb // 3)
        shapes = [(v,) * 3 for v in ns]
    else:
        shapes = [n] * nb
    out = []
    for s in shapes:
        h = (1.0 / 64) / 2 ** int(rng.integers(0, 3))
        out.append(_Blk(s, g, (h,) * 3, tuple(rng.uniform(0, 1 - max(s) * h, 3))))
    return out


def _groups(blocks):
    """[(first, count)] of runs of equal shapes."""
    out, i = [], 0
    while i < len(blocks):
        j = i
        while j < len(blocks) and blocks[j].n == blocks[i].n:
            j += 1
        out.append((i, j - i))
        i = j
    return out


def _up(x, a=32):
    return -(-x // a) * a


class _Pools:
    """Extents of the pools (the library's packing) and the strided views of a group of blocks."""

    def __init__(self, blocks):
        self.blocks, self.groups = blocks, _groups(blocks)
        self.L = G.Layout.of(blocks)

    def shape(self, i, stag):
        b = self.blocks[i]
        return tuple(b.n[a] + 2 * b.ng + stag[a] for a in (2, 1, 0))

    def view(self, pool, grp, stag=(0, 0, 0)):
        i, m = grp
        s = self.shape(i, stag)
        if stag == (0, 0, 0):
            off = int(self.L.cell_off[i])
        elif stag == (1, 1, 1):
            off = int(self.L.vert_off[i])
        else:
            off = int(self.L.face_off[i, stag.index(1)])
        st = _up(s[0] * s[1] * s[2])
        return pool.as_strided((m,) + s, (st, s[1] * s[2], s[2], 1), pool.storage_offset() + off)

    def cells(self, rows, dtype=F64):
        return torch.zeros((rows, self.L.ncell), dtype=dtype, device=_dev())

    def faces(self, dtype=F64):
        return [torch.zeros(self.L.nface[d], dtype=dtype, device=_dev()) for d in range(3)]

    def verts(self, rows):
        return torch.zeros((rows, self.L.nvert), dtype=F64, device=_dev())

    def axes(self, grp, stag):
        """Coordinates X, Y, Z of a group, broadcastable to (block, z, y, x)."""
        i, m = grp
        out = []
        for a in range(3):
            b0 = self.blocks[i]
            k = torch.arange(-b0.ng, b0.n[a] + b0.ng + stag[a], dtype=F64, device=_dev()) + (0.0 if stag[a] else 0.5)
            x0 = torch.tensor([self.blocks[j].x0[a] for j in range(i, i + m)], dtype=F64, device=_dev())
            dx = torch.tensor([self.blocks[j].dx[a] for j in range(i, i + m)], dtype=F64, device=_dev())
            v = x0[:, None] + k[None, :] * dx[:, None]
            out.append(v[:, None, None, :] if a == 0 else (v[:, None, :, None] if a == 1 else v[:, :, None, None]))
        return out

    def dx(self, grp, a):
        i, m = grp
        return torch.tensor([self.blocks[j].dx[a] for j in range(i, i + m)], dtype=F64, device=_dev())[:, None, None, None]


STAG = {"c": (0, 0, 0), "v": (1, 1, 1), 0: (1, 0, 0), 1: (0, 1, 0), 2: (0, 0, 1)}


# ---------------------------------------------------------------------------------------------------------------
# seeded inputs
# ---------------------------------------------------------------------------------------------------------------
class _Smooth:
    """Sum of a few random Fourier modes of the unit box, within [-1, 1]."""

    def __init__(self, rng, modes=4):
        k = rng.integers(-3, 4, size=(modes, 3))
        k[np.all(k == 0, axis=1)] = 1
        self.k = 2 * np.pi * k
        self.ph = rng.uniform(0, 2 * np.pi, modes)
        a = rng.uniform(0.5, 1.0, modes)
        self.a = a / a.sum()

    def __call__(self, X, Y, Z):
        out = 0.0
        for k, ph, a in zip(self.k, self.ph, self.a):
            out = out + a * torch.sin(k[0] * X + k[1] * Y + (k[2] * Z + ph))
        return out


@functools.lru_cache(None)
def _tov(rho_c):
    return I.solve_tov(rho_c=rho_c)


@functools.lru_cache(None)
def _table():
    return I.SyntheticEOS().table()


def _interp(x, xp, fp):
    j = torch.clamp(torch.searchsorted(xp, x.contiguous()) - 1, 0, xp.numel() - 2)
    t = (x - xp[j]) / (xp[j + 1] - xp[j])
    return fp[j] + torch.clamp(t, 0.0, 1.0) * (fp[j + 1] - fp[j])


def _curl(ax, dx):
    """Face field of an edge vector potential A(comp, X, Y, Z); ax(stag) gives the coordinates."""
    def A(c, f):
        return f(c, *ax(tuple(int(a != c) for a in range(3))))

    def of(f):
        Ax, Ay, Az = A(0, f), A(1, f), A(2, f)
        d = lambda q, dim: q.narrow(dim, 1, q.shape[dim] - 1) - q.narrow(dim, 0, q.shape[dim] - 1)  # noqa: E731
        return [d(Az, 2) / dx[1] - d(Ay, 1) / dx[2], d(Ax, 1) / dx[2] - d(Az, 3) / dx[0],
                d(Ay, 3) / dx[0] - d(Ax, 2) / dx[1]]
    return of


def _params(case):
    """Physical parameters of a case (plain numbers)."""
    if case["eos"] == "table":
        atm = 1e-14 if case["kind"] == "stage" else 1e-12
    else:
        atm = {"tube": 1e-10, "star": 1.28e-16, "stars": 1e-16}.get(case["inputs"], 1e-14)
    return dict(gamma=case["gamma"], rho_atm=atm, p_atm=100.0 * atm ** case["gamma"], T_atm=1e-6 if case["kind"] == "stage" else 1e-5,
                Ye_atm=0.5, band=1e-6 if case["precision"] == "mixed" and case["kind"] in ("stage", "step") else 1e-12,
                W_max=math.sqrt(401.0), M_max=1e4, tol=1e-10)


def _fill(case, seed, P):
    """Metric (16, nvert), W, [Bx, By, Bz] pools from the seed."""
    rng = np.random.default_rng(2311_04989 + seed)
    tab = case["eos"] == "table"
    M, W, B = P.verts(16), P.cells(7 if tab else 5), P.faces()
    kind = case["inputs"]
    if kind == "random":
        S = {k: _Smooth(rng) for k in ("rho", "th", "sig", "u0", "u1", "u2", "a0", "a1", "a2", "T", "ye")}
        Sm = [_Smooth(rng) for _ in range(16)]
        wide = case["kind"] == "con2prim"
        lr = np.log((1e-12, 1e-3) if wide and tab else (1e-10, 1e-3))
        ls = np.log((1e-3, 1e5) if wide and tab else (1e-3, 10.0))
        lt, lT = np.log((1e-3, 1e-1)), np.log((1e-4, 5e-2) if wide else (1e-5, 1e-2))
        umax, amp = (3.0 if wide and tab else 0.5), 1e-2
        eos = _table().eos if tab else None
        between = lambda l, f: torch.exp(l[0] + (l[1] - l[0]) * 0.5 * (1 + f))  # noqa: E731
    elif kind in ("star", "stars"):
        tov = _tov(1.28e-3 if kind == "star" else 1e-3)
        tt = {k: torch.tensor(getattr(tov, k), dtype=F64, device=_dev()) for k in ("rbar", "rho", "p", "alpha", "psi4")}
        h = P.blocks[0].dx[0]
        cs = [(0.0, 0.0, 0.0)] if kind == "star" else [(-20.0, 0.0, 0.0), (20.0, 0.0, 0.0)]
        cs = [tuple(c[a] + h * rng.uniform(-0.4, 0.4) for a in range(3)) for c in cs]
        Ab = (0.05 if kind == "star" else 16.0) * rng.uniform(0.8, 1.25)
        atm = _params(case)["rho_atm"]

        def at(r):
            ins = r < tov.R_iso
            rr = torch.clamp(r, min=0.5 * tov.R_iso)
            q = {k: _interp(r, tt["rbar"], tt[k]) for k in ("rho", "p", "alpha", "psi4")}
            z = torch.zeros_like(r)
            return (torch.where(ins, q["rho"], z), torch.where(ins, q["p"], z),
                    torch.where(ins, q["alpha"], (1 - tov.M / (2 * rr)) / (1 + tov.M / (2 * rr))),
                    torch.where(ins, q["psi4"], (1 + tov.M / (2 * rr)) ** 4))

        def dist(c, X, Y, Z):
            return torch.sqrt((X - c[0]) ** 2 + (Y - c[1]) ** 2 + (Z - c[2]) ** 2)
    for whole in P.groups:
        step = max(1, 8_000_000 // int(np.prod(P.shape(whole[0], (1, 1, 1)))))
        for o in range(0, whole[1], step):   # a bounded number of blocks at a time
            gr = (whole[0] + o, min(step, whole[1] - o))
            dx = [P.dx(gr, a) for a in range(3)]
            Mv = [P.view(M[c], gr, STAG["v"]) for c in range(16)]
            Wv = [P.view(w, gr) for w in W]
            Bv = [P.view(B[d], gr, STAG[d]) for d in range(3)]
            for c in (0, 4, 7, 9):
                Mv[c].fill_(1.0)
            Xv, Xc = P.axes(gr, STAG["v"]), P.axes(gr, STAG["c"])
            curl = _curl(lambda s: P.axes(gr, s), dx)  # noqa: B023
            if kind == "random":
                for c in range(16 if case["K"] else 10):
                    Mv[c].add_(amp * Sm[c](*Xv))

                def thermo(*X):
                    rho = between(lr, S["rho"](*X))
                    if not tab:
                        return rho, rho * between(lt, S["th"](*X)), None, None
                    T, ye = between(lT, S["T"](*X)), 0.05 + 0.45 * 0.5 * (1 + S["ye"](*X))
                    return rho, eos.p(rho, T, ye), ye, T
                for v, q in zip((0, 4, 5, 6), thermo(*Xc)):
                    if q is not None:
                        Wv[v].copy_(q)
                for c in range(3):
                    Wv[1 + c].copy_(umax / math.sqrt(3.0) * S["u%d" % c](*Xc))
                Bn = curl(lambda c, *X: torch.sqrt(between(ls, S["sig"](*X)) * thermo(*X)[1]) * S["a%d" % c](*X) / (2 * np.pi))
            elif kind == "tube":
                left = (Xc[0] < 0).expand(Wv[0].shape)
                pl, pr, by = rng.uniform(0.9, 1.1), rng.uniform(0.09, 0.11), rng.uniform(0.9, 1.1)
                Wv[0].copy_(torch.where(left, 1.0, 0.125))
                Wv[4].copy_(torch.where(left, pl, pr))
                Bn = [torch.full_like(Bv[0], 0.5), torch.where(P.axes(gr, STAG[1])[0] < 0, by, -by).expand(Bv[1].shape),
                      torch.zeros_like(Bv[2])]
            else:
                psi, apsi = 1.0, 1.0
                for c in cs:
                    _, _, a, q4 = at(dist(c, *Xv))
                    psi, apsi = psi + (q4 ** 0.25 - 1), apsi + (a * q4 ** 0.25 - 1)
                Mv[0].copy_(apsi / psi)
                for c in (4, 7, 9):
                    Mv[c].copy_(psi ** 4)
                rho = sum(at(dist(c, *Xc))[0] for c in cs)
                p = sum(at(dist(c, *Xc))[1] for c in cs)
                Wv[0].copy_(torch.clamp(rho, min=atm))
                Wv[4].copy_(torch.clamp(p, min=100.0 * atm ** 2))

                def A(comp, X, Y, Z):
                    out = torch.zeros(torch.broadcast_shapes(X.shape, Y.shape, Z.shape), dtype=F64, device=X.device)
                    for c in cs if comp < 2 else []:
                        f = Ab * torch.clamp(at(dist(c, X, Y, Z))[1] - 0.04 * float(tov.p[0]), min=0.0)
                        out = out + (-(Y - c[1]) * f if comp == 0 else (X - c[0]) * f)
                    return out
                Bn = curl(A)
            for d in range(3):
                Bv[d].copy_(Bn[d])
    return M, W, B


# ---------------------------------------------------------------------------------------------------------------
# prepare / run
# ---------------------------------------------------------------------------------------------------------------
class _State:
    """What a program holds between calls; the library's handles are given back with it."""
    drv = mesh = eos = ctx = None

    def __del__(self):
        if self.drv is not None:
            G.gr_driver_destroy(self.drv)
        if self.mesh is not None:
            G.gr_mesh_destroy(self.mesh)
        if self.eos is not None:
            G.gr_eos_destroy(self.eos)
        if self.ctx is not None:
            G.gr_context_destroy(self.ctx)


def _gr_params(case, s):
    q = _params(case)
    kw = dict(gamma_ad=q["gamma"], rho_atm=q["rho_atm"], p_atm=q["p_atm"], atm_band=q["band"], tol=q["tol"],
              recon=RECON[case["recon"]], emf=G.GR_EMF_MEAN if case["emf"] == "mean" else G.GR_EMF_UPWIND,
              precision=G.GR_PREC_MIXED if case["precision"] == "mixed" else G.GR_PREC_FP64,
              c2p_guess=G.GR_GUESS_FP32 if case["guess"] == "fp32" else G.GR_GUESS_NONE)
    if case["eos"] == "table":
        kw.update(eos=G.GR_EOS_TABLE, table=int(s.eos), T_atm=q["T_atm"], Ye_atm=q["Ye_atm"])
    if case["rk_mid"]:
        kw.update(rk_g0=0.75, rk_g1=0.25, rk_beta=0.25)
    return G.gr_params_default(**kw)


def _dt(P):
    return 0.2 * min(min(b.dx) for b in P.blocks)


def prepare(case, seed):
    s = _State()
    s.case = case
    s.ctx = G.gr_context_create(0)
    if case["eos"] == "table":
        s.eos = G.gr_eos_create(s.ctx, _table())
    P = s.P = _Pools(_blocks(case, seed))
    s.M, s.W, s.B = _fill(case, seed, P)
    s.mesh = G.gr_mesh_create(s.ctx, P.L.descriptors())
    s.p = _gr_params(case, s)
    kind = case["kind"]
    s.metric = G.metric_struct(s.M, order=case["order"], k_zero=not case["K"])
    nq = 6 if case["eos"] == "table" else 5
    if kind in ("stage", "step", "con2prim"):
        s.U = _ref_prim2con_pools(case, P, s.M, s.W, s.B)
    if kind == "stage":
        s.Uo, s.Wo, s.Bo = torch.zeros_like(s.U), torch.zeros_like(s.W), [torch.zeros_like(b) for b in s.B]
        s.status = torch.zeros(P.L.ncell, dtype=torch.uint8, device=_dev())
        s.state = G.state_struct(s.U, s.U, s.B, s.B, s.W, s.Uo, s.Bo, s.Wo, s.status)
        s.Wo32 = s.Bo32 = None
        if case["copies"]:   # the steady state of an evolution: FP32 copies of the inputs at hand, those of the outputs kept
            s.M32, s.W32, s.B32 = s.M.float(), s.W[:nq].float(), [b.float() for b in s.B]
            s.Wo32, s.Bo32 = torch.zeros_like(s.W32), [torch.zeros_like(b) for b in s.B32]
            s.metric = G.metric_struct(s.M, order=case["order"], k_zero=not case["K"], metric32=s.M32)
            G.set_fp32_copies(s.state, W32=s.W32, B32=s.B32, Wo32=s.Wo32, Bo32=s.Bo32)
        s.dt = _dt(P)
        if case["tune"]:
            G.gr_autotune(s.mesh, s.metric, s.state, s.dt, s.p, 2)
    elif kind == "step":
        s.status = torch.zeros(P.L.ncell, dtype=torch.uint8, device=_dev())
        s.drv = G.gr_driver_create(s.mesh, I.block_grid_neighbours((case["gx"], case["gy"], case["gz"])))
        s.keep = (s.U.clone(), s.W.clone(), [b.clone() for b in s.B])
    elif kind == "con2prim":
        s.Wo = torch.zeros_like(s.W)
        s.status = torch.zeros(P.L.ncell, dtype=torch.uint8, device=_dev())
    elif kind == "prim2con":
        s.U = P.cells(nq)
    else:
        s.out = P.verts(10)
    return s


def run(s):
    kind = s.case["kind"]
    if kind == "stage":
        G.gr_stage(s.mesh, s.metric, s.state, s.dt, s.p)
        out = {"U": list(s.Uo), "B": s.Bo, "W": list(s.Wo), "status": s.status}
        if s.Wo32 is not None:
            out["W32"], out["B32"] = list(s.Wo32), s.Bo32
        return out
    if kind == "step":   # from a saved state: what a program does that may repeat a step
        s.U.copy_(s.keep[0])
        s.W.copy_(s.keep[1])
        for d in range(3):
            s.B[d].copy_(s.keep[2][d])
        G.gr_driver_step(s.drv, s.metric, list(s.U), list(s.W), s.B, s.status, s.p, 0.2, G.GR_DT_GRID, s.case["rk_order"])
        return {"U": list(s.U), "B": s.B, "W": list(s.W), "status": s.status}
    if kind == "con2prim":
        G.gr_con2prim(s.mesh, s.metric, list(s.U), s.B, list(s.Wo), s.status, s.p)
        return {"U": list(s.U), "W": list(s.Wo), "status": s.status}
    if kind == "prim2con":
        G.gr_prim2con(s.mesh, s.metric, list(s.W), s.B, list(s.U), s.p)
        return {"U": list(s.U)}
    G.gr_adm_sources(s.mesh, s.metric, list(s.W), s.B, s.p, s.case["vc_order"], list(s.out))
    return {"sources": list(s.out)}


def work(case):
    cells = sum(b.n[0] * b.n[1] * b.n[2] for b in _blocks(case, 0))
    verts = sum((b.n[0] + 1) * (b.n[1] + 1) * (b.n[2] + 1) for b in _blocks(case, 0))
    tab = case["eos"] == "table"
    nq, nw, nm = (6, 6, 16 if case["K"] else 10) if tab else (5, 5, 16 if case["K"] else 10)
    kind = case["kind"]
    if kind in ("stage", "step"):
        # per stage: U, W, B and the metric read, U', W' (and T), B', status written; U0 and B0 of a later stage
        per = 8 * (nq + nw + 3) + 8 * (nq + nw + (1 if tab else 0) + 3) + 1
        if kind == "stage":
            b = cells * (per + (8 * (nq + 3) if case["rk_mid"] else 0)) + 8 * nm * verts
            stages = 1
        else:
            stages = case["rk_order"]
            b = stages * (cells * per + 8 * nm * verts) + (stages - 1) * cells * 8 * (nq + 3)
        # operations per cell of a stage: face fluxes (three faces: reconstruction and face physics), cell metric, field,
        # sources, corner fields and CT, con2prim
        rec = {"plm": 110, "wenoz": 870, "weno5": 840, "ppm": 900}[case["recon"]] * (8 / 7 if tab else 1)
        return {"bytes": b, "flops": stages * cells * (3 * (rec + 560 + (300 if tab else 0)) + 1800 + 300 + (1500 if tab else 0))}
    if kind == "con2prim":
        return {"bytes": cells * (8 * (2 * nq + 3 + nw + (1 if tab else 0)) + 1) + 8 * 6 * verts, "flops": cells * (900 if tab else 420)}
    if kind == "prim2con":
        return {"bytes": cells * 8 * (nw + 3 + nq) + 80 * verts, "flops": cells * 260}
    n4 = case["vc_order"] == 4
    return {"bytes": cells * 64 + verts * (48 + 80), "flops": cells * 200 + verts * 10 * (24 if n4 else 12)}


# ---------------------------------------------------------------------------------------------------------------
# the same pass in plain torch, 64 bits: (block, z, y, x) arrays; an array with its origin is (tensor, (lx, ly, lz))
# ---------------------------------------------------------------------------------------------------------------
DIM = (3, 2, 1)   # tensor dimension of x, y, z


def _cut(a, lo, rng):
    """Elements rng[x|y|z] = (first, last) of an array whose element 0 has index lo."""
    for d in range(3):
        a = a.narrow(DIM[d], rng[d][0] - lo[d], rng[d][1] - rng[d][0] + 1)
    return a


def _at(a, dim, i, k):
    return a.narrow(dim, i, k)


def _mid(a, dim, order):
    k = a.shape[dim] - 1
    out = 0.5 * (_at(a, dim, 0, k) + _at(a, dim, 1, k))
    if order == 4:
        out.narrow(dim, 1, k - 2).copy_((9 * (_at(a, dim, 1, k - 2) + _at(a, dim, 2, k - 2)) -
                                         (_at(a, dim, 0, k - 2) + _at(a, dim, 3, k - 2))) / 16)
    return out


def _der(a, dim, order, dx):
    k = a.shape[dim] - 1
    out = _at(a, dim, 1, k) - _at(a, dim, 0, k)
    if order == 4:
        out.narrow(dim, 1, k - 2).copy_((27 * (_at(a, dim, 2, k - 2) - _at(a, dim, 1, k - 2)) -
                                         (_at(a, dim, 3, k - 2) - _at(a, dim, 0, k - 2))) / 24)
    return out / dx


def _cells(a, order):
    return _mid(_mid(_mid(a, 3, order), 2, order), 1, order)


def _lower(g, u):
    return [g[0] * u[0] + g[1] * u[1] + g[2] * u[2], g[1] * u[0] + g[3] * u[1] + g[4] * u[2],
            g[2] * u[0] + g[4] * u[1] + g[5] * u[2]]


def _det(g):
    return g[0] * (g[3] * g[5] - g[4] ** 2) - g[1] * (g[1] * g[5] - g[4] * g[2]) + g[2] * (g[1] * g[4] - g[3] * g[2])


def _inv(g):
    d = _det(g)
    return [c / d for c in (g[3] * g[5] - g[4] ** 2, g[2] * g[4] - g[1] * g[5], g[1] * g[4] - g[2] * g[3],
                            g[0] * g[5] - g[2] ** 2, g[1] * g[2] - g[0] * g[4], g[0] * g[3] - g[1] ** 2)]


def _dot(a, b):
    return a[0] * b[0] + a[1] * b[1] + a[2] * b[2]


SYM = ((0, 1, 2), (1, 3, 4), (2, 4, 5))


class _Eos:
    """rho h and c_s^2 of (rho, p[, Y_e]); the table's trilinear interpolant and its inverse in log T."""

    def __init__(self, case):
        self.q = _params(case)
        self.tab = None
        if case["eos"] == "table":
            t = self.tab = _table()
            lr = t.x0[0] + t.dx[0] * np.arange(t.n[0])
            f = lambda a: torch.tensor(np.ascontiguousarray(a), dtype=F64, device=_dev()).reshape(-1)  # noqa: E731
            self.lp, self.le, self.cs2 = f(t.lp - lr), f(t.le - lr), f(t.cs2)
            self.h0 = float((torch.exp(self.le) + torch.exp(self.lp)).min())
            self.end = [t.x0[a] + t.dx[a] * (t.n[a] - 1) for a in range(3)]
        else:
            self.h0 = 1.0

    def locate(self, a, x):
        t = self.tab
        s = (torch.clamp(x, t.x0[a], self.end[a]) - t.x0[a]) / t.dx[a]
        i = torch.clamp(s.to(torch.int64), 0, t.n[a] - 2)
        return i, s - i

    def loc(self, lrho, ye):
        (ir, wr), (iy, wy) = self.locate(0, lrho), self.locate(2, ye)
        return iy * self.tab.n[1] * self.tab.n[0] + ir, wr, wy

    def node(self, f, L, k):
        o = L[0] + k * self.tab.n[0]
        sy = self.tab.n[1] * self.tab.n[0]
        return (1 - L[2]) * ((1 - L[1]) * f[o] + L[1] * f[o + 1]) + L[2] * ((1 - L[1]) * f[o + sy] + L[1] * f[o + sy + 1])

    def inv_T(self, f, L, y):
        n = self.tab.n[1]
        lo, hi = torch.zeros_like(L[0]), torch.full_like(L[0], n - 1)
        for _ in range(int(math.ceil(math.log2(n - 1))) + 1):
            mid = (lo + hi) // 2
            up = (self.node(f, L, mid) <= y) & (mid < hi)
            lo, hi = torch.where(up, torch.maximum(mid, lo), lo), torch.where(up, hi, torch.maximum(mid, lo + 1))
        k = torch.clamp(lo, 0, n - 2)
        a, b = self.node(f, L, k), self.node(f, L, k + 1)
        return k, torch.clamp((y - a) / (b - a), 0.0, 1.0)

    def on_T(self, f, L, k, w):
        a = self.node(f, L, k)
        return a + w * (self.node(f, L, k + 1) - a)

    def thermo(self, rho, p, ye):
        if self.tab is None:
            gam = self.q["gamma"]
            rhoh = rho + gam * p / (gam - 1)
            return rhoh, gam * p / rhoh
        L = self.loc(torch.log(rho), ye)
        k, w = self.inv_T(self.lp, L, torch.log(p / rho))
        return rho * torch.exp(self.on_T(self.le, L, k, w)) + p, self.on_T(self.cs2, L, k, w)

    def p_eps(self, rho, lT, ye):
        L = self.loc(torch.log(rho), ye)
        k, w = self.locate(1, lT)
        return rho * torch.exp(self.on_T(self.lp, L, k, w)), torch.expm1(self.on_T(self.le, L, k, w))

    def atm(self, like):
        """(rho, p, internal energy density) of the atmosphere."""
        r = torch.full_like(like, self.q["rho_atm"])
        if self.tab is None:
            p = torch.full_like(like, self.q["p_atm"])
            return r, p, p / (self.q["gamma"] - 1)
        p, eps = self.p_eps(r, torch.full_like(r, math.log(self.q["T_atm"])), torch.full_like(r, self.q["Ye_atm"]))
        return r, p, r * eps


def _fluid(g, alpha, beta, eos, w, Bd, ye=None):
    """Quantities of a state: W, v, b and the conserved variables over sqrt(gamma)."""
    sg = torch.sqrt(_det(g))
    ut, rho, p = w[1:4], w[0], w[4]
    utl = _lower(g, ut)
    W = torch.sqrt(1 + _dot(ut, utl))
    v, vl, Bu = [u / W for u in ut], [u / W for u in utl], [b / sg for b in Bd]
    Bl = _lower(g, Bu)
    ab0 = W * _dot(Bu, vl)
    b2 = (ab0 ** 2 + _dot(Bu, Bl)) / W ** 2
    bl = [Bl[i] / W + ab0 * vl[i] for i in range(3)]
    rhoh, cs2 = eos.thermo(rho, p, ye)
    e, pt = rhoh + b2, p + 0.5 * b2
    q = [sg * rho * W] + [sg * (e * W * utl[j] - ab0 * bl[j]) for j in range(3)]
    q.append(sg * ((rhoh * W * W - rho * W - p) + b2 * W * W - 0.5 * b2 - ab0 ** 2))
    vt = [v[i] - beta[i] / alpha for i in range(3)] if beta is not None else None
    return dict(sg=sg, W=W, v=v, vl=vl, vt=vt, Bu=Bu, bl=bl, ab0=ab0, b2=b2, e=e, pt=pt, cs2=cs2, q=q, rhoh=rhoh)


def _cell_B(B):
    return [0.5 * (B[d].narrow(DIM[d], 0, B[d].shape[DIM[d]] - 1) + B[d].narrow(DIM[d], 1, B[d].shape[DIM[d]] - 1))
            for d in range(3)]


def _weno_parts(v):
    a, b, c, d, e = v
    q = ((2 * a - 7 * b + 11 * c) / 6, (-b + 5 * c + 2 * d) / 6, (2 * c + 5 * d - e) / 6)
    k = (13 / 12 * (a - 2 * b + c) ** 2 + 0.25 * (a - 4 * b + 3 * c) ** 2,
         13 / 12 * (b - 2 * c + d) ** 2 + 0.25 * (b - d) ** 2,
         13 / 12 * (c - 2 * d + e) ** 2 + 0.25 * (3 * c - 4 * d + e) ** 2)
    return q, k


def _weno(v, z, eps=1e-40):
    q, k = _weno_parts(v)
    if z:
        t5 = (k[0] - k[2]).abs()
        w = [c * (1 + t5 / (b + eps)) for c, b in zip((0.1, 0.6, 0.3), k)]
    else:   # scaled by the smallest indicator so that squares neither underflow nor overflow
        m = torch.minimum(torch.minimum(k[0], k[1]), k[2]) + eps
        w = [c * (m / (b + eps)) ** 2 for c, b in zip((0.1, 0.6, 0.3), k)]
    return (w[0] * q[0] + w[1] * q[1] + w[2] * q[2]) / (w[0] + w[1] + w[2])


def _ppm_face(a, b, c, d):
    q = 7 / 12 * (b + c) - (a + d) / 12
    d2f, d2l, d2r = 3 * (b - 2 * q + c), a - 2 * b + c, b - 2 * c + d
    s = torch.sign(d2f)
    same = (s == torch.sign(d2l)) & (s == torch.sign(d2r)) & (d2f != 0)
    lim = torch.where(same, s * torch.minimum(1.25 * torch.minimum(d2l.abs(), d2r.abs()), d2f.abs()), torch.zeros_like(q))
    return torch.where((q - b) * (c - q) < 0, 0.5 * (b + c) - lim / 6, q)


def _ppm_cell(v):
    a, b, q, d, e = v
    l, r = _ppm_face(a, b, q, d), _ppm_face(b, q, d, e)
    ext = ((r - q) * (q - l) <= 0) | ((b - q) * (q - d) <= 0)
    d2, d2c, d2l, d2r = 6 * (l - 2 * q + r), b - 2 * q + d, a - 2 * b + q, q - 2 * d + e
    s = torch.sign(d2)
    same = (s == torch.sign(d2c)) & (s == torch.sign(d2l)) & (s == torch.sign(d2r)) & (d2 != 0)
    lim = torch.minimum(torch.minimum(1.25 * torch.minimum(d2l.abs(), d2r.abs()), 1.25 * d2c.abs()), d2.abs())
    ratio = torch.where(same, s * lim / torch.where(d2 == 0, torch.ones_like(d2), d2), torch.zeros_like(q))
    el, er = q + (l - q) * ratio, q + (r - q) * ratio
    nr = torch.where((r - q).abs() >= 2 * (l - q).abs(), q - 2 * (l - q), r)
    nl = torch.where((l - q).abs() >= 2 * (nr - q).abs(), q - 2 * (nr - q), l)
    return torch.where(ext, el, nl), torch.where(ext, er, nr)


def _recon(s, method):
    """Left and right state of the face between s[2] and s[3]."""
    if method == "plm":
        def slope(a, b, c):
            l, r = b - a, c - b
            return torch.where(l * r > 0, 2 * l * r / torch.where(l + r == 0, torch.ones_like(l), l + r), torch.zeros_like(l))
        return s[2] + 0.5 * slope(s[1], s[2], s[3]), s[3] - 0.5 * slope(s[2], s[3], s[4])
    if method == "ppm":
        return _ppm_cell(s[0:5])[1], _ppm_cell(s[1:6])[0]
    z = method == "wenoz"
    return _weno(s[0:5], z), _weno(s[5:0:-1], z)


def _c2p_master(eos, I, mu, vmax2):
    """f(mu) and what goes with it (the reading of the KKC master function)."""
    x = 1 / (1 + mu * I["b2"])
    rb2 = x * x * I["r2"] + mu * x * (1 + x) * I["rb"] ** 2
    qb = I["q"] - 0.5 * I["b2"] - 0.5 * mu ** 2 * x ** 2 * (I["b2"] * I["r2"] - I["rb"] ** 2)
    v2 = mu ** 2 * rb2
    cap = v2 > vmax2
    v2 = torch.clamp(v2, max=vmax2)
    iW = torch.sqrt(1 - v2)
    qm = qb - mu * rb2
    eps = (qm * (1 + iW) + v2) / (iW * (1 + iW))
    rho = I["D"] * iW
    if eos.tab is None:
        eps = torch.clamp(eps, min=0.0)
        p = (eos.q["gamma"] - 1) * rho * eps
        h, lT = 1 + eos.q["gamma"] * eps, None
    else:
        rho = torch.clamp(rho, math.exp(eos.tab.x0[0]), math.exp(eos.end[0]))
        L = eos.loc(torch.log(rho), I["ye"])
        y = torch.where(eps > -1, torch.log1p(torch.clamp(eps, min=-1 + 1e-300)), torch.full_like(eps, -math.inf))
        k, w = eos.inv_T(eos.le, L, y)
        ye = eos.on_T(eos.le, L, k, w)
        eps = torch.where((y <= eos.node(eos.le, L, torch.zeros_like(k))) | (y >= eos.node(eos.le, L, torch.full_like(k, eos.tab.n[1] - 1))),
                          torch.expm1(ye), eps)
        p = rho * torch.exp(eos.on_T(eos.lp, L, k, w))
        h, lT = 1 + eps + p / rho, eos.tab.x0[1] + eos.tab.dx[1] * (k + w)
    nu = torch.maximum(h * iW, h * (1 + qm) / (1 + eps))
    return mu - 1 / (nu + mu * rb2), dict(x=x, rb2=rb2, v2=v2, cap=cap, iW=iW, eps=eps, rho=rho, p=p, lT=lT)


def _con2prim(case, eos, g, q, Bd):
    """(U, W) of con2prim with the atmosphere and the limits."""
    P, tab = eos.q, eos.tab is not None
    sg = torch.sqrt(_det(g))
    thr = P["rho_atm"] * (1 + P["band"])
    atm = q[0] < thr * sg
    q = [torch.where(atm, sg if v == 0 else torch.zeros_like(sg), q[v]) for v in range(len(q))]   # placeholder where reset
    D, tau, S, Bu = q[0] / sg, q[4] / sg, [q[1 + i] / sg for i in range(3)], [b / sg for b in Bd]
    BB = _dot(Bu, _lower(g, Bu))
    ye = ye_raw = None
    if tab:
        ye_raw = torch.where(atm, torch.full_like(D, P["Ye_atm"]), q[5] / q[0])
        ye = torch.clamp(ye_raw, eos.tab.x0[2], eos.end[2])
    lim = BB > P["M_max"] * D
    D = torch.where(lim, BB / P["M_max"], D)
    tmin = 0.5 * BB
    if tab:
        tmin = tmin + D * eos.p_eps(D, torch.full_like(D, eos.tab.x0[1]), ye)[1]
    low = tau < tmin
    tau = torch.maximum(tau, tmin)
    mod = lim | low | ((ye_raw != ye) if tab else lim)
    gi = _inv(g)
    rl, bu = [s / D for s in S], [b / torch.sqrt(D) for b in Bu]
    ru = [gi[SYM[i][0]] * rl[0] + gi[SYM[i][1]] * rl[1] + gi[SYM[i][2]] * rl[2] for i in range(3)]
    I_ = dict(D=D, q=tau / D, r2=_dot(rl, ru), rb=_dot(rl, bu), b2=BB / D, ye=ye)
    vmax2 = 1 - 1 / P["W_max"] ** 2
    lo, hi = torch.zeros_like(D), torch.full_like(D, 1 / eos.h0)
    for it in range(100):
        if it % 8 == 0 and bool(((hi - lo) <= 2 ** -51 * hi).all()):
            break
        mid = 0.5 * (lo + hi)
        up = _c2p_master(eos, I_, mid, vmax2)[0] < 0
        lo, hi = torch.where(up, mid, lo), torch.where(up, hi, mid)
    mu = 0.5 * (lo + hi)
    _, E = _c2p_master(eos, I_, mu, vmax2)
    vu = [mu * E["x"] * (ru[i] + mu * I_["rb"] * bu[i]) for i in range(3)]
    s = torch.where(E["cap"], torch.sqrt(E["v2"] / torch.clamp(mu ** 2 * E["rb2"], min=1e-300)), torch.ones_like(mu))
    atm = atm | (E["rho"] < thr)
    w = [E["rho"]] + [v * s / E["iW"] for v in vu] + [E["p"]]
    out = [torch.where(mod & ~atm, sg * D, q[0]), q[1], q[2], q[3], torch.where(mod & ~atm, sg * tau, q[4])]
    if tab:
        T = torch.exp(E["lT"])
        cold = T < P["T_atm"]
        lTa = torch.full_like(T, math.log(P["T_atm"]))
        w[4] = torch.where(cold, eos.p_eps(E["rho"], lTa, ye)[0], w[4])
        w += [ye, torch.clamp(T, min=P["T_atm"])]
        out.append(torch.where(mod & ~atm, sg * D * ye, q[5]))
        f = _fluid(g, None, None, eos, [torch.where(atm, P["rho_atm"] + 0 * v, v) if k == 0 else v for k, v in enumerate(w[:5])], Bd, ye)
        cold = cold & ~atm
        out = [torch.where(cold, a, b) for a, b in zip(f["q"] + [f["q"][0] * ye], out)]
    ra, pa, ea = eos.atm(D)
    BBd = 0.5 * _dot(Bd, _lower(g, Bd)) / sg
    za = torch.zeros_like(D)
    qa = [sg * ra, za, za, za, sg * ea + BBd] + ([sg * ra * P["Ye_atm"]] if tab else [])
    wa = [ra, za, za, za, pa] + ([torch.full_like(D, P["Ye_atm"]), torch.full_like(D, P["T_atm"])] if tab else [])
    return [torch.where(atm, a, b) for a, b in zip(qa, out)], [torch.where(atm, a, b) for a, b in zip(wa, w)]


def _ref_stage(case, eos, dx, n, g, M, W, B, U, U0, B0, rk, dt):
    """U', W' (interior) and B' (faces of interior cells) of one stage; rk = (g0, g1, beta)."""
    order, tab = case["order"], eos.tab is not None
    lo = (-g,) * 3
    ring = [(-1, n[a]) for a in range(3)]
    inner = [(0, n[a] - 1) for a in range(3)]
    val = [_cells(M[c], order) for c in range(16 if case["K"] else 10)]
    gam = val[4:10]
    sgc = torch.sqrt(_det(gam))
    Bd = _cell_B(B)
    bcc = [b / sgc for b in Bd]
    utl = _lower(gam, W[1:4])
    Wl = torch.sqrt(1 + _dot(W[1:4], utl))
    vt = [W[1 + a] / Wl - val[1 + a] / val[0] for a in range(3)]
    ecc = [_cut(val[0] * (vt[(m + 2) % 3] * Bd[(m + 1) % 3] - vt[(m + 1) % 3] * Bd[(m + 2) % 3]), lo, ring) for m in range(3)]
    flux, flo = [], []
    for D in range(3):
        t1, t2 = (D + 1) % 3, (D + 2) % 3
        reg = [(-1, n[a]) for a in range(3)]
        reg[D] = (0, n[D])
        st = list(reg)
        st[D] = (-3, n[D] + 2)
        met = [_cut(_mid(_mid(M[c], DIM[t1], order), DIM[t2], order), lo, reg) for c in range(10)]
        q = list(W[:5]) + [bcc[t1], bcc[t2]] + ([W[5]] if tab else [])
        Ls, Rs, s2 = [], [], []
        for a in q:
            a = _cut(a, lo, st)
            s = [a.narrow(DIM[D], t, n[D] + 1) for t in range(6)]
            l, r = _recon(s, case["recon"])
            Ls.append(l), Rs.append(r), s2.append((s[2], s[3]))
        bad = ~((Ls[0] > 0) & (Rs[0] > 0) & (Ls[4] > 0) & (Rs[4] > 0))
        Ls = [torch.where(bad, s2[v][0], x) for v, x in enumerate(Ls)]
        Rs = [torch.where(bad, s2[v][1], x) for v, x in enumerate(Rs)]
        gf, al, be = met[4:], met[0], met[1:4]
        sg, gdd = torch.sqrt(_det(gf)), _inv(gf)[SYM[D][D]]
        Bn = _cut(B[D], lo, reg)
        side = []
        for s in (Ls, Rs):
            Bf = [None] * 3
            Bf[D], Bf[t1], Bf[t2] = Bn, s[5] * sg, s[6] * sg
            f = _fluid(gf, al, be, eos, s[:5], Bf, s[7] if tab else None)
            av, asg, BW = al * f["vt"][D], al * sg, f["Bu"][D] / f["W"]
            F = [f["q"][0] * av] + [f["q"][1 + j] * av - asg * f["bl"][j] * BW for j in range(3)]
            F[1 + D] = F[1 + D] + f["pt"] * asg
            F.append(f["q"][4] * av + asg * (f["pt"] * f["v"][D] - f["ab0"] * BW))
            F += [al * (Bf[t] * f["vt"][D] - Bf[D] * f["vt"][t]) for t in (t1, t2)]
            ca2 = f["b2"] / f["e"]
            c2 = f["cs2"] + ca2 - f["cs2"] * ca2
            v2, vd = _dot(f["v"], f["vl"]), f["v"][D]
            disc = torch.clamp((1 - v2) * (gdd * (1 - v2 * c2) - vd ** 2 * (1 - c2)), min=0.0)
            cr, den, vc = torch.sqrt(c2) * torch.sqrt(disc), 1 - v2 * c2, vd * (1 - c2)
            side.append((f["q"] + [Bf[t1], Bf[t2]], F, al * (vc - cr) / den - be[D], al * (vc + cr) / den - be[D]))
        (UL, FL, lmL, lpL), (UR, FR, lmR, lpR) = side
        lp, lm = torch.clamp(torch.maximum(lpL, lpR), min=0.0), torch.clamp(torch.minimum(lmL, lmR), max=0.0)
        den = torch.where(lp - lm == 0, torch.ones_like(lp), lp - lm)
        F = [torch.where(lp - lm == 0, 0.5 * (a + b), (lp * a - lm * b + lp * lm * (r - l)) / den)
             for a, b, l, r in zip(FL, FR, UL, UR)]
        if tab:
            F.append(F[0] * torch.where(F[0] > 0, Ls[7], Rs[7]))
        flux.append(F)
        flo.append(tuple(r[0] for r in reg))
    edge = []
    for m in range(3):
        a, b = (m + 1) % 3, (m + 2) % 3

        def pick(F, l0, d, back):   # elements at edge positions, one back along direction `d` where asked
            rng = [(0, n[x] if x != m else n[x] - 1) for x in range(3)]
            if back:
                rng[d] = (-1, n[d] - 1)
            return _cut(F, l0, rng)

        def cell(ba, bb):
            rng = [(0, n[x] if x != m else n[x] - 1) for x in range(3)]
            if ba:
                rng[a] = (-1, n[a] - 1)
            if bb:
                rng[b] = (-1, n[b] - 1)
            return _cut(ecc[m], (-1,) * 3, rng)
        Ea1, Ea0 = -pick(flux[a][5], flo[a], b, False), -pick(flux[a][5], flo[a], b, True)
        Eb1, Eb0 = pick(flux[b][6], flo[b], a, False), pick(flux[b][6], flo[b], a, True)
        E = 0.25 * (Ea1 + Ea0 + Eb1 + Eb0)
        if case["emf"] == "upwind":
            up = lambda v, l, h: torch.where(v > 0, l, torch.where(v < 0, h, 0.5 * (l + h)))  # noqa: E731
            va1, va0 = pick(flux[a][0], flo[a], b, False), pick(flux[a][0], flo[a], b, True)
            vb1, vb0 = pick(flux[b][0], flo[b], a, False), pick(flux[b][0], flo[b], a, True)
            C11, C01, C10, C00 = cell(0, 0), cell(1, 0), cell(0, 1), cell(1, 1)
            E = E + 0.25 * (up(va0, Eb0 - C00, Eb1 - C10) - up(va1, C01 - Eb0, C11 - Eb1)) + \
                0.25 * (up(vb0, Ea0 - C00, Ea1 - C01) - up(vb1, C10 - Ea0, C11 - Ea1))
        edge.append(E)
    bdt = rk[2] * dt
    Bo = []
    for D in range(3):
        t1, t2 = (D + 1) % 3, (D + 2) % 3
        dif = lambda E, t: (E.narrow(DIM[t], 1, n[t]) - E.narrow(DIM[t], 0, n[t]))  # noqa: E731
        curl = dif(edge[t2], t1) / dx[t1] - dif(edge[t1], t2) / dx[t2]
        reg = [(0, n[a] - 1) for a in range(3)]
        reg[D] = (0, n[D])
        b = rk[1] * _cut(B[D], lo, reg) - bdt * curl
        Bo.append(b + rk[0] * _cut(B0[D], lo, reg) if rk[0] else b)
    # sources
    ci = lambda a: _cut(a, lo, inner)  # noqa: E731
    met = [ci(v) for v in val]
    gi_, be, al = met[4:10], met[1:4], met[0]
    w = [ci(x) for x in W]
    f = _fluid(gi_, al, be, eos, w[:5], [ci(x) for x in Bd], w[5] if tab else None)
    dm = []
    for k in range(3):
        row = []
        for c in range(10):
            d = _der(M[c], DIM[k], order, dx[k])
            for o in range(3):
                if o != k:
                    d = _mid(d, DIM[o], order)
            row.append(ci(d))
        dm.append(row)
    gu = _inv(gi_)
    u = [f["W"] / al] + [f["W"] * f["vt"][i] for i in range(3)]
    bb = [f["ab0"] / al] + [f["Bu"][i] / f["W"] + f["ab0"] * f["vt"][i] for i in range(3)]
    T00 = f["e"] * u[0] ** 2 - f["pt"] / al ** 2 - bb[0] ** 2
    T0 = [f["e"] * u[0] * u[1 + i] + f["pt"] * be[i] / al ** 2 - bb[0] * bb[1 + i] for i in range(3)]
    Tij = [[f["e"] * u[1 + i] * u[1 + j] + f["pt"] * (gu[SYM[i][j]] - be[i] * be[j] / al ** 2) - bb[1 + i] * bb[1 + j]
            for j in range(3)] for i in range(3)]
    bl_, T0l = _lower(gi_, be), _lower(gi_, T0)
    T0l = [T0l[i] + T00 * bl_[i] for i in range(3)]
    src = [0.0]
    for k in range(3):
        s = -T00 * al * dm[k][0] + _dot(T0l, dm[k][1:4])
        for i in range(3):
            for j in range(3):
                s = s + (0.5 * T00 * be[i] * be[j] + T0[i] * be[j] + 0.5 * Tij[i][j]) * dm[k][4 + SYM[i][j]]
        src.append(al * f["sg"] * s)
    s = -sum((T00 * be[i] + T0[i]) * dm[i][0] for i in range(3))
    if case["K"]:
        for i in range(3):
            for j in range(3):
                s = s + (T00 * be[i] * be[j] + 2 * T0[i] * be[j] + Tij[i][j]) * met[10 + SYM[i][j]]
    src += [al * f["sg"] * s, 0.0]
    q = []
    for v in range(6 if tab else 5):
        cv = v if v < 5 else 7
        div = 0.0
        for d in range(3):
            hi_, lo_ = list(inner), list(inner)
            hi_[d] = (1, n[d])
            div = div + (_cut(flux[d][cv], flo[d], hi_) - _cut(flux[d][cv], flo[d], lo_)) / dx[d]
        x = rk[1] * ci(U[v]) + bdt * (src[v] - div)
        q.append(x + rk[0] * ci(U0[v]) if rk[0] else x)
    Uo, Wo = _con2prim(case, eos, gi_, q, _cell_B(Bo))
    return Uo, Wo, Bo


def _ref_prim2con_pools(case, P, M, W, B):
    """Conserved pools (interior cells) of primitive pools."""
    eos, tab = _Eos(case), case["eos"] == "table"
    U = P.cells(6 if tab else 5)
    for gr, n, g, _ in _chunks(P):
        inner, lo = [(0, n[a] - 1) for a in range(3)], (-g,) * 3
        met = [_cut(_cells(P.view(M[c], gr, STAG["v"]), case["order"]), lo, inner) for c in range(4, 10)]
        w = [_cut(P.view(x, gr), lo, inner) for x in W]
        Bd = [_cut(x, lo, inner) for x in _cell_B([P.view(B[d], gr, STAG[d]) for d in range(3)])]
        q = _fluid(met, None, None, eos, w[:5], Bd, w[5] if tab else None)["q"]
        if tab:
            q = q + [q[0] * w[5]]
        for v, x in enumerate(q):
            _cut(P.view(U[v], gr), lo, inner).copy_(x)
    return U


def _chunks(P, cells=2_500_000):
    for whole in P.groups:
        b = P.blocks[whole[0]]
        step = max(1, cells // int(np.prod(P.shape(whole[0], (0, 0, 0)))))
        for o in range(0, whole[1], step):
            gr = (whole[0] + o, min(step, whole[1] - o))
            yield gr, b.n, b.ng, [P.dx(gr, a) for a in range(3)]


def _stage_pools(case, eos, P, M, W, B, U, U0, B0, rk, dt, out):
    Uo, Wo, Bo = out
    for gr, n, g, dx in _chunks(P):
        v = lambda a, s="c": P.view(a, gr, STAG[s])  # noqa: B023, E731
        lo, inner = (-g,) * 3, [(0, n[a] - 1) for a in range(3)]
        q, w, b = _ref_stage(case, eos, dx, n, g, [v(m, "v") for m in M], [v(x) for x in W], [v(B[d], d) for d in range(3)],
                             [v(x) for x in U], [v(x) for x in U0], [v(B0[d], d) for d in range(3)], rk, dt)
        for pool, vals in ((Uo, q), (Wo, w)):
            for i, x in enumerate(vals):
                _cut(v(pool[i]), lo, inner).copy_(x)
        for d in range(3):
            reg = list(inner)
            reg[d] = (0, n[d])
            _cut(v(Bo[d], d), lo, reg).copy_(b[d])


def _wrap_fill(case, P, W, B):
    """Ghost cells and faces of a periodic grid of equal blocks from the owned elements."""
    m, b = (case["gx"], case["gy"], case["gz"]), P.blocks[0]
    n, g, gr = b.n, b.ng, (0, len(P.blocks))

    def fill(pool, stag):
        a = P.view(pool, gr, stag)
        a = a.reshape((m[2], m[1], m[0]) + a.shape[1:])
        own = a[..., g:g + n[2], g:g + n[1], g:g + n[0]]
        G_ = own.permute(0, 3, 1, 4, 2, 5).reshape(m[2] * n[2], m[1] * n[1], m[0] * n[0])
        idx = []
        for ax in (2, 1, 0):
            k = torch.arange(-g, n[ax] + g + stag[ax], device=a.device)
            idx.append((torch.arange(m[ax], device=a.device)[:, None] * n[ax] + k[None, :]) % (m[ax] * n[ax]))
        new = G_[idx[0][:, None, None, :, None, None], idx[1][None, :, None, None, :, None], idx[2][None, None, :, None, None, :]]
        keep = P.view(pool, gr, stag)
        new = new.reshape(keep.shape).clone()
        # faces on a block's own planes stay its own
        for ax in range(3):
            if stag[ax]:
                sl = [slice(None)] + [slice(g, g + n[x] + (x == ax)) for x in (2, 1, 0)]
                new[tuple(sl)] = keep[tuple(sl)]
        keep.copy_(new)
    for w in W:
        fill(w, STAG["c"])
    for d in range(3):
        fill(B[d], STAG[d])


def _adm(case, eos, P, M, W, B):
    out = P.verts(10)
    r = case["vc_order"] // 2
    for gr, n, g, _ in _chunks(P):
        lo, reg = (-g,) * 3, [(-r, n[a] + r - 1) for a in range(3)]
        met = [_cut(_cells(P.view(M[c], gr, STAG["v"]), case["order"]), lo, reg) for c in range(4, 10)]
        w = [_cut(P.view(x, gr), lo, reg) for x in W]
        Bd = [_cut(x, lo, reg) for x in _cell_B([P.view(B[d], gr, STAG[d]) for d in range(3)])]
        f = _fluid(met, None, None, eos, w[:5], Bd)
        eW2 = f["e"] * f["W"] ** 2
        s = [eW2 - f["pt"] - f["ab0"] ** 2] + [eW2 * f["vl"][i] - f["ab0"] * f["bl"][i] for i in range(3)]
        for i in range(3):
            for j in range(i, 3):
                s.append(eW2 * f["vl"][i] * f["vl"][j] + f["pt"] * met[SYM[i][j]] - f["bl"][i] * f["bl"][j])
        wt = (0.5, 0.5) if r == 1 else (-1 / 16, 9 / 16, 9 / 16, -1 / 16)
        for c, a in enumerate(s):
            for d in range(3):
                k = n[d] + 1
                a = sum(x * a.narrow(DIM[d], i, k) for i, x in enumerate(wt))
            _cut(P.view(out[c], gr, STAG["v"]), lo, [(0, n[d]) for d in range(3)]).copy_(a)
    return out


def exact(case, seed):
    P, kind = _Pools(_blocks(case, seed)), case["kind"]
    M, W, B = _fill(case, seed, P)
    eos = _Eos(case)
    if kind == "adm":
        return {"sources": list(_adm(case, eos, P, M, W, B))}
    U = _ref_prim2con_pools(case, P, M, W, B)
    if kind == "prim2con":
        return {"U": list(U)}
    if kind == "con2prim":
        Uo, Wo = U.clone(), torch.zeros_like(W)
        for gr, n, g, _ in _chunks(P):
            inner, lo = [(0, n[a] - 1) for a in range(3)], (-g,) * 3
            met = [_cut(_cells(P.view(M[c], gr, STAG["v"]), case["order"]), lo, inner) for c in range(4, 10)]
            Bd = [_cut(x, lo, inner) for x in _cell_B([P.view(B[d], gr, STAG[d]) for d in range(3)])]
            q, w = _con2prim(case, eos, met, [_cut(P.view(x, gr), lo, inner) for x in U], Bd)
            for pool, vals in ((Uo, q), (Wo, w)):
                for i, x in enumerate(vals):
                    _cut(P.view(pool[i], gr), lo, inner).copy_(x)
        return {"U": list(Uo), "W": list(Wo), "status": None}
    if kind == "stage":
        Uo, Wo, Bo = torch.zeros_like(U), torch.zeros_like(W), [torch.zeros_like(b) for b in B]
        rk = (0.75, 0.25, 0.25) if case["rk_mid"] else (0.0, 1.0, 1.0)
        _stage_pools(case, eos, P, M, W, B, U, U, B, rk, _dt(P), (Uo, Wo, Bo))
        out = {"U": list(Uo), "B": Bo, "W": list(Wo), "status": None}
        if case["copies"]:
            out["W32"], out["B32"] = list(Wo[:6 if eos.tab is not None else 5]), Bo
        return out
    # a whole step: ghosts before every stage, the last stage written over the input
    _wrap_fill(case, P, W, B)
    dt = 0.2 * min(min(b.dx) for b in P.blocks)
    co = ((0.0, 1.0, 1.0), (0.5, 0.5, 0.5)) if case["rk_order"] == 2 else ((0.0, 1.0, 1.0), (0.75, 0.25, 0.25), (1 / 3, 2 / 3, 2 / 3))
    iU, iW, iB = U, W, B
    for k, rk in enumerate(co):
        oU, oW, oB = U.clone(), W.clone(), [b.clone() for b in B]   # ghosts of the outputs: those of the step's input
        _stage_pools(case, eos, P, M, iW, iB, iU, U, B, rk, dt, (oU, oW, oB))
        if k < len(co) - 1:
            _wrap_fill(case, P, oW, oB)
        iU, iW, iB = oU, oW, oB
    return {"U": list(iU), "B": iB, "W": list(iW), "status": None}
