"""Workloads of the library through its public entry points.

A case is one kind of call a user's program makes, at one size:

  fs       a formal solution of a new source on opacities set before (a
           program that drives its own outer iteration)
  fs_new   new opacities, then a formal solution with Lambda* (the first
           iteration of every wavelength)
  solve    new opacities, thermalisation and Planck function, then the outer
           iteration to convergence (one wavelength)
  os       one operator-splitting step with given J_fs and J_old
  batch    several wavelengths solved together from J = B
  noalloc  the allocation-free formal solution

``form`` is the arithmetic (fp64, fp32: the FP32 sweep, df64: double-float),
``method`` the discretisation (long, parabolic, short), ``law`` the slab
(lognormal: chi spread per voxel, eps per voxel over four decades; smooth:
chi with 20% noise, one eps).  Grids are nx x ny x nz with n_theta x n_phi
directions; the opacity rises by eight decades from the top to the bottom,
as in the workloads module.
"""

from __future__ import annotations

import math

import numpy as np
import torch

from paper_1107_5719_gb300 import rt3d as R
from paper_1107_5719_gb300 import workloads as W

FORMS = {"fp64": R.RT_FP64, "fp32": R.RT_FP32_SWEEP, "df64": R.RT_DF64}
DEV = "cuda:0"
NG_PERIOD = 4
TOL_INNER = 1e-12
MAX_ITER = 500


def _case(name, call, form, method, law, nx, ny, nz, n_theta, n_phi, bottom="planck",
          os_method="jacobi", tol=1e-8):
    c = dict(call=call, form=form, method=method, law=law, nx=nx, ny=ny, nz=nz, n_theta=n_theta,
             n_phi=n_phi, bottom=bottom, os_method=os_method, tol=tol)
    return dict(c, name=name) if name else c


def listed():
    return [
        # a program's own iteration on a small slab: one call is a few launches
        _case("fs_17_fp64", "fs", "fp64", "long", "smooth", 17, 17, 17, 16, 16),
        # the small slab converged: many short launches, mostly sweeps
        _case("solve_17_fp64", "solve", "fp64", "long", "smooth", 17, 17, 17, 16, 16),
        # the default benchmark: one wavelength of the 65^3 slab in FP64
        _case("solve_65_fp64", "solve", "fp64", "long", "lognormal", 65, 65, 65, 32, 32),
        # the same slab in the FP32-sweep form, to a tolerance its finishing stage reaches
        _case("solve_65_fp32", "solve", "fp32", "long", "lognormal", 65, 65, 65, 32, 32, tol=1e-10),
        # a ragged grid in double-float with the LTE-diffusion boundary, Gauss-Seidel sweeps
        _case("solve_ragged_df64", "solve", "df64", "long", "lognormal", 61, 45, 52, 16, 24,
              bottom="diffusion", os_method="gauss_seidel"),
        # first formal solution and Lambda* of a wavelength on a mid-sized grid
        _case("fs_new_33_fp64", "fs_new", "fp64", "long", "lognormal", 33, 33, 33, 16, 16),
        # the strong-scattering slab at full size: its recording does not fit
        # the device, every formal solution marches
        _case("fs_129_fp32", "fs", "fp32", "long", "smooth", 129, 129, 129, 64, 64),
        # short characteristics, double-float, converged
        _case("solve_short_65_df64", "solve", "df64", "short", "lognormal", 65, 65, 65, 32, 32),
        # second-order source, converged
        _case("solve_parabolic_33_fp64", "solve", "fp64", "parabolic", "smooth", 33, 33, 33, 16, 16),
        # operator splitting on the 129^3 grid
        _case("os_129", "os", "fp64", "long", "lognormal", 129, 129, 129, 8, 8),
        # six wavelengths of uneven size in one FP32-sweep batch
        _case("batch_fp32", "batch", "fp32", "long", "lognormal", 41, 41, 41, 16, 16, tol=1e-10),
        # a caller that may not allocate
        _case("noalloc_33", "noalloc", "fp64", "long", "lognormal", 33, 33, 33, 16, 16),
    ]


# Steps of the uncut march, directions x voxels x planes / 2, that a drawn
# case of each kind may take (at most the largest listed case of the kind).
_STEPS = {"fs": (1e5, 8e9), "fs_new": (1e5, 5e9), "solve": (3e5, 4e9), "batch": (3e6, 5e8),
          "noalloc": (1e5, 1.5e9)}


def draw(rng):
    call = rng.choice(["fs", "fs_new", "solve", "solve", "os", "batch", "noalloc"])
    form, method = "fp64", "long"
    if call in ("fs", "fs_new", "solve"):
        form, method = rng.choice([("fp64", "long"), ("fp64", "long"), ("fp32", "long"),
                                   ("df64", "long"), ("fp64", "short"), ("df64", "short"),
                                   ("fp64", "parabolic")])
    elif call == "batch":
        form = rng.choice(["fp32", "fp32", "fp64", "df64"])
    law = "smooth" if method == "parabolic" else rng.choice(["smooth", "lognormal"])
    bottom = "planck" if call == "noalloc" else rng.choice(["planck", "planck", "diffusion"])
    os_method = rng.choice(["jacobi", "jacobi", "gauss_seidel"])
    tol = 1e-10 if form == "fp32" else 1e-8
    if call == "os":
        lo, hi = math.log(9), math.log(128)
        n_theta = n_phi = 4
        nx, ny, nz = (max(3, int(math.exp(rng.uniform(lo, hi)))) for _ in range(3))
        return _case("", call, form, method, law, nx, ny, nz, n_theta, n_phi, bottom, os_method, tol)
    s_lo, s_hi = _STEPS[call]
    if method == "parabolic":
        s_hi = min(s_hi, 1e9)
    target = math.exp(rng.uniform(math.log(s_lo), math.log(s_hi)))
    while True:
        n_theta = 2 * rng.randint(2, 16)
        n_phi = rng.randint(5, 32)
        # N nz / 2 = target / directions, with ragged sides around its fourth root
        n = (2.0 * target / (n_theta * n_phi)) ** 0.25
        nx, ny, nz = (int(round(n * 2.0 ** rng.uniform(-0.4, 0.4))) for _ in range(3))
        steps = n_theta * n_phi * nx * ny * nz * nz / 2.0
        fits = call != "noalloc" or (64 * nx * ny * nz + 88 * n_theta * n_phi * (nz + 1)
                                     < R.RT_NOALLOC_SCRATCH_BYTES - 4096)
        if min(nx, ny) >= 5 and nz >= 4 and max(nx, ny, nz) <= 110 and steps <= s_hi and fits:
            return _case("", call, form, method, law, nx, ny, nz, n_theta, n_phi, bottom, os_method,
                         tol)


# ---- inputs -----------------------------------------------------------------

def _gen(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed))
    return g


def _slab(law, nx, ny, nz, g, scale=1.0):
    """chi, eps, B of one wavelength (FP64 CUDA tensors [nz][ny][nx])."""
    shape = (nz, ny, nx)
    k = torch.arange(nz, dtype=torch.float64, device=DEV)[:, None, None] / (nz - 1)
    if law == "lognormal":
        z = torch.randn(shape, dtype=torch.float64, device=DEV, generator=g)
        chi = scale * 10.0 ** (-4.0 + 8.0 * k) * torch.exp(0.3 * z)
        eps = 10.0 ** (-4.0 * torch.rand(shape, dtype=torch.float64, device=DEV, generator=g))
        B = ((1.0 + k) ** 4).expand(shape).contiguous()
    else:
        u = torch.rand(shape, dtype=torch.float64, device=DEV, generator=g)
        chi = scale * 10.0 ** (-4.0 + 8.0 * k) * (1.0 + 0.2 * (u - 0.5))
        eps = torch.full(shape, 1e-2, dtype=torch.float64, device=DEV)
        B = torch.ones(shape, dtype=torch.float64, device=DEV)
    return chi.contiguous(), eps.contiguous(), B


def _batch_shapes(c):
    """Six wavelengths: two at the case's grid, four at about half of it."""
    h = tuple(max(5, v // 2) for v in (c["nx"], c["ny"], c["nz"]))
    return [(c["nx"], c["ny"], c["nz"])] * 2 + [h] * 4


def _fields(c, seed):
    """The inputs of a case, from the seed alone."""
    g = _gen(seed)
    if c["call"] == "batch":
        out = []
        for nx, ny, nz in _batch_shapes(c):
            s = 10.0 ** float(-1.0 + 2.0 * torch.rand((), device=DEV, dtype=torch.float64, generator=g))
            e = 10.0 ** float(-2.0 * torch.rand((), device=DEV, dtype=torch.float64, generator=g))
            chi, _, B = _slab(c["law"], nx, ny, nz, g, s)
            out.append((chi, torch.full_like(chi, e), B))
        return out
    chi, eps, B = _slab(c["law"], c["nx"], c["ny"], c["nz"], g)
    f = {"chi": chi, "eps": eps, "B": B}
    if c["call"] in ("fs", "fs_new", "noalloc"):
        # the source of some iteration: B attenuated towards the surface, with structure
        u = torch.rand(chi.shape, dtype=torch.float64, device=DEV, generator=g)
        f["S"] = (B * (0.2 + 0.8 * eps) * (1.0 + 0.3 * (u - 0.5))).contiguous()
    if c["call"] == "os":
        u = torch.rand(chi.shape, dtype=torch.float64, device=DEV, generator=g)
        f["J_old"] = (B * (0.4 + 0.5 * u)).contiguous()
    return f


def _quadrature(c):
    return W.quadrature(c["n_theta"], c["n_phi"])


BOTTOM = {"planck": W.BC_PLANCK, "diffusion": W.BC_DIFFUSION}


class _Context:
    """A context handle, destroyed with the state."""

    def __init__(self, c):
        self.h = R.rt_create(0, FORMS[c["form"]])
        h = self.h
        R.rt_set_grid(h, c["nx"], c["ny"], c["nz"])
        R.rt_set_boundary(h, W.BC_ZERO, BOTTOM[c["bottom"]])
        R.rt_set_quadrature(h, *_quadrature(c))
        R.rt_set_ng(h, NG_PERIOD, 1e-6 if c["form"] == "fp32" else 0.0)
        if c["method"] == "short":
            R.rt_set_fs_method(h, R.RT_FS_SHORT)
        if c["method"] == "parabolic":
            R.rt_set_source_order(h, R.RT_SRC_PARABOLIC)
        if c["os_method"] == "gauss_seidel":
            R.rt_set_os_method(h, R.RT_OS_GAUSS_SEIDEL)

    def set(self, f):
        R.rt_set_opacity_dev(self.h, f["chi"])
        R.rt_set_epsilon_dev(self.h, f["eps"])
        R.rt_set_planck_dev(self.h, f["B"])

    def __del__(self):
        h, self.h = getattr(self, "h", None), None
        if h:
            R.rt_destroy(h)


class _Batch:
    """A batch handle, destroyed with the state."""

    def __init__(self, c, fields):
        mu, phi, w = _quadrature(c)
        probs = []
        for (chi, eps, B) in fields:
            nz, ny, nx = chi.shape
            probs.append(W.Problem(nx, ny, nz, chi.cpu().numpy(), eps.cpu().numpy(), B.cpu().numpy(),
                                   mu, phi, w, bottom_bc=BOTTOM[c["bottom"]]))
        self.n = len(probs)
        self.h = R.rt_batch_create(probs, precision=FORMS[c["form"]])
        R.rt_batch_set_ng(self.h, NG_PERIOD, 1e-6 if c["form"] == "fp32" else 0.0)
        if c["os_method"] == "gauss_seidel":
            R.rt_batch_set_os_method(self.h, R.RT_OS_GAUSS_SEIDEL)

    def __del__(self):
        h, self.h = getattr(self, "h", None), None
        if h:
            R.rt_batch_destroy(h)


def prepare(case, seed):
    c = case
    f = _fields(c, seed)
    st = {"case": c, "f": f}
    if c["call"] == "batch":
        st["batch"] = _Batch(c, f)
        st["J"] = [torch.empty_like(chi) for chi, _, _ in f]
        return st
    st["J"] = torch.empty_like(f["chi"])
    if c["call"] == "noalloc":
        st["quad"] = _quadrature(c)
        torch.cuda.synchronize()
        return st
    torch.cuda.synchronize()      # the context works on a stream of its own
    st["ctx"] = _Context(c)
    if c["call"] in ("fs", "os"):
        st["ctx"].set(f)
    if c["call"] == "fs_new":
        R.rt_set_epsilon_dev(st["ctx"].h, f["eps"])
        R.rt_set_planck_dev(st["ctx"].h, f["B"])
        st["L"] = torch.empty((27,) + tuple(f["chi"].shape), dtype=torch.float64, device=DEV)
    if c["call"] == "os":
        st["J_fs"] = torch.empty_like(f["chi"])
        R.rt_formal_solution_dev(st["ctx"].h, f["J_old"], st["J_fs"])
    return st


def run(state):
    c, f, J = state["case"], state["f"], state["J"]
    if c["call"] == "fs":
        R.rt_formal_solution_dev(state["ctx"].h, f["S"], J)
        return J
    if c["call"] == "fs_new":
        h = state["ctx"].h
        R.rt_set_opacity_dev(h, f["chi"])
        R.rt_formal_solution_dev(h, f["S"], J, state["L"])
        return {"J": J, "lstar": state["L"]}
    if c["call"] == "solve":
        state["ctx"].set(f)
        R.rt_solve_dev(state["ctx"].h, J, tol=c["tol"], max_iter=MAX_ITER, tol_inner=TOL_INNER)
        return J
    if c["call"] == "os":
        R.rt_os_step_dev(state["ctx"].h, state["J_fs"], f["J_old"], J, tol_inner=TOL_INNER)
        return J
    if c["call"] == "batch":
        b = state["batch"]
        R.rt_batch_reset(b.h, rebuild_lstar=True)
        R.rt_batch_solve(b.h, b.n, tol=c["tol"], max_iter=MAX_ITER, tol_inner=TOL_INNER)
        for p in range(b.n):
            R.rt_batch_get_J_dev(b.h, p, J[p])
        return J
    mu, phi, w = state["quad"]
    rc = R.rt_formal_solution_noalloc(c["nx"], c["ny"], c["nz"], 1.0, 1.0, 1.0, W.BC_ZERO,
                                      BOTTOM[c["bottom"]], mu, phi, w, f["chi"], f["S"], f["B"], J,
                                      torch.cuda.current_stream())
    if rc != R.RT_OK:
        raise R.RtError(rc, "rt_formal_solution_noalloc")
    return J


# ---- cost -------------------------------------------------------------------

_WIDTH = {"fp64": 8, "df64": 8, "fp32": 4}      # bytes of a value in the form's arithmetic


def _segments(nx, ny, nz, ndir, method):
    """(voxel, direction, segment) triples a formal solution integrates: one
    per pair for short characteristics; for long ones the segments up to the
    boundary or to an optical depth of 40 in the slab's mean opacity."""
    if method == "short":
        return float(nx * ny * (nz - 1)) * ndir
    chi = 10.0 ** (-4.0 + 8.0 * np.arange(nz) / (nz - 1))
    amu = np.array([0.2, 0.5, 0.8])
    n = 0.0
    for s in (1, -1):
        c = chi if s > 0 else chi[::-1]
        tau = np.concatenate([[0.0], np.cumsum(0.5 * (c[1:] + c[:-1]))])
        for m in amu:
            # upstream of plane k: planes k-1 .. 0
            n += sum(np.count_nonzero(tau[k] - tau[:k] <= 40.0 * m) + (tau[k] - tau[0] > 40.0 * m)
                     for k in range(nz)) / (2.0 * len(amu))
    return n * nx * ny * ndir


def _fs_work(c, nx, ny, nz):
    """A formal solution: chi, S, B read and J written once; per segment the
    bilinear chi and S (14), the optical depth (2), the exponential and the
    weights (about 25) and the update (6)."""
    seg = _segments(nx, ny, nz, c["n_theta"] * c["n_phi"], c["method"])
    per = 80.0 if c["method"] == "parabolic" else 47.0
    return 32.0 * nx * ny * nz, per * seg


def _iterations(c):
    return {"smooth": 17, "lognormal": 18}[c["law"]] * (1.25 if c["tol"] < 1e-8 else 1.0)


def work(case):
    c = case
    nx, ny, nz = c["nx"], c["ny"], c["nz"]
    N = nx * ny * nz
    sweep = (232.0 * N, 52.0 * N)               # 26 coefficients, r, J in, J out
    if c["call"] == "os":
        n = 30                                   # sweeps to 1e-12
        return {"bytes": 27 * 8.0 * N + 32.0 * N, "flops": n * sweep[1]}
    if c["call"] == "solve" or c["call"] == "batch":
        shapes = _batch_shapes(c) if c["call"] == "batch" else [(nx, ny, nz)]
        by = fl = 0.0
        for (x, y, z) in shapes:
            _, f = _fs_work(c, x, y, z)
            n = x * y * z
            it = _iterations(c)
            # the segments' weights once per opacity, then per iteration the
            # interpolation and accumulation of S (9 per segment) and ~25 sweeps
            seg = _segments(x, y, z, c["n_theta"] * c["n_phi"], c["method"])
            by += 32.0 * n
            fl += f + it * (9.0 * seg + 25 * 52.0 * n)
        return {"bytes": by, "flops": fl}
    by, fl = _fs_work(c, nx, ny, nz)
    if c["call"] == "fs":                        # opacities set before: their weights are at hand
        fl = 9.0 * _segments(nx, ny, nz, c["n_theta"] * c["n_phi"], c["method"])
    if c["call"] == "fs_new":
        by += 216.0 * N
    return {"bytes": by, "flops": fl}


# ---- 64-bit values ------------------------------------------------------------
# The definitions of include/rt3d.h in plain torch, vectorised over voxels and
# directions.

def _dirs(c):
    mu, phi, w = _quadrature(c)
    amu = np.abs(mu)
    st = np.sqrt(1.0 - mu * mu)
    return mu, amu, st * np.cos(phi) / amu, st * np.sin(phi) / amu, w


def _t(a, dtype=torch.float64):
    return torch.as_tensor(a, dtype=dtype, device=DEV)


class _Shift:
    """Bilinear interpolation at (i + X, j + Y) of every voxel, one shift per
    direction: nodes and weights."""

    def __init__(self, X, Y, nx, ny):
        fx, fy = np.floor(X), np.floor(Y)
        tx, ty = X - fx, Y - fy
        ix = (np.arange(nx)[None, :] + fx[:, None].astype(np.int64)) % nx
        iy = (np.arange(ny)[None, :] + fy[:, None].astype(np.int64)) % ny
        self.x = [_t(ix, torch.int64), _t((ix + 1) % nx, torch.int64)]
        self.y = [_t(iy, torch.int64), _t((iy + 1) % ny, torch.int64)]
        self.b = [(a, e, _t(u * v)[None, :, None, None])
                  for e, v in ((0, 1.0 - ty), (1, ty)) for a, u in ((0, 1.0 - tx), (1, tx))]

    def field(self, p):
        """p [K, ny, nx], the same for every direction -> [K, D, ny, nx]."""
        return sum(b * p[:, self.y[e][:, :, None], self.x[a][:, None, :]] for a, e, b in self.b)

    def per_direction(self, p):
        """p [D, ny, nx], one plane per direction -> the same shape."""
        d = torch.arange(p.shape[0], device=DEV)[:, None, None]
        return sum(b[0] * p[d, self.y[e][:, :, None], self.x[a][:, None, :]] for a, e, b in self.b)


def _weights(x):
    """w_cur, w_up, e of a segment of optical depth x (linear source)."""
    e = torch.exp(-x)
    z = torch.clamp(x, max=1.0)
    E, Q, t = torch.zeros_like(z), torch.zeros_like(z), torch.ones_like(z)
    for j in range(9):
        E = E + t / math.factorial(2 * j + 2)
        Q = Q + t / math.factorial(2 * j + 3)
        t = t * z * z
    q = -torch.expm1(-x) / x
    small = x < 0.5
    return torch.where(small, z * (E - z * Q), 1.0 - q), torch.where(small, e * z * (E + z * Q), q - e), e


def _moments(a):
    """E_0, E_1, E_2 of t^n e^-t over [0, a]."""
    e = torch.exp(-a)
    z = torch.clamp(a, max=1.0)
    t2, term = torch.zeros_like(z), z ** 3 / 6.0
    for k in range(4, 24):
        t2 = t2 + term
        term = term * z / k
    t1 = 0.5 * z * z + t2
    e0 = -torch.expm1(-a)
    e1 = torch.where(a < 1.0, e * t1, e0 - a * e)
    return e0, e1, torch.where(a < 1.0, 2.0 * e * t2, 2.0 * e1 - a * a * e), e


def _boundary(c, f, top, dtau):
    """[1, ny, nx] incoming intensity of the entry plane without its |mu|
    term, and the gradient that multiplies |mu| (or None)."""
    if top:
        return None, None
    return f["B"][-1:], (dtau if c["bottom"] == "diffusion" else None)


def _gradient(f):
    chi, B = f["chi"], f["B"]
    return ((B[-1] - B[-2]) / (0.5 * (chi[-1] + chi[-2])))[None]


def _fs_exact(c, f, S):
    """J of the formal solution of source S."""
    nz, ny, nx = S.shape
    mu, amu, ax, ay, w = _dirs(c)
    J = torch.zeros_like(S)
    chunk = max(1, int(3e7 // (nz * ny * nx)))
    grad = _gradient(f)
    for top in (True, False):
        sel = np.nonzero(mu > 0 if top else mu < 0)[0]
        chi = f["chi"] if top else f["chi"].flip(0)
        s = S if top else S.flip(0)
        ibc, gr = _boundary(c, f, top, grad)
        acc = torch.zeros_like(S)
        for i in range(0, len(sel), chunk):
            d = sel[i:i + chunk]
            ds = _t(1.0 / amu[d])[None, :, None, None]
            wd = _t(w[d])[None, :, None, None]
            am = _t(amu[d])[None, :, None, None]
            shift = lambda m: _Shift(-m * ax[d], -m * ay[d], nx, ny)  # noqa: E731
            if c["method"] == "short":
                I = torch.zeros((len(d), ny, nx), dtype=torch.float64, device=DEV)
                if ibc is not None:
                    I = I + ibc + (am[0] * gr if gr is not None else 0.0)
                acc[0] += (wd[0] * I).sum(0)
                sh = shift(1)
                for k in range(1, nz):
                    x = 0.5 * ds[0] * (chi[k] + sh.field(chi[k - 1:k])[0])
                    wc, wu, e = _weights(x)
                    I = sh.per_direction(I) * e + wc * s[k] + wu * sh.field(s[k - 1:k])[0]
                    acc[k] += (wd[0] * I).sum(0)
                continue
            I = torch.zeros((nz, len(d), ny, nx), dtype=torch.float64, device=DEV)
            T = torch.ones_like(I)
            ca, sa = chi[:, None], s[:, None]
            xprev = sprev = None
            if c["method"] == "parabolic":       # the point one plane downstream, where it exists
                dn = _Shift(ax[d], ay[d], nx, ny)
                xprev = torch.ones_like(I)
                sprev = torch.zeros_like(I)
                xprev[:-1] = 0.5 * ds * (chi[:-1, None] + dn.field(chi[1:]))
                sprev[:-1] = dn.field(s[1:])
            for m in range(nz):
                if ibc is not None:              # voxels of plane m have reached the entry plane
                    sh = shift(m)
                    b = sh.field(ibc) + (am * sh.field(gr) if gr is not None else 0.0)
                    I[m] += (T[m:m + 1] * b)[0]
                if m == nz - 1:
                    break
                sh = shift(m + 1)
                cb, sb = sh.field(chi[:nz - m - 1]), sh.field(s[:nz - m - 1])
                ca, sa = (ca[1:], sa[1:])
                x = 0.5 * ds * (ca + cb)
                wc, wu, e = _weights(x)
                t = T[m + 1:]
                add = wc * sa + wu * sb
                if c["method"] == "parabolic":
                    xp, sp = xprev[-(nz - m - 1):], sprev[-(nz - m - 1):]
                    e0, e1, e2, _ = _moments(x)
                    par = ((e2 + xp * e1) / (x * (x + xp)) * sb
                           + (x * xp * e0 - (xp - x) * e1 - e2) / (x * xp) * sa
                           + (e2 - x * e1) / (xp * (x + xp)) * sp)
                    if m == 0:                   # the last plane has no downstream point
                        par[-1] = add[-1]
                    add, xprev, sprev = par, x, sa.expand_as(sb)
                I[m + 1:] += t * add
                T[m + 1:] = t * e
                ca, sa = cb, sb
            acc += (wd * I).sum(1)
        J += acc if top else acc.flip(0)
    return J


def _lstar_exact(c, f):
    """Lambda* [27, nz, ny, nx] (long characteristics, linear source)."""
    chi = f["chi"]
    nz, ny, nx = chi.shape
    mu, amu, ax, ay, w = _dirs(c)
    L = torch.zeros((27, nz, ny, nx), dtype=torch.float64, device=DEV)
    near = lambda r, n: {0: 0, 1: 1, n - 1: -1}.get(r)  # noqa: E731
    for top in (True, False):
        ch = chi if top else chi.flip(0)
        Lt = torch.zeros((27, nz, ny, nx), dtype=torch.float64, device=DEV)
        oz = -1 if top else 1
        for d in np.nonzero(mu > 0 if top else mu < 0)[0]:
            one, two = (_Shift(-m * ax[d:d + 1], -m * ay[d:d + 1], nx, ny) for m in (1, 2))
            c1 = one.field(ch[:-1])[:, 0]
            wc, wu, e = _weights(0.5 / amu[d] * (ch[1:] + c1))
            up = wu.clone()
            wc1, _, _ = _weights(0.5 / amu[d] * (c1[1:] + two.field(ch[:-2])[:, 0]))
            up[1:] += e[1:] * wc1
            Lt[13, 1:] += w[d] * wc
            fx, fy = math.floor(-ax[d]), math.floor(-ay[d])
            for a, b_y, b in one.b:
                ox, oy = near((fx + a) % nx, nx), near((fy + b_y) % ny, ny)
                if ox is not None and oy is not None:
                    Lt[(oz + 1) * 9 + (oy + 1) * 3 + ox + 1, 1:] += float(b) * w[d] * up
        L += Lt if top else Lt.flip(1)
    return L


def _neighbours(J):
    """[27, nz, ny, nx] values at the 27 offsets (0 outside in z)."""
    out = []
    for o in range(27):
        ox, oy, oz = o % 3 - 1, (o // 3) % 3 - 1, o // 9 - 1
        v = torch.roll(J, (-oy, -ox), (1, 2))
        if oz:
            z = torch.zeros_like(v)
            if oz > 0:
                z[:-1] = v[1:]
            else:
                z[1:] = v[:-1]
            v = z
        out.append(v)
    return out


def _os_exact(L, eps, J_fs, J_old, tol):
    """J_new of (1 - Lambda* D) J_new = J_fs - Lambda* D J_old by Jacobi sweeps."""
    one = [a * b for a, b in zip(L, _neighbours(1.0 - eps))]
    diag = 1.0 - one[13]
    r = (J_fs - sum(a * b for a, b in zip(one, _neighbours(J_old)))) / diag
    one = [a / diag for a in one]
    J = J_old
    for _ in range(1000):
        nb = _neighbours(J)
        Jn = r + sum(one[o] * nb[o] for o in range(27) if o != 13)
        done = float(((Jn - J) / Jn).abs().max()) < tol
        J = Jn
        if done:
            break
    return J


def _solve_exact(c, f):
    """The fixed point J = J_FS(eps B + (1 - eps) J), iterated with operator
    splitting and Ng to rounding."""
    L = _lstar_exact(c, f)
    eps, B = f["eps"], f["B"]
    J, hist = B, []
    for it in range(1, 120):
        Jn = _os_exact(L, eps, _fs_exact(c, f, eps * B + (1.0 - eps) * J), J, 1e-13)
        hist = [J] + hist[:2]
        if it % NG_PERIOD == 0 and len(hist) == 3:
            d0, d1, d2 = Jn - hist[0], hist[0] - hist[1], hist[1] - hist[2]
            q1, q2, wt = d0 - d1, d0 - d2, 1.0 / (Jn * Jn)
            a11, a12, a22, b1, b2 = (float((wt * u * v).sum()) for u, v in
                                     ((q1, q1), (q1, q2), (q2, q2), (d0, q1), (d0, q2)))
            det = a11 * a22 - a12 * a12
            if det != 0.0:
                a, b = (b1 * a22 - b2 * a12) / det, (b2 * a11 - b1 * a12) / det
                Jn = (1.0 - a - b) * Jn + a * hist[0] + b * hist[1]
            hist = []
        delta = float(((Jn - J) / Jn).abs().max())
        J = Jn
        if delta < 1e-12:
            break
    return J


def exact(case, seed):
    c = case
    ndir = c["n_theta"] * c["n_phi"]
    steps = ndir * c["nx"] * c["ny"] * c["nz"] ** 2 / 2.0
    f = _fields(c, seed)
    if c["call"] == "os":
        if c["nx"] < 4 or c["ny"] < 4 or c["nz"] < 3:
            return None
        L = _lstar_exact(c, f)
        return _os_exact(L, f["eps"], _fs_exact(c, f, f["J_old"]), f["J_old"], TOL_INNER)
    if c["method"] == "short":
        steps = steps / c["nz"]
    if c["call"] in ("fs", "noalloc"):
        return _fs_exact(c, f, f["S"]) if steps < 1.2e10 else None
    if c["call"] == "fs_new":
        if steps >= 1.2e10:
            return None
        J = _fs_exact(c, f, f["S"])
        return {"J": J, "lstar": _lstar_exact(c, f) if c["method"] == "long" else None}
    if c["method"] != "long":
        return None          # the fixed point needs that method's own Lambda* only for speed
    if c["call"] == "batch":
        if steps > 4e7:
            return None
        return [_solve_exact(c, dict(chi=chi, eps=eps, B=B)) for chi, eps, B in f]
    return _solve_exact(c, f) if steps < 4e7 else None
