"""What a user of the library has it do: the calls whose time matters.

Every case goes through the public binding (paper_2102_01734_gb300.rt3d and
.warmstart). Sizes are those of the repository's own configurations, tests and
benchmark (33^3 with 8 x 16 solid angles, 97^3 with 16 x 32, 129^3 with
32 x 64, the 65 x 65 x 257 box of the paper's periodic test, the 65 x 33 x 65
shell) and, in draw(), sizes between them.

Kinds:
  fs       one formal solution on the periodic box, in FP32, float-float (ff)
           or FP64, with or without the non-local Lambda* band
  ali      one ALI step (source, formal solution, Jacobi solve, update)
  os       one operator-splitting solve with a given Lambda* band
  solve    a converged solve, its Lambda* band built anew
  batched  converged solves of several wavelengths that share the geometry
  sph      one formal solution on the spherical shell
  train    forward, loss and backward pass of the warm-start network
  predict  the warm-start network's prediction

The atmospheres follow inputs.cartesian_config (vertical opacity over six
decades times a lognormal k^-3 field, B = 1 + 0.2 field), drawn on the GPU.
"""
import math

import numpy as np
import torch

from paper_2102_01734_gb300 import inputs, rt3d, warmstart

DEV = "cuda"
PRECISION = {"fp64": rt3d.FP64, "fp32": rt3d.FP32_FS_FP64_ALI, "ff": rt3d.FP32_FS_FF_REFINE}
SOLVER = {"jacobi": rt3d.OS_JACOBI, "gs": rt3d.OS_GAUSS_SEIDEL}


# --------------------------------------------------------------- the cases
def _box(kind, name=None, *, n, angles, precision="fp32", parabolic=True, eps=1e-6, **more):
    c = {"kind": kind, "nx": n[0], "ny": n[1], "nz": n[2], "ntheta": angles[0], "nphi": angles[1],
         "precision": precision, "parabolic": parabolic, "eps": eps, **more}
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # the small box of the plain method's configuration, one formal
        # solution in single precision: launches and latency
        _box("fs", "fs32_33", n=(33, 33, 33), angles=(8, 16), lstar=False),
        # the benchmark's box: the call that carries a solve's time
        _box("fs", "fs32_129", n=(129, 129, 129), angles=(32, 64), lstar=False),
        # first iteration of a solve on the paper's periodic test box: the
        # formal solution that also builds Lambda*
        _box("fs", "fs32_lstar_65x65x257", n=(65, 65, 257), angles=(16, 32), lstar=True),
        # the plain FP64 method on its own configuration (linear source)
        _box("fs", "fs64_33", n=(33, 33, 33), angles=(8, 16), precision="fp64", parabolic=False,
             eps=1e-2, lstar=False),
        # a refinement residual on the batched configuration's box
        _box("fs", "fsff_97", n=(97, 97, 97), angles=(16, 32), precision="ff", lstar=False),
        # an ALI iteration of a user who steps by hand, band already built
        _box("ali", "ali_97", n=(97, 97, 97), angles=(16, 32)),
        # the preconditioner's solve of the benchmark
        {"kind": "os", "name": "os_gs_129", "nx": 129, "ny": 129, "nz": 129, "precision": "fp32",
         "solver": "gs", "eps": 1e-6},
        # whole converged solves: the plain FP64 configuration, and the mixed
        # precision with float-float refinement on the field
        _box("solve", "solve64_33", n=(33, 33, 33), angles=(8, 16), precision="fp64",
             parabolic=False, eps=1e-2, solver="jacobi"),
        _box("solve", "solve_ff_65", n=(65, 65, 65), angles=(16, 32), precision="ff", eps=1e-4,
             solver="gs"),
        # wavelengths of uneven opacity and eps on one geometry
        _box("batched", "batched_8x33", n=(33, 33, 33), angles=(8, 16), precision="ff",
             nlambda=8),
        # the shell of the irradiated test case
        {"kind": "sph", "name": "sph32_65x33x65", "nr": 65, "nt": 33, "np": 65, "ntheta": 16,
         "nphi": 32, "precision": "fp32", "parabolic": True},
        # one training step of the warm start on its training box
        {"kind": "train", "name": "train_32x32x193", "nx": 32, "ny": 32, "nz": 193},
    ]


def draw(rng):
    """One more case of the same ranges."""
    def size(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(["fs", "fs", "fs", "fs", "ali", "os", "solve", "sph", "train", "predict"])
    if kind in ("train", "predict"):
        return {"kind": kind, "nx": size(16, 65), "ny": size(16, 65), "nz": size(16, 193)}
    if kind == "os":
        return {"kind": "os", "nx": size(12, 129), "ny": size(12, 129), "nz": size(8, 129),
                "precision": rng.choice(["fp32", "fp32", "fp64"]),
                "solver": rng.choice(["jacobi", "gs"]), "eps": 10.0 ** rng.uniform(-6, -3)}
    if kind == "sph":
        return {"kind": "sph", "nr": size(12, 65), "nt": size(9, 33), "np": size(12, 65),
                "ntheta": 2 * size(2, 8), "nphi": 4 * size(1, 8),
                "precision": rng.choice(["fp32", "fp32", "ff", "fp64"]),
                "parabolic": rng.random() < 0.75}
    big = 2.0e8 if kind == "solve" else 2.9e10
    while True:
        precision = rng.choice(["fp32", "fp32", "fp32", "ff", "fp64"])
        lstar = kind == "fs" and rng.random() < 0.3
        # the slower kinds stay below the time of the largest listed call
        cap = big
        if kind != "solve":
            cap = {"fp32": 2.9e10, "ff": 4.0e9, "fp64": 6.0e8}[precision] / (4.0 if lstar else 1.0)
        elif precision == "fp64":
            cap = 3.0e7
        angles = rng.choice([(4, 8), (8, 16), (16, 32), (32, 64)])
        hi = 65 if kind == "solve" else 129
        c = _box(kind, n=(size(12, hi), size(12, hi), size(9, 129)), angles=angles,
                 precision=precision, parabolic=rng.random() < 0.75, eps=10.0 ** rng.uniform(-6, -2))
        if kind == "fs":
            c["lstar"] = lstar and precision != "ff"
        if kind == "solve":
            c["solver"] = rng.choice(["jacobi", "gs"])
            c["eps"] = max(c["eps"], 1e-4)
        if 1e6 < _segments(c) < cap:
            return c


# ------------------------------------------------------------------ inputs
def _field(shape, gen):
    """Gaussian field with spectrum k^-3, unit variance, clipped at 4.5."""
    f = torch.fft.fftn(torch.randn(shape, generator=gen, dtype=torch.float64, device=DEV))
    k = [torch.fft.fftfreq(n, dtype=torch.float64, device=DEV) for n in shape]
    k2 = k[0][:, None, None] ** 2 + k[1][None, :, None] ** 2 + k[2][None, None, :] ** 2
    k2[0, 0, 0] = 1.0
    amp = k2 ** -0.75
    amp[0, 0, 0] = 0.0
    g = torch.fft.ifftn(f * amp).real
    g = g - g.mean()
    return (g / g.std()).clamp(-4.5, 4.5)


def _atmosphere(nx, ny, nz, eps, seed):
    """(chi, eps, B, J, I_bottom): J grows from the outer layer, where it is
    a few per cent of B, to B below optical depth one."""
    gen = torch.Generator(device=DEV).manual_seed(seed)
    shape = (nz, ny, nx)
    g = _field(shape, gen)
    chi = torch.from_numpy(inputs.vertical_chi(nz)).to(DEV)[:, None, None] * torch.exp(0.5 * g)
    B = 1.0 + 0.2 * g
    tau = torch.flip(torch.cumsum(torch.flip(chi, [0]), 0), [0]) - 0.5 * chi
    J = B * (0.02 + 0.98 * tau / (1.0 + tau))
    return chi.contiguous(), torch.full_like(B, eps), B.contiguous(), J.contiguous(), B[0].clone()


def _band(chi, gen):
    """A Lambda* band of the shape the formal solution gives: rows sum to the
    trapping probability of their voxel, most of it on the diagonal, and
    nothing outside the box."""
    nz, ny, nx = chi.shape
    trap = chi / (chi + 1.0)
    w = torch.rand((27, nz, ny, nx), generator=gen, dtype=torch.float64, device=DEV)
    w[13] = 0.0
    w[:9, 0] = 0.0
    w[18:, nz - 1] = 0.0
    w *= (0.3 * trap / w.sum(0))[None]
    w[13] = 0.7 * trap
    return w.view(27, -1)


class _State:
    pass


def prepare(case, seed):
    s = _State()
    s.case = c = dict(case)
    kind = c["kind"]
    if kind == "sph":
        gen = torch.Generator(device=DEV).manual_seed(seed)
        n = (c["nr"], c["nt"], c["np"])
        chi, eps, B, bc = inputs.spherical_config(n, 1e-4)
        f = _field((c["np"], c["nt"], c["nr"]), gen)
        s.chi = (torch.from_numpy(chi).to(DEV) * torch.exp(0.2 * f)).contiguous()
        s.S = (0.2 + 0.8 * s.chi / (1.0 + s.chi)) * (1.0 + 0.1 * f)
        s.bc = {"I_top": 0.0, "I_bottom": torch.from_numpy(bc["I_bottom"]).to(DEV),
                "I_irr": bc["I_irr"]}
        s.grid = rt3d.Grid(n, c["ntheta"], c["nphi"],
                           rt3d.PARABOLIC if c["parabolic"] else rt3d.LINEAR,
                           PRECISION[c["precision"]], geometry=rt3d.SPHERICAL)
        return s
    nx, ny, nz = c["nx"], c["ny"], c["nz"]
    if kind in ("train", "predict"):
        chi, eps, B, J, _ = _atmosphere(nx, ny, nz, 1e-6, seed)
        s.chi, s.eps, s.B, s.J = chi[None], eps[None], B[None], J[None]
        s.net = warmstart.UNet(seed=seed, device=DEV)
        return s
    if kind == "os":
        s.chi, s.eps, s.B, s.J, _ = _atmosphere(nx, ny, nz, c["eps"], seed)
        gen = torch.Generator(device=DEV).manual_seed(seed + 1)
        s.lstar = _band(s.chi, gen)
        s.r = 1e-2 * s.J * (1.0 + 0.3 * torch.randn(s.J.shape, generator=gen, dtype=torch.float64,
                                                     device=DEV))
        # the direction set plays no part in this call
        s.grid = rt3d.Grid((nx, ny, nz), 2, 4, rt3d.LINEAR, PRECISION[c["precision"]])
        s.grid.set_os_solver(SOLVER[c["solver"]])
        return s
    interp = rt3d.PARABOLIC if c["parabolic"] else rt3d.LINEAR
    if kind == "batched":
        one = [_atmosphere(nx, ny, nz, c["eps"], seed)] * c["nlambda"]
        eps, scale = inputs.batched_wavelengths(c["nlambda"], seed % (1 << 31))
        d = lambda v: torch.from_numpy(v).to(DEV)[:, None, None, None]
        s.chi = (torch.stack([a[0] for a in one]) * d(scale)).contiguous()
        s.B = torch.stack([a[2] for a in one]).contiguous()
        s.eps = (torch.ones_like(s.B) * d(eps)).contiguous()
        s.bc = {"I_top": 0.0, "I_bottom": torch.stack([a[4] for a in one]).contiguous()}
        s.grid = rt3d.Grid((nx, ny, nz), c["ntheta"], c["nphi"], interp, PRECISION[c["precision"]])
        return s
    s.chi, s.eps, s.B, s.J, bottom = _atmosphere(nx, ny, nz, c["eps"], seed)
    s.S = (1.0 - s.eps) * s.J + s.eps * s.B
    s.bc = {"I_top": 0.0, "I_bottom": bottom}
    s.grid = rt3d.Grid((nx, ny, nz), c["ntheta"], c["nphi"], interp, PRECISION[c["precision"]])
    if kind == "solve":
        s.grid.set_os_solver(SOLVER[c["solver"]])
    return s


# --------------------------------------------------------------- one pass
def run(s):
    c = s.case
    kind = c["kind"]
    if kind == "fs" or kind == "sph":
        if c["precision"] == "ff":
            return s.grid.formal_solution_ff(s.chi, s.S, s.bc)
        return s.grid.formal_solution(s.chi, s.S, s.bc, lstar=c.get("lstar", False))
    if kind == "ali":
        J = s.J.clone()
        rel = s.grid.ali_step(s.chi, s.eps, s.B, s.bc, J)
        return J, rel
    if kind == "os":
        return s.grid.os_solve(s.lstar, s.eps, s.r)
    if kind == "solve":
        J = s.B.clone()
        s.grid.invalidate_lstar()
        s.grid.solve(s.chi, s.eps, s.B, s.bc, J)
        return J
    if kind == "batched":
        J = s.B.clone()
        s.grid.solve_batched(s.chi, s.eps, s.B, s.bc, J)
        return J
    if kind == "predict":
        return s.net.predict(s.chi, s.eps, s.B, s.B)
    X = s.net.features(s.chi, s.eps, s.B, s.B)
    y = s.net.forward(X, tuple(s.chi.shape[1:]))
    sse, dY = s.net.loss_grad(y, s.J, s.B)
    gW, gb = s.net.backward(dY)
    return {"sse": sse, "gW": [gW[l[0]] for l in warmstart.LAYERS],
            "gb": [gb[l[0]] for l in warmstart.LAYERS]}


# ------------------------------------------------------- work and tolerance
def _directions(ntheta, nphi):
    mu = -1.0 + (2 * np.arange(ntheta) + 1) / ntheta
    ph = (2 * np.arange(nphi) + 1) * np.pi / nphi
    st = np.sqrt((1.0 - mu) * (1.0 + mu))
    return np.stack([(st[:, None] * np.cos(ph)).ravel(), (st[:, None] * np.sin(ph)).ravel(),
                     np.repeat(mu, nphi)], 1)


def _segments(c):
    d = np.abs(_directions(c["ntheta"], c["nphi"]))
    span = c["nz"] / d[:, 2]
    points = c["nz"] + np.floor(d[:, 0] * span + 0.5) + np.floor(d[:, 1] * span + 0.5)
    return float(points.sum()) * c["nx"] * c["ny"]


# operations of one segment (interval functions, parabolic weights, update
# and J weight), and of the up to nine window entries of Lambda*
SEG_OPS, LSTAR_OPS = 28, 18


def work(case):
    c = case
    kind = c["kind"]
    if kind in ("train", "predict"):
        v = c["nx"] * c["ny"] * c["nz"]
        per = {"e1a": 1, "e1b": 1, "e2a": 8, "e2b": 8, "b_a": 64, "b_b": 64, "d2a": 8, "d2b": 8,
               "d1a": 1, "d1b": 1, "out": 1}
        mac = sum(27 * l[1] * l[2] * v / per[l[0]] for l in warmstart.LAYERS)
        weights = sum(27 * l[1] * l[2] + l[2] for l in warmstart.LAYERS)
        if kind == "predict":
            return {"bytes": 40 * v + 2 * weights, "flops": 2 * mac}
        return {"bytes": 40 * v + 6 * weights, "flops": 6 * mac}
    if kind == "sph":
        v = c["nr"] * c["nt"] * c["np"]
        # a cell is crossed by 1.4 to 1.9 rays of every direction
        return {"bytes": 24 * v, "flops": 1.5 * SEG_OPS * v * c["ntheta"] * c["nphi"]}
    v = c["nx"] * c["ny"] * c["nz"]
    if kind == "os":
        return {"bytes": 8 * v * (27 + 3), "flops": 2.0 * 27 * v * 50}
    seg = _segments(c)
    if kind == "fs":
        lstar = c["lstar"]
        return {"bytes": 8 * v * (3 + (27 if lstar else 0)),
                "flops": seg * (SEG_OPS + (LSTAR_OPS if lstar else 0))}
    if kind == "ali":
        return {"bytes": 8 * v * 5, "flops": seg * SEG_OPS + 2.0 * 27 * v * 50}
    # converged solves: some thirty formal solutions, the first with Lambda*
    nl = c.get("nlambda", 1)
    return {"bytes": 8 * v * 5 * nl, "flops": nl * seg * (30 * SEG_OPS + LSTAR_OPS)}


def tolerance(case):
    c = case
    kind = c["kind"]
    if kind in ("fs", "sph"):
        # measured against exact(): 2e-8 (fp32, the rounding of a segment
        # averaged over the directions; more with few of them), 3e-15 (ff),
        # 1e-15 (fp64)
        return {"fp32": {"rel": 4e-7, "max": 4e-6}, "ff": {"rel": 2e-14, "max": 1e-11},
                "fp64": {"rel": 1e-14, "max": 1e-13}}[c["precision"]]
    if kind == "ali":
        # measured against exact(): 3e-6, the FP32 formal solution's rounding
        # as the solve of the nearly singular system amplifies it
        return {"rel": 1.2e-5, "max": 1.2e-4} if c["precision"] != "fp64" else {"rel": 1e-12, "max": 1e-11}
    if kind == "os":
        # measured against exact(): 8e-8 (FP32 coefficients)
        return {"rel": 4e-7, "max": 4e-6} if c["precision"] != "fp64" else {"rel": 1e-13, "max": 1e-12}
    if kind in ("solve", "batched"):
        # each solve certifies an estimated relative error of 1e-8; the
        # batch's wavelengths reach down to eps = 1e-8, where the estimate is
        # loosest (2e-8, at most 3e-7 between two runs)
        return {"rel": 2e-8, "max": 1e-7} if kind == "solve" else {"rel": 8e-8, "max": 1e-6}
    # BF16 activations: 3e-3 to 1e-2 against exact(), and a sum in another
    # order rounds some of them the other way
    return {"rel": 1e-2, "max": 0.2}


# -------------------------------------------------------- the same in 64 bits
def _trace(nx, ny, nz, d):
    """Points of the characteristic from face cell (0, 0): unwrapped x, y,
    layer, chord, and the chord sum of the point's layer."""
    a = np.abs(d)
    end = nz / a[2]
    m = lambda q: (np.arange(1, int(q * end + 0.5) + 2) - 0.5) / q
    tx, ty, tz = m(a[0]), m(a[1]), np.arange(1, nz + 1) / a[2]
    t = np.unique(np.concatenate([tx, ty, tz]))
    t = np.concatenate([[0.0], t[t <= tz[-1]]])
    s = np.sign(d).astype(np.int64)
    x = s[0] * np.searchsorted(tx, t[:-1], side="right")
    y = s[1] * np.searchsorted(ty, t[:-1], side="right")
    z = np.searchsorted(tz, t[:-1], side="right") * s[2] + (0 if d[2] > 0 else nz - 1)
    length = np.diff(t)
    return x, y, z, length, np.bincount(z, length, nz)[z]


def _windows(x, y, z, nx, ny):
    """Ring positions 0..8 (points k-7 .. k+1) of the passage window of every
    point: the neighbour's index in 0..26, or -1."""
    k = len(x)
    out = -np.ones((9, k), np.int64)
    alive = np.ones(k, bool)
    for r in range(8, -1, -1):
        j = np.arange(k) + r - 7
        ok = (j >= 0) & (j < k)
        jc = np.clip(j, 0, k - 1)
        dd = []
        for p, n in ((x, nx), (y, ny)):
            q = (p[jc] - p) % n
            dd.append(np.where(q == n - 1, -1, q))
        dz = z[jc] - z
        near = ok & (dd[0] <= 1) & (dd[1] <= 1) & (np.abs(dz) <= 1)
        if r == 8:  # the last point's window ends at itself
            use, alive = near, near | ~ok
        else:
            alive = alive & near
            use = alive
        out[r] = np.where(use, (dd[0] + 1) + 3 * (dd[1] + 1) + 9 * (dz + 1), -1)
    return out


def _interval(u):
    """e0, a = e1/u, d = a - e2/u^2 of the interval of optical depth u."""
    small = u < 0.1
    us = torch.where(small, u, torch.zeros_like(u))
    p = torch.zeros_like(u)
    for m in range(9, -1, -1):
        p = p * us + (-2.0 if m % 2 else 2.0) / math.factorial(m + 3)
    b = us * p
    a = 0.5 * us * (1.0 - b)
    ub = torch.where(small, torch.ones_like(u), u)
    e0 = -torch.expm1(-ub)
    ab = 1.0 - e0 / ub
    return (torch.where(small, us * (1.0 - a), e0), torch.where(small, a, ab),
            torch.where(small, a - b, (2.0 * ab - e0) / ub))


def _formal_solution(c, chi, S, bottom, lstar):
    """J (and the Lambda* band) by marching all characteristics of all
    directions a point at a time, in double precision."""
    nx, ny, nz = c["nx"], c["ny"], c["nz"]
    dirs = _directions(c["ntheta"], c["nphi"])
    tr = [_trace(nx, ny, nz, d) for d in dirs]
    order = sorted(range(len(tr)), key=lambda i: -len(tr[i][0]))
    K = [len(tr[i][0]) for i in order]
    A, kmax, nray, N = len(tr), max(K), nx * ny, nx * ny * nz

    def table(rows, dtype):
        t = np.zeros((kmax, A), dtype)
        for a, r in enumerate(rows):
            t[:len(r), a] = r
        return torch.from_numpy(t).to(DEV)

    w = 1.0 / A
    X = table([tr[i][0] % nx for i in order], np.int32)
    Y = table([tr[i][1] % ny for i in order], np.int32)
    Z = table([tr[i][2] for i in order], np.int32)
    L = table([tr[i][3] for i in order], np.float64)
    C = table([w * tr[i][3] / tr[i][4] for i in order], np.float64)
    live = np.array([sum(1 for q in K if q > k) for k in range(kmax + 1)])
    win = None
    if lstar:
        wd = -np.ones((kmax, 9, A), np.int8)
        for a, i in enumerate(order):
            wd[:K[a], :, a] = _windows(*tr[i][:3], nx, ny).T
        win = torch.from_numpy(wd).to(DEV)
    ray = torch.arange(nray, device=DEV)
    x0, y0 = (ray % nx)[None], (ray // nx)[None]
    chif, Sf = chi.reshape(-1), S.reshape(-1)
    J = torch.zeros(N, dtype=torch.float64, device=DEV)
    band = torch.zeros(27 * N, dtype=torch.float64, device=DEV) if lstar else None
    up = torch.tensor([dirs[i][2] > 0 for i in order], device=DEV)
    chunk = max(1, int((6e6 if not lstar else 3e6) // nray))
    for a0 in range(0, A, chunk):
        na = min(chunk, A - a0)

        def at(k, n):
            sl = slice(a0, a0 + n)
            xi = x0 + X[k, sl, None]
            yi = y0 + Y[k, sl, None]
            v = (xi - nx * (xi >= nx)) + nx * ((yi - ny * (yi >= ny)) + ny * Z[k, sl, None])
            return v.long(), 0.5 * L[k, sl, None]

        I = torch.where(up[a0:a0 + na, None], bottom.reshape(1, -1), torch.zeros(1, 1, device=DEV,
                                                                                 dtype=torch.float64))
        v, hl = at(0, na)
        hc = chif[v] * hl
        u = hc
        Sc = Sf[v]
        Sp = Sc
        ring = [torch.zeros_like(I) for _ in range(9)] if lstar else None
        for k in range(K[a0]):
            n = int(min(max(live[k] - a0, 0), na))
            nn = int(min(max(live[k + 1] - a0, 0), na))
            I, u, hc, Sc, Sp, v = (q[:n] for q in (I, u, hc, Sc, Sp, v))
            e0, a, d = _interval(u)
            al, be = e0 - a, a
            ga = torch.zeros_like(u)
            Sn = Sc
            if nn:
                vn, hl = at(k + 1, nn)
                hn = chif[vn] * hl
                Sn = torch.cat([Sf[vn], Sc[nn:]]) if nn < n else Sf[vn]
                wn = hc[:nn] + hn
                if c["parabolic"]:
                    q = u[:nn] / wn
                    f = (2.0 - 2.0 * u[:nn]).clamp(0, 1) * (2.0 - 0.5 * q).clamp(0, 1)
                    sd = f * (u[:nn] / (u[:nn] + wn)) * d[:nn]
                    if nn < n:
                        pad = torch.zeros((n - nn, nray), dtype=torch.float64, device=DEV)
                        sd, q = torch.cat([sd, pad]), torch.cat([q, pad])
                    ga = -q * sd
                    al = al - sd
                    be = be + sd
            E = 1.0 - e0
            I = E * I + al * Sp + be * Sc + ga * (Sn - Sc)
            cw = C[k, a0:a0 + n, None]
            J.index_add_(0, v.reshape(-1), (cw * I).reshape(-1))
            if lstar:
                ring = [E * r[:n] for r in ring[1:]] + [ga]
                ring[7 if k == 0 else 6] = ring[7 if k == 0 else 6] + al
                ring[7] = ring[7] + be - ga
                codes = win[k, :, a0:a0 + n]
                for r in range(9):
                    pick = (codes[r] >= 0).nonzero()[:, 0]
                    if len(pick):
                        at_ = v[pick] + codes[r][pick].long()[:, None] * N
                        band.index_add_(0, at_.reshape(-1), (cw[pick] * ring[r][pick]).reshape(-1))
            if nn:
                u, Sp, Sc, hc, v = wn, Sc[:nn], Sn[:nn], hn, vn
    return J.view(nz, ny, nx), (band.view(27, N) if lstar else None)


def _shift(x, d):
    """x_{v+d}, zero outside the box."""
    dx, dy, dz = d % 3 - 1, (d // 3) % 3 - 1, d // 9 - 1
    x = torch.roll(x, (-dy, -dx), (1, 2))
    if dz:
        y = torch.zeros_like(x)
        if dz > 0:
            y[:-1] = x[1:]
        else:
            y[1:] = x[:-1]
        return y
    return x


def _os(band, eps, r, solver, max_sweeps=50, tol=1e-3):
    """Jacobi or eight-colour Gauss-Seidel sweeps from r / diag."""
    nz, ny, nx = r.shape
    band = band.view(27, nz, ny, nx)
    a = [band[d] * _shift(1.0 - eps, d) for d in range(27)]
    diag = 1.0 - a[13]
    z, y, x = (torch.arange(n, device=DEV) & 1 for n in (nz, ny, nx))
    colour = x[None, None, :] + 2 * y[None, :, None] + 4 * z[:, None, None]
    cur = r / diag
    for m in range(1, max_sweeps + 1):
        new = cur
        for col in range(8 if solver == "gs" else 1):
            acc = r.clone()
            for d in range(27):
                if d != 13:
                    acc += a[d] * _shift(new, d)
            acc /= diag
            new = torch.where(colour == col, acc, new) if solver == "gs" else acc
        change, size = float((new - cur).abs().max()), float(new.abs().max())
        cur = new
        if change <= tol * size:
            return cur, m
    return cur, max_sweeps


def _network(s):
    """Loss and gradients of the network with its BF16 weights, in FP64."""
    F = torch.nn.functional
    nz, ny, nx = s.chi.shape[1:]
    W = {n: s.net.Wt[n].double().requires_grad_() for n in s.net.Wt}
    b = {n: s.net.b32[n].double().requires_grad_() for n in s.net.b32}

    def conv(x, name, relu):
        w = W[name].view(3, 3, 3, *W[name].shape[1:]).permute(4, 3, 0, 1, 2)
        x = F.pad(F.pad(x, (1, 1, 1, 1, 0, 0), mode="circular"), (0, 0, 0, 0, 1, 1))
        x = F.conv3d(x, w, b[name])
        return x.relu() if relu else x

    def pool(x):
        g = x.shape[2:]
        x = F.pad(x, (0, 0, 0, 0, 0, g[0] & 1))
        if g[1] & 1:
            x = torch.cat([x, x[:, :, :, :1]], 3)
        if g[2] & 1:
            x = torch.cat([x, x[:, :, :, :, :1]], 4)
        return F.avg_pool3d(x, 2)

    def up(x, skip):
        g = skip.shape[2:]
        for i in range(3):
            x = x.repeat_interleave(2, 2 + i)
        return torch.cat([x[:, :, :g[0], :g[1], :g[2]], skip], 1)

    f = [torch.log10(s.chi) / 3.0, torch.log10(s.eps) / 4.0, s.B - 1.0, torch.log(s.B)]
    X = torch.zeros((1, 16, nz, ny, nx), dtype=torch.float64, device=DEV)
    for i, q in enumerate(f):
        X[:, i] = q
    s1 = conv(conv(X, "e1a", True), "e1b", True)
    s2 = conv(conv(pool(s1), "e2a", True), "e2b", True)
    z = conv(conv(pool(s2), "b_a", True), "b_b", True)
    z = conv(conv(up(z, s2), "d2a", True), "d2b", True)
    z = conv(conv(up(z, s1), "d1a", True), "d1b", True)
    y = conv(z, "out", False)[:, 0]
    if s.case["kind"] == "predict":
        return s.B * torch.exp(y.detach())
    sse = ((y - torch.log(s.J / s.B)) ** 2).sum()
    (sse / y.numel()).backward()
    return {"sse": sse.detach().reshape(1), "gW": [W[l[0]].grad for l in warmstart.LAYERS],
            "gb": [b[l[0]].grad for l in warmstart.LAYERS]}


def exact(case, seed):
    """run()'s outputs in 64 bits. Converged solves and the spherical rays
    have none here, nor boxes of more segments than a few seconds allow."""
    c = case
    kind = c["kind"]
    if kind in ("solve", "batched", "sph"):
        return None
    if kind in ("fs", "ali") and _segments(c) > (3.3e9 if c.get("lstar") or kind == "ali" else 6e9):
        return None
    s = prepare(case, seed)
    if kind in ("train", "predict"):
        return _network(s)
    if kind == "os":
        return _os(s.lstar, s.eps, s.r, c["solver"])
    if kind == "ali":
        J, band = _formal_solution(c, s.chi, s.S, s.bc["I_bottom"], True)
        dJ, _ = _os(band, s.eps, J - s.J, "jacobi")
        new = s.J + dJ
        return new, float((dJ.abs() / new.abs()).max())
    J, band = _formal_solution(c, s.chi, s.S, s.bc["I_bottom"], c["lstar"])
    return (J, band) if c["lstar"] else J
