"""The calls this library is timed on: what programs that use it have it do.

Every case goes through the public binding (`paper_1305_6497_gb300.binding`).
The kinds, and what each stands for:

  matvec_dev  y = A x on a caller's device buffers (`dda_matvec_noalloc`): a
              program with its own Krylov method calls it once per iteration,
              so launches and latency count on small boxes;
  solve       one batch of right-hand sides on a target that is kept
              (`Target.solve`): the same particle for another beam direction,
              the dipole moments returned;
  request     a target that was not seen before: create, solve for both
              polarizations, free -- one request of the serving stream;
  spectrum    one target at several wavelengths in turn, where every wavelength
              needs its own Green-tensor transform;
  orient      orientation averages with a Mueller matrix (`orient_average`):
              one batch of 2 NBETA NTHETA right-hand sides;
  nearfield   fields in and around the target on an extended box.

Refined solves (FP32 inside FP64 refinement) run to 1e-11, FP64 ones to 1e-10,
so that results do not depend on the rounding of the iterations in between.
Boxes, materials and size parameters are those of this repository's workloads
and tests (16^3, 64^3 and 256^3 spheres, the 48x96x144 ellipsoid, the 32x64x64
Au brick, the 48^3 sphere, the serving stream's shapes) or generic ones with
odd sides.
"""
from __future__ import annotations

import math

import numpy as np
import torch

LDR_B = (-1.8915316, 0.1648469, -1.7700004)


def listed():
    return [
        # a caller's own Krylov method on a small particle: launch latency
        dict(name="matvec16_dev_fp32", kind="matvec_dev", shape="ellipsoid", nx=16, ny=16, nz=16,
             mre=1.33, mim=0.01, kd=0.4, method="LDR", precision="fp32"),
        # the same on a box near the scratch limit, sides without a power of two
        dict(name="matvec75x60x50_dev_fp32", kind="matvec_dev", shape="ellipsoid", nx=75, ny=60,
             nz=50, mre=1.5, mim=0.02, kd=0.3, method="GKDLDR", precision="fp32"),
        # the smallest workload: 16^3 sphere, x = 1, FP64 (the binding's default)
        dict(name="sphere16_fp64", kind="solve", shape="ellipsoid", nx=16, ny=16, nz=16, mre=1.33,
             mim=0.01, kd=0.1238, method="LDR", precision="fp64", solver="bicgstab", tuned=False),
        # the guide's 48^3 sphere, x = 5, FP64, its recommended polarizability
        dict(name="sphere48_fp64", kind="solve", shape="ellipsoid", nx=48, ny=48, nz=48, mre=1.5,
             mim=0.01, kd=0.2062, method="GKDLDR", precision="fp64", solver="bicgstab",
             tuned=False),
        # the 64^3 sphere, x = 5, refined, with a tuned schedule as bench.py has it
        dict(name="sphere64_refined", kind="solve", shape="ellipsoid", nx=64, ny=64, nz=64,
             mre=1.5, mim=0.02, kd=0.1562, method="LDR", precision="fp32_refined",
             solver="bicgstab", tuned=True),
        # the guide's Au brick with its recommended method (PBCGS2, GKDLDR)
        dict(name="au_brick_bicgstab2", kind="solve", shape="rect", nx=32, ny=64, nz=64,
             mre=0.9656, mim=1.8628, kd=0.1963, method="GKDLDR", precision="fp32_refined",
             solver="bicgstab2", tuned=False),
        # a million dipoles (the top of the serving range) in a box of odd sides, QMR
        dict(name="rect100x75x135_qmr", kind="solve", shape="rect", nx=100, ny=75, nz=135,
             mre=1.33, mim=0.05, kd=0.09, method="LDR", precision="fp32_refined", solver="qmr",
             tuned=False),
        # one request of the serving stream: an unseen hexagonal prism
        dict(name="request_hex_prism", kind="request", shape="hex", nx=36, ny=41, nz=36, mre=1.6,
             mim=0.1, kd=0.2, method="LDR", precision="fp32_refined", solver="bicgstab"),
        # a spectrum: the Green transform is built anew for every wavelength
        dict(name="spectrum_cylinder", kind="spectrum", shape="cylinder", nx=70, ny=54, nz=54,
             mre=1.4, mim=0.03, kd=0.12, method="GKDLDR", precision="fp32_refined",
             solver="bicgstab", nkd=3),
        # the 1:2:3 ellipsoid's orientation average (2 x 2 orientations, 8 right-hand sides)
        dict(name="orient_ellipsoid", kind="orient", shape="ellipsoid", nx=48, ny=96, nz=144,
             mre=1.7, mim=0.1, kd=0.1, method="FCD", precision="fp32_refined",
             solver="bicgstab", nbeta=2, ntheta=2, tuned=True),
        # fields in and around a sphere of 32^3 sites, on a box of twice its sides
        dict(name="nearfield_sphere32", kind="nearfield", shape="ellipsoid", nx=32, ny=32, nz=32,
             mre=0.96, mim=1.01, kd=0.3, method="LDR"),
        # the largest: the 256^3 sphere (grid 512^3), efficiencies and amplitudes only
        dict(name="sphere256_refined", kind="solve", shape="ellipsoid", nx=256, ny=256, nz=256,
             mre=1.33, mim=0.01, kd=0.0465, method="LDR", precision="fp32_refined",
             solver="bicgstab", tuned=False, want_P=False),
    ]


def draw(rng):
    kind = rng.choice(["matvec_dev", "solve", "solve", "solve", "request", "spectrum", "orient",
                       "nearfield"])

    def side(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    hi = {"matvec_dev": 72, "solve": 150, "request": 90, "spectrum": 90,
          "orient": 64, "nearfield": 40}[kind]
    c = dict(kind=kind, shape=rng.choice(["ellipsoid", "rect", "cylinder", "hex"]),
             nx=side(10, hi), ny=side(10, hi), nz=side(10, hi))
    mre, mim = rng.uniform(1.2, 1.8), rng.uniform(0.0, 0.3)
    # |m| k d <= 0.6 and a size parameter of at most about 4
    kmax = min(0.6 / abs(complex(mre, mim)), 4.0 / (0.62 * (c["nx"] * c["ny"] * c["nz"]) ** (1 / 3)))
    c.update(mre=round(mre, 4), mim=round(mim, 4), kd=round(kmax * rng.uniform(0.4, 1.0), 5),
             method=rng.choice(["LDR", "GKDLDR", "FCD", "CM"]))
    if kind == "matvec_dev":
        c["precision"] = rng.choice(["fp32", "fp32", "fp64"])
        if c["precision"] == "fp64":
            c.update(nx=min(c["nx"], 56), ny=min(c["ny"], 56), nz=min(c["nz"], 56))
    elif kind != "nearfield":
        small = c["nx"] * c["ny"] * c["nz"] < 120000
        c["precision"] = rng.choice(["fp32_refined", "fp32_refined",
                                     "fp64" if small and kind == "solve" else "fp32_refined"])
        c["solver"] = rng.choice(["bicgstab", "bicgstab", "qmr", "bicgstab2", "gpbicg"])
    if kind == "solve":
        c["tuned"] = False
    if kind == "spectrum":
        c["nkd"] = rng.choice([2, 3])
    if kind == "orient":
        c.update(nbeta=rng.choice([1, 2]), ntheta=2, tuned=False, solver="bicgstab")
    return c


# ---- inputs ---------------------------------------------------------------------
def _occupancy(c):
    nx, ny, nz = c["nx"], c["ny"], c["nz"]
    z, y, x = np.meshgrid(*[np.arange(n) - 0.5 * (n - 1) for n in (nz, ny, nx)], indexing="ij")
    if c["shape"] == "rect":
        m = np.ones(x.shape, bool)
    elif c["shape"] == "ellipsoid":
        m = (x / nx) ** 2 + (y / ny) ** 2 + (z / nz) ** 2 <= 0.25
    elif c["shape"] == "cylinder":   # axis along x
        m = (y / ny) ** 2 + (z / nz) ** 2 <= 0.25
    else:                            # hexagonal cross-section in the y-z plane
        u, v = np.abs(y) / (0.5 * ny), np.abs(z) / (0.5 * nz)
        m = (v <= 0.87) & (u + v * math.tan(math.pi / 6) <= 1.0)
    return m.astype(np.uint8)


def _axes(rng):
    """A random beam direction and its transverse axes."""
    q, _ = np.linalg.qr(rng.standard_normal((3, 3)))
    if np.linalg.det(q) < 0:
        q[:, 0] *= -1
    return q[:, 0].copy(), q[:, 1].copy(), q[:, 2].copy()


def _inputs(case, seed):
    """What the caller starts from: occupancy, refractive index, k d, beam, vectors."""
    rng = np.random.default_rng([int(seed), 1305])
    c = dict(case)
    occ = _occupancy(c)
    m = complex(c["mre"], c["mim"]) * (1 + 0.01 * rng.uniform(-1, 1))
    kd = c["kd"] * (1 + 0.02 * rng.uniform(-1, 1))
    khat, yhat, _ = _axes(rng)
    th = np.deg2rad([30.0, 90.0, 150.0, 180.0])
    s = dict(case=c, occ=occ, m=m, kd=kd, khat=khat[None], yhat=yhat[None],
             e01=yhat[None].astype(np.complex128),
             dirs=np.array([(t, p) for p in (0.0, 0.5 * math.pi) for t in th]))
    if c["kind"] == "matvec_dev":
        shp = (3,) + occ.shape
        v = (rng.standard_normal(shp) + 1j * rng.standard_normal(shp)) * (occ != 0)
        s["xbox"] = v.astype(np.complex64 if c["precision"] == "fp32" else np.complex128)
    if c["kind"] == "nearfield":
        # dipoles of the first Born approximation, alpha E_inc
        pos = _positions(occ)
        ph = np.exp(1j * kd * pos @ khat)
        a = 3 / (4 * math.pi) * (m * m - 1) / (m * m + 2)
        e2 = np.cross(khat, yhat)
        s["P"] = np.stack([a * ph[:, None] * e[None].astype(np.complex128) for e in (yhat, e2)])
        s["ext"] = np.full(6, 0.5)
    return s


def prepare(case, seed):
    from paper_1305_6497_gb300 import binding as B
    s = _inputs(case, seed)
    c = s["case"]
    s["B"] = B
    if c["kind"] == "request":
        return s
    t = s["t"] = B.Target(s["occ"], None, [s["m"]], method=c["method"])
    if c["kind"] == "matvec_dev":
        s["x"] = torch.from_numpy(s["xbox"]).cuda()
        s["y"] = torch.zeros_like(s["x"])
        # builds the Green-tensor transform the allocation-free call needs
        t.matvec(s["kd"], np.zeros((t.num_dipoles, 3), np.complex128), s["khat"][0],
                 s["e01"][0], precision=c["precision"])
        torch.cuda.synchronize()
    elif c["kind"] == "nearfield":
        t.nearfield(s["kd"], s["khat"], s["e01"], s["P"], s["ext"])
    elif c.get("tuned"):
        t.autotune(s["kd"], 2 * c["nbeta"] * c["ntheta"] if c["kind"] == "orient" else 2)
    return s


def _solve(s, t, kd, want_P):
    c = s["case"]
    out = t.solve(kd, s["khat"], s["e01"], yhat=s["yhat"], npol=2,
                  tol=1e-10 if c["precision"] == "fp64" else 1e-11, max_iter=4000,
                  precision=c["precision"], dirs=s["dirs"], want_P=want_P, solver=c["solver"])
    return {k: out[k] for k in ("P", "Qext", "Qabs", "Qsca", "famp") if out[k] is not None}


def run(s):
    c, B = s["case"], s["B"]
    kind = c["kind"]
    if kind == "matvec_dev":
        B.dda_matvec_noalloc(s["t"].h, s["kd"], s["x"].data_ptr(), s["y"].data_ptr(),
                             s["khat"][0], s["e01"][0], precision=c["precision"])
        return s["y"]
    if kind == "solve":
        return _solve(s, s["t"], s["kd"], c.get("want_P", True))
    if kind == "request":
        t = B.Target(s["occ"], None, [s["m"]], method=c["method"])
        out = _solve(s, t, s["kd"], False)
        t.close()
        return out
    if kind == "spectrum":
        return [_solve(s, s["t"], kd, False) for kd in _spectrum(s)]
    if kind == "orient":
        out = s["t"].orient_average(s["kd"], beta=(0.0, 2 * math.pi), nbeta=c["nbeta"],
                                    theta=(0.0, math.pi), ntheta=c["ntheta"], tol=1e-11,
                                    max_iter=4000, precision=c["precision"],
                                    solver=c["solver"], eta=1.0, sel=s["dirs"])
        return {k: out[k] for k in ("Qext", "Qabs", "Qsca", "Qpha", "Qbk", "g", "cos2",
                                    "mueller")}
    out = s["t"].nearfield(s["kd"], s["khat"], s["e01"], s["P"], s["ext"])
    return {k: out[k] for k in ("E_inc", "E_sca", "E_macro")}


def _spectrum(s):
    return [s["kd"] * (1 + 0.15 * i) for i in range(s["case"]["nkd"])]


# ---- what a pass cannot do without -------------------------------------------------
def _smooth(n):
    while True:
        m = n
        for p in (2, 3, 5):
            while m % p == 0:
                m //= p
        if m == 1:
            return n
        n += 1


def work(case):
    c = case
    n = [c["nx"], c["ny"], c["nz"]]
    kind = c["kind"]
    if kind == "nearfield":
        n = [2 * v for v in n]
    L = [_smooth(2 * v - 1) for v in n]
    nb, M = float(np.prod(n)), float(np.prod(L))
    octant = float(np.prod([v // 2 + 1 for v in L]))
    el = 16 if c.get("precision", "fp64") == "fp64" else 8
    # the pruned transforms forward and back, and the 3x3 multiply; vectors in
    # and out, and the Green transform read once
    fl = 2 * 3 * (5 * n[1] * n[2] * L[0] * math.log2(L[0]) + 5 * n[2] * L[0] * L[1] * math.log2(L[1])
                  + 5 * M * math.log2(L[2])) + 66 * M
    by = el * (6 * nb + 6 * octant)
    # a Green-tensor transform: six even/odd functions on an octant, in FP64
    gfl = 6 * 2.5 * octant * math.log2(M) + 150 * nb
    gby = 16 * 6 * octant
    if kind == "matvec_dev":
        return {"bytes": by, "flops": fl}
    if kind == "nearfield":
        return {"bytes": 2 * (by + 2 * 16 * 3 * nb), "flops": 2 * fl}
    # Krylov products per right-hand side, roughly: they grow with the phase
    # shift across the particle
    x = c["kd"] * (0.75 / math.pi * nb) ** (1 / 3)
    mv = 2 * (10 + 8 * x * abs(complex(c["mre"], c["mim"]) - 1)) * (1 if c["precision"] == "fp64" else 1.5)
    R = 2 * c.get("nbeta", 1) * c.get("ntheta", 1)
    k = c.get("nkd", 1)
    w = {"bytes": k * R * mv * by, "flops": k * R * mv * fl}
    if kind in ("request", "spectrum"):
        w["bytes"] += k * gby
        w["flops"] += k * gfl
    return w


# ---- the same in 64 bits, in plain numpy and torch ----------------------------------
def _positions(occ):
    iz, iy, ix = np.nonzero(occ)
    nz, ny, nx = occ.shape
    return np.stack([ix - 0.5 * (nx - 1), iy - 0.5 * (ny - 1), iz - 0.5 * (nz - 1)], 1)


def _alpha(method, m, kd, khat, e):
    """The diagonal of the polarizability on the lattice axes."""
    m2, k3 = m * m, kd ** 3
    a0 = 3 / (4 * math.pi) * (m2 - 1) / (m2 + 2)
    if method == "CM":
        return np.full(3, a0 / (1 - 2j / 3 * k3 * a0))
    if method == "FCD":
        lg = math.log((math.pi - kd) / (math.pi + kd))
        return np.full(3, a0 / (1 - a0 * (4 / 3 * kd ** 2 + 2 / (3 * math.pi) * lg * k3 + 2j / 3 * k3)))
    S = khat ** 2
    if method == "LDR":
        S = np.full(3, np.sum(khat ** 2 * np.abs(e) ** 2) / np.sum(np.abs(e) ** 2))
    b1, b2, b3 = LDR_B
    return a0 / (1 + a0 * ((b1 + m2 * b2 + m2 * b3 * S) * kd ** 2 - 2j / 3 * k3))


def _sici(x):
    """Si, Ci for x > 1 from the continued fraction of E1(ix), evaluated backwards."""
    z = torch.complex(torch.zeros_like(x), x)
    f = torch.zeros_like(z)
    for n in range(600, 0, -1):
        f = -(float(n) * n) / (z + (2 * n + 1) + f)
    e1 = torch.exp(-z) / (z + 1 + f)
    return 0.5 * math.pi + e1.imag, -e1.real


class _Operator:
    """A x = x / alpha - sum G x by circular convolution, complex128 on the GPU."""

    def __init__(self, n, kd, filtered):
        self.n, self.L = n, [_smooth(2 * v - 1) for v in n]
        dev = "cuda"
        ax = []
        for v, L in zip(n, self.L):
            i = torch.arange(L, device=dev)
            d = torch.where(i < v, i, i - L)
            ax.append((d.double(), ((i < v) | (i > L - v)).double()))
        Z, Y, X = torch.meshgrid(ax[2][0], ax[1][0], ax[0][0], indexing="ij")
        keep = ax[2][1][:, None, None] * ax[1][1][None, :, None] * ax[0][1][None, None, :]
        r2 = X * X + Y * Y + Z * Z
        keep[0, 0, 0] = 0.0
        r2[0, 0, 0] = 1.0
        u, inv = torch.unique(r2, return_inverse=True)
        r = torch.sqrt(u)
        if not filtered:
            e = torch.exp(1j * kd * r) / r ** 3
            A = e * ((kd * r) ** 2 - 1 + 1j * kd * r)
            Bf = e * (3 - (kd * r) ** 2 - 3j * kd * r)
        else:
            # r g = i sin kr + [cos kr S + sin kr C] / pi and its derivatives
            k, a, b = kd, math.pi - kd, math.pi + kd
            sa, ca = _sici(a * r)
            sb, cb = _sici(b * r)
            S, C = sa + sb, ca - cb
            S1 = (torch.sin(a * r) + torch.sin(b * r)) / r
            C1 = (torch.cos(a * r) - torch.cos(b * r)) / r
            S2 = (a * torch.cos(a * r) + b * torch.cos(b * r)) / r - S1 / r
            C2 = (-a * torch.sin(a * r) + b * torch.sin(b * r)) / r - C1 / r
            s, co = torch.sin(k * r), torch.cos(k * r)
            h = 1j * s + (co * S + s * C) / math.pi
            h1 = 1j * k * co + (-k * s * S + co * S1 + k * co * C + s * C1) / math.pi
            h2 = -1j * k * k * s + (-k * k * co * S - 2 * k * s * S1 + co * S2 - k * k * s * C
                                    + 2 * k * co * C1 + s * C2) / math.pi
            g, g1 = h / r, h1 / r - h / r ** 2
            g2 = h2 / r - 2 * h1 / r ** 2 + 2 * h / r ** 3
            A, Bf = k * k * g + g1 / r, g2 - g1 / r
        A, Bf = A[inv] * keep, Bf[inv] * keep / r2
        self.g = {}
        for i, p in enumerate((X, Y, Z)):
            for j, q in enumerate((X, Y, Z)):
                if j >= i:
                    v = Bf * (p * q)
                    self.g[i, j] = torch.fft.fftn(v + A if i == j else v)

    def field(self, x):
        """sum_{l != j} G x_l on every box site; x: [3, nz, ny, nx]."""
        nx, ny, nz = self.n
        s = [torch.fft.fftn(x[i], s=self.L[::-1]) for i in range(3)]
        out = torch.empty_like(x)
        for i in range(3):
            v = sum(self.g[min(i, j), max(i, j)] * s[j] for j in range(3))
            out[i] = torch.fft.ifftn(v)[:nz, :ny, :nx]
        return out


def _bicgstab(mv, b, tol, cap):
    x = torch.zeros_like(b)
    bn = torch.linalg.norm(b)
    for _ in range(4):
        r = b - mv(x)
        if float(torch.linalg.norm(r) / bn) <= tol:
            break
        rh, p, v = r.clone(), torch.zeros_like(b), torch.zeros_like(b)
        rho = al = om = torch.ones((), dtype=b.dtype, device=b.device)
        for _ in range(cap):
            rn = torch.vdot(rh, r)
            p = r + rn / rho * al / om * (p - om * v)
            rho = rn
            v = mv(p)
            al = rho / torch.vdot(rh, v)
            s = r - al * v
            t = mv(s)
            om = torch.vdot(t, s) / torch.vdot(t, t)
            x = x + al * p + om * s
            r = s - om * t
            if float(torch.linalg.norm(r) / bn) <= 0.3 * tol:
                break
    return x


def _frames(s):
    """(khat, yhat, zhat) of every incidence."""
    c = s["case"]
    if c["kind"] != "orient":
        return [(s["khat"][0], s["yhat"][0], np.cross(s["khat"][0], s["yhat"][0]))]
    nb, nt = c["nbeta"], c["ntheta"]
    out = []
    for i in range(nb):
        b = (i + 0.5) * 2 * math.pi / nb
        for j in range(nt):
            ct = 1.0 - 2.0 * (j + 0.5) / nt
            st, cb, sb = math.sqrt(1 - ct * ct), math.cos(b), math.sin(b)
            out.append((np.array([ct, -st * cb, st * sb]), np.array([st, ct * cb, -ct * sb]),
                        np.array([0.0, sb, cb])))
    return out


def _observe(s, kd):
    """P, efficiencies and amplitudes of every incidence and both polarizations."""
    c, occ, m = s["case"], s["occ"], s["m"]
    n = [c["nx"], c["ny"], c["nz"]]
    op = _Operator(n, kd, c["method"] == "FCD")
    pos = _positions(occ)
    N = len(pos)
    mask = torch.from_numpy(occ != 0).cuda()
    geo = math.pi * (0.75 / math.pi * N) ** (2 / 3)
    Ps, Qe, Qa, fa = [], [], [], []
    for kh, y, z in _frames(s):
        ph = np.exp(1j * kd * pos @ kh)
        per_pol = []
        for e in (y.astype(np.complex128), np.cross(kh, y).astype(np.complex128)):
            al = _alpha(c["method"], m, kd, kh, e)
            E = ph[:, None] * e[None]
            box = torch.zeros((3,) + occ.shape, dtype=torch.complex128, device="cuda")
            box[:, mask] = torch.from_numpy(np.ascontiguousarray(E.T)).cuda()
            ai = torch.from_numpy(1 / al).cuda()[:, None, None, None]

            def mv(v):
                v = v.reshape(box.shape)
                return ((ai * v - op.field(v)) * mask).reshape(-1)
            P = _bicgstab(mv, box.reshape(-1), 1e-13, 400).reshape(box.shape)[:, mask].T.cpu().numpy()
            Ps.append(P)
            Qe.append(4 * math.pi * kd * np.sum(np.imag(np.conj(E) * P)) / geo)
            Qa.append(4 * math.pi * kd * np.sum(np.abs(P) ** 2 * (-np.imag(1 / al) - 2 / 3 * kd ** 3)) / geo)
            rows = []
            for t, f in [(0.0, 0.0)] + [tuple(d) for d in s["dirs"]]:
                nv = kh * math.cos(t) + y * math.sin(t) * math.cos(f) + z * math.sin(t) * math.sin(f)
                F = np.exp(-1j * kd * pos @ nv) @ P
                et = -kh * math.sin(t) + (y * math.cos(f) + z * math.sin(f)) * math.cos(t)
                rows.append([kd ** 3 * et @ F, kd ** 3 * (z * math.cos(f) - y * math.sin(f)) @ F])
            per_pol.append(np.array(rows))
        fa.append(np.stack(per_pol, -1))
    Qe, Qa = np.array(Qe), np.array(Qa)
    return dict(P=np.array(Ps), Qext=Qe, Qabs=Qa, Qsca=Qe - Qa, famp=np.array(fa))


def exact(case, seed):
    s = _inputs(case, seed)
    c, kd = s["case"], s["kd"]
    kind = c["kind"]
    n = [c["nx"], c["ny"], c["nz"]]
    if n[0] * n[1] * n[2] > 3_000_000:
        return None
    if kind == "matvec_dev":
        op = _Operator(n, kd, c["method"] == "FCD")
        mask = torch.from_numpy(s["occ"] != 0).cuda()
        ai = torch.from_numpy(1 / _alpha(c["method"], s["m"], kd, s["khat"][0], s["e01"][0])).cuda()
        x = torch.from_numpy(s["xbox"].astype(np.complex128)).cuda()
        return (ai[:, None, None, None] * x - op.field(x)) * mask
    if kind == "nearfield":
        lo = [int(math.floor(0.5 * v + 0.5)) for v in n]
        big = [v + 2 * w for v, w in zip(n, lo)]
        op = _Operator(big, kd, c["method"] == "FCD")
        occ = np.zeros(big[::-1], np.uint8)
        occ[lo[2]:lo[2] + n[2], lo[1]:lo[1] + n[1], lo[0]:lo[0] + n[0]] = s["occ"]
        mask = torch.from_numpy(occ != 0).cuda()
        ax = [torch.arange(b, device="cuda").double() - w - 0.5 * (v - 1)
              for b, w, v in zip(big, lo, n)]
        kh = s["khat"][0]
        ph = torch.exp(1j * kd * (kh[2] * ax[2][:, None, None] + kh[1] * ax[1][None, :, None]
                                  + kh[0] * ax[0][None, None, :]))
        fac = torch.where(mask, torch.tensor(3 / (s["m"] ** 2 + 2), dtype=torch.complex128,
                                             device="cuda"), 1.0 + 0j)
        out = dict(E_inc=[], E_sca=[], E_macro=[])
        for l, e in enumerate((s["yhat"][0], np.cross(kh, s["yhat"][0]))):
            x = torch.zeros((3,) + occ.shape, dtype=torch.complex128, device="cuda")
            x[:, mask] = torch.from_numpy(np.ascontiguousarray(s["P"][l].T)).cuda()
            es = op.field(x)
            ei = torch.from_numpy(e.astype(np.complex128)).cuda()[:, None, None, None] * ph
            for k, v in (("E_inc", ei), ("E_sca", es), ("E_macro", fac * (ei + es))):
                out[k].append(v.cpu().numpy())
        return {k: np.array(v) for k, v in out.items()}
    if kind == "orient":
        q = _observe(s, kd)
        return dict(Qpha=None, Qbk=None, g=None, cos2=None, mueller=None,
                    **{k: q[k].reshape(-1, 2).mean(0) for k in ("Qext", "Qabs", "Qsca")})
    if kind == "spectrum":
        got = [_observe(s, k) for k in _spectrum(s)]
    else:
        got = [_observe(s, kd)]
    if kind != "solve" or not c.get("want_P", True):
        for g in got:
            del g["P"]
    return got if kind == "spectrum" else got[0]
