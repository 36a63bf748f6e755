"""The work whose speed this repository watches, through its public entry points.

Every case is a dict of plain values; `prepare` makes its inputs and handles
from a seed, `run` is one call as a user's program makes it, `exact` is the
same result from plain torch in 64 bits (no code of this package but the
geometry generators), and `work` is what the call cannot do without.

Paths: "product" (Problem.matvec), "update" (a geometry step: new centres and
radii, then the factors, the generators and one product of the new operator),
"farfield", "nearfield", "solve" (GMRES and the far field), "gradient" (the
far-field misfit and its adjoint gradient), "dort" (time reversal).
Geometries: "four" (the four-disk example), "random" (sound-soft disks of
uneven radii), "unit" (batched clusters of unit disks, sound-soft or
sound-hard each, uneven sizes), "lattice" (jittered square lattice), "three"
(the time-reversal example).  Sizes are those of the workloads module.
"""
import math

import numpy as np
import torch

from paper_1409_8186_gb300 import msd
from paper_1409_8186_gb300 import workloads as W

PREC = {"fp64": msd.MSD_FP64, "fp32": msd.MSD_FP32, "mixed": msd.MSD_MIXED}


# ---------------------------------------------------------------- the cases

def listed():
    return [
        # the smallest whole call: the four-disk example solved to 1e-12, 360 far-field angles
        {"name": "solve_four_disks", "path": "solve", "geometry": "four", "configs": 1, "disks": 4, "k": 1.0,
         "columns": 1, "precision": "fp64", "angles": 360},
        # one operator product inside the plain FP64 solve of the 400-disk cluster
        {"name": "product_fp64_random400", "path": "product", "geometry": "random", "configs": 1, "disks": 400,
         "k": 2 * math.pi, "columns": 1, "precision": "fp64"},
        # the same product inside the FP32 sweeps of its mixed solve
        {"name": "product_fp32_random400", "path": "product", "geometry": "random", "configs": 1, "disks": 400,
         "k": 2 * math.pi, "columns": 1, "precision": "fp32"},
        # FP64 product with 16 incidences: the gradient workload's operator
        {"name": "product_fp64_random200_r16", "path": "product", "geometry": "random", "configs": 1, "disks": 200,
         "k": 10.0, "columns": 16, "precision": "fp64"},
        # the largest operator: 4000-disk lattice, 64 incidences, FP32 sweeps
        {"name": "product_fp32_lattice4000_r64", "path": "product", "geometry": "lattice", "configs": 1,
         "disks": 4000, "k": 5.0, "columns": 64, "precision": "fp32"},
        # a group of the batched workload: clusters of uneven size, 32 incidences each
        {"name": "product_fp32_batch8_r32", "path": "product", "geometry": "unit", "configs": 8, "disks": 400,
         "k": 8.0, "columns": 32, "precision": "fp32"},
        # a step of a geometry loop: new centres and radii, new operator, its first product
        {"name": "update_random400", "path": "update", "geometry": "random", "configs": 1, "disks": 400,
         "k": 2 * math.pi, "columns": 1, "precision": "fp64"},
        # far field of one solution at 360 angles
        {"name": "farfield_random400", "path": "farfield", "geometry": "random", "configs": 1, "disks": 400,
         "k": 2 * math.pi, "columns": 1, "angles": 360},
        # near-field map of one solution on a 512 x 512 grid
        {"name": "nearfield_random400", "path": "nearfield", "geometry": "random", "configs": 1, "disks": 400,
         "k": 2 * math.pi, "columns": 1, "points": 512 * 512},
        # batched mixed-precision solve: eight clusters, 32 incidences each
        {"name": "solve_mixed_batch8_r32", "path": "solve", "geometry": "random", "configs": 8, "disks": 60,
         "k": 5.0, "columns": 32, "precision": "mixed", "angles": 360},
        # one gradient of an inverse problem: forward and adjoint FP64 solves, 16 incidences
        {"name": "gradient_fp64_random40", "path": "gradient", "geometry": "random", "configs": 1, "disks": 40,
         "k": 10.0, "columns": 16, "precision": "fp64", "angles": 360},
        # time reversal of the three-disk example with 512 mirror angles
        {"name": "dort_three_512", "path": "dort", "geometry": "three", "configs": 1, "disks": 3,
         "k": 2 * math.pi, "columns": 512, "precision": "fp64"},
    ]


def _logint(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    path = rng.choice(["product", "product", "product", "update", "farfield", "nearfield", "solve", "gradient",
                       "dort"])
    k = rng.choice([1.0, 2.0, 3.5, 5.0, 2 * math.pi, 8.0, 10.0])
    if path == "product":
        prec = rng.choice(["fp64", "fp32"])
        geometry = rng.choice(["random", "unit", "lattice"])
        configs = rng.randint(1, 12) if geometry == "unit" else 1
        disks = _logint(rng, 5, 800 if geometry == "unit" else 3000 if geometry == "lattice" else 400)
        if geometry == "lattice":
            k = 5.0
        elif geometry == "unit":
            k = float(rng.randint(2, 8))
        columns = rng.choice([1, 1, 1, 2, 3, 4, 7, 8, 12, 16, 16, 24, 32, 32, 33, 48, 64])
        case = {"path": path, "geometry": geometry, "configs": configs, "disks": disks, "k": k, "columns": columns,
                "precision": prec}
        most = 4e10 if prec == "fp64" else 1.5e12
        while work(case)["flops"] > most and case["columns"] > 1:
            case["columns"] = max(1, case["columns"] // 2)
        while work(case)["flops"] > most:
            case["disks"] = case["disks"] * 3 // 4
        return case
    if path == "update":
        return {"path": path, "geometry": "random", "configs": 1, "disks": _logint(rng, 5, 400), "k": k, "columns": 1,
                "precision": "fp64"}
    if path == "farfield":
        configs = rng.choice([1, 1, 2, 5])
        return {"path": path, "geometry": "unit" if configs > 1 else "random", "configs": configs,
                "disks": _logint(rng, 5, 400), "k": max(2.0, float(round(k))) if configs > 1 else k,
                "columns": rng.choice([1, 2, 3, 8, 16, 17, 32]), "angles": _logint(rng, 8, 720)}
    if path == "nearfield":
        return {"path": path, "geometry": "random", "configs": 1, "disks": _logint(rng, 5, 300), "k": k,
                "columns": rng.choice([1, 1, 2, 4, 5]), "points": _logint(rng, 100, 40000)}
    if path == "solve":
        mixed = rng.random() < 0.5
        return {"path": path, "geometry": "random", "configs": rng.randint(1, 4),
                "disks": _logint(rng, 4, 60 if mixed else 40), "k": min(k, 5.0),
                "columns": rng.choice([1, 2, 3, 8, 16] if mixed else [1, 2, 4]),
                "precision": "mixed" if mixed else "fp64", "angles": rng.choice([90, 180, 360])}
    if path == "gradient":
        return {"path": path, "geometry": "random", "configs": 1, "disks": _logint(rng, 4, 40), "k": k,
                "columns": rng.choice([1, 2, 4, 8, 16]), "precision": "fp64", "angles": rng.choice([90, 180, 360])}
    return {"path": path, "geometry": "three", "configs": 1, "disks": 3, "k": 2 * math.pi,
            "columns": _logint(rng, 16, 512), "precision": "fp64"}


# ---------------------------------------------------------------- inputs

def _sizes(case):
    """(disks, whole wavenumber, truncation order) of every configuration, from the case alone."""
    C, M, k = case["configs"], case["disks"], case["k"]
    out = []
    for c in range(C):
        m = M if C == 1 or case["geometry"] != "unit" else max(2, round(M * (0.25 + 0.75 * c / (C - 1))))
        if case["geometry"] == "four":
            out.append((4, k, 12))
        elif case["geometry"] == "three":
            out.append((3, k, 4))
        elif case["geometry"] == "lattice":
            out.append((m, k, 15))
        elif case["geometry"] == "unit":
            kc = 2 + (3 * c + int(k) - 2) % (int(k) - 1) if k > 2 else 2
            out.append((m, float(kc), kc + 8))
        elif _even_radii(case):
            out.append((m, k, math.ceil(1.2 * k) + 10))
        else:
            out.append((m, k, math.ceil(1.5 * k) + 10))
    return out


def _even_radii(case):
    return case["path"] in ("solve", "gradient") or case["k"] >= 10.0


def _clusters(case, seed):
    out = []
    for c, (M, k, N) in enumerate(_sizes(case)):
        rng = np.random.default_rng([seed, c])
        if case["geometry"] == "four":
            cl = W.four_disks()
        elif case["geometry"] == "three":
            cl = W.dort_three_disks()
            cl.centres = cl.centres + 0.2 * rng.standard_normal(cl.centres.shape)
        elif case["geometry"] == "lattice":
            cl = W.lattice_4000(seed=seed, M=M)
        elif case["geometry"] == "unit":
            o, a = W.random_disks(rng, M, max(0.5 * math.sqrt(M * math.pi / 0.2), 3.0), 1.0, 1.0, 0.01)
            cl = W.Cluster(o, a, rng.integers(0, 2, size=M).astype(np.int8), k - float(rng.uniform(0.05, 0.95)), N)
        else:
            lo, hi = (0.8, 1.2) if _even_radii(case) else (0.5, 1.5)
            o, a = W.random_disks(rng, M, max(2.5 * math.sqrt(M), 5.0), lo, hi, 0.2)
            cl = W.Cluster(o, a, np.zeros(M, np.int8), k, N)
        out.append(cl)
    return out


def _normal(rng, shape, scale=1.0):
    return scale * (rng.standard_normal(shape) + 1j * rng.standard_normal(shape))


def _inputs(case, seed):
    """Geometry and host inputs of one call, from the case and the seed alone."""
    cls = _clusters(case, seed)
    rng = np.random.default_rng([seed, 1000])
    R, ntot = case["columns"], sum(c.ntot for c in cls)
    s = {"clusters": cls, "path": case["path"]}
    if "angles" in case:
        s["thetas"] = W.angles(case["angles"])
    if case["path"] in ("product", "update"):
        s["x"] = _normal(rng, (ntot, R)).astype(np.complex64 if case["precision"] == "fp32" else np.complex128)
    if case["path"] in ("farfield", "nearfield"):
        # densities fall off with the mode number as those of a solution do
        damp = np.concatenate([np.tile(0.7 ** np.abs(np.arange(-c.N, c.N + 1)), c.M) for c in cls])
        s["rho"] = _normal(rng, (ntot, R)) * damp[:, None]
    if case["path"] == "update":
        # the next step of a loop: every disk moved and resized a little
        new = W.Cluster(cls[0].centres + 0.02 * rng.uniform(-1, 1, cls[0].centres.shape),
                        cls[0].radii * (1 + 0.02 * rng.uniform(-1, 1, cls[0].M)), cls[0].bc, cls[0].k, cls[0].N)
        s["next"] = new
    if case["path"] == "nearfield":
        half = np.abs(cls[0].centres).max() + 5.0
        side = math.isqrt(case["points"])
        if side * side == case["points"]:  # a map: a shifted grid
            g = np.linspace(-half, half, side)
            pts = np.stack(np.meshgrid(g, g), -1).reshape(-1, 2) + 0.01 * rng.standard_normal(2)
        else:
            pts = rng.uniform(-half, half, (case["points"], 2))
        s["points"] = pts
    if case["path"] in ("solve", "gradient"):
        s["betas"] = W.angles(R) + float(rng.uniform(0, 2 * math.pi))
    if case["path"] == "gradient":
        s["target"] = _normal(rng, (1, case["angles"], R))
    return s


def prepare(case, seed):
    s = _inputs(case, seed)
    s["case"] = case
    s["pb"] = pb = msd.Problem(s["clusters"])
    if "x" in s:
        # a program that multiplies holds the operator's generators and plan
        s["x"] = torch.from_numpy(s["x"]).cuda()
        pb.matvec(s["x"], PREC[case["precision"]])
    if "rho" in s:
        s["rho"] = torch.from_numpy(s["rho"]).cuda()
    if "target" in s:
        s["target"] = torch.from_numpy(s["target"]).cuda()
    if "next" in s:
        s["centres"] = torch.from_numpy(s["next"].centres).cuda()
        s["radii"] = torch.from_numpy(s["next"].radii).cuda()
    return s


def run(s):
    case, pb = s["case"], s["pb"]
    if case["path"] == "product":
        return pb.matvec(s["x"], PREC[case["precision"]])
    if case["path"] == "update":
        pb.update_geometry(s["centres"], s["radii"])
        return [pb.diagonals(), pb.generators(), pb.matvec(s["x"])]
    if case["path"] == "farfield":
        return pb.farfield(s["rho"], s["thetas"])
    if case["path"] == "nearfield":
        return pb.nearfield(s["rho"], s["points"])
    if case["path"] == "solve":
        r = pb.solve(s["betas"], tol=1e-12, restart=500, precision=PREC[case["precision"]])
        return [r.rho, pb.farfield(r.rho, s["thetas"])]
    if case["path"] == "gradient":
        return list(pb.grad_farfield_misfit(s["betas"], s["thetas"], s["target"], tol=1e-12, restart=500))
    eig, F, T, _ = pb.dort(case["columns"], restart=200)
    return [eig, F, T]


# ---------------------------------------------------------------- what a call cannot do without

def work(case):
    sizes, R = _sizes(case), case["columns"]
    single = case.get("precision") == "fp32"
    elem = 8 if single else 16
    ntot = sum(M * (2 * N + 1) for M, _, N in sizes)
    gens = sum(M * (M - 1) * (4 * N + 1) for M, _, N in sizes)
    macs = sum(M * (M - 1) * (2 * N + 1) ** 2 for M, _, N in sizes)
    product = {"bytes": elem * (gens + 2 * ntot * R), "flops": 8 * R * macs}
    if case["path"] == "product":
        return product
    if case["path"] == "update":  # generators made and read out, one product
        return {"bytes": 16 * (3 * gens + 6 * ntot), "flops": product["flops"] + 20 * gens}
    if case["path"] == "farfield":
        T = case["angles"]
        return {"bytes": 16 * (ntot * R + len(sizes) * T * R), "flops": 8 * ntot * T * R}
    if case["path"] == "nearfield":
        P = case["points"]
        return {"bytes": 16 * (ntot * R + P + P * R), "flops": (8 * R + 10) * ntot * P}
    if case["path"] == "dort":  # T = conj(F)^T F and its reduction (4/3 n^3 complex multiply-adds)
        return {"bytes": 16 * (2 * R * R + R), "flops": 8 * R ** 3 * 7 // 3}
    # a Krylov solve needs at least one product per right-hand side; how many it
    # takes is the system's own matter
    T = case["angles"]
    twice = 2 if case["path"] == "gradient" else 1
    return {"bytes": twice * product["bytes"] + 16 * len(sizes) * T * R,
            "flops": twice * product["flops"] + 8 * ntot * T * R}


# ---------------------------------------------------------------- the same in plain torch, 64 bits

class _Bessel(torch.autograd.Function):
    """J_l(x), Y_l(x), l = 0..lmax, stacked first: J by Miller's backward
    recurrence, Y_0 and Y_1 by Neumann's series over the same orders
    (Abramowitz and Stegun 9.1.88 and its derivative), Y_l by the forward
    recurrence."""

    @staticmethod
    def forward(ctx, x, lmax):
        top = max(lmax + 1, float(x.max()))
        start = int(top + math.sqrt(60 * top)) + 16
        start += start & 1
        J = [None] * (lmax + 2)
        hi, lo = torch.zeros_like(x), torch.full_like(x, 1e-30)
        norm, s0, s1 = torch.zeros_like(x), torch.zeros_like(x), torch.zeros_like(x)
        for l in range(start, 0, -1):
            if l <= lmax + 1:
                J[l] = lo
            h = l // 2
            if l % 2 == 0:
                norm = norm + 2 * lo
                s0 = s0 + (-1.0) ** h / h * lo
            else:  # (-1)^k (J_{2k-1} - J_{2k+1}) / k, collected by the order l = 2h + 1
                s1 = s1 - (-1.0) ** h * (1.0 / (h + 1) + (1.0 / h if h else 0.0)) * lo
            hi, lo = lo, (2.0 * l / x) * lo - hi
            big = lo.abs() > 1e150
            if bool(big.any()):
                f = torch.where(big, torch.full_like(x, 1e-150), torch.ones_like(x))
                hi, lo, norm, s0, s1 = hi * f, lo * f, norm * f, s0 * f, s1 * f
                J = [None if j is None else j * f for j in J]
        J[0] = lo
        norm = norm + lo
        J = [j / norm for j in J]
        log = torch.log(0.5 * x) + 0.57721566490153286061
        Y = [(log * J[0] - 2 * s0 / norm) * (2 / math.pi), (log * J[1] - J[0] / x + s1 / norm) * (2 / math.pi)]
        for l in range(1, lmax + 1):
            Y.append((2.0 * l / x) * Y[l] - Y[l - 1])
        ctx.J, ctx.Y, ctx.lmax = J, Y, lmax
        return torch.stack(J[:lmax + 1]), torch.stack(Y[:lmax + 1])

    @staticmethod
    def backward(ctx, gJ, gY):
        g = 0
        for l in range(ctx.lmax + 1):
            for z, gz in ((ctx.J, gJ), (ctx.Y, gY)):
                d = -z[1] if l == 0 else 0.5 * (z[l - 1] - z[l + 1])
                g = g + gz[l] * d
        return g, None


def _orders(z, lmax):
    """Rows l = -lmax..lmax of Z_l from l >= 0 (Z_{-l} = (-1)^l Z_l)."""
    sign = torch.tensor([(-1.0) ** l for l in range(lmax, 0, -1)], dtype=z.dtype, device=z.device)
    neg = torch.flip(z[1:], [0]) * sign.reshape(-1, *([1] * (z.dim() - 1)))
    return torch.cat([neg, z])


class _Dense:
    """One configuration: Bessel factors and generators in 64 bits (centres, radii, k: tensors)."""

    def __init__(self, O, a, k, N, bc):
        self.O, self.a, self.k, self.N, self.n, self.M = O, a, k, N, 2 * N + 1, len(a)
        J, Y = _Bessel.apply(k * a, N + 1)
        J, Y = _orders(J, N + 1), _orders(Y, N + 1)
        self.J, self.H = J[1:-1].T, torch.complex(J, Y)[1:-1].T  # [M, n]
        self.dJ = (0.5 * (J[:-2] - J[2:])).T
        H = torch.complex(J, Y)
        self.dH = (0.5 * (H[:-2] - H[2:])).T
        self.hard = torch.as_tensor(np.asarray(bc) == 1, device=a.device)[:, None]
        sa = torch.sqrt(a)[:, None]
        self.r = sa * self.J
        base = torch.where(self.hard, self.dJ / (self.J * self.dH), 1 / self.H)
        self.l = base / sa
        self.rhs_scale = 2j / (math.pi * a[:, None]) * base

    def pairs(self):
        """J, Y [2N+1][M, M] of k b_pq and e^{i alpha_pq}; the diagonal is a dummy."""
        d = self.O[:, None, :] - self.O[None, :, :]
        eye = torch.eye(self.M, dtype=torch.float64, device=d.device)
        d = d + eye[..., None]
        b = torch.sqrt((d * d).sum(-1))
        J, Y = _Bessel.apply((self.k * b).reshape(-1), 2 * self.N)
        e = torch.complex(d[..., 0] / b, d[..., 1] / b)
        return J.reshape(-1, self.M, self.M), Y.reshape(-1, self.M, self.M), e, 1.0 - eye

    def shifts(self):
        """(l, g_l [M, M]) for l = -2N..2N, zero on the diagonal."""
        J, Y, e, off = self.pairs()
        p = torch.ones_like(e)
        for l in range(2 * self.N + 1):
            H = torch.complex(J[l], Y[l]) * off
            yield l, H * p
            if l:
                yield -l, (-1.0) ** l * H * p.conj()
            p = p * e

    def apply(self, x):
        """(I + l T(g) r) x for x [M n, R]."""
        X = x.reshape(self.M, self.n, -1)
        xs = X * self.r[..., None]
        s = torch.zeros_like(xs)
        for l, g in self.shifts():  # s_m += g_l xs_{m + l}
            lo, hi = max(0, -l), min(self.n, self.n - l)
            if lo < hi:
                s[:, lo:hi] += (g @ xs[:, lo + l:hi + l].reshape(self.M, -1)).reshape(self.M, hi - lo, -1)
        return (X + self.l[..., None] * s).reshape(x.shape)

    def matrix(self):
        G = torch.stack([g for _, g in sorted(self.shifts(), key=lambda t: t[0])])  # [4N+1, M, M]
        m = torch.arange(self.n, device=G.device)
        blocks = G[(m[None, :] - m[:, None]) + 2 * self.N]  # [m, n', p, q]
        A = blocks.permute(2, 0, 3, 1) * self.l[:, :, None, None] * self.r[None, None]
        A = A.reshape(self.M * self.n, -1)
        return A + torch.eye(len(A), dtype=A.dtype, device=A.device)

    def modes(self):
        return torch.arange(-self.N, self.N + 1, device=self.O.device, dtype=torch.float64)

    def rhs(self, betas):
        proj = self.O[:, :1] * torch.cos(betas) + self.O[:, 1:] * torch.sin(betas)  # [M, R]
        d = torch.exp(1j * self.k * proj)[:, None, :] * torch.exp(
            1j * self.modes()[:, None] * (0.5 * math.pi - betas))[None]
        amp = torch.sqrt(2 * math.pi * self.a)[:, None, None]
        return (self.rhs_scale[..., None] * amp * d).reshape(self.M * self.n, -1)

    def farfield(self, rho, thetas):
        proj = thetas.cos()[:, None] * self.O[:, 0] + thetas.sin()[:, None] * self.O[:, 1]  # [T, M]
        c = torch.exp(1j * self.modes() * (thetas[:, None] - 0.5 * math.pi))[:, None, :] * self.J[None]
        pre = 1j * np.exp(-0.25j * math.pi) / (2 * torch.sqrt(self.k)) * torch.sqrt(self.a) * torch.exp(
            -1j * self.k * proj)
        return (pre[..., None] * c).reshape(len(thetas), -1) @ rho

    def nearfield(self, rho, pts):
        w = (0.5j * math.pi * self.a / torch.sqrt(2 * math.pi * self.a))[:, None] * self.J
        w = w[..., None] * rho.reshape(self.M, self.n, -1)
        u = torch.zeros(len(pts), rho.shape[1], dtype=torch.complex128, device=pts.device)
        step = max(1, 4_000_000 // len(pts))
        for p in range(0, self.M, step):  # a few disks at a time
            d = pts[None] - self.O[p:p + step, None]  # [disks, points, 2]
            r = torch.sqrt((d * d).sum(-1))
            a = self.a[p:p + step, None]
            inside = (r <= a).any(0)
            J, Y = _Bessel.apply(self.k * torch.maximum(r, a), self.N)
            H = torch.complex(_orders(J, self.N), _orders(Y, self.N))
            H = H * torch.exp(1j * self.modes()[:, None, None] * torch.atan2(d[..., 1], d[..., 0]))
            u += torch.einsum("mdt,dmr->tr", H, w[p:p + step])
            u[inside] = complex(float("nan"), 0.0)
        return torch.where(torch.isnan(u.real), torch.zeros_like(u), u)


def _dense(cl, dev, grad=False):
    t = [torch.tensor(v, dtype=torch.float64, device=dev, requires_grad=grad) for v in (cl.centres, cl.radii, cl.k)]
    return _Dense(t[0], t[1], t[2], cl.N, cl.bc), t


def exact(case, seed):
    dev = torch.device("cuda" if torch.cuda.is_available() else "cpu")
    s = _inputs(case, seed)
    cls, R = s["clusters"], case["columns"]

    def put(v):
        return torch.from_numpy(np.ascontiguousarray(v)).to(dev)

    def rows(v):
        return torch.split(put(v).to(torch.complex128), [c.ntot for c in cls])

    if case["path"] == "product":
        return torch.cat([_dense(c, dev)[0].apply(x) for c, x in zip(cls, rows(s["x"]))])
    if case["path"] == "update":
        D, _ = _dense(s["next"], dev)
        diag = torch.stack([D.J + 0j, D.dJ + 0j, D.H, D.dH]).reshape(4, -1)
        G = torch.empty(D.M, D.M, 4 * D.N + 1, dtype=torch.complex128, device=dev)
        for l, g in D.shifts():
            G[:, :, l + 2 * D.N] = g.T  # [q][p][l]
        return [diag, G, D.apply(put(s["x"]))]
    if case["path"] == "farfield":
        return torch.stack([_dense(c, dev)[0].farfield(r, put(s["thetas"])) for c, r in zip(cls, rows(s["rho"]))])
    if case["path"] == "nearfield":
        return _dense(cls[0], dev)[0].nearfield(put(s["rho"]), put(s["points"]))
    if case["path"] == "gradient":
        D, t = _dense(cls[0], dev, grad=True)
        rho = torch.linalg.solve(D.matrix(), D.rhs(put(s["betas"])))
        m = (D.farfield(rho, put(s["thetas"])) - put(s["target"][0])).abs().square().sum()
        m.backward()
        return [m.detach().reshape(1), t[0].grad, t[1].grad, t[2].grad.reshape(1)]
    if case["path"] == "solve":
        D = [_dense(c, dev)[0] for c in cls]
        rho = [torch.linalg.solve(d.matrix(), d.rhs(put(s["betas"]))) for d in D]
        return [torch.cat(rho), torch.stack([d.farfield(r, put(s["thetas"])) for d, r in zip(D, rho)])]
    D, al = _dense(cls[0], dev)[0], put(W.angles(R))
    F = D.farfield(torch.linalg.solve(D.matrix(), D.rhs(al)), al + math.pi)
    T = F.conj().T @ F
    return [torch.flip(torch.linalg.eigvalsh(T), [0])[None], F[None], T[None]]
