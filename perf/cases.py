"""What a user of the library has it do, as timed cases: products and delayed sums of the
ET-AIM operator, marches, and the far-field post-processing, through the public binding.

A context (mesh, grid, tables, preconditioner) is what a program sets up once and keeps;
the vectors, histories, plane waves and spectra it feeds to it are the inputs and are drawn
from the seed.  Results of the complex64 grid path are kept in complex64, the precision
that path has; the plain path's stay complex128.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_1408_7060_gb300 import AimContext, abi
from paper_1408_7060_gb300.inputs import icosphere, place_grid, plate_mesh, random_plane_waves, sphere_array
from paper_1408_7060_gb300.rcs import sphere_grid

C0 = 299792458.0
BETA = 0.25  # dt = BETA / half band, the step of every workload of the repository

DEFAULTS = dict(op="matvec", mesh="sphere", size=4, grid=64, precision="c64", waves=1, f_mhz=600.0, band=0.1,
                order=2, delay=0, steps=0, tol=1e-6, precond="diag", sai_scale=1.0, refine=0, blocked=0,
                directions=0, freqs=0)


def listed():
    return [
        # the smallest product: the 480-RWG parity sphere, plain path, one vector; launches count
        dict(name="matvec_sphere480_c128", op="matvec", mesh="sphere", size=2, grid=16, precision="c128", f_mhz=150.0,
             band=0.5),
        # an open surface (2 m plate, 4 grid planes deep), a delayed term, an odd batch
        dict(name="matvec_plate1160_c64", op="matvec", mesh="plate", size=20, grid=32, f_mhz=285.0, band=0.0526,
             order=3, waves=3, delay=1),
        # one vector on the 7680-RWG sphere: the product inside a single-wave march
        dict(name="matvec_sphere7680_c64", op="matvec", size=4, grid=64, f_mhz=600.0, band=0.3),
        # the 64 plane waves of the batched sphere
        dict(name="matvec_sphere7680_b64_c64", op="matvec", size=4, grid=64, f_mhz=600.0, band=0.1, waves=64),
        # the plain path at a length with a factor 3: reference products, FP64 throughout
        dict(name="matvec_sphere7680_n96_c128", op="matvec", size=4, grid=96, precision="c128", f_mhz=600.0, band=0.3),
        # the 4 x 4 sphere array on the 384^3 grid (768 x 768 x 192 transforms), four waves
        dict(name="matvec_array_n384_c64", op="matvec", mesh="array", size=4, grid=384, f_mhz=1000.0, band=0.05,
             waves=4),
        # the right-hand side of a step with many delays (N_g = 12), power-of-two z transforms
        dict(name="rhs_sphere7680_wide_c64", op="rhs", size=4, grid=64, f_mhz=600.0, band=0.6),
        # the right-hand side at a length with a factor 3, a small batch
        dict(name="rhs_sphere7680_n96_c64", op="rhs", size=4, grid=96, f_mhz=600.0, band=0.3, waves=4),
        # a whole march on the plain path: the small sphere, pulse and all
        dict(name="march_sphere480_c128", op="march", size=2, grid=16, precision="c128", f_mhz=150.0, band=0.2,
             steps=32, tol=1e-6),
        # a whole march on the production path: complex64 grid stages, near-zone SAI, FP64 refinement
        dict(name="march_sphere7680_c64", op="march", size=4, grid=64, f_mhz=600.0, band=0.1, waves=4, steps=24,
             tol=1e-6, precond="sai", sai_scale=2.5, refine=4),
        # the far-field envelopes of a current history and the adjoint map back (gradients)
        dict(name="farfield_sphere1920", op="farfield", size=3, grid=32, precision="c128", f_mhz=300.0, band=0.3,
             steps=60, directions=16),
        # bistatic RCS of two waves at three frequencies over the whole sphere of directions
        dict(name="rcs_sphere7680", op="rcs", size=4, grid=64, f_mhz=600.0, band=0.3, waves=2, freqs=3,
             directions=288),
    ]


# meshes and the grids that resolve them: (mesh, size, grids, carrier in MHz, RWGs)
_SHAPES = [("sphere", 2, (16,), 150.0), ("sphere", 3, (32, 64), 300.0), ("sphere", 4, (64, 96, 128), 600.0)]


def _log_int(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    """One more case of these ranges: spheres of 480 to 7680 RWGs and plates of 65 to 7400,
    grids of 16 to 128, one wave to a batch of 64, both precisions, every operation."""
    op = rng.choice(["matvec"] * 5 + ["rhs"] * 3 + ["march"] * 3 + ["farfield", "rcs"])
    c = dict(op=op)
    if rng.random() < 0.35:
        cells = _log_int(rng, 5, 50)
        grid = 16 if cells <= 9 else 32 if cells <= 24 else rng.choice((64, 96))
        c.update(mesh="plate", size=cells, grid=grid, f_mhz=round(rng.uniform(250.0, 300.0), 2),
                 band=round(rng.uniform(0.05, 0.15), 4), order=rng.choice((2, 3)))
    else:
        mesh, size, grids, f = rng.choice(_SHAPES)
        grid = rng.choice(grids)
        c.update(mesh=mesh, size=size, grid=grid, f_mhz=round(f * rng.uniform(0.8, 1.0), 2),
                 band=round(rng.uniform(0.1, 0.5), 4), order=rng.choice((2, 2, 3)))
    c["precision"] = rng.choice(("c64", "c64", "c128"))
    most = 64 if grid <= 64 else 8
    if c["precision"] == "c128":
        most = max(1, most // 16)
    if op == "matvec":
        c.update(waves=_log_int(rng, 1, most), delay=rng.choice((0, 0, 1, 2)))
    elif op == "rhs":
        c.update(waves=_log_int(rng, 1, max(1, most // 4)))
    elif op == "march":
        # grids up to 64 (plain path: 32); the pulse's band kept narrow so that the currents decay
        if c["grid"] > 64 or (c["precision"] == "c128" and c["grid"] > 32):
            c.update(mesh="sphere", size=3, grid=32, f_mhz=round(300.0 * rng.uniform(0.8, 1.0), 2), precision="c128")
        c.update(waves=rng.randint(1, 3), steps=rng.randint(8, 24), band=round(rng.uniform(0.05, 0.2), 4),
                 blocked=rng.choice((0, 0, 1)))
        if c["precision"] == "c64":
            sai = c["mesh"] == "plate" or c["size"] == 4 or rng.random() < 0.5
            c.update(refine=4, precond="sai" if sai else "diag", tol=1e-6)
        else:
            c.update(tol=rng.choice((1e-6, 1e-8)))
    elif op == "farfield":
        if c["mesh"] == "sphere":
            c.update(size=rng.choice((2, 3)), grid=32, f_mhz=200.0)
        c.update(precision="c128", steps=rng.randint(10, 60), directions=rng.randint(1, 16))
    else:
        c.update(waves=rng.randint(1, 4), freqs=rng.randint(1, 4), directions=_log_int(rng, 20, 300))
    return c


# ------------------------------------------------------------------ what a program keeps

_KEPT: dict = {}   # the contexts of the last two set-ups, as a program keeps its own


def _full(case):
    c = dict(DEFAULTS)
    c.update(case)
    return c


def _geometry(c):
    if c["mesh"] == "plate":
        V, F = plate_mesh(0.1 * c["size"], c["size"])
    elif c["mesh"] == "array":
        V, F = sphere_array(c["size"], 0.5, 1.5)
    else:
        V, F = icosphere(c["size"], 1.0)
    h, origin = place_grid(V, c["grid"], 0.15 if c["mesh"] == "sphere" and c["grid"] == 16 else None)
    return V, F, h, origin


def _dt(c):
    return BETA / (c["band"] * c["f_mhz"] * 1e6)


def _context(c):
    key = tuple((k, c[k]) for k in ("mesh", "size", "grid", "precision", "waves", "f_mhz", "band", "order", "precond",
                                    "sai_scale", "refine", "blocked"))
    if key not in _KEPT:
        V, F, h, origin = _geometry(c)
        near = 2 * h if c["grid"] == 16 and c["mesh"] == "sphere" else 3 * h
        while len(_KEPT) >= 2:
            _KEPT.pop(next(iter(_KEPT)))
        _KEPT[key] = AimContext(V=V, F=F, grid_n=c["grid"], origin=origin, h=h, near_radius=near, dt=_dt(c),
                                f_c=c["f_mhz"] * 1e6, order=c["order"], precision=c["precision"],
                                batch_max=c["waves"], precond=c["precond"], precond_radius=c["sai_scale"] * near,
                                refine=c["refine"], rhs_blocked=c["blocked"])
    return _KEPT[key]


def _normal(shape, seed):
    """Standard normal complex128 values on the GPU."""
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    return torch.view_as_complex(torch.randn(*shape, 2, generator=g, dtype=torch.float64, device="cuda"))


def _directions(n, seed):
    """n observation directions with two transverse unit vectors each."""
    r, e1 = random_plane_waves(n, seed)
    return r, e1, np.cross(r, e1)


def _far_times(c, ctx):
    """First far-field time and the number of them: the marched steps and the surface's reach."""
    V = _geometry(c)[0]
    reach = int(math.ceil(np.linalg.norm(V, axis=1).max() / (C0 * _dt(c))))
    return 1 - reach, c["steps"] + 2 * reach + c["order"]


def prepare(case, seed):
    c = _full(case)
    ctx = _context(c)
    ns, nb = ctx.ns, c["waves"]
    s = dict(c=c, ctx=ctx)
    if c["op"] == "matvec":
        s["m"] = min(c["delay"], ctx.n_delays)
        s["x"] = _normal((nb, ns), seed)
        s["out"] = torch.empty_like(s["x"])
    elif c["op"] == "rhs":
        s["hist"] = _normal((ctx.n_delays, nb, ns), seed)
        s["out"] = torch.empty((nb, ns), dtype=torch.complex128, device="cuda")
    elif c["op"] == "march":
        s["k"], s["p"] = random_plane_waves(nb, seed)
        s["sigma"] = 3.0 / (2.0 * math.pi * c["band"] * c["f_mhz"] * 1e6)
        s["out"] = torch.empty((c["steps"], nb, ns), dtype=torch.complex128, device="cuda")
    elif c["op"] == "farfield":
        s["dirs"] = _directions(c["directions"], 7 + seed % 1000)
        s["I"] = _normal((c["steps"], ns), seed)
        s["n0"], s["n_out"] = _far_times(c, ctx)
    else:
        n_th = max(2, int(round(math.sqrt(c["directions"] / 2))))
        rhat, pol, _, _, _ = sphere_grid(n_th, max(1, c["directions"] // n_th))
        s["rhat"], s["pol"] = rhat, pol
        f = c["f_mhz"] * 1e6
        s["f"] = f * (1.0 + c["band"] * np.linspace(-0.5, 0.5, c["freqs"])) if c["freqs"] > 1 else np.array([f])
        s["spec"] = _normal((c["freqs"], nb, ns), seed)
        s["out"] = torch.empty((c["freqs"], nb, len(rhat)), dtype=torch.float64, device="cuda")
    return s


def _kept(c, y):
    return y.to(torch.complex64) if c["precision"] == "c64" else y


def run(s):
    c, ctx = s["c"], s["ctx"]
    if c["op"] == "matvec":
        return _kept(c, ctx.matvec(s["m"], s["x"], out=s["out"]))
    if c["op"] == "rhs":
        return _kept(c, ctx.rhs(ctx.n_delays + 1, s["hist"], out=s["out"]))
    if c["op"] == "march":
        cur, _, _ = ctx.march(s["k"], s["p"], s["sigma"], 8.0 * s["sigma"], c["steps"], c["tol"], out=s["out"])
        return _kept(c, cur)
    if c["op"] == "farfield":
        F = abi.aim_farfield(ctx.handle, *s["dirs"], s["I"], s["n0"], s["n_out"])
        G = abi.aim_farfield_adjoint(ctx.handle, *s["dirs"], c["steps"], s["n0"], F)
        return F, G
    return ctx.rcs(s["f"], s["spec"], s["rhat"], s["pol"], out=s["out"])


# ------------------------------------------------------------------ the work of one pass

def _sizes(c):
    """RWGs, near pairs, z transform length, delays and triangles, from the geometry."""
    area = {"plate": (0.1 * c["size"]) ** 2, "array": 16 * math.pi, "sphere": 4 * math.pi}[c["mesh"]]
    span = {"plate": 0.1 * c["size"], "array": 5.5, "sphere": 2.0}[c["mesh"]]
    depth = {"plate": 0.0, "array": 1.0, "sphere": 2.0}[c["mesh"]]
    ns = (3 * c["size"] ** 2 - 2 * c["size"] if c["mesh"] == "plate" else
          30 * 4 ** c["size"] * (16 if c["mesh"] == "array" else 1))
    h = 0.15 if c["mesh"] == "sphere" and c["grid"] == 16 else span / (c["grid"] - 5)
    near = 2 * h if c["grid"] == 16 and c["mesh"] == "sphere" else 3 * h
    nnz = ns * (1 + ns / area * math.pi * near * near)
    lz = 2 * (int(depth / h) + 4)          # no circular z transform of the box is shorter
    diag = math.sqrt(2 * span * span) if c["mesh"] != "sphere" else span
    ng = int((diag + 3 * h) / (C0 * _dt(c)) + c["order"])
    return ns, nnz, lz, ng, 2 * ns / 3


def work(case):
    c = _full(case)
    ns, nnz, lz, ng, nt = _sizes(c)
    nb, N = c["waves"], c["grid"]
    es = 8 if c["precision"] == "c64" else 16
    M = (2 * N) * (2 * N) * lz
    fft = 4 * 5 * M * math.log2(M)                       # one 3-D transform of the four grids
    product = 2 * fft / 2 + 6 * 4 * M + 2 * 4 * 256 * ns  # half the inputs and outputs are padding
    tables = 2 * (N + 1) ** 2 * (lz / 2 + 1) * es + ns * 256 * es / 2 + nnz * 20
    one = dict(flops=nb * (product + 8 * nnz), bytes=2 * nb * ns * 16 + tables)
    if c["op"] == "matvec":
        return one
    if c["op"] == "rhs":
        # every history vector to its spectrum, the spectral sum, one inverse transform
        flops = nb * ((ng + 1) * fft / 2 + 8 * 4 * M * ng + ng * 8 * nnz + (ng + 1) * 4 * 256 * ns)
        return dict(flops=flops, bytes=(ng + 1) * nb * ns * 16 + ng * (tables - ns * 256 * es / 2) + ns * 256 * es / 2)
    if c["op"] == "march":
        its = 12 if c["precond"] == "sai" else 25
        return dict(flops=c["steps"] * (its + ng) * one["flops"], bytes=c["steps"] * (its + ng) * one["bytes"])
    if c["op"] == "farfield":
        n_out = c["steps"] + 2 * int(2.0 / (C0 * _dt(c)) + 1)
        pts, taps = 7 * nt * c["directions"], c["order"] + 1
        return dict(flops=2 * pts * (40 + c["steps"] * taps * 16),
                    bytes=16.0 * (2 * c["steps"] * ns + 2 * n_out * c["directions"] * 2) + 7 * nt * 32)
    pts = 7 * nt * c["freqs"] * c["directions"]
    return dict(flops=pts * (40 + nb * 16), bytes=16.0 * c["freqs"] * nb * ns + 7 * nt * 32)


# ------------------------------------------------------------------ the same in plain 64-bit torch

class _Plain:
    """The operator of a context from its tables (stencil weights, kernel spectra, near
    values: what set-up computed), with torch's FFTs and sums in complex128."""

    def __init__(self, ctx):
        self.ctx, i = ctx, ctx.info
        dev = "cuda"
        anchor, lam = ctx.anterp()
        a = torch.from_numpy(anchor.astype(np.int64)).to(dev)
        L, self.LZ = 2 * i["grid_n"], i["z_len"]
        self.shape = (self.LZ, L, L)
        t = torch.arange(64, device=dev)
        x, y, z = a[:, :1] + (t & 3), a[:, 1:2] + ((t >> 2) & 3), a[:, 2:] - i["box_lo"][2] + (t >> 4)
        self.node = (z * L + y) * L + x                     # [ns][64]
        self.lam = torch.from_numpy(lam).to(dev)            # [ns][4][64]
        rowptr, col, self.val = ctx.near()
        self.row = torch.repeat_interleave(torch.arange(ctx.ns, device=dev),
                                           torch.from_numpy(np.diff(rowptr).astype(np.int64)).to(dev))
        self.col = torch.from_numpy(col.astype(np.int64)).to(dev)

    def spectrum(self, m, kind):
        o = torch.from_numpy(self.ctx.kernel_spectrum(m, kind)).cuda()
        for d, n in enumerate(self.shape):
            k = torch.arange(n, device="cuda")
            o = o.index_select(d, torch.minimum(k, n - k))
        return o * float(np.prod(self.shape))

    def apply(self, m, x):
        """Z_m x for x [nb][ns]."""
        y = torch.zeros_like(x)
        val = torch.from_numpy(self.val[m]).cuda()
        y.index_add_(1, self.row, val * x[:, self.col])
        for c in range(4):
            if c in (0, 3):
                G = self.spectrum(m, c // 3)
            w = self.lam[:, c]
            for b in range(x.shape[0]):
                g = torch.zeros(int(np.prod(self.shape)), dtype=torch.complex128, device="cuda")
                g.index_add_(0, self.node.reshape(-1), (w * x[b][:, None]).reshape(-1))
                g = torch.fft.ifftn(torch.fft.fftn(g.view(self.shape)) * G).reshape(-1)
                y[b] += (w * g[self.node]).sum(1)
        return y

    def dense(self, m):
        """Z_m as a matrix, from its columns."""
        ns = self.ctx.ns
        Z = torch.zeros(ns, ns, dtype=torch.complex128, device="cuda")
        Z[self.row, self.col] = torch.from_numpy(self.val[m]).cuda()
        G = [self.spectrum(m, 0), self.spectrum(m, 1)]
        step = 16
        for k0 in range(0, ns, step):
            n = min(step, ns - k0)
            cols = torch.arange(n, device="cuda")[:, None]
            for c in range(4):
                g = torch.zeros(n, int(np.prod(self.shape)), dtype=torch.complex128, device="cuda")
                g[cols, self.node[k0:k0 + n]] = self.lam[k0:k0 + n, c].to(torch.complex128)
                g = torch.fft.fftn(g.view(n, *self.shape), dim=(1, 2, 3)) * G[c // 3]
                g = torch.fft.ifftn(g, dim=(1, 2, 3)).reshape(n, -1)
                for j in range(n):
                    Z[:, k0 + j] += (self.lam[:, c] * g[j][self.node]).sum(1)
        return Z


class _Surface:
    """The cubature points of every RWG side in plain torch: r [ns][2][7][3], the basis
    function there and the weights (7-point degree-5 rule of Radon)."""

    def __init__(self, ctx, V, F):
        s15 = math.sqrt(15.0)
        b, w = [(1 / 3, 1 / 3, 1 / 3)], [9 / 40]
        for sg in (-1.0, 1.0):
            p = (6.0 + sg * s15) / 21.0
            for i in range(3):
                q = [p, p, p]
                q[i] = 1.0 - 2.0 * p
                b.append(tuple(q))
                w.append((155.0 + sg * s15) / 1200.0)
        b, w = np.array(b), np.array(w)
        edge, tri, free = ctx.rwg_table()
        T = V[F]                                             # [nt][3][3]
        area = 0.5 * np.linalg.norm(np.cross(T[:, 1] - T[:, 0], T[:, 2] - T[:, 0]), axis=1)
        ln = np.linalg.norm(V[edge[:, 0]] - V[edge[:, 1]], axis=1)
        r = np.einsum("qv,kavd->kaqd", b, T[tri])            # [ns][2][7][3]
        sign = np.array([1.0, -1.0])[None, :]
        coef = sign * ln[:, None] / (2.0 * area[tri])
        S = coef[:, :, None, None] * (r - V[free][:, :, None, :])
        wt = w[None, None, :] * area[tri][:, :, None]
        self.r = torch.from_numpy(r.reshape(ctx.ns, 14, 3)).cuda()
        self.wS = torch.from_numpy((wt[..., None] * S).reshape(ctx.ns, 14, 3)).cuda()


def _excitation(sf, c, k, p, l):
    """V_l of the modulated Gaussian plane waves [nb][ns]."""
    wc, dt = 2 * math.pi * c["f_mhz"] * 1e6, _dt(c)
    sigma = 3.0 / (2.0 * math.pi * c["band"] * c["f_mhz"] * 1e6)
    out = []
    for kb, pb in zip(k, p):
        delay = (sf.r @ torch.from_numpy(kb).cuda()) / C0
        tau = l * dt - delay - 8.0 * sigma
        g = torch.exp(-tau ** 2 / (2 * sigma ** 2))
        e = torch.complex(-tau / sigma ** 2 * g, wc * g) * torch.exp(-1j * wc * (delay + 8.0 * sigma))
        out.append(((sf.wS @ torch.from_numpy(pb).cuda()) * e).sum(1))
    return torch.stack(out)


def _d_basis(u, Q, dt, wc):
    """(DT)(u) = T'(u)/dt + j wc T(u) of the piecewise Lagrange basis of order Q."""
    T, D = torch.zeros_like(u), torch.zeros_like(u)
    for j in range(Q + 1):
        nodes = [i for i in range(j - Q, j + 1) if i != 0]
        on = (u > j - 1) & (u <= j)
        t, d = torch.ones_like(u), torch.zeros_like(u)
        for i in nodes:
            d = d * (u - i) / (-i) + t / (-i)
            t = t * (u - i) / (-i)
        T, D = torch.where(on, t, T), torch.where(on, d, D)
    return torch.complex(D / dt, wc * T)


def _far_terms(sf, s, d):
    """Direction d: delays in steps and the two weighted transverse components, per point."""
    c = s["c"]
    rh, e1, e2 = (torch.from_numpy(np.ascontiguousarray(v[d])).cuda() for v in s["dirs"])
    rr = sf.r @ rh
    ph = torch.exp(1j * (2 * math.pi * c["f_mhz"] * 1e6 / C0) * rr)
    cf = -4e-7 * math.pi / (4 * math.pi)
    return rr / (C0 * _dt(c)), cf * (sf.wS @ e1) * ph, cf * (sf.wS @ e2) * ph


def _exact_far(s):
    """F[n][d][q] = sum_l sum_k I_l[k] A_{n-l}[k] and its adjoint, through the taps A_s."""
    c, ctx = s["c"], s["ctx"]
    V, F_, _, _ = _geometry(c)
    sf = _Surface(ctx, V, F_)
    nl, no, n0 = c["steps"], s["n_out"], s["n0"]
    wc = 2 * math.pi * c["f_mhz"] * 1e6
    F = torch.zeros(no, c["directions"], 2, dtype=torch.complex128, device="cuda")
    G = torch.zeros(nl, ctx.ns, dtype=torch.complex128, device="cuda")
    for d in range(c["directions"]):
        u, a1, a2 = _far_terms(sf, s, d)
        top = int(u.abs().max().item()) + c["order"] + 2
        taps = {}
        for sh in range(-top, top + 1):                      # sh = n - l
            t = _d_basis(sh + u, c["order"], _dt(c), wc)
            taps[sh] = torch.stack([(t * a1).sum(1), (t * a2).sum(1)], 1)   # [ns][2]
        for i in range(no):
            for j in range(nl):
                sh = (n0 + i) - (j + 1)
                if sh in taps:
                    F[i, d] += s["I"][j] @ taps[sh]
        for i in range(no):
            for j in range(nl):
                sh = (n0 + i) - (j + 1)
                if sh in taps:
                    G[j] += taps[sh].conj() @ F[i, d]
    return F, G


def _exact_rcs(s):
    c, ctx = s["c"], s["ctx"]
    V, F_, _, _ = _geometry(c)
    sf = _Surface(ctx, V, F_)
    rh, pol = torch.from_numpy(s["rhat"]).cuda(), torch.from_numpy(s["pol"]).cuda()
    out = torch.empty_like(s["out"])
    for i, f in enumerate(s["f"]):
        w = 2 * math.pi * float(f)
        for d in range(len(rh)):
            ph = torch.exp(1j * (w / C0) * (sf.r @ rh[d]))
            v = (sf.wS.to(torch.complex128) * ph[..., None]).sum(1)          # [ns][3]
            proj = pol[d] - rh[d] * (rh[d] @ pol[d])
            e = s["spec"][i] @ (v @ proj.to(torch.complex128))
            out[i, :, d] = 4 * math.pi * (w * 4e-7 * math.pi / (4 * math.pi)) ** 2 * e.abs() ** 2
    return out


def _exact_march(s):
    c, ctx = s["c"], s["ctx"]
    if ctx.ns > 2000:
        return None  # a dense solve of the larger systems takes too long
    V, F_, _, _ = _geometry(c)
    sf, op = _Surface(ctx, V, F_), _Plain(ctx)
    Z = [op.dense(m) for m in range(ctx.n_delays + 1)]
    LU = torch.linalg.lu_factor(Z[0])
    I = []
    for l in range(1, c["steps"] + 1):
        b = _excitation(sf, c, s["k"], s["p"], l)
        for m in range(1, ctx.n_delays + 1):
            if l - m >= 1:
                b = b - I[l - m - 1] @ Z[m].T
        I.append(torch.linalg.lu_solve(*LU, b.T).T)
    return torch.stack(I)


def exact(case, seed):
    s = prepare(case, seed)
    op = s["c"]["op"]
    if op == "matvec":
        return _Plain(s["ctx"]).apply(s["m"], s["x"])
    if op == "rhs":
        p = _Plain(s["ctx"])
        return sum(p.apply(m, s["hist"][m - 1]) for m in range(1, s["ctx"].n_delays + 1))
    if op == "march":
        return _exact_march(s)
    return _exact_far(s) if op == "farfield" else _exact_rcs(s)
