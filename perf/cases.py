"""Performance cases of the library: the calls its users make, over the sizes they make them on.

Every case is a dict of plain values; ``prepare`` builds what a program holds before the call (the
microstructure, the context / batch / server with its workspace, the vectors), ``run`` makes the
call through the public binding, ``work`` states the bytes and operations the path cannot do
without, and ``exact`` computes the same outputs in 64-bit torch without the library.

Kinds:
  apply       one operator product (elas_apply in FP64, elas_apply_f32 in FP32)
  residual    the FP64 residual A w + b with its norm
  stress      voxel stress, von Mises and macroscopic stress of a fluctuation
  hotspot     the smoothed maximum stress of a von Mises field
  generate    one microstructure: grain assignment, orientations, pore overwrite
  solve       one PCG solve and the stress of its solution
  batch       several RVEs under the six unit load cases, advanced together
  serve       a burst of requests through the continuous-batching server until all are collected

Iterated cases stop at a true relative residual of 1e-11, so that two correct solves of the same
inputs agree well beyond their stopping error.  A fluctuation is determined up to a rigid
translation, which rounding in the single-precision iteration moves: programs that take
displacements from a mixed-precision solve refer them to the solid's mean, and so do the cases.
"""
import math

import numpy as np
import torch

from paper_2602_07354_gb300 import binding as B
from paper_2602_07354_gb300 import synth

TOL = 1e-11
MAX_ITER = 20000
CUBIC = (204.6, 137.7, 126.2)          # C11, C12, C44 (GPa) of the polycrystal workload
UNIT_LOADS = 1e-3 * np.eye(6)          # e11, e22, e33, e23, e13, e12
MEAN_PORE = 4.0 / 3.0 * math.pi * 80   # voxels of a sphere with radius uniform in 2..6 (E[r^3] = 80)


# --- the cases -----------------------------------------------------------------------------------
def listed():
    return [
        # the 20^3 inclusion cell's product: launches and latency count
        dict(name="apply_fp64_20", kind="apply", f32=False, micro="inclusion", nx=20, ny=20, nz=20, grains=2, pores=0.0),
        # the operator of the 100^3 polycrystal workload
        dict(name="apply_fp64_100", kind="apply", f32=False, micro="poly", nx=100, ny=100, nz=100, grains=500, pores=0.01),
        # a cropped scan: odd, ragged dimensions
        dict(name="apply_f32_ragged", kind="apply", f32=True, micro="poly", nx=131, ny=87, nz=59, grains=336, pores=0.02),
        # one product of a large single solve (voxels per grain of the 500^3 cell)
        dict(name="apply_f32_300", kind="apply", f32=True, micro="poly", nx=300, ny=300, nz=300, grains=4320, pores=0.02),
        # post-processing of the 200^3 repeat of the polycrystal workload
        dict(name="stress_200", kind="stress", micro="poly", nx=200, ny=200, nz=200, grains=4000, pores=0.01),
        # stress concentration extraction on a 200^3 field with the study's kernel width
        dict(name="hotspot_200", kind="hotspot", micro="poly", nx=200, ny=200, nz=200, grains=4000, pores=0.01, s=0.4, solid=False),
        # what every served request of the largest edge generates before its solve
        dict(name="generate_160", kind="generate", nx=160, ny=160, nz=160, grains=2048, pores=0.015, weighted=False),
        # the smallest solve: 20^3 inclusion cell, Algorithm 2's stopping rule
        dict(name="solve_fp64_20", kind="solve", mixed=False, micro="inclusion", nx=20, ny=20, nz=20, grains=2, pores=0.0),
        # plain FP64 solve of the 100^3 polycrystal workload
        dict(name="solve_fp64_100", kind="solve", mixed=False, micro="poly", nx=100, ny=100, nz=100, grains=500, pores=0.01),
        # mixed-precision solve of a 128^3 polycrystal
        dict(name="solve_mixed_128", kind="solve", mixed=True, micro="poly", nx=128, ny=128, nz=128, grains=1048, pores=0.015),
        # uneven RVEs, six load cases each: the columns of their effective stiffness
        dict(name="batch_5x6", kind="batch", edges="32,48,64,80,96", pores=0.015),
        # a burst of requests of the served sizes
        dict(name="serve_6", kind="serve", edges="48,96,64,128,48,64", pores=0.015),
    ]


def _dims(rng, lo, hi):
    """A ragged grid around an edge whose logarithm is uniform."""
    n = math.exp(rng.uniform(math.log(lo), math.log(hi)))
    d = [max(lo, min(hi, int(round(n * math.exp(rng.uniform(-0.35, 0.35)))))) for _ in range(3)]
    return dict(nx=d[0], ny=d[1], nz=d[2])


def _poly(rng, lo, hi):
    c = _dims(rng, lo, hi)
    N = c["nx"] * c["ny"] * c["nz"]
    c.update(micro="poly", grains=max(1, min(6000, N // rng.choice((2000, 2000, 6250)))), pores=round(rng.uniform(0.0, 0.03), 4))
    return c


def draw(rng):
    kind = rng.choice(("apply", "apply", "apply", "residual", "stress", "hotspot", "generate", "solve", "solve", "batch", "serve"))
    if kind == "apply":
        f32 = rng.random() < 0.5
        return dict(kind=kind, f32=f32, **_poly(rng, 17, 280 if f32 else 180))
    if kind == "residual":
        return dict(kind=kind, **_poly(rng, 17, 160))
    if kind == "stress":
        return dict(kind=kind, **_poly(rng, 17, 200))
    if kind == "hotspot":
        return dict(kind=kind, **_poly(rng, 17, 200), s=rng.choice((0.4, 0.4, 0.5, 0.8)), solid=rng.random() < 0.5)
    if kind == "generate":
        c = _poly(rng, 24, 180)
        del c["micro"]
        return dict(kind=kind, **c, weighted=rng.random() < 0.5)
    if kind == "solve":
        mixed = rng.random() < 0.5
        return dict(kind=kind, mixed=mixed, **_poly(rng, 17, 128 if mixed else 100))
    sizes, most = ((32, 48, 64, 80), 1.0e6) if kind == "batch" else ((48, 64, 96, 128), 5.5e6)
    edges = [rng.choice(sizes) for _ in range(rng.randint(2, 6))]
    while sum(n ** 3 for n in edges) > most:  # no more than the listed ones
        edges.pop()
    return dict(kind=kind, edges=",".join(map(str, edges)), pores=round(rng.uniform(0.0, 0.03), 4))


def _edges(case):
    return [int(e) for e in case["edges"].split(",")]


def _grid(case):
    return case["nx"], case["ny"], case["nz"]


# --- inputs --------------------------------------------------------------------------------------
def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed) & 0x7FFFFFFF)
    return g


def _rand(g, *shape):
    return torch.rand(*shape, generator=g, device="cuda", dtype=torch.float64)


def _pore_draws(dims, frac, g):
    """Centres and radii of spherical pores (r uniform in 2..6) of about this volume fraction."""
    N = dims[0] * dims[1] * dims[2]
    k = int(round(frac * N / MEAN_PORE))
    c = _rand(g, k, 3) * torch.tensor(dims, device="cuda", dtype=torch.float64)
    r = 2.0 + 4.0 * _rand(g, k)
    return c, r.clamp(max=0.45 * min(dims))


def _voronoi(dims, seeds):
    """Nearest seed of every voxel centre in the periodic cell (int32, x fastest)."""
    nx, ny, nz = dims
    G = seeds.shape[0]
    sq = []
    for d, n in enumerate(dims):
        x = torch.arange(n, device="cuda", dtype=torch.float64)[:, None] + 0.5 - seeds[None, :, d]
        x = x - n * torch.round(x / n)
        sq.append((x * x).float())
    out = torch.empty(nz * ny, nx, device="cuda", dtype=torch.int32)
    rows = max(1, (1 << 28) // (nx * G))
    for r0 in range(0, nz * ny, rows):
        r = torch.arange(r0, min(nz * ny, r0 + rows), device="cuda")
        yz = sq[2][r // ny] + sq[1][r % ny]
        out[r0:r0 + rows] = (yz[:, None, :] + sq[0][None]).argmin(-1).int()
    return out.reshape(-1)


def _stamp(phase, dims, c, r):
    """Voxels whose centre lies in a pore get the id -1 (periodic cell)."""
    nx, ny, nz = dims
    o = torch.arange(-7, 8, device="cuda")
    off = torch.stack(torch.meshgrid(o, o, o, indexing="ij"), -1).reshape(-1, 3)
    for p in range(0, c.shape[0], 256):
        at = torch.floor(c[p:p + 256]).long()[:, None, :] + off[None]
        d = at + 0.5 - c[p:p + 256, None, :]
        inside = (d * d).sum(-1) <= (r[p:p + 256] ** 2)[:, None]
        at = at[inside]
        phase[at[:, 0] % nx + nx * (at[:, 1] % ny + ny * (at[:, 2] % nz))] = -1
    return phase


def _rodrigues(g, n):
    u = _rand(g, n, 3).cpu().numpy()
    qw = np.sqrt(1 - u[:, 0]) * np.sin(2 * np.pi * u[:, 1])
    q = np.stack([np.sqrt(1 - u[:, 0]) * np.cos(2 * np.pi * u[:, 1]), np.sqrt(u[:, 0]) * np.sin(2 * np.pi * u[:, 2]),
                  np.sqrt(u[:, 0]) * np.cos(2 * np.pi * u[:, 2])], 1)
    return q / np.where(np.abs(qw) < 1e-8, 1e-8, qw)[:, None]


def _polycrystal(dims, grains, pores, g):
    """Phase ids on the device, material rows and Rodrigues vectors of a seeded polycrystal."""
    seeds = _rand(g, grains, 3) * torch.tensor(dims, device="cuda", dtype=torch.float64)
    phase = _voronoi(dims, seeds)
    _stamp(phase, dims, *_pore_draws(dims, pores, g))
    return phase, np.tile(synth.cubic_mat(*CUBIC), (grains, 1)), _rodrigues(g, grains)


def _micro(case, g, dims=None):
    """(phase on the device, materials, Rodrigues vectors or None) of a case's grid."""
    if dims is None:
        dims = _grid(case)
    if case.get("micro") == "inclusion":  # spherical inclusion of a quarter edge, isotropic phases
        x = torch.arange(dims[0], device="cuda", dtype=torch.float64) + 0.5 - dims[0] / 2
        r2 = x[:, None, None] ** 2 + x[None, :, None] ** 2 + x[None, None, :] ** 2
        phase = (r2 <= (dims[0] / 4) ** 2).int().reshape(-1)
        return phase, np.stack([synth.iso_mat(200.0, 0.3), synth.iso_mat(400.0, 0.25)]), None
    grains = case["grains"] if "grains" in case else max(1, dims[0] * dims[1] * dims[2] // 2000)
    return _polycrystal(dims, grains, case["pores"], g)


def _strain(g):
    e = _rand(g, 6).cpu().numpy() - 0.5
    return 1e-3 * e / math.sqrt(float((e[:3] ** 2).sum() + 2 * (e[3:] ** 2).sum()))


def _field(dims, g, scale):
    """A displacement-like vector field: long waves and node-to-node noise."""
    N = dims[0] * dims[1] * dims[2]
    f = torch.randn(3, N, generator=g, device="cuda", dtype=torch.float64).mul_(0.3 * scale)
    a = _rand(g, 3, 3, 2)
    for c in range(3):
        for d in range(3):
            n = dims[d]
            wave = torch.sin(2 * math.pi * (torch.arange(n, device="cuda", dtype=torch.float64) / n + a[c, d, 0])) * (scale * a[c, d, 1])
            f[c].view(dims[2], dims[1], dims[0]).add_(wave.view([-1 if d == 2 else 1, -1 if d == 1 else 1, -1 if d == 0 else 1]))
    return f.reshape(-1)


def _inputs(case, seed):
    """The case's inputs, from its seed alone; used by prepare and by exact."""
    g = _gen(seed)
    kind = case["kind"]
    if kind in ("batch", "serve"):
        problems = []
        for n in _edges(case):
            phase, mats, rho = _micro(case, g, (n, n, n))
            problems.append(dict(dims=(n, n, n), phase=phase, mats=mats, rho=rho, strain=_strain(g)))
        return dict(problems=problems)
    dims = _grid(case)
    if kind == "generate":
        seeds = (_rand(g, case["grains"], 3) * torch.tensor(dims, device="cuda", dtype=torch.float64)).cpu().numpy()
        semi = None
        if case["weighted"]:  # prolate grains, 10% spread
            rt = torch.exp(0.1 * torch.randn(case["grains"], generator=g, device="cuda", dtype=torch.float64))
            al = 1.0 + 0.1 * torch.randn(case["grains"], generator=g, device="cuda", dtype=torch.float64)
            semi = torch.stack([rt, rt * al.clamp(0.5, 1.5)], 1).cpu().numpy()
        c, r = _pore_draws(dims, case["pores"], g)
        eye = torch.eye(3, device="cuda", dtype=torch.float64).reshape(1, 9).expand(c.shape[0], 9)
        pores = torch.cat([c, r[:, None].expand(-1, 3), eye], 1).cpu().numpy()
        return dict(seeds=seeds, semi=semi, pores=pores, u=_rand(g, case["grains"], 3))
    phase, mats, rho = _micro(case, g)
    s = dict(phase=phase, mats=mats, rho=rho, strain=_strain(g))
    if kind == "apply":
        s["u"] = _field(dims, g, 1e-3)
        if case["f32"]:
            s["u"] = s["u"].float()
    elif kind in ("residual", "stress"):
        s["w"] = _field(dims, g, 1e-4)
    elif kind == "hotspot":  # a von Mises field (GPa): positive, rough, zero in the pores
        vm = 0.2 + 0.05 * torch.randn(phase.shape[0], generator=g, device="cuda", dtype=torch.float64)
        s["vm"] = torch.where(phase >= 0, vm.abs(), torch.zeros_like(vm))
    return s


def _microstructure(dims, p):
    return synth.Microstructure(*dims, p["phase"].cpu().numpy(), p["mats"], p["rho"])


def _solid_nodes(dims, phase):
    """1 for every node that touches a solid voxel, else 0; and their number."""
    m = (phase >= 0).view(dims[2], dims[1], dims[0])
    for d in range(3):
        m = m | torch.roll(m, 1, d)
    m = m.reshape(-1).double()
    return m, float(m.sum())


def _about_mean(w, solid):
    """Displacements relative to the mean over the solid's nodes, in place."""
    w = w.view(3, -1)
    w -= ((w * solid[0]).sum(1) / solid[1])[:, None] * solid[0]
    return w


def _f64(n):
    return torch.empty(n, dtype=torch.float64, device="cuda")


def prepare(case, seed):
    kind = case["kind"]
    s = _inputs(case, seed)
    s["case"] = case
    if kind == "batch":
        micros = [_microstructure(p["dims"], p) for p in s["problems"]]
        s["batch"] = B.elas_batch_create(micros, 6, B.PREC_MIXED)
        s["strains"] = np.tile(UNIT_LOADS.reshape(-1), len(micros))
        s["stress"] = [_f64(6 * m.N) for m in micros for _ in range(6)]
    elif kind == "serve":
        s["micros"] = [_microstructure(p["dims"], p) for p in s["problems"]]
        s["server"] = B.elas_server_create(2 << 30, 16, B.PREC_MIXED)
        s["w"] = [_f64(3 * m.N) for m in s["micros"]]
        s["solid"] = [_solid_nodes(p["dims"], p["phase"]) for p in s["problems"]]
    elif kind == "generate":
        s["phase"] = torch.empty(case["nx"] * case["ny"] * case["nz"], dtype=torch.int32, device="cuda")
        s["rho"] = _f64(3 * case["grains"]).reshape(-1, 3)
    else:
        dims = _grid(case)
        N = dims[0] * dims[1] * dims[2]
        mixed = case.get("mixed", False) or case.get("f32", False)
        s["ctx"] = B.create_from_micro(_microstructure(dims, s), B.PREC_MIXED if mixed else B.PREC_FP64)
        if kind == "apply":
            s["y"] = torch.empty_like(s["u"])
        elif kind == "residual":
            s["g"] = _f64(3 * N)
        elif kind == "hotspot":
            s["smooth"] = _f64(N)
        else:
            s["stress"], s["vm"] = _f64(6 * N), _f64(N)
            if kind == "solve":
                s["w"] = _f64(3 * N)
                s["solid"] = _solid_nodes(dims, s["phase"])
    return s


def run(s):
    case = s["case"]
    kind = case["kind"]
    if kind == "apply":
        (B.elas_apply_f32 if case["f32"] else B.elas_apply)(s["ctx"], s["u"], s["y"])
        return s["y"]
    if kind == "residual":
        return s["g"], B.elas_residual(s["ctx"], s["strain"], s["w"], s["g"])
    if kind == "stress":
        macro = B.elas_stress(s["ctx"], s["strain"], s["w"], s["stress"], s["vm"])
        return s["stress"], s["vm"], macro
    if kind == "hotspot":
        top, at, smooth = B.elas_hotspot(s["ctx"], s["vm"], case["s"], s["smooth"],
                                         B.HOTSPOT_SOLID if case["solid"] else B.HOTSPOT_ALL)
        return smooth, top, at
    if kind == "generate":
        phase = B.elas_assign_grains(_grid(case), s["seeds"], s["semi"], phase=s["phase"])
        rho = B.elas_orientations(B.TEXTURE_RANDOM, s["u"], rho=s["rho"])
        carved = B.elas_stamp_pores(_grid(case), s["pores"], phase)
        return phase, rho, carved
    if kind == "solve":
        if case["mixed"]:
            B.elas_pcg_solve(s["ctx"], s["strain"], TOL, MAX_ITER, w_out=s["w"], replace_every=1000, replace_drop=3)
        else:
            rule = B.STOP_PRECOND if case["micro"] == "inclusion" else B.STOP_TRUE
            B.elas_pcg_solve(s["ctx"], s["strain"], TOL, MAX_ITER, w_out=s["w"], stop_rule=rule)
        macro = B.elas_stress(s["ctx"], s["strain"], None, s["stress"], s["vm"])
        return _about_mean(s["w"], s["solid"]) if case["mixed"] else s["w"], s["stress"], s["vm"], macro
    if kind == "batch":
        B.elas_batch_solve(s["batch"], s["strains"], TOL, MAX_ITER, replace_every=1000, replace_drop=3)
        macro = [B.elas_batch_stress(s["batch"], k // 6, k % 6, UNIT_LOADS[k % 6], stress) for k, stress in enumerate(s["stress"])]
        return s["stress"], np.stack(macro)
    srv = s["server"]
    ids = [B.elas_server_submit(srv, m, p["strain"], TOL, MAX_ITER) for m, p in zip(s["micros"], s["problems"])]
    left = set(range(len(ids)))
    while left:
        B.elas_server_step(srv)
        left -= {k for k in left if B.elas_server_poll(srv, ids[k], s["w"][k]) is not None}
    return [_about_mean(w, solid) for w, solid in zip(s["w"], s["solid"])]


# --- bytes and operations a pass cannot do without -----------------------------------------------
def _iterations(n, micro):
    return (4 if micro == "inclusion" else 7) * n  # PCG iterations grow with the longest edge


def work(case):
    kind = case["kind"]
    if kind in ("batch", "serve"):
        loads = 6 if kind == "batch" else 1
        vi = sum(loads * n ** 3 * _iterations(n, "poly") for n in _edges(case))
        return dict(bytes=148 * vi, flops=480 * vi)
    nx, ny, nz = _grid(case)
    N = nx * ny * nz
    if kind == "apply":
        return dict(bytes=N * (28 if case["f32"] else 52), flops=432 * N)  # u, ids in; A u out
    if kind == "residual":
        return dict(bytes=52 * N, flops=438 * N)
    if kind == "stress":
        return dict(bytes=84 * N, flops=150 * N)  # w, ids in; 6 stresses and von Mises out
    if kind == "hotspot":
        r = max(1, math.ceil(2 * case["s"]))
        return dict(bytes=20 * N, flops=3 * (2 * r + 1) ** 3 * N)  # field, ids in; smoothed field out
    if kind == "generate":
        return dict(bytes=4 * N, flops=27 * 8 * N)  # ids out; a voxel's nearest seed is among 27 cells' seeds
    it = _iterations(max(nx, ny, nz), case["micro"])
    return dict(bytes=N * (56 + it * (148 if case["mixed"] else 244)), flops=480 * it * N)


# --- 64-bit values of the outputs ----------------------------------------------------------------
def _stiffness(mats, rho):
    """Sample-frame Voigt stiffness (engineering shear) of every phase, on the device."""
    out = []
    vi, vj = [0, 1, 2, 1, 0, 0], [0, 1, 2, 2, 2, 1]
    for p in range(len(mats)):
        kind, a, b, c = mats[p]
        if kind == synth.ISO:
            mu, lam = a / (2 * (1 + b)), a * b / ((1 + b) * (1 - 2 * b))
            c11, c12, c44 = lam + 2 * mu, lam, mu
        else:
            c11, c12, c44 = a, b, c
        d = np.eye(3)
        C = c12 * np.einsum("ij,kl->ijkl", d, d) + c44 * (np.einsum("ik,jl->ijkl", d, d) + np.einsum("il,jk->ijkl", d, d))
        for q in range(3):
            C[q, q, q, q] += c11 - c12 - 2 * c44
        if rho is not None:
            r = rho[p]
            K = np.array([[0, -r[2], r[1]], [r[2], 0, -r[0]], [-r[1], r[0], 0]])
            R = np.eye(3) + 2 / (1 + r @ r) * (K + K @ K)
            for _ in range(4):  # rotate one index at a time, the rotated index last
                C = np.tensordot(C, R, axes=([0], [1]))
        out.append([[C[vi[i], vj[i], vi[j], vj[j]] for j in range(6)] for i in range(6)])
    return torch.tensor(np.array(out), device="cuda", dtype=torch.float64)


def _b_matrices():
    """B (6 x 24, Voigt rows with engineering shear) of the unit voxel at its 8 Gauss points, and at
    its centre; corner a = ax + 2 ay + 4 az, degree of freedom 3 a + c."""
    def at(x):
        Bm = torch.zeros(6, 24, dtype=torch.float64)
        for a in range(8):
            s = [(a >> d) & 1 for d in range(3)]
            f = [x[d] if s[d] else 1 - x[d] for d in range(3)]
            gr = [(1.0 if s[d] else -1.0) * f[(d + 1) % 3] * f[(d + 2) % 3] for d in range(3)]
            for c, rows in enumerate(((0, 5, 4), (5, 1, 3), (4, 3, 2))):
                for d in range(3):
                    Bm[rows[d], 3 * a + c] += gr[d]
        return Bm
    h = 0.5 / math.sqrt(3.0)
    pts = [[0.5 + h * (1 if (q >> d) & 1 else -1) for d in range(3)] for q in range(8)]
    return torch.cat([at(p) for p in pts]).cuda(), at([0.5] * 3).cuda()


class _Cell:
    """Plain 64-bit evaluation of one periodic cell, a block of z layers at a time."""

    def __init__(self, dims, phase, mats, rho):
        self.dims, self.N = dims, dims[0] * dims[1] * dims[2]
        C = _stiffness(mats, rho)
        self.C = torch.cat([C, torch.zeros(1, 6, 6, device="cuda", dtype=torch.float64)])
        self.phase = torch.where(phase >= 0, phase, torch.full_like(phase, len(mats))).long().view(dims[2], dims[1], dims[0])
        self.B8, self.Bc = _b_matrices()
        self.layers = max(1, 1500000 // (dims[0] * dims[1]))
        # the per-phase element matrices' diagonal 3x3 blocks, for the preconditioner
        K = torch.einsum("gia,pij,gjb->pab", self.B8.view(8, 6, 24), self.C, self.B8.view(8, 6, 24)) / 8
        self.diag = torch.stack([K[:, 3 * a:3 * a + 3, 3 * a:3 * a + 3] for a in range(8)], 1)

    def corners(self, u, k0, k1):
        """(24, voxels) corner values of the voxels of layers k0 .. k1 - 1; u: (3, nz, ny, nx)."""
        nz = self.dims[2]
        idx = torch.arange(k0, k1 + 1, device="cuda") % nz
        v = u[:, idx]
        out = []
        for a in range(8):
            t = v[:, 1:] if a & 4 else v[:, :-1]
            if a & 1:
                t = torch.roll(t, -1, 3)
            if a & 2:
                t = torch.roll(t, -1, 2)
            out.append(t.reshape(3, -1))
        return torch.stack(out).reshape(24, -1)

    def product(self, u, strain=None):
        """A u + b(strain) as (3, nz, ny, nx)."""
        nx, ny, nz = self.dims
        y = torch.zeros(3, nz, ny, nx, device="cuda", dtype=torch.float64)
        e0 = None
        if strain is not None:
            e0 = torch.tensor([*strain[:3], *(2 * strain[3:])], device="cuda", dtype=torch.float64)
        for k0 in range(0, nz, self.layers):
            k1 = min(nz, k0 + self.layers)
            ph = self.phase[k0:k1].reshape(-1)
            eps = (self.B8 @ self.corners(u, k0, k1)).view(8, 6, -1)
            if e0 is not None:
                eps = eps + e0[None, :, None]
            sig = torch.bmm(self.C[ph], eps.permute(2, 1, 0)).permute(2, 1, 0).reshape(48, -1)
            f = ((self.B8.T @ sig) / 8).view(8, 3, k1 - k0, ny, nx)
            for a in range(8):
                t = f[a]
                if a & 1:
                    t = torch.roll(t, 1, 3)
                if a & 2:
                    t = torch.roll(t, 1, 2)
                lo, hi = (k0 + 1, k1 + 1) if a & 4 else (k0, k1)
                if hi <= nz:
                    y[:, lo:hi] += t
                else:
                    y[:, lo:nz] += t[:, :nz - lo]
                    y[:, :hi - nz] += t[:, nz - lo:]
        return y

    def stress(self, w, strain):
        nx, ny, nz = self.dims
        e0 = torch.tensor([*strain[:3], *(2 * strain[3:])], device="cuda", dtype=torch.float64)
        S = torch.empty(6, nz, ny, nx, device="cuda", dtype=torch.float64)
        for k0 in range(0, nz, self.layers):
            k1 = min(nz, k0 + self.layers)
            eps = self.Bc @ self.corners(w, k0, k1) + e0[:, None]
            ph = self.phase[k0:k1].reshape(-1)
            S[:, k0:k1] = torch.bmm(self.C[ph], eps.T[:, :, None])[:, :, 0].T.reshape(6, k1 - k0, ny, nx)
        S = S.reshape(6, -1)
        vm = torch.sqrt(0.5 * ((S[0] - S[1]) ** 2 + (S[1] - S[2]) ** 2 + (S[2] - S[0]) ** 2) + 3 * (S[3] ** 2 + S[4] ** 2 + S[5] ** 2))
        return S.reshape(-1), vm, S.mean(1).cpu().numpy()

    def solve(self, strain, tol=1e-13):
        """Point-block Jacobi preconditioned conjugate gradients from zero."""
        nx, ny, nz = self.dims
        D = torch.zeros(nz, ny, nx, 3, 3, device="cuda", dtype=torch.float64)
        solid = torch.zeros(nz, ny, nx, device="cuda", dtype=torch.float64)
        for a in range(8):
            sh = ((a >> 2) & 1, (a >> 1) & 1, a & 1)
            D += torch.roll(self.diag[self.phase, a], sh, (0, 1, 2))
            solid += torch.roll((self.phase < self.C.shape[0] - 1).double(), sh, (0, 1, 2))
        D[solid == 0] = torch.eye(3, device="cuda", dtype=torch.float64)
        M = torch.linalg.inv(D).permute(3, 4, 0, 1, 2).contiguous()
        prec = lambda g: (M * g[None]).sum(1)  # noqa: E731
        w = torch.zeros(3, nz, ny, nx, device="cuda", dtype=torch.float64)
        g = self.product(w, strain)
        b2 = float((g * g).sum())
        h = prec(g)
        gg = (g * h).sum()
        for it in range(20 * max(self.dims)):
            Ah = self.product(h)
            lam = gg / (h * Ah).sum()
            w -= lam * h
            g -= lam * Ah
            z = prec(g)
            new = (g * z).sum()
            h = z + (new / gg) * h
            gg = new
            if it % 16 == 15 and float((g * g).sum()) <= tol * tol * b2:
                break
        return w


def _solve_cost(dims):
    return dims[0] * dims[1] * dims[2] * max(dims)


def exact(case, seed):
    kind = case["kind"]
    s = _inputs(case, seed)
    if kind == "generate":  # ids and counts are whole numbers; the orientations are Shoemake's
        u = s["u"]
        a, b, t, p = torch.sqrt(1 - u[:, 0]), torch.sqrt(u[:, 0]), 2 * math.pi * u[:, 1], 2 * math.pi * u[:, 2]
        return None, torch.stack([a * torch.cos(t), b * torch.sin(p), b * torch.cos(p)], 1) / (a * torch.sin(t))[:, None], None
    if kind in ("batch", "serve"):
        # the small cells only, and one load case of each: the rest would take minutes
        out = []
        for p in s["problems"]:
            cell = _Cell(p["dims"], p["phase"], p["mats"], p["rho"])
            small = max(p["dims"]) <= 64
            if kind == "serve":
                out.append(_about_mean(cell.solve(p["strain"]).view(3, -1), _solid_nodes(p["dims"], p["phase"])) if small else None)
            else:
                out += [cell.stress(cell.solve(UNIT_LOADS[0]), UNIT_LOADS[0])[0] if small else None] + [None] * 5
        return out if kind == "serve" else (out, None)
    dims = _grid(case)
    nx, ny, nz = dims
    if kind == "hotspot":
        r = max(1, math.ceil(2 * case["s"]))
        k = torch.exp(-torch.arange(-r, r + 1, device="cuda", dtype=torch.float64) ** 2 / (2 * case["s"] ** 2))
        k = k / k.sum()
        m = (s["phase"] >= 0).double().view(nz, ny, nx)
        num, den = m * s["vm"].view(nz, ny, nx), m
        for d in range(3):
            num = sum(k[o + r] * torch.roll(num, -o, d) for o in range(-r, r + 1))
            den = sum(k[o + r] * torch.roll(den, -o, d) for o in range(-r, r + 1))
        smooth = torch.where(den > 0, num / den.clamp(min=1e-300), torch.zeros_like(num))
        field = torch.where(m > 0, smooth, torch.full_like(smooth, -1.0)) if case["solid"] else smooth
        best = field
        for d in range(3):
            best = torch.maximum(best, torch.maximum(torch.roll(best, 1, d), torch.roll(best, -1, d)))
        hot = (m > 0) & (field >= best)
        return smooth.reshape(-1), float(smooth[hot].max()) if bool(hot.any()) else 0.0, None
    cell = _Cell(dims, s["phase"], s["mats"], s["rho"])
    if kind == "apply":
        return cell.product(s["u"].double().view(3, nz, ny, nx)).reshape(-1)
    if kind == "residual":
        g = cell.product(s["w"].view(3, nz, ny, nx), s["strain"]).reshape(-1)
        return g, float(torch.linalg.norm(g))
    if kind == "stress":
        return cell.stress(s["w"].view(3, nz, ny, nx), s["strain"])
    if _solve_cost(dims) > 3e8:
        return None
    w = cell.solve(s["strain"])
    rest = cell.stress(w, s["strain"])
    return (_about_mean(w.view(3, -1), _solid_nodes(dims, s["phase"])) if case["mixed"] else w.reshape(-1), *rest)
