"""The solver's work over its range of use, as cases that can be measured.

A case is one pass through the public entry points with a fixed budget of residual evaluations
(``tol`` = 0), so that every pass does the same work:

* ``solve``     Solver.solve on a bound microstructure (strain control, fields written);
* ``stress``    Solver.solve_stress with a per-phase eigenstrain;
* ``served``    Solver.set_material of a new microstructure on a resident context, then solves;
* ``batch``     Batch.solve of several RVEs under the six unit strains each;
* ``residual``  hs_residual_noalloc, the FP64 equilibrium residual alone.

The listed sizes are those of the repository's tests, benchmark and serving stream: 32^3 (the
iterate-by-iterate configuration) to 512^3 (the polycrystal), cubic and ragged, with lengths that
are powers of two, multiples of 3 and multiples of 5, 7 and 11.  Solvers run on a stream of their
own, as the benchmark and the server run them.

Values computed in FP32 (the FP32 precision, and the refined precision's fields and stresses after
a fixed number of FP32 iterations) are returned as FP32; those of the FP64 precision as FP64.  The
error history belongs to the FP64 outputs only: near the FP32 floor it is a sum of squared roundings.
"""
from __future__ import annotations

import ctypes
import math

import numpy as np
import torch

from paper_2405_11168_gb300 import hs

PRECISION = {"fp64": hs.HS_FP64, "fp32": hs.HS_FP32, "refined": hs.HS_FP32_REFINED}
INNER_RATIO = 1e-3  # the library's default


def listed():
    def case(name, kind, precision, grid, micro, **kw):
        c = {"name": name, "kind": kind, "precision": precision, "n1": grid[0], "n2": grid[1], "n3": grid[2],
             "micro": micro, "radius": 0.0, "fraction": 0.0, "contrast": 1.0, "grains": 0, "evals": 64, "inner_max": 200}
        c.update(kw)
        return c

    return [
        # the iterate-by-iterate configuration: one centred sphere, FP64; launches and latency count
        case("sphere_32_fp64", "solve", "fp64", (32, 32, 32), "sphere", fraction=0.2, contrast=10.0),
        # the cell of the paper's contrast study (a length with a factor 11)
        case("sphere_44_fp32", "solve", "fp32", (44, 44, 44), "sphere", radius=17.6, contrast=10.0),
        # a small served RVE: FP32 iterations with FP64 sweeps and correction solves between them
        case("spheres_64_refined", "solve", "refined", (64, 64, 64), "spheres", radius=8.0, fraction=0.2, contrast=1e-3,
             evals=123, inner_max=40),
        # a request of the serving stream: a 50-grain polycrystal bound to a resident context, three loads
        case("grains_96_served", "served", "refined", (96, 96, 96), "voronoi", grains=50, evals=24),
        # applied stress with an eigenstrain on a ragged cell (factors 5, 7 and 11)
        case("stress_160x112x88_fp32", "stress", "fp32", (160, 112, 88), "spheres", radius=9.0, fraction=0.25, contrast=10.0,
             evals=32),
        # the residual alone, as a caller with a fixed memory budget asks for it
        case("residual_128", "residual", "fp64", (128, 128, 128), "spheres", radius=8.0, fraction=0.3, contrast=1e-3, evals=1),
        # five sizes of the batched configuration, six unit strains each, in shared launches
        case("batch_32_to_128", "batch", "refined", (128, 128, 128), "mixed", grains=50, evals=32),
        # voids in FP32, the middle of the serving range
        case("voids_128_fp32", "solve", "fp32", (128, 128, 128), "spheres", radius=16.0, fraction=0.2, contrast=0.0),
        # plain FP64, the precision of parity checks and tight tolerances
        case("spheres_128_fp64", "solve", "fp64", (128, 128, 128), "spheres", radius=8.0, fraction=0.3, contrast=10.0,
             evals=24),
        # a served size that is a multiple of 3
        case("spheres_192_refined", "solve", "refined", (192, 192, 192), "spheres", radius=12.0, fraction=0.2,
             contrast=1e-2, evals=48),
        # the benchmark's workload
        case("spheres_256_refined", "solve", "refined", (256, 256, 256), "spheres", radius=8.0, fraction=0.3, contrast=1e-3),
        # the large polycrystal: 500 grains, the full anisotropic law
        case("grains_512_refined", "solve", "refined", (512, 512, 512), "voronoi", grains=500, evals=16),
    ]


# even lengths with prime factors 2, 3, 5, 7 and 11
def _lengths(lo, hi):
    out = []
    for n in range(lo + (lo & 1), hi + 1, 2):
        m = n
        for p in (2, 3, 5, 7, 11):
            while m % p == 0:
                m //= p
        if m == 1:
            out.append(n)
    return out


def draw(rng):
    kind = rng.choice(["solve", "solve", "solve", "solve", "stress", "served", "batch", "residual"])
    precision = {"residual": "fp64", "served": "refined", "batch": "refined"}.get(kind) or rng.choice(
        ["fp32", "refined", "refined", "fp64"])
    if kind == "stress" and precision == "refined":
        precision = "fp32"
    top = {"batch": 128, "served": 192, "residual": 256}.get(kind, 256 if precision != "fp64" else 160)
    side = math.exp(rng.uniform(math.log(24), math.log(top)))
    n = [rng.choice([m for m in _lengths(16, 320) if abs(math.log(m / side)) < 0.4 and m <= 1.2 * top] or [32])
         for _ in range(3)]
    if rng.random() < 0.4:
        n = [n[0]] * 3
    micro = "mixed" if kind == "batch" else rng.choice(["spheres", "spheres", "voronoi"])
    if kind == "served":
        micro = "voronoi"
    if kind == "stress":
        micro = "spheres"
    evals = 1 if kind == "residual" else rng.choice([16, 24, 32, 40, 48])
    return {"kind": kind, "precision": precision, "n1": n[0], "n2": n[1], "n3": n[2], "micro": micro,
            "radius": round(max(2.5, min(n) / rng.choice([8.0, 10.0, 12.0])), 2), "fraction": rng.choice([0.15, 0.2, 0.25]),
            "contrast": rng.choice([0.0, 1e-3, 1e-2, 1e-1, 3.0, 10.0]) if kind != "stress" else rng.choice([0.3, 3.0, 10.0]),
            "grains": rng.choice([20, 50, 100]), "evals": evals, "inner_max": rng.choice([12, 200])}


# ---- inputs -----------------------------------------------------------------------------------
def _grid(case):
    return int(case["n1"]), int(case["n2"]), int(case["n3"])


def _isotropic(E, nu):
    lam, mu = E * nu / ((1 + nu) * (1 - 2 * nu)), E / (2 * (1 + nu))
    C = np.zeros((6, 6))
    C[:3, :3] = lam
    C[range(3), range(3)] = lam + 2 * mu
    C[range(3, 6), range(3, 6)] = mu
    return C


def _centres(grid, radius, fraction, rng):
    """Random sequential addition of non-overlapping periodic spheres."""
    n = np.array(grid, dtype=np.float64)
    want = max(1, int(fraction * n.prod() / (4.0 / 3.0 * math.pi * radius ** 3)))
    kept = np.zeros((0, 3))

    def clash(a, b):
        d = a[:, None, :] - b[None, :, :]
        d -= n * np.round(d / n)
        return (d * d).sum(-1) < (2 * radius) ** 2

    for _ in range(400):
        c = rng.random((512, 3)) * n
        if len(kept):
            c = c[~clash(c, kept).any(1)]
        if not len(c):
            continue
        near, ok = clash(c, c), []
        for i in range(len(c)):
            if not near[i, ok].any():
                ok.append(i)
        kept = np.vstack([kept, c[ok]])
        if len(kept) >= want:
            return kept[:want]
    return kept


def _stamp(grid, centres, radius):
    """Voxels (centres at l + 1/2) inside a sphere, minimum image: uint8 [N3][N2][N1] on the GPU."""
    n = torch.tensor(grid, device="cuda", dtype=torch.int64)
    c = torch.from_numpy(np.ascontiguousarray(centres)).cuda()
    span = min(int(math.ceil(radius)) + 1, min(grid) // 2)
    o = torch.arange(-span, span + 1, device="cuda")
    ids = torch.zeros(grid[0] * grid[1] * grid[2], dtype=torch.uint8, device="cuda")
    for part in c.split(max(1, (1 << 24) // len(o) ** 3)):
        at = part.floor().long()[:, :, None] + o  # [k][axis][offset]
        d2 = (at + 0.5 - part[:, :, None]) ** 2
        at = at % n[:, None]
        inside = d2[:, 2, :, None, None] + d2[:, 1, None, :, None] + d2[:, 0, None, None, :] <= radius * radius
        flat = (at[:, 2, :, None, None] * n[1] + at[:, 1, None, :, None]) * n[0] + at[:, 0, None, None, :]
        ids[flat[inside]] = 1
    return ids.view(grid[2], grid[1], grid[0])


def _voronoi(grid, grains, rng):
    """Periodic Voronoi cells of uniform centres: int16 [N3][N2][N1] on the GPU."""
    n = np.array(grid, dtype=np.float64)
    c = rng.random((grains, 3)) * n
    best = torch.full((grid[2], grid[1], grid[0]), 1e30, device="cuda")
    ids = torch.zeros(best.shape, dtype=torch.int16, device="cuda")
    d = []
    for a in range(3):
        x = np.arange(grid[a]) + 0.5 - c[:, a:a + 1]
        d.append(torch.from_numpy((x - n[a] * np.round(x / n[a])) ** 2).float().cuda())
    for g in range(grains):
        r2 = d[2][g][:, None, None] + (d[1][g][:, None] + d[0][g][None, :])[None]
        near = r2 < best
        best = torch.where(near, r2, best)
        ids[near] = g
    return ids


def _cubic_grains(grains, rng):
    """Cubic crystals (C11, C12, C44 = 168.4, 121.4, 75.4 GPa) in uniformly random orientations."""
    V = np.array([[0, 5, 4], [5, 1, 3], [4, 3, 2]])
    C6 = np.zeros((6, 6))
    C6[:3, :3] = 121.4
    C6[range(3), range(3)] = 168.4
    C6[range(3, 6), range(3, 6)] = 75.4
    C4 = C6[V[:, :, None, None], V[None, None]]
    q = rng.standard_normal((grains, 4))
    w, x, y, z = (q / np.linalg.norm(q, axis=1, keepdims=True)).T
    R = np.array([[1 - 2 * (y * y + z * z), 2 * (x * y - z * w), 2 * (x * z + y * w)],
                  [2 * (x * y + z * w), 1 - 2 * (x * x + z * z), 2 * (y * z - x * w)],
                  [2 * (x * z - y * w), 2 * (y * z + x * w), 1 - 2 * (x * x + y * y)]]).transpose(2, 0, 1)
    T = np.einsum("gip,gjq,gkr,gls,pqrs->gijkl", R, R, R, R, C4, optimize=True)
    P = [(0, 0), (1, 1), (2, 2), (1, 2), (0, 2), (0, 1)]
    out = np.array([[T[:, i, j, k, l] for (k, l) in P] for (i, j) in P]).transpose(2, 0, 1)
    return 0.5 * (out + out.transpose(0, 2, 1))


def _micro(kind, grid, case, rng):
    if kind == "voronoi":
        return _voronoi(grid, case["grains"], rng), _cubic_grains(case["grains"], rng)
    table = np.stack([_isotropic(1.0, 0.3), _isotropic(case["contrast"], 0.3)])
    if kind == "sphere":
        R = case["radius"] or (3 * case["fraction"] * grid[0] * grid[1] * grid[2] / (4 * math.pi)) ** (1 / 3)
        return _stamp(grid, np.array([grid]) / 2 + rng.uniform(-1, 1, (1, 3)), R), table
    return _stamp(grid, _centres(grid, case["radius"], case["fraction"], rng), case["radius"]), table


def _rves(case, rng):
    """The batched configuration's mix: sizes up to the case's, random spheres and polycrystals."""
    sizes = [tuple(m for m in _lengths(4, n) if m <= n * f)[-1] for n in _grid(case) for f in (0.25, 0.375, 0.5, 0.75, 1.0)]
    grids = [tuple(sizes[5 * a + k] for a in range(3)) for k in range(5)]
    out = []
    for k, g in enumerate(grids):
        c = dict(case, radius=max(2.0, min(g) / 8), fraction=0.2, contrast=(10.0, 0.0, 0.1, 3.0, 1e-2)[k], grains=50)
        out.append((g,) + _micro("voronoi" if k in (1, 3) else "spheres", g, c, rng))
    return out


def _inputs(case, seed):
    """Everything a pass takes, from the seed alone (device ids, host tables and loads)."""
    rng = np.random.Generator(np.random.PCG64(seed))
    x = {"grid": _grid(case)}
    if case["kind"] == "batch":
        x["rves"] = _rves(case, rng)
        x["loads"] = 1e-3 * np.eye(6) * rng.uniform(0.5, 1.0, 6)
        return x
    x["ids"], x["table"] = _micro(case["micro"], x["grid"], case, rng)
    E = rng.standard_normal((3, 6))
    x["loads"] = 1e-3 * E / np.linalg.norm(E, axis=1, keepdims=True)
    if case["kind"] == "stress":
        x["eigen"] = 1e-4 * rng.standard_normal((len(x["table"]), 6))
    if case["kind"] == "residual":
        g = torch.Generator(device="cuda").manual_seed(seed)
        x["u"] = 1e-3 * torch.randn((3,) + tuple(x["ids"].shape), generator=g, device="cuda", dtype=torch.float64)
    return x


# ---- passes -----------------------------------------------------------------------------------
def prepare(case, seed):
    x = _inputs(case, seed)
    s = {"case": case, "x": x}
    stream = torch.cuda.Stream()
    stream.wait_stream(torch.cuda.current_stream())
    s["stream"] = stream
    if case["kind"] == "residual":
        s["ids16"] = x["ids"].to(torch.int16).contiguous()
        s["table"] = np.ascontiguousarray(x["table"], dtype=np.float64)
        s["force"] = torch.empty_like(x["u"], dtype=torch.float32)
        torch.cuda.current_stream().synchronize()
        return s
    opt = {"precision": PRECISION[case["precision"]], "stream": stream, "inner_max": case["inner_max"],
           "out_f32": 0 if case["precision"] == "fp64" else 1}
    if case["kind"] == "batch":
        rves = [(ids.cpu().numpy().astype(np.uint16), table) for _, ids, table in x["rves"]]
        opt.pop("out_f32")
        s["batch"] = hs.Batch(rves, [r for r in range(len(rves)) for _ in range(6)], **opt)
        s["E"] = np.concatenate([x["loads"]] * len(rves))
        return s
    if case["kind"] == "served":
        # the resident context holds an earlier request's material; the new one comes from the host
        s["host_ids"] = x["ids"].cpu().numpy().astype(np.uint16)
        old = np.zeros_like(s["host_ids"])
        s["solver"] = hs.Solver(old, x["table"][:1], layout_nphase=64 if case["grains"] <= 64 else 128, **opt)
        return s
    s["solver"] = hs.Solver(x["ids"], x["table"], **opt)
    if case["kind"] == "stress":
        s["solver"].set_eigenstrain(x["eigen"])
        s["S"] = x["loads"][0] * 1e3
    return s


def _typed(case, a):
    return np.asarray(a, dtype=np.float64 if case["precision"] == "fp64" else np.float32)


def run(s):
    case, x = s["case"], s["x"]
    n = int(case["evals"])
    if case["kind"] == "residual":
        sig, l2 = np.zeros(6), ctypes.c_double()
        dp = ctypes.POINTER(ctypes.c_double)
        E = np.ascontiguousarray(x["loads"][0])
        st = hs.load().hs_residual_noalloc(
            (ctypes.c_int * 3)(*x["grid"]), ctypes.c_void_p(s["ids16"].data_ptr()), s["table"].ctypes.data_as(dp),
            len(s["table"]), E.ctypes.data_as(dp), ctypes.c_void_p(x["u"].data_ptr()),
            ctypes.c_void_p(s["force"].data_ptr()), sig.ctypes.data_as(dp), ctypes.byref(l2),
            ctypes.c_void_p(s["stream"].cuda_stream))
        return {"status": int(st), "force": s["force"], "sig": sig, "l2": l2.value}
    if case["kind"] == "batch":
        r = s["batch"].solve(s["E"], tol=0.0, max_iter=n)
        return {"iters": r["iters"], "status": r["item_status"], "sig_eff": _typed(case, r["sig_eff"])}
    sv = s["solver"]

    def answer(r):
        out = {"iters": r["iters"], "status": r["status"], "eps": r["eps"], "sig": r["sig"],
               "sig_eff": _typed(case, r["sig_eff"])}
        if "E" in r:
            out["E"] = _typed(case, r["E"])
        if case["precision"] == "fp64":
            out["history"] = sv.err_history(n)
        return out

    if case["kind"] == "stress":
        return answer(sv.solve_stress(s["S"], tol=0.0, max_iter=n))
    if case["kind"] == "served":
        sv.set_material(s["host_ids"], x["table"])
        return [answer(sv.solve(E, tol=0.0, max_iter=n)) for E in x["loads"]]
    return answer(sv.solve(x["loads"][0], tol=0.0, max_iter=n))


def work(case):
    """Per evaluation the displacement spectrum is read and written once and the phase ids are read
    once; the fields are written once at the end.  Operations: two real transforms of 3 components, the
    two tetrahedra's strains, stresses and adjoints (about 300) and the Green update (about 110 per
    complex point)."""
    real = 8 if case["precision"] == "fp64" else 4
    grids = [_grid(case)]
    if case["kind"] == "batch":
        grids = [tuple(_lengths(4, n)[-1] if f == 1 else [m for m in _lengths(4, n) if m <= n * f][-1] for n in _grid(case))
                 for f in (0.25, 0.375, 0.5, 0.75, 1.0)]
    b = f = 0.0
    for g in grids:
        N = float(g[0]) * g[1] * g[2]
        if case["kind"] == "residual":
            return {"bytes": N * (24 + 2 + 12), "flops": 300.0 * N}
        solves = {"batch": 6, "served": 3}.get(case["kind"], 1)
        out = 0 if case["kind"] == "batch" else 12 * real
        b += solves * N * (case["evals"] * (6 * real + 2) + out)
        f += solves * N * case["evals"] * (2 * 3 * 2.5 * math.log2(N) + 300 + 55)
    return {"bytes": b, "flops": f}


# ---- the same passes in 64 bits ---------------------------------------------------------------
_T1 = ((0, 0, 0), (0, 1, 1), (1, 1, 0), (1, 0, 1))  # offsets (x, y, z) of the corner below: coordinate - 1


class _Scheme:
    """The basic scheme on one microstructure in FP64 with torch operations."""

    def __init__(self, grid, ids, table, eigen=None):
        self.grid, self.N = grid, grid[0] * grid[1] * grid[2]
        self.ids = ids.to("cuda", torch.int64)
        self.iso = all(np.allclose(C, _iso_of(C), rtol=0, atol=1e-12 * max(np.abs(C).max(), 1e-300)) for C in table)
        self.C = torch.from_numpy(np.ascontiguousarray(table)).cuda()
        self.s0 = None
        if eigen is not None:
            eng = eigen * np.array([1, 1, 1, 2, 2, 2.0])
            self.s0 = torch.from_numpy(np.einsum("pij,pj->pi", table, eng)).cuda()
        self.lam0, self.mu0 = _reference(table)
        C0 = np.zeros((6, 6))
        C0[:3, :3] = self.lam0
        C0[range(3), range(3)] += 2 * self.mu0
        C0[range(3, 6), range(3, 6)] = self.mu0
        self.S0 = np.array([1, 1, 1, .5, .5, .5])[:, None] * np.linalg.inv(C0)
        n1, n2, n3 = grid
        ph = [torch.exp(-2j * math.pi * torch.arange(m, device="cuda", dtype=torch.float64) / n)
              for m, n in ((n1 // 2 + 1, n1), (n2, n2), (n3, n3))]
        x, y, z = ph[0][None, None, :], ph[1][None, :, None], ph[2][:, None, None]
        yz, xy, xz = y * z, x * y, x * z
        D = [0.5 * (1 + yz - xy - xz), 0.5 * (1 - yz - xy + xz), 0.5 * (1 - yz + xy - xz)]
        tr = sum(2 * (d.real ** 2 + d.imag ** 2) for d in D)
        a, m = self.lam0 + self.mu0, self.mu0
        A = {}
        for i in range(3):
            for j in range(i, 3):
                A[i, j] = a * 2 * (D[i] * D[j].conj()).real + (m * tr if i == j else 0)
        c11, c22, c33 = A[1, 1] * A[2, 2] - A[1, 2] ** 2, A[0, 0] * A[2, 2] - A[0, 2] ** 2, A[0, 0] * A[1, 1] - A[0, 1] ** 2
        c12, c13, c23 = (A[0, 2] * A[1, 2] - A[0, 1] * A[2, 2], A[0, 1] * A[1, 2] - A[0, 2] * A[1, 1],
                         A[0, 1] * A[0, 2] - A[0, 0] * A[1, 2])
        det = A[0, 0] * c11 + A[0, 1] * c12 + A[0, 2] * c13
        trans = [(0, 0, 0), (n3 // 2, n2 // 2, n1 // 2)]
        for t in trans:
            det[t] = 1
        self.Om = [[c / det for c in row] for row in ((c11, c12, c13), (c12, c22, c23), (c13, c23, c33))]
        for row in self.Om:
            for o in row:
                for t in trans:
                    o[t] = 0
        self.u = torch.zeros((3, n3, n2, n1), device="cuda", dtype=torch.float64)

    def _stress(self, e):
        if self.iso:
            lam, mu = self.C[:, 0, 1][self.ids], self.C[:, 3, 3][self.ids]
            t = lam * (e[0] + e[1] + e[2])
            s = [t + 2 * mu * e[i] for i in range(3)] + [mu * e[i] for i in range(3, 6)]
        else:
            s = [0, 0, 0, 0, 0, 0]
            for i in range(6):
                for j in range(i, 6):
                    c = self.C[:, i, j][self.ids]
                    s[i] = s[i] + c * e[j]
                    if j != i:
                        s[j] = s[j] + c * e[i]
        if self.s0 is not None:
            s = [s[i] - self.s0[:, i][self.ids] for i in range(6)]
        return s

    def evaluate(self, E, fields=False):
        """Force, mean stress, L2 norm and (asked for) the fields at the current displacement."""
        F = torch.zeros_like(self.u)
        mean = np.zeros(6)
        eps = sig = None
        for flip in (0, 1):
            corner = [tuple(o ^ flip for o in c) for c in _T1]
            g = [[None] * 3 for _ in range(3)]
            for j in range(3):
                a, b, c, d = (torch.roll(self.u[j], (o[2], o[1], o[0]), (0, 1, 2)) for o in corner)
                sgn = -0.5 if flip else 0.5
                g[0][j], g[1][j], g[2][j] = sgn * ((a + b) - (c + d)), sgn * ((a - b) - (c - d)), sgn * ((a - b) + (c - d))
            e = [E[0] + g[0][0], E[1] + g[1][1], E[2] + g[2][2], 2 * E[3] + g[1][2] + g[2][1],
                 2 * E[4] + g[0][2] + g[2][0], 2 * E[5] + g[0][1] + g[1][0]]
            del g
            s = self._stress(e)
            mean += np.array([float(v.sum()) for v in s])
            if fields:
                h = [0.5 * e[i] * (1 if i < 3 else 0.5) for i in range(6)]
                if eps is None:
                    eps, sig = torch.stack(h), torch.stack([0.5 * v for v in s])
                else:
                    for i in range(6):
                        eps[i] += h[i]
                        sig[i] += 0.5 * s[i]
                del h
            del e
            for k, (i1, i2, i3) in enumerate(((0, 5, 4), (5, 1, 3), (4, 3, 2))):
                sgn = -0.25 if flip else 0.25
                for o, w in zip(corner, ((1, 1, 1), (1, -1, -1), (-1, -1, 1), (-1, 1, -1))):
                    f = sgn * (w[0] * s[i1] + w[1] * s[i2] + w[2] * s[i3])
                    F[k] += torch.roll(f, (-o[2], -o[1], -o[0]), (0, 1, 2))
        mean *= 0.5 / self.N
        l2 = math.sqrt(float((F * F).sum()) / self.N)
        return F, mean, l2, eps, sig

    def update(self, F):
        n1, n2, n3 = self.grid
        f = torch.fft.rfftn(F, dim=(1, 2, 3), norm="forward")
        for j in range(3):
            d = sum(self.Om[j][k] * f[k] for k in range(3))
            self.u[j] -= 2 * torch.fft.irfftn(d, s=(n3, n2, n1), norm="forward")


def _iso_of(C):
    out = np.zeros((6, 6))
    out[:3, :3] = C[0, 1]
    out[range(3), range(3)] = C[0, 1] + 2 * C[3, 3]
    out[range(3, 6), range(3, 6)] = C[3, 3]
    return out


def _reference(table):
    """(lambda0, mu0) of the default reference medium."""
    iso = all(np.allclose(C, _iso_of(C), rtol=0, atol=1e-12 * max(np.abs(C).max(), 1e-300)) for C in table)
    if len(table) == 2 and iso:
        km, ki = (C[0, 1] + 2 * C[3, 3] / 3 for C in table)
        a = 0.55 if ki < km else 0.45
        nu = table[0][0, 1] / (2 * (table[0][0, 1] + table[0][3, 3]))
        k0 = a * km + (1 - a) * ki
        mu0 = 3 * k0 * (1 - 2 * nu) / (2 * (1 + nu))
        return k0 - 2 * mu0 / 3, mu0
    w = np.sqrt(np.array([1, 1, 1, 2, 2, 2.0]))
    B = np.zeros((5, 6))
    B[0, :2] = 1 / math.sqrt(2), -1 / math.sqrt(2)
    B[1, :3] = np.array([1, 1, -2]) / math.sqrt(6)
    B[range(2, 5), range(3, 6)] = 1
    K = [C[:3, :3].sum() / 9 for C in table]
    ev = np.concatenate([np.linalg.eigvalsh(B @ (C * w[:, None] * w) @ B.T) for C in table])
    k0, mu0 = 0.5 * (min(K) + max(K)), 0.25 * (ev.min() + ev.max())
    return k0 - 2 * mu0 / 3, mu0


def _norm(s):
    return math.sqrt(float((np.array([1, 1, 1, 2, 2, 2.0]) * s * s).sum()))


def _plain(sch, E, n, S=None):
    """n evaluations of the basic scheme; S: applied stress."""
    E = np.array(E, dtype=np.float64)
    if S is not None:
        E = sch.S0 @ S
    hist = []
    for k in range(n):
        F, mean, l2, eps, sig = sch.evaluate(E, fields=k == n - 1)
        hist.append(l2 / _norm(mean))
        if k < n - 1:
            sch.update(F)
            if S is not None:
                E = E + sch.S0 @ (S - mean)
        del F
    return hist, mean, eps, sig, E


def _refined(sch, E, n, inner_max, fields=True):
    """The refined solve in exact arithmetic: each restart repeats the evaluation at the state reached,
    and a run stops on its budget or when its error has fallen by the inner ratio."""
    total, stop, den = 0, None, None  # den: the last FP64 sweep's mean stress; None in the plain first run
    F, mean, l2, eps, sig = sch.evaluate(E)
    while True:
        budget = min(inner_max, n - 1) if den is None else min(inner_max, n - total)
        for k in range(budget):
            if k:
                sch.update(F)
                F, mean, l2, _, _ = sch.evaluate(E)
            err = l2 / (den or _norm(mean))
            if den is None and k == 0:
                stop = INNER_RATIO * err
            total += 1
            if err < stop:
                break
        total += 1
        last = total >= n
        F, mean, l2, eps, sig = sch.evaluate(E, fields=fields and last)
        if last:
            return mean, eps, sig
        den = _norm(mean)
        stop = INNER_RATIO * l2 / den


def exact(case, seed):
    x = _inputs(case, seed)
    n = int(case["evals"])
    if case["kind"] == "residual":
        sch = _Scheme(x["grid"], x["ids"], x["table"])
        sch.u = x["u"]
        F, mean, l2, _, _ = sch.evaluate(x["loads"][0])
        return {"status": None, "force": F, "sig": mean, "l2": l2}
    if case["kind"] == "batch":
        sig = []
        for g, ids, table in x["rves"]:
            for E in x["loads"]:
                sig.append(_refined(_Scheme(g, ids, table), E, n, case["inner_max"], fields=False)[0])
        return {"iters": None, "status": None, "sig_eff": np.array(sig)}

    def one(E):
        sch = _Scheme(x["grid"], x["ids"], x["table"], x.get("eigen"))
        if case["kind"] == "stress":
            h, mean, eps, sig, Ef = _plain(sch, np.zeros(6), n, S=E * 1e3)
        elif case["precision"] == "refined":
            mean, eps, sig = _refined(sch, E, n, case["inner_max"])
        else:
            h, mean, eps, sig, _ = _plain(sch, E, n)
        out = {"iters": None, "status": None, "eps": eps, "sig": sig, "sig_eff": mean}
        if case["precision"] == "fp64":
            out["history"] = np.array(h)
        if case["kind"] == "stress":
            out["E"] = Ef
        return out

    if case["kind"] == "served":
        return [one(E) for E in x["loads"]]
    return one(x["loads"][0])
