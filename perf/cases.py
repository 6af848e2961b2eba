"""Performance cases: the work that programs built on this library have it do.

Each case is a dict of plain values; `prepare` makes what a program holds before
the call (inputs on the GPU, the plan, batch or network), `run` is one pass
through the public entry points, `work` the bytes and operations that no
implementation can do without, `exact` the same result by plain torch in 64
bits.  The kinds:

  map       one far-field map: solve for an incident direction, then the far
            field over a set of outgoing angles (2D and 3D)
  vcycle    one V(1,1) cycle on a given iterate and right-hand side, FP32 or FP64
            (programs with their own outer iteration, and the inner loop of
            every solve)
  farfield  the far field of a given 2D solution
  gmres     a solve with GMRES(3) smoothing at the rotation of the paper's
            tables (9.9 degrees)
  batch     many uneven 2D problems in one batched solve
  net_fwd   the learned smoother's network applied to a residual field
  net_grad  loss and weight gradients of the network on a batch of patches

Potentials keep k^2 w (wavenumber, Gaussian width) moderate, as in the paper's
model problems: the far field's terms stay within a few thousand times its
value, so a map has digits to compare.  Whole solves ask for 1e-10, the
tolerance of the small configuration, so that a solution is fixed beyond the
rounding of its FP32 cycles.
"""
import math

import numpy as np
import torch

import paper_1211_4461_gb300 as csff
from paper_1211_4461_gb300.learned import init_weights

PI = math.pi
DEV = "cuda"


# ---------------------------------------------------------------------------
# the cases
# ---------------------------------------------------------------------------
def listed():
    return [
        # the smallest call: the plain FP64 configuration (Jacobi V(2,2), 360
        # angles), where launches and latency count
        {"name": "map2d_n65_fp64", "kind": "map", "dim": 2, "n": 65, "coarsest": 5, "R": 10.0, "k": 2.0,
         "k2w": 8.0, "gauss": 1, "smoother": "jacobi", "precision": "fp64", "ang": 360},
        # an ordinary map of a parameter scan: FP32 cycles, FP64 refinement
        {"name": "map2d_n257", "kind": "map", "dim": 2, "n": 257, "coarsest": 9, "R": 20.0, "k": 3.0,
         "k2w": 9.0, "gauss": 1, "smoother": "rbgs", "precision": "mixed", "ang": 360},
        # the main 2D workload's grid, levels and 720 angles
        {"name": "map2d_n1025", "kind": "map", "dim": 2, "n": 1025, "coarsest": 9, "R": 20.0, "k": 3.0,
         "k2w": 9.0, "gauss": 1, "smoother": "rbgs", "precision": "mixed", "ang": 720},
        # the 3D workload: one incident direction on 257^3, 64 x 32 angles
        {"name": "map3d_n257", "kind": "map", "dim": 3, "n": 257, "coarsest": 5, "R": 15.0, "k": 4.0,
         "k2w": 8.0, "gauss": 1, "smoother": "rbgs", "precision": "mixed", "ang": 32},
        # one plain FP64 cycle on the main 2D grid
        {"name": "vcycle2d_f64_n1025", "kind": "vcycle", "dim": 2, "n": 1025, "coarsest": 9, "R": 20.0, "k": 5.0,
         "k2w": 100.0, "gauss": 1, "dtype": "f64"},
        # the largest 2D grid: FP32 arrays beyond the L2 cache
        {"name": "vcycle2d_f32_n4097", "kind": "vcycle", "dim": 2, "n": 4097, "coarsest": 9, "R": 20.0, "k": 20.0,
         "k2w": 1600.0, "gauss": 1, "dtype": "f32"},
        # one FP32 cycle of the 3D workload
        {"name": "vcycle3d_f32_n257", "kind": "vcycle", "dim": 3, "n": 257, "coarsest": 5, "R": 15.0, "k": 4.0,
         "k2w": 48.0, "gauss": 1, "dtype": "f32"},
        # the far field alone, for a solution that the program already has, with
        # the main workload's potential width
        {"name": "farfield2d_n1025", "kind": "farfield", "n": 1025, "coarsest": 9, "R": 20.0, "k": 2.0,
         "k2w": 16.0, "gauss": 1, "ang": 720},
        # the paper's own solver setting: 3D, two Gaussians, V(1,1)/GMRES(3),
        # FP64, residual reduction 1e-6
        {"name": "gmres3d_n129", "kind": "gmres", "dim": 3, "n": 129, "k": 1.0, "precision": "fp64"},
        # a scan over uneven problems in one persistent launch
        {"name": "batch2d_32", "kind": "batch", "inst": 32, "n_min": 129, "n_max": 1025},
        # the learned smoother on the 2049^2 grid's residual
        {"name": "net_fwd_n2047", "kind": "net_fwd", "B": 1, "H": 2047, "W": 2047},
        # one gradient of its training, a batch of 32 patches of 64^2
        {"name": "net_grad_b32", "kind": "net_grad", "B": 32, "P": 64},
    ]


def _grids(lo, hi):
    """Grid sizes c 2^j + 1 in [lo, hi] (c = 4..7: coarsest grids of 5 to 8 nodes)."""
    return sorted((c * 2 ** j + 1, c + 1) for c in (4, 5, 6, 7) for j in range(1, 12) if lo <= c * 2 ** j + 1 <= hi)


def _grid(rng, lo, hi):
    """One of them, spread over the logarithm of the size."""
    x = math.exp(rng.uniform(math.log(lo), math.log(hi)))
    return min(_grids(lo, hi), key=lambda g: abs(math.log(g[0] / x)))


def _logu(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def draw(rng):
    kind = rng.choice(["map", "map", "map3", "vcycle", "vcycle", "farfield", "gmres", "batch", "net_fwd", "net_grad"])
    if kind == "map":
        n, cn = _grid(rng, 49, 1025)
        R = 20.0 if n >= 257 else 10.0
        fp64 = rng.random() < 0.35 and n <= 257
        ng = rng.choice([1, 1, 2])
        return {"kind": "map", "dim": 2, "n": n, "coarsest": cn, "R": R,
                "k": round(_logu(rng, 1.0, min(5.0, 0.65 * (n - 1) / (2 * R))), 3),
                "k2w": round(rng.uniform(4.0 if ng == 2 else 2.0, 9.0), 2), "gauss": ng,
                "smoother": rng.choice(["jacobi", "rbgs"]) if fp64 else "rbgs",
                "precision": "fp64" if fp64 else "mixed", "ang": int(_logu(rng, 90, 721))}
    if kind == "map3":
        n, cn = _grid(rng, 33, 161)
        R = 15.0 if n >= 129 else 5.0
        return {"kind": "map", "dim": 3, "n": n, "coarsest": cn, "R": R,
                "k": round(_logu(rng, 1.0, min(4.0, 0.5 * (n - 1) / (2 * R))), 3),
                "k2w": round(rng.uniform(2.0, 8.0), 2), "gauss": 1, "smoother": "rbgs", "precision": "mixed",
                "ang": rng.choice([8, 12, 16, 24, 32])}
    if kind == "vcycle":
        dim = rng.choice([2, 2, 3])
        f64 = rng.random() < 0.4
        n, cn = _grid(rng, 129, 2049 if f64 else 3585) if dim == 2 else _grid(rng, 33, 129 if f64 else 257)
        R = 20.0 if dim == 2 else 15.0
        k = round(_logu(rng, 1.0, max(1.1, 0.5 * (n - 1) / (2 * R))), 3)
        return {"kind": "vcycle", "dim": dim, "n": n, "coarsest": cn, "R": R, "k": k,
                "k2w": round(rng.uniform(1.0, 4.0) * k * k, 2), "gauss": rng.choice([1, 1, 2]),
                "dtype": "f64" if f64 else "f32"}
    if kind == "farfield":
        n, cn = _grid(rng, 129, 1025)
        return {"kind": "farfield", "n": n, "coarsest": cn, "R": 20.0,
                "k": round(_logu(rng, 1.0, min(4.0, 0.65 * (n - 1) / 40.0)), 3), "k2w": round(rng.uniform(4.0, 16.0), 2),
                "gauss": rng.choice([1, 2]), "ang": int(_logu(rng, 90, 721))}
    if kind == "gmres":
        dim = rng.choice([2, 3])
        n = rng.choice([65, 129, 257]) if dim == 2 else rng.choice([33, 65])
        return {"kind": "gmres", "dim": dim, "n": n, "k": round(_logu(rng, 0.5, 1.0), 3),
                "precision": "fp64"}
    if kind == "batch":
        return {"kind": "batch", "inst": int(_logu(rng, 3, 32)), "n_min": 129, "n_max": rng.choice([257, 513, 1025])}
    if kind == "net_fwd":
        return {"kind": "net_fwd", "B": rng.choice([1, 1, 2]), "H": int(_logu(rng, 127, 1400)),
                "W": int(_logu(rng, 127, 1400))}
    return {"kind": "net_grad", "B": int(_logu(rng, 4, 32)), "P": rng.choice([32, 33, 47, 48, 64])}


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------
def _angles_2d(n):
    a = np.arange(n)
    mirror = a > n // 2
    t = 2 * np.pi * np.where(mirror, n - a, a) / n
    return np.ascontiguousarray(np.stack([np.cos(t), np.where(mirror, -np.sin(t), np.sin(t))], axis=1))


def _angles_3d(n_theta):
    n_phi = 2 * n_theta
    i = np.arange(n_phi)
    mirror = i > n_phi // 2
    ph = 2 * np.pi * np.where(mirror, n_phi - i, i) / n_phi
    sgn = np.where(mirror, -1.0, 1.0)
    th = np.pi * (np.arange(n_theta) + 0.5) / n_theta
    T, P = np.meshgrid(th, ph, indexing="ij")
    S = np.broadcast_to(sgn, T.shape)
    return np.ascontiguousarray(
        np.stack([np.sin(T) * np.cos(P), S * np.sin(T) * np.sin(P), np.cos(T)], axis=-1).reshape(-1, 3))


def _direction(rng, dim):
    if dim == 2:
        t = rng.uniform(0.0, 2 * PI)
        return np.array([[math.cos(t), math.sin(t)]])
    z, t = rng.uniform(-0.9, 0.9), rng.uniform(0.0, 2 * PI)
    s = math.sqrt(1.0 - z * z)
    return np.array([[s * math.cos(t), s * math.sin(t), z]])


def _problem(case, rng, dim):
    """One or two Gaussians of width k2w / k^2 (two: 3/k apart, after the
    paper's eq. chi2D), amplitudes near -1 by the seed; rotation pi/6."""
    k = case["k"]
    w = case["k2w"] / k ** 2
    amp = rng.uniform(0.8, 1.2, size=case["gauss"])
    off = [0.0] if case["gauss"] == 1 else [1.5 / k, -1.5 / k]
    gs = [{"amp": complex(-a / case["gauss"]), "width": w, "center": (0.0, o, 0.0)} for a, o in zip(amp, off)]
    return {"dim": dim, "n": case["n"], "lo": -case["R"], "hi": case["R"], "gamma": PI / 6, "k": k, "gaussians": gs}


def _opts(case):
    smoother = case.get("smoother", "rbgs")
    nu = 2 if smoother == "jacobi" else 1
    return {"smoother": smoother, "omega": 2.0 / 3.0 if smoother == "jacobi" else 1.0, "nu1": nu, "nu2": nu,
            "coarsest_n": case["coarsest"], "rel_tol": 1e-10, "max_cycles": 200,
            "precision": case.get("precision", "mixed"), "inner_cycles": 10, "adaptive_inner": 1, "refine_fp64": 1}


def _gmres_setup(case, rng):
    k = case["k"]
    amp = -0.2 / k ** 2 * rng.uniform(0.9, 1.1, size=2)
    gs = [{"amp": complex(a), "width": 1.0, "center": (0.0, o, 0.0)} for a, o in zip(amp, (4.0, -4.0))]
    prob = {"dim": case["dim"], "n": case["n"], "lo": -20.0, "hi": 20.0, "gamma": 9.9 * PI / 180, "k": k,
            "gaussians": gs}
    opts = {"smoother": "gmres", "krylov_m": 3, "nu1": 1, "nu2": 1, "coarsest_n": 5, "rel_tol": 1e-6,
            "max_cycles": 60, "precision": case["precision"], "inner_cycles": 2}
    return prob, opts, _direction(rng, case["dim"])


def _batch_setup(case, rng):
    sizes = [n for n in (129, 257, 513, 1025) if case["n_min"] <= n <= case["n_max"]]
    probs, etas = [], []
    for i in range(case["inst"]):
        n = sizes[i % len(sizes)]
        probs.append({"dim": 2, "n": n, "lo": -20.0, "hi": 20.0, "gamma": PI / 6, "k": rng.uniform(2.0, 10.0),
                      "gaussians": [{"amp": complex(rng.uniform(-2.0, -0.2)), "width": rng.uniform(1.0, 4.0),
                                     "center": (0.0, 0.0, 0.0)}]})
        etas.append(_direction(rng, 2)[0])
    opts = {"smoother": "rbgs", "omega": 1.0, "nu1": 1, "nu2": 1, "coarsest_n": 5, "rel_tol": 1e-10,
            "max_cycles": 200, "inner_cycles": 6, "adaptive_inner": 1, "refine_fp64": 1}
    return probs, opts, np.array(etas)


def _randc(shape, seed, dtype):
    g = torch.Generator(device=DEV).manual_seed(int(seed))
    return torch.randn(tuple(shape), generator=g, device=DEV, dtype=dtype)


def _field(case, problem, rng):
    """A scattered field as a program hands it in: a few plane waves on the grid."""
    n = case["n"]
    x = torch.linspace(-case["R"], case["R"], n, dtype=torch.float64, device=DEV)[1:-1]
    u = torch.zeros((n - 2, n - 2), dtype=torch.complex128, device=DEV)
    for _ in range(4):
        t, a = rng.uniform(0.0, 2 * PI), 0.2 * complex(rng.standard_normal(), rng.standard_normal())
        u += a * torch.outer(torch.exp(1j * problem["k"] * math.sin(t) * x), torch.exp(1j * problem["k"] * math.cos(t) * x))
    return u.reshape(-1).contiguous()


def _net_grad_inputs(case, seed):
    B, P = case["B"], case["P"]
    r = _randc((B, P, P), seed, torch.complex64)
    q = 1.37 * (1.0 + 0.1 * _randc((B, P, P), seed + 7, torch.complex64))
    c = np.full(B, complex(math.cos(PI / 3), -math.sin(PI / 3)))
    return r, q, c


def prepare(case, seed):
    rng = np.random.Generator(np.random.PCG64(seed))
    kind = case["kind"]
    s = {"kind": kind}
    if kind == "map":
        dim = case["dim"]
        s["plan"] = csff.Plan(_problem(case, rng, dim), _opts(case))
        s["eta"] = _direction(rng, dim)
        s["al"] = _angles_2d(case["ang"]) if dim == 2 else _angles_3d(case["ang"])
        s["u"] = torch.zeros(s["plan"].N, dtype=torch.complex128, device=DEV)
        s["F"] = torch.zeros(len(s["al"]), dtype=torch.complex128, device=DEV)
        s["E"] = torch.zeros(len(s["al"]), dtype=torch.int32, device=DEV)
    elif kind == "vcycle":
        opts = dict(_opts(case), precision="fp64" if case["dtype"] == "f64" else "mixed")
        s["plan"] = csff.Plan(_problem(case, rng, case["dim"]), opts)
        dt = torch.complex128 if case["dtype"] == "f64" else torch.complex64
        s["b"] = _randc((s["plan"].N,), seed, dt)
        s["u"] = _randc((s["plan"].N,), seed + 1, dt) * 1e-3
    elif kind == "farfield":
        prob = _problem(case, rng, 2)
        s["plan"] = csff.Plan(prob, _opts(case))
        s["eta"] = _direction(rng, 2)
        s["al"] = _angles_2d(case["ang"])
        s["u"] = _field(case, prob, rng)
        s["F"] = torch.zeros(case["ang"], dtype=torch.complex128, device=DEV)
        s["E"] = torch.zeros(case["ang"], dtype=torch.int32, device=DEV)
    elif kind == "gmres":
        prob, opts, s["eta"] = _gmres_setup(case, rng)
        s["plan"] = csff.Plan(prob, opts)
        s["u"] = torch.zeros(s["plan"].N, dtype=torch.complex128, device=DEV)
    elif kind == "batch":
        probs, opts, s["eta"] = _batch_setup(case, rng)
        s["batch"] = csff.Batch(probs, opts)
        s["batch"].set_tiles(16)
        s["n"] = len(probs)
    elif kind == "net_fwd":
        s["net"] = csff.Net(init_weights(seed))
        s["r"] = _randc((case["B"], case["H"], case["W"]), seed, torch.complex64)
        s["y"] = torch.zeros_like(s["r"])
    else:
        s["net"] = csff.Net(init_weights(seed))
        s["r"], s["q"], s["c"] = _net_grad_inputs(case, seed)
    return s


def run(s):
    kind = s["kind"]
    if kind == "map":
        s["plan"].solve(s["eta"], s["u"])
        s["plan"].far_field(s["eta"], s["u"], s["al"], s["F"], s["E"])
        return {"u": s["u"], "F": s["F"], "F_exp": s["E"]}
    if kind == "vcycle":
        s["plan"].vcycle(s["u"], s["b"])
        return s["u"]
    if kind == "farfield":
        s["plan"].far_field(s["eta"], s["u"], s["al"], s["F"], s["E"])
        return {"F": s["F"], "F_exp": s["E"]}
    if kind == "gmres":
        s["plan"].solve(s["eta"], s["u"])
        return s["u"]
    if kind == "batch":
        s["batch"].solve(s["eta"])
        return [s["batch"].solution(i) for i in range(s["n"])]
    if kind == "net_fwd":
        s["net"].forward(s["r"], s["y"])
        return s["y"]
    loss, g = s["net"].loss_grad(s["r"], s["q"], s["c"], margin=4)
    return {"loss": np.float32(loss), "grad": g}


# ---------------------------------------------------------------------------
# what a pass cannot do without
# ---------------------------------------------------------------------------
def _cycle_work(dim, N, el):
    """One V(1,1) cycle with el-byte complex values: the finest level's iterate
    and right-hand side read, the iterate written; per unknown of every level
    two sweeps and a residual (a complex neighbour sum and three complex
    products each)."""
    return 3.0 * el * N, 2.0 ** dim / (2.0 ** dim - 1) * N * 3 * (4 * dim + 22)


def _far_work(dim, m, n_ang):
    """u read once; the sum factorised over the axes, mirrored angles sharing
    their first stage."""
    N = m ** dim
    rows = n_ang // 2 + 1 if dim == 2 else max(1, int(round(math.sqrt(n_ang / 2))))
    flops = 8.0 * rows * N + 8.0 * n_ang * m * (1 if dim == 2 else m + 1) + 20.0 * N
    return 16.0 * N + 16.0 * n_ang, flops


def work(case):
    kind = case["kind"]
    if kind == "map":
        m = case["n"] - 2
        N = float(m ** case["dim"])
        n_ang = case["ang"] if case["dim"] == 2 else 2 * case["ang"] ** 2
        b0, f0 = _cycle_work(case["dim"], N, 16 if case["precision"] == "fp64" else 8)
        b1, f1 = _far_work(case["dim"], m, n_ang)
        # a solve to 1e-10 takes about 20 cycles; u is written once
        return {"bytes": 20 * b0 + 16 * N + b1, "flops": 20 * f0 + f1}
    if kind == "vcycle":
        b, f = _cycle_work(case["dim"], float((case["n"] - 2) ** case["dim"]), 16 if case["dtype"] == "f64" else 8)
        return {"bytes": b, "flops": f}
    if kind == "farfield":
        b, f = _far_work(2, case["n"] - 2, case["ang"])
        return {"bytes": b, "flops": f}
    if kind == "gmres":
        N = float((case["n"] - 2) ** case["dim"])
        el = 16 if case["precision"] == "fp64" else 8
        # about 10 cycles; two smoothing steps a cycle, each 4 operator
        # applications, 10 inner products and 10 updates of whole vectors
        return {"bytes": 10 * 2 * el * N * 12, "flops": 10 * 2 * N * (4 * (4 * case["dim"] + 16) + 20 * 8)}
    if kind == "batch":
        b = f = 0.0
        sizes = [n for n in (129, 257, 513, 1025) if case["n_min"] <= n <= case["n_max"]]
        for i in range(case["inst"]):
            N = float((sizes[i % len(sizes)] - 2) ** 2)
            b0, f0 = _cycle_work(2, N, 8)
            b, f = b + 22 * b0 + 16 * N, f + 22 * f0
        return {"bytes": b, "flops": f}
    if kind == "net_fwd":
        n = float(case["B"] * case["H"] * case["W"])
        return {"bytes": 16.0 * n, "flops": 2.0 * 2880 * n}
    n = float(case["B"] * case["P"] ** 2)
    return {"bytes": 16.0 * n, "flops": 3 * 2.0 * 2880 * n}


# ---------------------------------------------------------------------------
# the same results by plain torch in 64 bits
# ---------------------------------------------------------------------------
def _shift_sum(u, dim):
    """Sum of the 2 dim neighbours over the last dim axes, zero outside."""
    s = torch.zeros_like(u)
    for a in range(1, dim + 1):
        n = u.shape[-a]
        s.narrow(-a, 1, n - 1).add_(u.narrow(-a, 0, n - 1))
        s.narrow(-a, 0, n - 1).add_(u.narrow(-a, 1, n - 1))
    return s


class _Grid:
    """Levels of the rotated-grid operator A u = c (2 d u - sum u) - k^2 (1 + chi) u."""

    def __init__(self, prob, coarsest, smoother, omega=1.0, nu=1):
        self.dim, self.smoother, self.omega, self.nu = prob["dim"], smoother, omega, nu
        rot = complex(math.cos(prob["gamma"]), math.sin(prob["gamma"]))
        self.lv = []
        n = prob["n"]
        while True:
            h = (prob["hi"] - prob["lo"]) / (n - 1)
            chi = _chi(prob, n, rot)
            c = (1 / rot) ** 2 / h ** 2
            q = prob["k"] ** 2 * (1.0 + chi)
            L = {"n": n, "h": h, "c": c, "q": q, "d": 2 * self.dim * c - q}
            if smoother == "rbgs":
                idx = torch.arange(1, n - 1, device=DEV)
                par = sum(idx.reshape([-1 if i == a else 1 for i in range(self.dim)]) for a in range(self.dim)) % 2
                L["red"] = par == 0
            self.lv.append(L)
            if n == coarsest:
                break
            n = (n + 1) // 2
        L, m = self.lv[-1], self.lv[-1]["n"] - 2
        eye = torch.eye(m ** self.dim, dtype=torch.complex128, device=DEV).reshape((-1,) + (m,) * self.dim)
        self.dense = self.apply(L, eye).reshape(m ** self.dim, -1).T.contiguous()

    def apply(self, L, u):
        return L["d"] * u - L["c"] * _shift_sum(u, self.dim)

    def smooth(self, L, u, b):
        for _ in range(self.nu):
            if self.smoother == "jacobi":
                u = u + self.omega * (b - self.apply(L, u)) / L["d"]
            elif self.smoother == "rbgs":
                for colour in (L["red"], ~L["red"]):
                    u = torch.where(colour, (b + L["c"] * _shift_sum(u, self.dim)) / L["d"], u)
            else:
                u = self.gmres(L, u, b, 3)
        return u

    def gmres(self, L, u, b, m):
        r = b - self.apply(L, u)
        beta = torch.linalg.vector_norm(r).item()
        if beta == 0.0:
            return u
        V = [r / beta]
        H = np.zeros((m + 1, m), complex)
        for j in range(m):
            w = self.apply(L, V[j])
            for i in range(j + 1):
                hij = torch.vdot(V[i].reshape(-1), w.reshape(-1)).item()
                H[i, j] = hij
                w = w - hij * V[i]
            H[j + 1, j] = torch.linalg.vector_norm(w).item()
            if abs(H[j + 1, j]) == 0.0:
                m = j + 1
                break
            V.append(w / H[j + 1, j])
        rhs = np.zeros(m + 1, complex)
        rhs[0] = beta
        y = np.linalg.lstsq(H[:m + 1, :m], rhs, rcond=None)[0]
        for j in range(m):
            u = u + complex(y[j]) * V[j]
        return u

    def restrict(self, r):
        for a in range(1, self.dim + 1):
            m = r.shape[-a]
            mc = (m - 1) // 2
            pick = lambda s: torch.narrow(r, -a, s, 2 * mc - 1).index_select(  # noqa: E731
                r.dim() - a, torch.arange(0, 2 * mc - 1, 2, device=DEV))
            r = 0.5 * pick(1) + 0.25 * (pick(0) + pick(2))
        return r

    def prolong(self, e):
        for a in range(1, self.dim + 1):
            mc = e.shape[-a]
            shape = list(e.shape)
            shape[-a] = 2 * mc + 1
            out = torch.zeros(shape, dtype=e.dtype, device=DEV)
            ev = torch.arange(0, 2 * mc + 1, 2, device=DEV)
            ax = e.dim() - a
            half = 0.5 * e
            out.index_add_(ax, ev[:-1], half)
            out.index_add_(ax, ev[1:], half)
            out.index_add_(ax, torch.arange(1, 2 * mc + 1, 2, device=DEV), e)
            e = out
        return e

    def cycle(self, l, u, b):
        L = self.lv[l]
        if l == len(self.lv) - 1:
            return torch.linalg.solve(self.dense, b.reshape(-1)).reshape(b.shape)
        u = self.smooth(L, u, b)
        bc = self.restrict(b - self.apply(L, u))
        u = u + self.prolong(self.cycle(l + 1, torch.zeros_like(bc), bc))
        return self.smooth(L, u, b)

    def solve(self, b):
        u = torch.zeros_like(b)
        nb = torch.linalg.vector_norm(b).item()
        best = math.inf
        for _ in range(90):
            u = self.cycle(0, u, b)
            rel = torch.linalg.vector_norm(b - self.apply(self.lv[0], u)).item() / nb
            if rel < 1e-13 or rel > 0.98 * best:
                break
            best = rel
        return u


def _axis(prob, n):
    h = (prob["hi"] - prob["lo"]) / (n - 1)
    return prob["lo"] + h * torch.arange(1, n - 1, dtype=torch.float64, device=DEV)


def _outer(fs):
    """Product over the axes of per-axis factors given x first; x is the last axis."""
    out = fs[0]
    for f in fs[1:]:
        out = f.reshape([-1] + [1] * out.dim()) * out
    return out


def _chi(prob, n, rot):
    z = _axis(prob, n) * rot
    out = 0.0
    for g in prob["gaussians"]:
        out = out + complex(g["amp"]) * _outer([torch.exp(-(z - g["center"][a]) ** 2 / g["width"])
                                                for a in range(prob["dim"])])
    return out


def _chi_uin(prob, eta):
    rot = complex(math.cos(prob["gamma"]), math.sin(prob["gamma"]))
    z = _axis(prob, prob["n"]) * rot
    out = 0.0
    for g in prob["gaussians"]:
        out = out + complex(g["amp"]) * _outer(
            [torch.exp(-(z - g["center"][a]) ** 2 / g["width"] + 1j * prob["k"] * float(eta[a]) * z)
             for a in range(prob["dim"])])
    return out


def _far(prob, u, eta, al):
    dim, n = prob["dim"], prob["n"]
    rot = complex(math.cos(prob["gamma"]), math.sin(prob["gamma"]))
    h = (prob["hi"] - prob["lo"]) / (n - 1)
    z = _axis(prob, n) * rot
    g = _chi_uin(prob, eta) + _chi(prob, n, rot) * u
    pref = prob["k"] ** 2 * (rot * h) ** dim
    F = []
    for a0 in range(0, len(al), 256):
        A = torch.from_numpy(al[a0:a0 + 256]).to(DEV)
        P = [torch.exp(-1j * prob["k"] * A[:, c:c + 1] * z[None, :]) for c in range(dim)]
        T = P[0] @ g.reshape(-1, n - 2).T                       # sum over x
        if dim == 3:
            T = torch.einsum("azy,ay->az", T.reshape(len(A), n - 2, n - 2), P[1])
        F.append(pref * (T * P[dim - 1]).sum(1))
    return torch.cat(F)


def _conv(x, w):
    """3x3 cross-correlation, zero outside; x (B, C, H, W), w (O, C, 3, 3), 64 bits."""
    B, C, H, W = x.shape
    xp = torch.nn.functional.pad(x, (1, 1, 1, 1))
    out = torch.zeros((B, w.shape[0], H, W), dtype=x.dtype, device=x.device)
    for a in range(3):
        for b in range(3):
            out = out + torch.einsum("oc,bchw->bohw", w[:, :, a, b], xp[:, :, a:a + H, b:b + W])
    return out


def _net(w, r):
    w1, w2, w3 = w[:288].reshape(16, 2, 3, 3), w[288:2592].reshape(16, 16, 3, 3), w[2592:].reshape(2, 16, 3, 3)
    x = torch.stack([r.real, r.imag], dim=1)
    y = _conv(torch.relu(_conv(torch.relu(_conv(x, w1)), w2)), w3)
    return torch.complex(y[:, 0], y[:, 1])


def exact(case, seed):
    rng = np.random.Generator(np.random.PCG64(seed))
    kind = case["kind"]
    if kind == "map":
        dim = case["dim"]
        prob = _problem(case, rng, dim)
        eta = _direction(rng, dim)[0]
        o = _opts(case)
        G = _Grid(prob, case["coarsest"], o["smoother"], o["omega"], o["nu1"])
        u = G.solve(prob["k"] ** 2 * _chi_uin(prob, eta))
        al = _angles_2d(case["ang"]) if dim == 2 else _angles_3d(case["ang"])
        return {"u": u.reshape(-1), "F": _far(prob, u, eta, al), "F_exp": None}
    if kind == "vcycle":
        prob = _problem(case, rng, case["dim"])
        shape = (case["n"] - 2,) * case["dim"]
        dt = torch.complex128 if case["dtype"] == "f64" else torch.complex64
        N = (case["n"] - 2) ** case["dim"]
        b = _randc((N,), seed, dt).to(torch.complex128).reshape(shape)
        u = (_randc((N,), seed + 1, dt) * 1e-3).to(torch.complex128).reshape(shape)
        return _Grid(prob, case["coarsest"], "rbgs").cycle(0, u, b).reshape(-1)
    if kind == "farfield":
        prob = _problem(case, rng, 2)
        eta = _direction(rng, 2)[0]
        u = _field(case, prob, rng).reshape(case["n"] - 2, case["n"] - 2)
        return {"F": _far(prob, u, eta, _angles_2d(case["ang"])), "F_exp": None}
    if kind == "gmres":
        prob, _, eta = _gmres_setup(case, rng)
        u = _Grid(prob, 5, "gmres").solve(prob["k"] ** 2 * _chi_uin(prob, eta[0]))
        return u.reshape(-1)
    if kind == "batch":
        probs, _, etas = _batch_setup(case, rng)
        return [_Grid(p, 5, "rbgs").solve(p["k"] ** 2 * _chi_uin(p, e)).reshape(-1) for p, e in zip(probs, etas)]
    w = torch.from_numpy(init_weights(seed)).to(DEV).double()
    if kind == "net_fwd":
        return _net(w, _randc((case["B"], case["H"], case["W"]), seed, torch.complex64).to(torch.complex128))
    r, q, c = _net_grad_inputs(case, seed)
    r, q = r.to(torch.complex128), q.to(torch.complex128)
    w.requires_grad_(True)
    y = _net(w, r)
    cc = torch.from_numpy(c).to(DEV).reshape(-1, 1, 1)
    E = (r - (cc * (4 * y - _shift_sum_diff(y)) - q * y))[:, 4:-4, 4:-4]
    R = r[:, 4:-4, 4:-4]
    loss = ((E.real ** 2 + E.imag ** 2).sum((1, 2)) / (R.real ** 2 + R.imag ** 2).sum((1, 2))).mean()
    loss.backward()
    return {"loss": float(loss.item()), "grad": w.grad}


def _shift_sum_diff(y):
    """The 2D neighbour sum as padded slices (no writes in place, for autograd)."""
    p = torch.nn.functional.pad(torch.view_as_real(y), (0, 0, 1, 1, 1, 1))
    s = p[:, :-2, 1:-1] + p[:, 2:, 1:-1] + p[:, 1:-1, :-2] + p[:, 1:-1, 2:]
    return torch.view_as_complex(s.contiguous())
