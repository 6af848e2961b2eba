"""Per-level calls in place and cycles outside the ordinary coefficients,
against the CPU oracle and 64-bit restatements."""
import math

import numpy as np
import pytest

import workloads as W
from oracle import csff_oracle as O

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def csff():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1211_4461_gb300 as m
    return m


# the coarsest solve in place and with overlapping buffers, in one CTA of four
# lanes a row, two of them (64 and 81 unknowns) and a warp a row (225)
@pytest.mark.parametrize("n,coarsest", [(9, 5), (17, 9), (19, 10), (21, 11), (33, 17)])
@pytest.mark.parametrize("dtype", [torch.complex128, torch.complex64])
@pytest.mark.parametrize("shift", [0, 1, -1])
def test_coarse_solve_in_place(csff, n, coarsest, dtype, shift):
    prob = W.problem(2, n, 3.0, math.pi / 6, 1.0, [W.gauss(-0.7, 1.5)])
    plan = csff.Plan(prob, {"smoother": "rbgs", "nu1": 1, "nu2": 1, "coarsest_n": coarsest, "rel_tol": 1e-8,
                            "precision": "fp64"})
    N = (coarsest - 2) ** 2
    b = torch.from_numpy(W.rand_complex(N, 5)).to(dtype).cuda()
    apart = torch.zeros_like(b)
    plan.coarse_solve(b, apart)
    buf = torch.zeros(N + 2, dtype=dtype, device="cuda")
    src, dst = buf[1:N + 1], buf[1 + shift:N + 1 + shift]
    for _ in range(20):
        src.copy_(b)
        plan.coarse_solve(src, dst)
        assert torch.equal(dst, apart)
    plan.close()


class Cycle3D:
    """One V(1,1) RB-GS cycle without a potential, in the given complex type
    (numpy's long double where FP64 itself is on trial)."""

    def __init__(self, n, coarsest, R, k, dtype, q=None):
        self.t, self.lv = np.dtype(dtype).type, []
        g = self.t(math.pi / 6)
        q = np.full((n - 2,) * 3, k * k, dtype=dtype) if q is None else q.astype(dtype)
        while True:
            m = n - 2
            h = self.t(2 * R) / self.t(n - 1)
            c = np.exp(self.t(-2j) * g) / (h * h)
            red = np.indices((m,) * 3).sum(0) % 2 == 1
            self.lv.append((m, c, q, 1 / (6 * c - q), red))
            if n == coarsest:
                break
            n, q = (n + 1) // 2, q[1::2, 1::2, 1::2]
        m, c, q, _, _ = self.lv[-1]
        eye = np.eye(m ** 3).reshape((-1,) + (m,) * 3)
        self.A = np.array([self._apply(c, q, e.astype(dtype)).ravel() for e in eye]).T
        self.lu = np.linalg.inv(self.A.astype(np.complex128))

    @staticmethod
    def _sum(u):
        p = np.pad(u, 1)
        i = slice(1, -1)
        return p[2:, i, i] + p[:-2, i, i] + p[i, 2:, i] + p[i, :-2, i] + p[i, i, 2:] + p[i, i, :-2]

    def _apply(self, c, q, u):
        return c * (6 * u - self._sum(u)) - q * u

    def _coarse(self, b):
        x = np.zeros_like(b.ravel())
        for _ in range(4):                      # refined in the type itself
            x = x + (self.lu @ (b.ravel() - self.A @ x).astype(np.complex128)).astype(x.dtype)
        return x.reshape(b.shape)

    def _sweep(self, l, u, b):
        _, c, _, dinv, red = self.lv[l]
        for colour in (red, ~red):
            u = np.where(colour, dinv * (b + c * self._sum(u)), u)
        return u

    def __call__(self, u, b, l=0):
        if l == len(self.lv) - 1:
            return self._coarse(b)
        m, c, q, _, _ = self.lv[l]
        u = self._sweep(l, u, b)
        r = b - self._apply(c, q, u)
        for ax in range(3):
            p = np.moveaxis(np.pad(r, [(1, 1) if a == ax else (0, 0) for a in range(3)]), ax, 0)
            r = np.moveaxis((p[:-2] + 2 * p[1:-1] + p[2:]) / 4, 0, ax)
        bc = r[1::2, 1::2, 1::2]
        e = self(np.zeros_like(bc), bc, l + 1)
        f = np.zeros((m + 2,) * 3, dtype=e.dtype)
        f[2:-1:2, 2:-1:2, 2:-1:2] = e
        for ax in range(3):
            v = np.moveaxis(f, ax, 0)
            v[1:-1:2] = (v[0:-2:2] + v[2::2]) / 2
        return self._sweep(l, u + f[1:-1, 1:-1, 1:-1], b)


# a cycle from an iterate that earlier cycles left.  A few dozen roundings a
# point, most of them averaged: 1.0 to 2.4 units of the type in the norm for
# per-level passes restated on the CPU
@pytest.mark.parametrize("prec,R", [("fp64", 5.0), ("fp64", 15.0), ("mixed", 5.0), ("mixed", 15.0)])
def test_vcycle_3d_rounding_from_an_iterate(csff, prec, R):
    n, coarsest, k = 65, 5, 1.0
    unit, ct, nt = (2.0 ** -53, np.clongdouble, np.complex128) if prec == "fp64" else (2.0 ** -24, np.complex128,
                                                                                       np.complex64)
    if np.finfo(ct).eps > unit / 256:
        pytest.skip("no wider type here")
    plan = csff.Plan(W.problem(3, n, R, math.pi / 6, k, []),
                     {"smoother": "rbgs", "omega": 1.0, "nu1": 1, "nu2": 1, "coarsest_n": coarsest, "rel_tol": 1e-8,
                      "precision": "fp64" if prec == "fp64" else "mixed"})
    m = plan.m
    b = W.rand_complex((m,) * 3, 4).astype(nt)
    start = Cycle3D(n, coarsest, R, k, np.complex128)
    u = start(np.zeros((m,) * 3, complex), b.astype(complex)).astype(nt)
    ref = Cycle3D(n, coarsest, R, k, ct)(u.astype(ct), b.astype(ct))
    ug = torch.from_numpy(u.ravel()).cuda()
    plan.vcycle(ug, torch.from_numpy(b.ravel()).cuda())
    plan.close()
    err = np.linalg.norm((ug.cpu().numpy().reshape(ref.shape) - ref).astype(complex)) / np.linalg.norm(ref.astype(complex))
    assert err <= 4 * unit


def _cycle_error(csff, plan, n, coarsest, R, k, q, before=4):
    """Error of one FP32 cycle, in units of 2^-24, from an iterate that `before` cycles left."""
    m = plan.m
    b = W.rand_complex((m,) * 3, 4).astype(np.complex64)
    exact = Cycle3D(n, coarsest, R, k, np.complex128, q)
    u = np.zeros((m,) * 3, complex)
    for _ in range(before):
        u = exact(u, b.astype(complex))
    u = u.astype(np.complex64)
    ref = exact(u.astype(complex), b.astype(complex))
    ug = torch.from_numpy(u.ravel()).cuda()
    plan.vcycle(ug, torch.from_numpy(b.ravel()).cuda())
    got = ug.cpu().numpy().reshape(ref.shape)
    return np.linalg.norm(got - ref) / np.linalg.norm(ref) * 2.0 ** 24


# one level above the direct solve (its right-hand side goes out in natural order)
# and several, rows of a slot pair up to several blocks' worth
@pytest.mark.parametrize("n,coarsest,R", [(5, 3, 3.0), (7, 4, 3.0), (13, 4, 3.0), (19, 10, 3.0), (37, 10, 5.0),
                                          (41, 6, 5.0), (65, 5, 5.0), (73, 10, 5.0)])
def test_vcycle_3d_from_an_iterate_over_grids(csff, n, coarsest, R):
    k, opts = 1.0, dict(OPTS3, coarsest_n=coarsest)
    plan = csff.Plan(W.problem(3, n, R, math.pi / 6, k, []), opts)
    levels = O.make_hierarchy(O.problem_from_dict(W.problem(3, n, R, math.pi / 6, k, [])), coarsest)
    lu, o, m = O.coarse_factor(levels[-1]), O.opts_from_dict(opts), plan.m
    b = W.rand_complex((m,) * 3, 4).astype(np.complex64)
    u = O.vcycle(levels, lu, 0, np.zeros((m,) * 3, complex), b.astype(complex), o).astype(np.complex64)
    ref = O.vcycle(levels, lu, 0, u.astype(complex), b.astype(complex), o)
    ug = torch.from_numpy(u.ravel()).cuda()
    plan.vcycle(ug, torch.from_numpy(b.ravel()).cuda())
    plan.close()
    # rounding as above (at most 4 units), and the coarsest product's in FP32, a
    # few units of a correction that on two levels is most of the result
    assert np.linalg.norm(ug.cpu().numpy().reshape(ref.shape) - ref) <= 16 * 2.0 ** -24 * np.linalg.norm(ref)


OPTS3 = {"smoother": "rbgs", "nu1": 1, "nu2": 1, "coarsest_n": 5, "rel_tol": 1e-8, "precision": "mixed"}


# coefficients far from the plan's k^2: an energy of 20 on a plan of k = 1, and
# barriers whose diagonal 6 c - q comes near zero on a level (|6 c / d| = 10.8),
# as samples and as a Gaussian plan.  Per-level passes restated: 0.7 to 2.4 units
@pytest.mark.parametrize("E,V,kind", [(20.0, 2.0, "sampled"), (1.0, 40.0, "sampled"), (1.0, 40.0, "gauss"),
                                      (1.0, 20.0, "sampled")])
def test_vcycle_3d_rounding_on_other_coefficients(csff, E, V, kind):
    n, R, w = 33, 15.0, 1.5
    g = math.pi / 6
    k = math.sqrt(2 * E) if kind == "gauss" else 1.0
    plan = csff.Plan(W.problem(3, n, R, g, k, [W.gauss(-V / E, w)] if kind == "gauss" else []), OPTS3)
    z = (-R + np.arange(1, n - 1) * 2 * R / (n - 1)) * np.exp(1j * g)
    ax = np.exp(-z * z / w)
    q = 2 * E - 2 * V * ax[:, None, None] * ax[None, :, None] * ax[None, None, :]
    if kind == "sampled":
        plan.set_potential(torch.from_numpy(q.ravel()).cuda())
    assert _cycle_error(csff, plan, n, 5, R, k, q) <= 4.0
    plan.close()


def test_plan_3d_without_room_for_the_split_arrays(csff):
    """A device with room for the plan but not for the colour-split arrays gives
    a plan that cycles per level."""
    n, R, k = 257, 15.0, 1.0
    prob = W.problem(3, n, R, math.pi / 6, k, [])
    plan = csff.Plan(prob, OPTS3)
    m, full = plan.m, plan.describe()["device_bytes"]
    b = torch.from_numpy(W.rand_complex((m,) * 3, 4).astype(np.complex64)).cuda().ravel()
    want = torch.zeros_like(b)
    plan.vcycle(want, b)
    plan.set_potential(torch.full((m ** 3,), k * k, dtype=torch.complex128, device="cuda"))
    split = full - plan.describe()["device_bytes"]        # what the plan gave back
    plan.close()
    assert split > 400 << 20
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    # all but the plan's own arrays and some room for their granules
    fill = torch.empty(torch.cuda.mem_get_info()[0] - (full - split) - (200 << 20), dtype=torch.uint8, device="cuda")
    plan = csff.Plan(prob, OPTS3)
    assert plan.describe()["device_bytes"] == full - split
    got = torch.zeros_like(b)
    plan.vcycle(got, b)
    plan.close()
    del fill
    torch.cuda.empty_cache()
    assert torch.linalg.vector_norm(got - want) <= 1e-5 * torch.linalg.vector_norm(want)


# amplitudes at which the residual of a converging solve is subnormal in FP64
# (below 2^-1022 from a relative 1e-8 on): its rounding to FP32 keeps it
@pytest.mark.parametrize("batch", [False, True])
def test_refinement_of_tiny_amplitudes(csff, batch):
    prob = W.problem(2, 65, 5.0, math.pi / 6, 1.0, [W.gauss(1e-300, 1.5)])
    opts = {"smoother": "rbgs", "nu1": 1, "nu2": 1, "coarsest_n": 5, "rel_tol": 1e-10, "max_cycles": 60,
            "precision": "mixed", "refine_fp64": 1}
    eta = np.array([[1.0, 0.0]])
    if batch:
        b = csff.Batch([prob], opts)
        st, infos = b.solve(eta)
        b.close()
    else:
        plan = csff.Plan(prob, opts)
        u = torch.zeros(plan.N, dtype=torch.complex128, device="cuda")
        st, infos = plan.solve(eta, u)
        plan.close()
    assert st == csff.OK and infos[0]["rel_res"] <= 1e-10


# the coarsest product in FP32: the restated rms error of a row in 32 lanes (or
# four of eight chains) is 1.2 to 1.5 units of 2^-24 of the result, of four lanes
# with a chain each 2.1; the rounding of the inverse adds 0.4 in the square
@pytest.mark.parametrize("coarsest", [11, 12, 13])
def test_coarse_product_rounding(csff, coarsest):
    n, R, g = 2 * coarsest - 1, 5.0, math.pi / 6
    plan = csff.Plan(W.problem(2, n, R, g, 1.0, []), {"smoother": "rbgs", "nu1": 1, "nu2": 1, "coarsest_n": coarsest,
                                                      "rel_tol": 1e-8, "precision": "fp64"})
    m, h = coarsest - 2, 2 * R / (coarsest - 1)
    T = 2 * np.eye(m) - np.eye(m, k=1) - np.eye(m, k=-1)
    A = np.exp(-2j * g) / h ** 2 * (np.kron(np.eye(m), T) + np.kron(T, np.eye(m))) - np.eye(m * m)
    err = []
    for seed in range(8):
        b = W.rand_real(m * m, seed).astype(np.complex64)
        u = torch.zeros(m * m, dtype=torch.complex64, device="cuda")
        plan.coarse_solve(torch.from_numpy(b).cuda(), u)
        ref = np.linalg.solve(A, b.astype(complex))
        err.append(np.linalg.norm(u.cpu().numpy() - ref) / np.linalg.norm(ref))
    plan.close()
    assert np.sqrt(np.mean(np.square(err))) <= 1.7 * 2.0 ** -24
