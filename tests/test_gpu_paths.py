"""Edges of the kernels' size ranges against the CPU oracle: one V-cycle on
grids whose coarse-level block has one to four levels, even and odd coarsest
grids, staged and unstaged coarsest inverses, and the far-field and learned
paths at tile remainders."""
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


def _problem(dim, n, k, R=5.0):
    return W.problem(dim, n, R, math.pi / 6, k, [W.gauss(-0.7, 1.5), W.gauss(-0.3, 1.0, (0.5, -0.4, 0.2))])


def _vcycle_pair(csff, prob, opts, dtype, seed=3):
    plan = csff.Plan(prob, opts)
    u0 = W.rand_complex(plan.N, seed)
    b = W.rand_complex(plan.N, seed + 1)
    np_t = np.complex128 if dtype == torch.complex128 else np.complex64
    u = torch.from_numpy(u0.astype(np_t)).cuda()
    bt = torch.from_numpy(b.astype(np_t)).cuda()
    plan.vcycle(u, bt)
    plan.close()
    levels = O.make_hierarchy(O.problem_from_dict(prob), opts["coarsest_n"])
    shape = (levels[0].m,) * prob["dim"]
    ref = O.vcycle(levels, O.coarse_factor(levels[-1]), 0, u0.astype(np_t).astype(np.complex128).reshape(shape),
                   b.astype(np_t).astype(np.complex128).reshape(shape), O.opts_from_dict(opts))
    return u.cpu().numpy().astype(np.complex128).ravel(), ref.ravel()


# coarsest grids of 3 (one unknown), 4 and 6 (even), 9 (inverse staged), 17 and
# 18 (the FP64 inverse does not fit shared memory; 18: the block is the direct
# solve alone)
@pytest.mark.parametrize("n,coarsest", [(65, 3), (49, 4), (41, 6), (65, 9), (65, 17), (69, 18)])
@pytest.mark.parametrize("prec", ["fp64", "df", "mixed64"])
def test_vcycle_over_coarse_blocks(csff, n, coarsest, prec):
    opts = {"smoother": "rbgs", "omega": 1.0, "nu1": 1, "nu2": 1, "coarsest_n": coarsest, "rel_tol": 1e-8,
            "max_cycles": 100, "precision": "fp64" if prec == "fp64" else "mixed",
            "refine_fp64": int(prec == "mixed64")}
    got, ref = _vcycle_pair(csff, _problem(2, n, 1.0), opts,
                            torch.complex128 if prec == "fp64" else torch.complex64)
    # FP64: rounding of a cycle's few dozen operations a point and of the
    # coarsest inverse; FP32: the same in 2^-24, coefficients included
    tol = 1e-11 if prec == "fp64" else 1e-4
    assert np.linalg.norm(got - ref) <= tol * np.linalg.norm(ref)


# 3D V(1,1) cycles on colour-split arrays: rows of one slot pair (5 nodes) up
# to several, row lengths that are no multiple of the pitch's four slots, one
# level above the direct solve and several, even coarsest grids
@pytest.mark.parametrize("n,coarsest", [(5, 3), (7, 4), (9, 3), (13, 4), (21, 6), (29, 8), (33, 5)])
@pytest.mark.parametrize("prec", ["fp64", "df", "mixed64"])
def test_vcycle_3d_by_colour(csff, n, coarsest, prec):
    opts = {"smoother": "rbgs", "omega": 1.0, "nu1": 1, "nu2": 1, "coarsest_n": coarsest, "rel_tol": 1e-8,
            "max_cycles": 100, "precision": "fp64" if prec == "fp64" else "mixed",
            "refine_fp64": int(prec == "mixed64")}
    got, ref = _vcycle_pair(csff, _problem(3, n, 1.0, R=3.0), opts,
                            torch.complex128 if prec == "fp64" else torch.complex64)
    tol = 1e-11 if prec == "fp64" else 1e-4
    assert np.linalg.norm(got - ref) <= tol * np.linalg.norm(ref)


# training gradients: one patch and several, widths around the 256-thread loss
# blocks and the weight gradient's row groups, non-square patches
@pytest.mark.parametrize("B,H,Wd,margin", [(1, 9, 9, 4), (1, 1, 1, 0), (2, 17, 15, 3), (5, 16, 16, 2), (3, 33, 40, 4),
                                           (40, 12, 11, 1)])
def test_net_gradient_over_patch_shapes(csff, B, H, Wd, margin):
    import oracle.net_oracle as NO
    theta = NO.init_params(8)
    net = csff.Net(theta)
    r = W.rand_complex((B, H, Wd), 21).astype(np.complex64)
    q = (W.rand_complex((B, H, Wd), 22, scale=0.3) + 1.4).astype(np.complex64)
    c = np.array([complex(np.exp(-1j * math.pi / 3) * (1.0 + 0.1 * b)) for b in range(B)])
    L, g = net.loss_grad(torch.from_numpy(r).cuda(), torch.from_numpy(q).cuda(), c, margin=margin)
    tb = torch.from_numpy(theta.astype(np.float32)).to(torch.bfloat16).to(torch.float64).numpy()
    Lo, go = NO.batch_loss_and_grad(tb, list(r.astype(complex)), list(q.astype(complex)), list(c), margin=margin)
    net.close()
    # the BF16 rounding of input and activations (2^-9 a value) bounds both
    assert abs(L - Lo) <= 2e-2 * abs(Lo)
    assert np.linalg.norm(g - go) <= 5e-2 * np.linalg.norm(go)


# Jacobi sweeps from a zero and a non-zero iterate, odd and even counts (the
# second buffer holds the result of one of them), and the per-level passes in
# blocks of both shapes: 2D levels of 31 to 255 points a side, 3D of 7 to 31
@pytest.mark.parametrize("dim,n,coarsest", [(2, 33, 5), (2, 161, 6), (2, 257, 9), (3, 17, 5), (3, 33, 9)])
@pytest.mark.parametrize("nu1,nu2", [(1, 2), (2, 1), (3, 0), (0, 3)])
@pytest.mark.parametrize("prec", ["fp64", "df"])
def test_vcycle_jacobi(csff, dim, n, coarsest, nu1, nu2, prec):
    opts = {"smoother": "jacobi", "omega": 0.6, "nu1": nu1, "nu2": nu2, "coarsest_n": coarsest, "rel_tol": 1e-8,
            "max_cycles": 100, "precision": "fp64" if prec == "fp64" else "mixed"}
    got, ref = _vcycle_pair(csff, _problem(dim, n, 1.0, R=4.0), opts,
                            torch.complex128 if prec == "fp64" else torch.complex64)
    tol = 1e-11 if prec == "fp64" else 1e-4
    assert np.linalg.norm(got - ref) <= tol * np.linalg.norm(ref)


# the 2D far-field contraction: row counts below, at and above its tiles of 128
# rows and 16 phase rows, block counts of one and several, odd angle sets; k =
# 8 on the small box varies too fast per block for the digit form
@pytest.mark.parametrize("n,coarsest,n_ang,k,R", [(5, 3, 1, 1.0, 2.0), (33, 5, 33, 1.0, 5.0), (35, 18, 31, 1.0, 5.0),
                                                  (129, 5, 30, 2.0, 10.0), (137, 18, 97, 2.0, 10.0),
                                                  (273, 18, 64, 3.0, 10.0), (65, 5, 40, 8.0, 10.0)])
@pytest.mark.parametrize("scale", [1.0, 1e-200, 1e150])
def test_far_field_contraction(csff, n, coarsest, n_ang, k, R, scale):
    prob = W.problem(2, n, R, math.pi / 6, k, [W.gauss(-0.7, 1.5), W.gauss(-0.3, 3.0, (0.5, -0.4, 0.0))])
    opts = {"smoother": "jacobi", "nu1": 1, "nu2": 1, "coarsest_n": coarsest, "rel_tol": 1e-8, "precision": "fp64"}
    plan = csff.Plan(prob, opts)
    m = plan.m
    u0 = scale * W.rand_complex((m, m), 31)
    eta = np.array([[math.cos(0.4), math.sin(0.4)]])
    al = W.angle_set_2d(n_ang)
    F = torch.zeros(n_ang, dtype=torch.complex128, device="cuda")
    E = torch.zeros(n_ang, dtype=torch.int32, device="cuda")
    plan.far_field(eta, torch.from_numpy(u0.ravel()).cuda(), al, F, E)
    mant, e2, tn = O.far_field(O.problem_from_dict(prob), u0, eta[0], al, return_terms_norm=True)
    got = F.cpu().numpy() * 2.0 ** (E.cpu().numpy().astype(np.float64) - e2)
    plan.close()
    # the contraction's rounding (2^-47 of the sum of the terms' magnitudes for
    # the double-float form, less for digits) and the phase tables' few ulp
    assert np.all(np.abs(got - mant) <= 1e-13 * tn)


# the z contraction of the 3D far field: distinct z components below, at and
# above its tiles of 16, last rows of 32 nodes whose second scale block of 16 is
# empty (m = 71, 79) or short (63, 95), several column chunks (159) and phases
# too steep for its digits (k = 3 on the wide box: the FP64 kernel)
@pytest.mark.parametrize("n,coarsest,n_z,k,R", [(65, 5, 33, 1.0, 5.0), (73, 10, 48, 2.0, 5.0), (81, 6, 17, 2.0, 5.0),
                                                (97, 7, 16, 3.0, 10.0), (161, 6, 7, 2.0, 15.0), (65, 5, 40, 3.0, 10.0)])
@pytest.mark.parametrize("scale", [1.0, 1e-150])
def test_far_field_3d_contraction(csff, n, coarsest, n_z, k, R, scale):
    prob = W.problem(3, n, R, math.pi / 6, k, [W.gauss(-0.7, 1.5), W.gauss(-0.3, 3.0, (0.5, -0.4, 0.2))])
    opts = {"smoother": "jacobi", "nu1": 1, "nu2": 1, "coarsest_n": coarsest, "rel_tol": 1e-8, "precision": "fp64"}
    plan = csff.Plan(prob, opts)
    m = plan.m
    u0 = scale * W.rand_complex((m, m, m), 31)
    eta = np.array([[0.6, 0.0, 0.8]])
    th, ph = np.pi * (np.arange(n_z) + 0.5) / n_z, 0.7 * np.arange(n_z)
    al = np.ascontiguousarray(np.stack([np.sin(th) * np.cos(ph), np.sin(th) * np.sin(ph), np.cos(th)], axis=1))
    F = torch.zeros(n_z, dtype=torch.complex128, device="cuda")
    E = torch.zeros(n_z, dtype=torch.int32, device="cuda")
    plan.far_field(eta, torch.from_numpy(u0.ravel()).cuda(), al, F, E)
    plan.close()
    sel = np.unique(np.array([0, n_z // 2, n_z - 1]))
    mant, e2, tn = O.far_field(O.problem_from_dict(prob), u0, eta[0], al[sel], return_terms_norm=True)
    got = F.cpu().numpy()[sel] * 2.0 ** (E.cpu().numpy()[sel].astype(np.float64) - e2)
    # each stage's rounding is below 2^-48 of the sum of the terms' magnitudes
    assert np.all(np.abs(got - mant) <= 1e-13 * tn)
