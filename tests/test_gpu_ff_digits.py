"""The digit contractions of the far field where inputs or phases leave the
ordinary: non-finite directions, phases that vary over a block."""
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


def _plan(csff, dim, n, coarsest, R, k):
    prob = W.problem(dim, n, R, math.pi / 6, k, [W.gauss(-0.7, 1.5), W.gauss(-0.3, 3.0, (0.5, -0.4, 0.2))])
    return prob, csff.Plan(prob, {"smoother": "jacobi", "nu1": 1, "nu2": 1, "coarsest_n": coarsest,
                                  "rel_tol": 1e-8, "precision": "fp64"})


def _far(plan, eta, u, al):
    F = torch.zeros(len(al), dtype=torch.complex128, device="cuda")
    E = torch.zeros(len(al), dtype=torch.int32, device="cuda")
    plan.far_field(eta, torch.from_numpy(np.ascontiguousarray(u).ravel()).cuda(), al, F, E)
    return F.cpu().numpy(), E.cpu().numpy()


# a direction with a component that is not a number: no value for it, the same
# ones for all others (z and y contractions in digits: 64 angles a z component)
@pytest.mark.parametrize("component", [1, 0])
def test_nan_direction_3d_gives_nan(csff, component):
    prob, plan = _plan(csff, 3, 65, 5, 5.0, 1.0)
    u = W.rand_complex((plan.m,) * 3, 31)
    eta, al = np.array([[0.6, 0.0, 0.8]]), W.angle_set_3d(64, 33)
    F0, E0 = _far(plan, eta, u, al)
    bad = al.copy()
    bad[77, component] = np.nan
    F1, E1 = _far(plan, eta, u, bad)
    plan.close()
    others = np.arange(len(al)) != 77
    assert np.isnan(F1[77].real) and np.isnan(F1[77].imag)
    assert np.all(np.isfinite(F0)) and np.array_equal(F0[others], F1[others]) and np.array_equal(E0[others], E1[others])


# fields (far over the incident wave's) that live where the phases of a block of
# 32 nodes are smallest, so that the block's scales lie far over its terms: a
# single node of a row, three of them, or a fall three times the phases' growth;
# phases that vary by var binades over the block, below, around and above the
# digit form's line.  The contraction against the FP64 one of the same call (the
# waits made to run out), whose rounding is 2^-52: no further apart than the
# double-float form's rms error of 2^-48
@pytest.mark.parametrize("var", [2.0, 4.5, 6.5, 8.3, 9.5, 11.0, 12.5, 14.0])
@pytest.mark.parametrize("nodes", [1, 3, 32])
def test_far_field_2d_of_unbalanced_blocks(csff, var, nodes):
    n, R, g = 129, 10.0, math.pi / 6
    h = 2 * R / (n - 1)
    k = var * math.log(2.0) / (32 * h * math.sin(g))
    prob = W.problem(2, n, R, g, k, [W.gauss(1.0, 1e6)])
    plan = csff.Plan(prob, {"smoother": "jacobi", "nu1": 1, "nu2": 1, "coarsest_n": 5, "rel_tol": 1e-8,
                            "precision": "fp64"})
    m = plan.m
    u, i = np.zeros((m, m), dtype=complex), np.arange(nodes)
    u[60, 32:32 + nodes] = W.rand_complex(nodes, 7) * (1e40 * 2.0 ** (-3 * var * i / 32 * (nodes == 32)))
    t = np.linspace(-0.3, 0.3, 97)
    al = np.ascontiguousarray(np.stack([np.cos(t), np.sin(t)], axis=1))
    eta = np.array([[0.6, 0.8]])
    F, E = _far(plan, eta, u, al)
    plan.debug_far_field_waits(1, wait_ms=20)
    F64, E64 = _far(plan, eta, u, al)
    digits = plan.debug_far_field_waits(0)
    plan.close()
    assert digits or var > 9.5
    tn, e2 = O.far_field(O.problem_from_dict(prob), u, eta[0], al, return_terms_norm=True)[:0:-1]
    diff = np.abs(F * 2.0 ** (E.astype(np.float64) - e2) - F64 * 2.0 ** (E64.astype(np.float64) - e2)) / tn
    assert np.sqrt(np.mean(diff ** 2)) <= 2.0 ** -48


def test_far_field_2d_holds_one_set_of_operands(csff):
    """The digit and the double-float contraction share their operands' memory."""
    prob, plan = _plan(csff, 2, 513, 9, 10.0, 1.0)
    m, ang = plan.m, 300
    al = W.angle_set_2d(ang)
    before = plan.describe()["device_bytes"]
    _far(plan, np.array([[0.6, 0.8]]), np.zeros((m, m), dtype=complex), al)
    grown = plan.describe()["device_bytes"] - before
    plan.close()
    rows, nb = len(np.unique(al[:, 0])), (m + 31) // 32
    tiles_x, tiles_g = (rows + 15) // 16, (m + 127) // 128
    field = 16 * m * m + 16 * m * (rows + 2 * ang) + 16 * m * rows           # g, phase tables, sums
    digits = nb * (tiles_x * 8 * 4096 + tiles_g * 8 * 16384)
    words = 8 * nb * (rows + m) + tiles_x * ((m + 31) // 32) * nb + 8 * 3 * (rows + ang) + 4 * ang
    assert grown <= field + digits + words


def test_far_field_work_counts_the_tiles_of_the_contraction_that_ran(csff):
    """Rows 0-31 live in the first of four blocks, the others in the last: every
    double-float tile (32 rows) keeps one block of four, the digit form's one tile
    of 128 rows two.  At k = 6 the phases vary too much over a block for digits."""
    for k, fraction in ((0.5, 0.5), (6.0, 0.25)):
        prob = W.problem(2, 129, 10.0, math.pi / 6, k, [W.gauss(1.0, 1e6)])
        plan = csff.Plan(prob, {"smoother": "jacobi", "nu1": 1, "nu2": 1, "coarsest_n": 5, "rel_tol": 1e-8,
                                "precision": "fp64"})
        m = plan.m
        u = np.zeros((m, m), dtype=complex)
        u[:32, :32], u[32:, 96:] = 1e60, 1e60
        _far(plan, np.array([[0.6, 0.8]]), u, W.angle_set_2d(40))
        assert plan.far_field_work() == fraction
        plan.close()


# the y contraction in digits (angles that share z components, in numbers that are
# no multiple of its tiles of 16; rows of 63 to 127 nodes, whose second scale block
# of the last 32 is full, empty or short): against the oracle at selected angles.
# A y component too steep for digits takes its three launches away
@pytest.mark.parametrize("n,coarsest,per_z,n_z,k,R", [(65, 5, 40, 56, 1.0, 5.0), (73, 10, 24, 67, 2.0, 5.0),
                                                      (81, 6, 17, 80, 2.0, 5.0), (97, 7, 33, 30, 2.0, 10.0),
                                                      (129, 5, 9, 60, 2.0, 10.0)])
def test_far_field_3d_y_contraction(csff, n, coarsest, per_z, n_z, k, R):
    prob, plan = _plan(csff, 3, n, coarsest, R, k)
    u = W.rand_complex((plan.m,) * 3, 31)
    th, ph = np.pi * (np.arange(n_z) + 0.5) / n_z, 2 * np.pi * (np.arange(per_z) + 0.2) / per_z
    T, P = np.meshgrid(th, ph, indexing="ij")
    al = np.ascontiguousarray(np.stack([np.sin(T) * np.cos(P), np.sin(T) * np.sin(P), np.cos(T)], -1).reshape(-1, 3))
    eta = np.array([[0.6, 0.0, 0.8]])
    before = csff.kernel_launches()
    F, E = _far(plan, eta, u, al)
    launches = csff.kernel_launches() - before
    steep = al.copy()
    steep[5, 1] = 40.0
    _far(plan, eta, u, steep)
    plan.close()
    assert csff.kernel_launches() - before == 2 * launches - 3
    sel = np.array([0, per_z // 2, len(al) // 2 + 7, len(al) - 1])
    mant, e2, tn = O.far_field(O.problem_from_dict(prob), u, eta[0], al[sel], return_terms_norm=True)
    # each stage's rounding is below 2^-48 of the sum of the terms' magnitudes, the
    # phases' own k |z| and a few ulp
    assert np.all(np.abs(F[sel] * 2.0 ** (E[sel].astype(np.float64) - e2) - mant) <= 1e-13 * tn)
