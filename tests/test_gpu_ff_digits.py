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
