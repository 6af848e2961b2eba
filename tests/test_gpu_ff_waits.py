"""Bounded waits of the far field's digit contraction (the hook makes it wait
for an arrival that never comes)."""
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


class Case:
    """A far field that takes the digit contraction with at least three of its
    accumulations a tile, and the oracle's value at selected angles."""

    def __init__(self, csff, dim):
        n, coarsest = (129, 5) if dim == 2 else (65, 5)
        self.prob = W.problem(dim, n, 10.0 if dim == 2 else 5.0, math.pi / 6, 1.0,
                              [W.gauss(-0.7, 1.5), W.gauss(-0.3, 3.0, (0.5, -0.4, 0.2))])
        self.plan = csff.Plan(self.prob, {"smoother": "jacobi", "nu1": 1, "nu2": 1, "coarsest_n": coarsest,
                                          "rel_tol": 1e-8, "precision": "fp64"})
        m = self.plan.m
        u = W.rand_complex((m,) * dim, 31)
        self.u = torch.from_numpy(u.ravel()).cuda()
        self.eta = np.array([[0.6, 0.8]]) if dim == 2 else np.array([[0.6, 0.0, 0.8]])
        self.al = W.angle_set_2d(30) if dim == 2 else W.angle_set_3d(64, 33)
        self.sel = np.array([0, len(self.al) // 3, len(self.al) - 1])
        self.mant, self.e2, self.tn = O.far_field(O.problem_from_dict(self.prob), u, self.eta[0], self.al[self.sel],
                                                  return_terms_norm=True)

    def run(self, with_exp=True):
        F = torch.zeros(len(self.al), dtype=torch.complex128, device="cuda")
        E = torch.zeros(len(self.al), dtype=torch.int32, device="cuda")
        st = self.plan.far_field(self.eta, self.u, self.al, F, E if with_exp else None)
        return st, F.cpu().numpy()[self.sel] * 2.0 ** (E.cpu().numpy()[self.sel].astype(np.float64) - self.e2)

    def check(self, got):
        # the contraction's and the stages' rounding, below 2^-47 of the sum of the
        # terms' magnitudes, and the phase tables' few ulp
        assert np.all(np.abs(got - self.mant) <= 1e-13 * self.tn)


@pytest.mark.parametrize("dim", [2, 3])
def test_contraction_whose_waits_run_out_ends_and_leaves_the_next_call_whole(csff, dim):
    """A CTA that gives up waits for its own copies and matrix products before it
    ends, so the launch after it finds its shared and tensor memory whole."""
    c = Case(csff, dim)
    c.plan.debug_far_field_waits(1, wait_ms=20)
    c.run(with_exp=True)
    assert c.plan.debug_far_field_waits(0) is True
    st, got = c.run()
    assert st == csff.OK and c.plan.debug_far_field_waits(0) is False
    c.check(got)
    c.plan.close()


@pytest.mark.parametrize("with_exp", [True, False])
@pytest.mark.parametrize("dim", [2, 3])
def test_contraction_whose_waits_run_out_is_repeated_in_fp64(csff, dim, with_exp):
    """The map of the call itself is right, with and without exponents: both
    contractions of the 3D case (its angles share z components) give up."""
    c = Case(csff, dim)
    c.plan.debug_far_field_waits(1, wait_ms=20)
    st, got = c.run(with_exp)
    assert c.plan.debug_far_field_waits(0) is True
    assert st == csff.OK
    c.check(got)
    c.plan.close()
