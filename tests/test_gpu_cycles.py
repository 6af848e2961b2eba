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
