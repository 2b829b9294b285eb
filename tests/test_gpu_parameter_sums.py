"""The parameter block's right-hand side: sums over the chain's contributions by quads of
lanes, at parameter counts that leave part of a warp idle and element counts whose number of
partial sums (2 N up to 64) leaves a remainder to one lane; and the Schur complement's totals, by
the block that factors it up to 22 parameters and by the grid above."""
import numpy as np
import pytest

from paper_2607_12201_gb300 import workloads as W
from oracle import ipm as oipm
from oracle.nlp import Problem as OProblem
from gpu_helpers import newton_system

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def collo():
    from paper_2607_12201_gb300 import build
    build.build()
    from paper_2607_12201_gb300 import collo
    return collo


@pytest.mark.parametrize("mode", [0, 1])
@pytest.mark.parametrize("N", [1, 3, 17, 33])
@pytest.mark.parametrize("p", [2, 3, 11, 21, 22, 23, 67])
def test_solution_before_refinement(collo, p, N, mode):
    """FP64, no refinement.  A lost or doubled partial sum leaves a residual of the size of the
    parameter rows' right-hand side; rounding, with pivots that are not searched for, stays
    many orders below 1e-8 of it."""
    inst = (W.linear_cascade(N=N, T=0.2 * N) if p == 2 else
            W.random_network(max(2, p // 2), p, n_obs=2, M=5, T=0.1 * N, N=N, seed=900 + p,
                             theta0_spread=0.1))
    assert inst.p == p
    oprob = OProblem(inst)
    x, lam, zl, zu, _ = oipm.initial_point(oprob, inst.theta0, oipm.Options())
    mu, dw = 0.1, 1.0
    dc = 1e-8 * mu ** 0.25
    ref = newton_system(oprob, x, lam, zl, zu, mu, dw, dc)
    K, rhs = ref["K"], ref["rhs"].copy()
    rows = slice(oprob.nz, oprob.nz + p)
    rhs[rows] = np.cos(1.0 + np.arange(p)) * np.max(np.abs(rhs))
    with collo.Problem(inst, launch_mode=mode) as prob:
        prob.eval(x, lam)
        prob.kkt_factor(ref["sigma"], dw, dc, precision=collo.FP64)
        sol, _ = prob.kkt_solve(rhs, refine_max=0)
    assert np.max(np.abs(rhs - K @ sol)[rows]) <= 1e-8 * np.max(np.abs(rhs))
