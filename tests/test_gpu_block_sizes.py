"""Newton steps at the block sizes where the large-block kernels change: element blocks of
10 n + few rows (Radau) around the register-tile limit (124), around whole 32-row blocks of
the global slab, with whole and ragged last panels (3 n pairs in panels of 8 or 16), reduction
blocks and substitutions around 128 rows, odd parameter counts; and the sums over elements
around their blocks of 32 columns."""
import dataclasses

import numpy as np
import pytest

from paper_2607_12201_gb300 import workloads as W
from oracle import ipm as oipm
from oracle.nlp import Problem as OProblem
from gpu_helpers import assemble_J, assemble_W, newton_system, random_point, rel_max, sparse_rel

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def collo():
    from paper_2607_12201_gb300 import build
    build.build()
    from paper_2607_12201_gb300 import collo
    return collo


def _network(n, r, N, scheme="radau"):
    inst = W.random_network(n, r, n_obs=min(2, n), M=5, T=0.1 * N, N=N, seed=500 + n,
                            theta0_spread=0.1)
    return dataclasses.replace(inst, K=4, scheme="gauss") if scheme == "gauss" else inst


SIZES = [("radau", n, r) for n, r in ((12, 28), (13, 21), (16, 16), (16, 32), (17, 33), (21, 42),
                                      (22, 44), (27, 54), (28, 64), (29, 55), (32, 32), (32, 64),
                                      (33, 67))]
SIZES += [("gauss", n, r) for n, r in ((10, 24), (11, 25), (16, 32), (26, 53))]


@pytest.mark.parametrize("mode", [0, 1])
@pytest.mark.parametrize("scheme,n,r", SIZES)
def test_step_at_block_edges_matches_oracle(collo, scheme, n, r, mode):
    """Five elements: both ends of the chain, odd and even reduction blocks.  The step's
    backward error: the refinement stops at 1e-14 of the right-hand side (FP32 factors), two
    FP64 corrections of a backward-stable FP64 solution end at the rounding of the residual,
    a few eps; a wrong entry of a factor leaves its own size, whatever the condition."""
    inst = _network(n, r, 5, scheme)
    oprob = OProblem(inst)
    x, lam, zl, zu, _ = oipm.initial_point(oprob, inst.theta0, oipm.Options())
    mu, dw = 0.1, 1.0
    dc = 1e-8 * mu ** 0.25
    ref = newton_system(oprob, x, lam, zl, zu, mu, dw, dc)
    K, rhs = ref["K"], ref["rhs"]
    Kinf = abs(K).sum(axis=1).max()
    with collo.Problem(inst, launch_mode=mode) as prob:
        prob.eval(x, lam)
        for prec, refine, tol in ((collo.MIXED, 40, 1e-14), (collo.FP64, 2, 1e-15)):
            assert prob.kkt_factor(ref["sigma"], dw, dc, precision=prec) == ref["inertia"]
            sol, info = prob.kkt_solve(rhs, refine_max=refine, refine_tol=1e-14)
            err = np.max(np.abs(rhs - K @ sol))
            assert err <= tol * (Kinf * np.max(np.abs(sol)) + np.max(np.abs(rhs))), (prec, info)


@pytest.mark.parametrize("n,r,N", [(4, 31, 3), (4, 32, 257), (4, 33, 40), (10, 65, 40),
                                   (50, 100, 2)])
def test_evaluation_sums_at_block_edges_match_oracle(collo, n, r, N):
    """Parameter counts around 32 columns per block, more elements than a block has threads
    per column, and derivative rows larger than their shared-memory stage (50 species)."""
    inst = _network(n, r, N)
    oprob = OProblem(inst)
    x, lam = random_point(oprob, 11)
    ev = oprob.evaluate(x, lam, obj_factor=0.8)
    with collo.Problem(inst) as prob:
        out = prob.eval(x, lam, obj_factor=0.8)
    tol = 1e-13   # sums of N <= 257 FP64 terms in another order
    assert abs(out["phi"] - ev["phi"]) <= tol * max(1.0, abs(ev["phi"]))
    assert rel_max(out["c"], ev["c"]) <= tol
    assert rel_max(out["grad"], ev["grad"]) <= tol
    assert sparse_rel(assemble_J(oprob, out), ev["J"]) <= tol
    assert sparse_rel(assemble_W(oprob, out), ev["W"]) <= tol
