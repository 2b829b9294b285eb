"""The factors themselves, at the block sizes where the kernels change: solutions before any
refinement, which would hide an error of a factor's entry as long as it contracts.

The yardstick is the same elimination (pairs in the GPU's order, without pivoting) in NumPy in
the factor's precision.  Both are one algorithm with one growth of entries; they differ in the
order of the sums within a block only, so that their residuals are of one size: within 32 times,
or 16 units in the last place of the right-hand side.  An entry lost at the edge of a tile or
panel is off by its own size, seven (FP32) or sixteen (FP64) digits up."""
import numpy as np
import pytest
import scipy.linalg as sl

from oracle import ipm as oipm
from oracle.nlp import Problem as OProblem
from gpu_helpers import newton_system
from test_gpu_block_sizes import SIZES, _network
from test_static_pair_pivots import elimination_order

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def collo():
    from paper_2607_12201_gb300 import build
    build.build()
    from paper_2607_12201_gb300 import collo
    return collo


def _eliminated(K, p, rhs, dtype):
    """Solution of K x = rhs by pairs in the given order in dtype; the last p rows (parameters)
    in float64, their updates from dtype operands."""
    m = K.shape[0]
    c1 = m - p
    A = K.astype(dtype)
    S = K[c1:, c1:].copy()
    L = np.eye(m, dtype=dtype)
    D = []
    for c in range(0, c1, 2):
        P = A[c:c + 2, c:c + 2]
        det = P[0, 0] * P[1, 1] - P[0, 1] * P[0, 1]
        D.append(np.array([[P[1, 1], -P[0, 1]], [-P[0, 1], P[0, 0]]], dtype=dtype) / det)
        X = A[c + 2:, c:c + 2].copy()
        r = np.flatnonzero(X.any(axis=1))          # rows this pair touches
        Lb = X[r] @ D[-1]
        L[c + 2 + r, c:c + 2] = Lb
        A[np.ix_(c + 2 + r, c + 2 + r)] -= Lb @ X[r].T
        t = r[r + c + 2 >= c1]
        if t.size:
            at = t + c + 2 - c1
            S[np.ix_(at, at)] -= (Lb[r + c + 2 >= c1] @ X[t].T).astype(float)
    w = sl.solve_triangular(L[:c1, :c1], rhs[:c1].astype(dtype), lower=True, unit_diagonal=True)
    th = np.linalg.solve(S, rhs[c1:] - (L[c1:, :c1] @ w).astype(float)) if p else np.zeros(0)
    v = np.concatenate([Di @ w[2 * i:2 * i + 2] for i, Di in enumerate(D)])
    x = sl.solve_triangular(L[:c1, :c1].T, v - L[c1:, :c1].T @ th.astype(dtype), lower=False,
                            unit_diagonal=True)
    return np.concatenate([x.astype(float), th])


@pytest.mark.parametrize("scheme,n,r", SIZES)
def test_unrefined_residual_is_the_eliminations(collo, scheme, n, r):
    inst = _network(n, r, 3, scheme)    # three elements: reduction blocks with both neighbours
    oprob = OProblem(inst)
    x, lam, zl, zu, _ = oipm.initial_point(oprob, inst.theta0, oipm.Options())
    mu, dw = 0.1, 1.0
    dc = 1e-8 * mu ** 0.25
    ref = newton_system(oprob, x, lam, zl, zu, mu, dw, dc)
    rhs = ref["rhs"]
    K = ref["K"].toarray() if hasattr(ref["K"], "toarray") else np.asarray(ref["K"])
    perm = elimination_order(oprob, "radau3" if scheme == "radau" else "gauss4")

    def error(sol):
        return np.max(np.abs(rhs - K @ sol)) / np.max(np.abs(rhs))

    for name, dtype in (("MIXED", np.float32), ("FP64", np.float64)):
        sol = np.empty_like(rhs)
        sol[perm] = _eliminated(K[np.ix_(perm, perm)], oprob.p, rhs[perm], dtype)
        allowed = max(32 * error(sol), 16 * np.finfo(dtype).eps)
        for mode in (0, 1):
            with collo.Problem(inst, launch_mode=mode) as prob:
                prob.eval(x, lam)
                prob.kkt_factor(ref["sigma"], dw, dc, precision=getattr(collo, name))
                got, _ = prob.kkt_solve(rhs, refine_max=0)
            assert error(got) <= allowed, (name, mode, error(sol))
