"""Substitutions of a batch against the same problems alone: how many blocks a launch has, and
how large its largest one is, decide how many panels are in flight and how many CUDA blocks share
an SM, for narrow blocks (one warp) and wide ones; the arithmetic of a block stays the same, so
its problem's result does bit for bit."""
import numpy as np
import pytest

from paper_2607_12201_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def collo():
    from paper_2607_12201_gb300 import build
    build.build()
    from paper_2607_12201_gb300 import collo
    return collo


def _instance(n, N):
    if n == 2:
        return W.linear_cascade(N=N, T=0.1 * N)
    return W.random_network(n, 2 * n, n_obs=2, M=10, T=0.1 * N, N=N, seed=1100 + n,
                            theta0_spread=0.05)


def _solve(collo, insts, prec):
    probs = [collo.Problem(i) for i in insts]
    res = collo.batch_solve(probs, [i.theta0 for i in insts], want_x=True, precision=prec,
                            max_iter=2, refine_tol=1e-13, refine_max=3)
    for p in probs:
        p.close()
    return [(r["x"], r["lam"], r["iterations"]) for r in res]


# the problems looked at: narrow; narrow elements at the limit of a warp; wide elements with
# narrow and wide reduction blocks
LOOKED_AT = [(2, 7), (6, 40), (12, 33), (13, 21), (16, 30), (22, 17)]
# what else is in the batch: nothing; many narrow elements; many wide ones whose largest leaves
# room for two CUDA blocks per SM, with few or more panels; wide ones between; all of them
OTHERS = [[], [(10, 5000)], [(13, 700)], [(27, 700)], [(27, 1300)], [(50, 650)],
          [(10, 5000), (33, 1300)]]


# FP64 up to 27 species: the shared-memory sizes repeat at half the rows
CASES = [(i, "MIXED") for i in range(len(OTHERS))] + \
        [(i, "FP64") for i, o in enumerate(OTHERS) if all(n <= 27 for n, _ in o)]


@pytest.mark.parametrize("others,prec", CASES)
def test_batch_gives_each_problem_its_own_result(collo, others, prec):
    prec = getattr(collo, prec)
    looked_at = [_instance(*c) for c in LOOKED_AT]
    alone = [_solve(collo, [i], prec)[0] for i in looked_at]
    mixed = _solve(collo, looked_at + [_instance(*c) for c in OTHERS[others]], prec)
    for (x, lam, its), (xm, lamm, itsm), case in zip(alone, mixed, LOOKED_AT):
        assert its == itsm and np.array_equal(x, xm) and np.array_equal(lam, lamm), case
