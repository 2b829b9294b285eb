"""Collocation forward sweep at the sizes where its kernel changes: one and two unknowns per
lane, the block sizes (32 / 64 unknowns), every register tile of the kept inverse (96, 128,
160, 192) and the matrix in memory above, on both schemes and over several experimental
conditions; and meshes so coarse that elements are given up."""
import dataclasses

import numpy as np
import pytest

from paper_2607_12201_gb300 import workloads as W
from oracle.init import forward_sweep
from oracle.nlp import Problem as OProblem

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def collo():
    from paper_2607_12201_gb300 import build
    build.build()
    from paper_2607_12201_gb300 import collo
    return collo


def _check(collo, inst, theta):
    x, failures = None, None
    with collo.Problem(inst) as prob:
        x, failures = prob.initial_states(theta)
    z, nfail = forward_sweep(OProblem(inst), theta)
    z = np.asarray(z).reshape(-1)
    # both stop at a correction of 1e-12 max(1, |Z|) per element, and an element's error is
    # carried by the relaxing network without growth: N elements, two sides
    N = inst.N * inst.Nc
    assert failures == nfail
    assert np.max(np.abs(x[:z.size] - z)) <= 2e-12 * N * max(1.0, np.max(np.abs(z)))
    assert np.array_equal(x[z.size:], theta)


@pytest.mark.parametrize("scheme,n", [("radau", n) for n in (1, 10, 11, 21, 22, 32, 33, 42, 43,
                                                             53, 54, 64, 65)]
                         + [("gauss", n) for n in (1, 8, 9, 16, 17, 24, 40, 41, 48, 49)])
def test_sweep_matches_oracle_at_every_tile(collo, scheme, n):
    N = 12
    inst = W.random_network(n, 2 * n, n_obs=min(2, n), M=5, T=0.05 * N, N=N, seed=300 + n,
                            theta0_spread=0.1)
    if scheme == "gauss":
        inst = dataclasses.replace(inst, K=4, scheme="gauss")
    _check(collo, inst, inst.theta0)


def test_sweep_over_conditions_and_cascade(collo):
    inst = W.multi_condition(n=6, r=12, Nc=3, N=15, T=1.5, seed=1006)
    _check(collo, inst, inst.theta0)
    inst = W.linear_cascade(N=25, T=10.0)
    _check(collo, inst, inst.theta0)


@pytest.mark.parametrize("n,T,N,seed", [(27, 20.0, 4, 58), (15, 20.0, 4, 46)])
def test_sweep_gives_up_the_same_elements(collo, n, T, N, seed):
    """Elements of five units of time against rate constants up to 60: Newton's method fails
    on some or all of them, and they keep the constant guess."""
    inst = W.random_network(n, 2 * n, n_obs=4, M=20, T=T, N=N, seed=seed, theta0_spread=0.8)
    _check(collo, inst, inst.theta0)
