"""The forward sweep ends at rounding level: what an element leaves of its iteration adds up
along the chain, so it has to stay below the rounding of its states."""
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


@pytest.mark.parametrize("n,N,seed", [(10, 400, 3), (11, 400, 1011), (27, 120, 77),
                                      (27, 415, 4027), (50, 80, 4001), (66, 60, 66)])
def test_sweep_is_as_exact_as_newtons_method(collo, n, N, seed):
    """Relaxing networks: an element's error is carried on without growth.  An element leaves
    the rounding of its residual and of its states, an ulp of the largest state each, on
    both sides (the oracle's Newton iteration leaves nothing else): 2 sides x N x 2 x 2^-53.
    An iteration ended by an estimate from its last step alone left five times that at 27
    species, 120 elements."""
    inst = W.random_network(n, 2 * n, n_obs=4, M=50, T=min(20.0, 0.1 * N), N=N, seed=seed,
                            theta0_spread=0.1)
    theta = inst.theta_true + np.random.default_rng([5, seed]).uniform(-0.1, 0.1, inst.p)
    z, nfail = forward_sweep(OProblem(inst), theta)
    z = np.asarray(z).reshape(-1)
    with collo.Problem(inst) as prob:
        x, failures = prob.initial_states(theta)
    assert failures == nfail
    assert np.max(np.abs(x[:z.size] - z)) <= 4 * N * 2.0 ** -53 * max(1.0, np.max(np.abs(z)))
