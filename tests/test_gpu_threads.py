"""Problems of different sizes used at once from different host threads (each call's kernels
need another amount of shared memory): no call fails, and every result is the one the problem
gives alone."""
import threading

import numpy as np
import pytest
import torch

from paper_2607_12201_gb300 import workloads as W

pytestmark = pytest.mark.gpu

CALLS = 4000   # evaluations per thread: setting a kernel's limit per call failed some 30 of them


@pytest.fixture(scope="module")
def collo():
    from paper_2607_12201_gb300 import build
    build.build()
    from paper_2607_12201_gb300 import collo
    return collo


def _calls(prob, x, lam, theta):
    """An evaluation and a forward sweep."""
    out = [np.atleast_1d(v) for v in prob.eval(x, lam).values()]
    states, failures = prob.initial_states(theta)
    return out + [states, np.array([failures])]


def _step(collo, prob, x, lam):
    """A factorization and a solve (with one launch per phase: launch_mode 1)."""
    prob.eval_raw(x.ctypes.data, lam.ctypes.data)
    inertia = prob.kkt_factor(np.ones(prob.n_x), 1.0, 1e-8, precision=collo.MIXED)
    rhs = np.cos(np.arange(prob.n_x + prob.n_c))
    sol, _ = prob.kkt_solve(rhs, refine_max=1)
    return [np.array(inertia), sol]


@pytest.mark.parametrize("mode", [0, 1])
def test_threads_on_problems_of_different_sizes(collo, mode):
    jobs = []
    for n in (12, 40, 60):   # evaluation 24, 51, 57 KB; sweep below 16 KB, 25, 50 KB
        inst = W.random_network(n, 2 * n, n_obs=2, M=5, T=0.3, N=3, seed=700 + n,
                                theta0_spread=0.1)
        prob = collo.Problem(inst, launch_mode=mode)
        g = np.random.default_rng(n)
        x = g.uniform(0.2, 1.2, prob.n_x)
        x[prob.n_x - prob.p:] = inst.theta0
        lam = g.standard_normal(prob.n_c)
        jobs.append((prob, x, lam, np.asarray(inst.theta0, float)))
    step = _step if mode == 1 else (lambda *a: [])
    alone = [_calls(*j) + step(collo, *j[:3]) for j in jobs]
    dev = [[torch.as_tensor(v, device="cuda") for v in j[1:3]] for j in jobs]
    torch.cuda.synchronize()
    wrong, start = [], threading.Barrier(len(jobs))

    def loop(k):
        start.wait()
        for i in range(CALLS):
            try:
                jobs[k][0].eval_raw(dev[k][0].data_ptr(), dev[k][1].data_ptr())
                if i % 40:
                    continue
                got = _calls(*jobs[k]) + step(collo, *jobs[k][:3])
                if any(not np.array_equal(a, b) for a, b in zip(got, alone[k])):
                    wrong.append((k, i, "result differs"))
            except collo.ColloError as e:
                wrong.append((k, i, str(e)))

    threads = [threading.Thread(target=loop, args=(k,)) for k in range(len(jobs))]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    for j in jobs:
        j[0].close()
    assert not wrong, wrong[:5]
