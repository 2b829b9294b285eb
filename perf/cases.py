"""What the library is timed on: Newton steps, evaluations, forward sweeps and batched
solves of mass-action networks over the size ranges of the repository's configurations.

Every case goes through the public binding (``paper_2607_12201_gb300.collo``):

* ``step``: one interior-point Newton step of one problem, the three calls a driver of
  its own makes per iteration: evaluate at (x, lambda), factor the KKT matrix, solve with
  refinement.  Vectors are device tensors, as such a driver keeps them.
* ``eval``: all derivative arrays into caller-owned device buffers.
* ``sweep``: the collocation forward sweep that gives a solve its initial states.
* ``solve``: the first Newton iterations of a batched solve (multistart of one network,
  or networks of uneven sizes) from starts near a known fit, each step refined to the
  rounding level, from parameters to the iterates on the host.

The networks are the seeded generators of ``workloads``; a case's network is fixed by its
``net`` value and the seed moves the iterate, the multipliers and the starts.
"""
import dataclasses
import math

import numpy as np
import torch

from paper_2607_12201_gb300 import collo
from paper_2607_12201_gb300 import workloads as W

# A step's regularisation delta_w (what an inertia correction ends at; delta_c is the barrier
# method's at mu), the size of its multipliers, and the noise floor of the measurements.
DELTA_W, LAMBDA, NOISE_FLOOR = 1.0, 0.1, 1e-2
PREC = {"fp64": collo.FP64, "mixed": collo.MIXED}


def listed():
    return [
        # the smallest problem users start with: two species, 50 elements; launches and
        # host work decide it
        dict(name="step_cascade", kind="step", n=2, N=50, scheme="radau", prec="fp64", net=1001),
        # the multistart network (10 species, 20 parameters, 400 elements), one Newton step
        # of one solve, on Radau and on the paper's Gauss-Legendre points
        dict(name="step_n10", kind="step", n=10, N=400, scheme="radau", prec="mixed", net=3),
        dict(name="step_n10_gauss", kind="step", n=10, N=400, scheme="gauss", prec="mixed", net=3),
        # a network measured under three experimental conditions sharing theta
        dict(name="step_conditions", kind="step", n=6, N=30, scheme="radau", prec="mixed",
             conditions=3, net=1006),
        # the median and the largest network of the uneven multistart batch
        dict(name="step_n27", kind="step", n=27, N=415, scheme="radau", prec="mixed", net=4027),
        dict(name="step_n50", kind="step", n=50, N=2000, scheme="radau", prec="mixed", net=4001),
        # the plain FP64 path (no refinement to fall back on)
        dict(name="step_n20_fp64", kind="step", n=20, N=333, scheme="radau", prec="fp64", net=4020),
        # derivatives for a solver of the user's own
        dict(name="eval_n30", kind="eval", n=30, N=2000, scheme="radau", net=1030),
        # initial states of a start
        dict(name="sweep_n10", kind="sweep", n=10, N=400, scheme="radau", net=3),
        dict(name="sweep_n27", kind="sweep", n=27, N=415, scheme="radau", net=4027),
        # 32 starts of the multistart network solved together, first iterations
        dict(name="solve_multistart", kind="solve", n=10, N=400, scheme="radau", prec="mixed",
             starts=32, iters=4, net=3),
        # networks of uneven sizes solved together, first iterations
        dict(name="solve_uneven", kind="solve", n=50, N=300, scheme="radau", prec="mixed",
             starts=24, iters=3, uneven=True, net=606),
    ]


def _logint(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """A case of the same ranges: n 2..50 species, 1..2000 elements."""
    kind = rng.choice(["step", "step", "step", "step", "eval", "sweep", "solve"])
    n, net = _logint(rng, 2, 50), rng.randrange(1 << 20)
    scheme = rng.choice(["radau", "radau", "gauss"])
    prec = rng.choice(["mixed", "mixed", "fp64"])
    N = _logint(rng, 1, 2000)
    if kind == "eval":
        return dict(kind=kind, n=n, N=N, scheme=scheme, net=net)
    if kind == "sweep":   # sequential over the elements
        return dict(kind=kind, n=n, N=min(N, 12000 // n), scheme=scheme, net=net)
    if kind == "solve":
        if rng.random() < 0.5:
            return dict(kind=kind, n=max(n, 5), N=_logint(rng, 100, 300), scheme=scheme,
                        prec="mixed", starts=rng.randint(2, 12), iters=1, uneven=True, net=net)
        n = min(n, 12)
        return dict(kind=kind, n=n, N=max(20, min(N, 4000 // n)), scheme=scheme, prec="mixed",
                    starts=rng.randint(1, 40), iters=rng.randint(1, 2), net=net)
    if prec == "fp64":
        n = min(n, 32)
        N = min(N, 8000 // n)
    if scheme == "gauss":
        N = min(N, 40000 // n)
    c = dict(kind=kind, n=n, N=N, scheme=scheme, prec=prec, net=net)
    if n <= 12 and rng.random() < 0.3:
        c.update(conditions=rng.randint(2, 4), N=max(1, min(N, 200)))
    return c


# ---- problems -------------------------------------------------------------------------

def _instance(case, n=None, N=None, net=None):
    n, N, net = n or case["n"], N or case["N"], case["net"] if net is None else net
    # meshes below 200 elements cover a shorter horizon, so that an element stays short
    # against the fastest reactions (10 per unit of time)
    T = min(20.0, 0.1 * N)
    if n == 2:
        inst = W.linear_cascade(N=N, T=min(10.0, T), seed=net)
    elif case.get("conditions"):
        inst = W.multi_condition(n=n, r=2 * n, Nc=case["conditions"], N=N, T=T, seed=net)
    else:
        inst = W.random_network(n, 2 * n, n_obs=min(4, n), M=50, T=T, N=N, seed=net,
                                theta0_spread=0.1)
    inst = dataclasses.replace(inst, obs_sigma=np.maximum(inst.obs_sigma, NOISE_FLOOR))
    if case["scheme"] == "gauss":
        inst = dataclasses.replace(inst, K=4, scheme="gauss")
    return inst


def _tables(K, gauss):
    """Interpolation points tau, derivative matrix D[k][j] = l_j'(tau_k), end weights b."""
    if gauss:
        x, _ = np.polynomial.legendre.leggauss(K)
        tau = np.concatenate([[0.0], (x + 1) / 2])
    else:
        tau = np.array([0.0, (4 - math.sqrt(6)) / 10, (4 + math.sqrt(6)) / 10, 1.0])
    w = np.array([1 / np.prod([a - b for b in tau if b != a]) for a in tau])
    D = np.array([[w[j] / w[k] / (tau[k] - tau[j]) if j != k else 0.0 for j in range(K + 1)]
                  for k in range(K + 1)])
    D -= np.diag(D.sum(1))
    if gauss:
        b = np.array([np.prod([(1 - c) / (a - c) for c in tau if c != a]) for a in tau])
    else:
        b = np.array([0.0] * K + [1.0])
    return tau, D, b


def _iterate(inst, seed):
    """An iterate as a solve meets it: rate constants near the truth, positive states that
    relax from the initial state to some level (not on a trajectory: the constraints are
    violated), multipliers of order one, barrier terms of the parameters' bounds."""
    g = np.random.default_rng([int(seed), inst.seed, inst.N, inst.n])
    n, K, Nc = inst.n, inst.K, inst.Nc
    tau, _, _ = _tables(K, inst.scheme == "gauss")
    t = (np.arange(inst.N)[:, None] + tau[None]) * (inst.T / inst.N)
    x0 = inst.x0[None] if inst.cond_x0 is None else inst.cond_x0
    end = g.uniform(0.05, 1.0, (Nc, n))
    rate = np.exp(g.uniform(math.log(1 / inst.T), math.log(20 / inst.T), (Nc, n)))
    f = np.exp(-t[None, :, :, None] * rate[:, None, None])
    z = x0[:, None, None] * f + end[:, None, None] * (1 - f)
    z = z * (1 + 0.01 * g.standard_normal(z.shape))
    spread = 0.2 if inst.logscale else 0.1
    th = inst.theta_true + g.uniform(-spread, spread, inst.p)
    zl, zu, mu = g.uniform(0.5, 2.0, inst.p), g.uniform(0.5, 2.0, inst.p), 0.05
    sl, su = th - inst.theta_lo, inst.theta_hi - th
    sigma = np.concatenate([np.zeros(z.size), zl / sl + zu / su])
    bar = -mu / sl + mu / su
    lam = LAMBDA * g.standard_normal(z.size)
    return np.concatenate([z.reshape(-1), th]), lam, sigma, bar, mu


# ---- the NLP in plain torch (right-hand sides and exact values) -------------------------

class _Model:
    """Residuals and derivative blocks of the collocation NLP, float64, in the layouts of
    collo_eval (elements of all conditions, K points each)."""

    def __init__(self, inst, dev):
        self.inst, self.dev = inst, dev
        f = lambda a: torch.as_tensor(np.ascontiguousarray(a, dtype=np.float64), device=dev)
        self.f = f
        n, r, p = inst.n, inst.r, inst.p
        nu, ra, rb = np.zeros((n, r)), np.zeros((r, n)), np.zeros((r, n))
        for j in range(r):
            for k in range(2):
                if inst.react[j, k] >= 0:
                    nu[inst.react[j, k], j] -= 1
                if inst.prod[j, k] >= 0:
                    nu[inst.prod[j, k], j] += 1
            ra[j, inst.react[j, 0]] = 1
            if inst.react[j, 1] >= 0:
                rb[j, inst.react[j, 1]] = 1
        Q = np.zeros((r, p))
        for j in range(r):
            if inst.pidx[j] >= 0:
                Q[j, inst.pidx[j]] = 1
        self.nu, self.ra, self.rb, self.Q = f(nu), f(ra), f(rb), f(Q)
        self.two = f((inst.react[:, 1] >= 0).astype(float))
        self.est = f((inst.pidx >= 0).astype(float))
        self.kfix = f(inst.kfix)
        tau, D, b = _tables(inst.K, inst.scheme == "gauss")
        self.tau, self.D, self.b = tau, f(D), f(b)
        self.h = inst.T / inst.N
        self.E, self.Nc = inst.N * inst.Nc, inst.Nc
        sc = np.ones((inst.Nc, r)) if inst.cond_scale is None else inst.cond_scale
        self.scale = f(np.repeat(sc, inst.N, axis=0))                      # [E, r]
        self.x0 = f(inst.x0[None] if inst.cond_x0 is None else inst.cond_x0)
        cond = np.zeros(inst.M, dtype=np.int64) if inst.obs_cond is None else inst.obs_cond
        el, w = [], []
        for m in range(inst.M):
            u = inst.obs_t[m] * inst.N / inst.T
            i = min(max(math.ceil(u) - 1, 0), inst.N - 1)
            s = u - i
            w.append([np.prod([(s - c) / (a - c) for c in tau if c != a]) for a in tau])
            el.append(int(cond[m]) * inst.N + i)
        self.oe = torch.as_tensor(np.array(el, dtype=np.int64), device=dev)
        self.os = torch.as_tensor(np.array(inst.obs_s, dtype=np.int64), device=dev)
        self.ow = f(np.array(w).reshape(inst.M, inst.K + 1))
        self.oy, self.og = f(inst.obs_y), f(inst.obs_sigma)

    def __call__(self, x, lam):
        i, h = self.inst, self.h
        n, p, K, E = i.n, i.p, i.K, self.E
        z, th = x[:E * (K + 1) * n].reshape(E, K + 1, n), x[E * (K + 1) * n:]
        la = lam.reshape(E, K + 1, n)
        t = self.Q @ th
        if i.logscale:
            k0, l10 = 10.0 ** t, math.log(10.0)
            k1, k2 = l10 * k0, l10 * l10 * k0
        else:
            k0, k1, k2 = t, torch.ones_like(t), torch.zeros_like(t)
        kr = (self.est * k0 + (1 - self.est) * self.kfix) * self.scale      # [E, r]
        dk, d2k = self.est * k1 * self.scale, self.est * k2 * self.scale
        zk = z[:, 1:]
        za, zb = zk @ self.ra.T, zk @ self.rb.T                               # [E, K, r]
        da = torch.where(self.two > 0, zb, torch.ones_like(zb))
        db = za * self.two
        mon = za * da
        om = la[:, 1:] @ self.nu                                              # [E, K, r]
        o = {}
        c = torch.empty_like(z)
        c[:, 1:] = torch.einsum("kj,ejs->eks", self.D[1:], z) - h * (kr[:, None] * mon) @ self.nu.T
        prev = torch.einsum("j,ejs->es", self.b, z).roll(1, 0)
        prev[::i.N] = self.x0
        c[:, 0] = z[:, 0] - prev
        o["c"] = c.reshape(-1)
        dmon = da[..., None] * self.ra + db[..., None] * self.rb              # [E, K, r, n]
        o["jac_z"] = -h * torch.einsum("sr,er,ekrt->ekst", self.nu, kr, dmon)
        o["jac_theta"] = -h * torch.einsum("sr,er,ekr,rq->eksq", self.nu, dk, mon, self.Q)
        pair = self.ra[:, :, None] * self.rb[:, None, :]
        pair = pair + pair.transpose(1, 2)
        ck = om * kr[:, None]
        o["hess_zz"] = -h * torch.einsum("ekr,rtu->ektu", ck, pair)
        o["hess_ztheta"] = -h * torch.einsum("ekr,er,ekrt,rq->ektq", om, dk, dmon, self.Q)
        o["hess_thth"] = -h * torch.einsum("ekr,er,ekr,rq->q", om, d2k, mon, self.Q)
        yh = (self.ow * z[self.oe, :, self.os]).sum(1)
        res = (yh - self.oy) / self.og
        o["phi"] = 0.5 * (res * res).sum().reshape(1)
        gz = torch.zeros_like(z)
        gz.index_put_((self.oe[:, None], torch.arange(K + 1, device=self.dev)[None],
                       self.os[:, None]), self.ow * (res / self.og)[:, None], accumulate=True)
        o["grad"] = torch.cat([gz.reshape(-1), torch.zeros_like(th)])
        wo = torch.zeros(E, n, K + 1, K + 1, dtype=z.dtype, device=self.dev)
        wo.index_put_((self.oe, self.os), self.ow[:, :, None] * self.ow[:, None, :]
                      / (self.og ** 2)[:, None, None], accumulate=True)
        o["hess_obj"] = wo
        return o

    def jt(self, o, v):
        """J^T v as [states, parameters]."""
        i = self.inst
        v = v.reshape(self.E, i.K + 1, i.n)
        y = torch.einsum("kj,eks->ejs", self.D[1:], v[:, 1:])
        y[:, 1:] += torch.einsum("ekst,eks->ekt", o["jac_z"], v[:, 1:])
        y[:, 0] += v[:, 0]
        nxt = v[:, 0].roll(-1, 0)
        nxt[i.N - 1::i.N] = 0
        y -= self.b[None, :, None] * nxt[:, None]
        return torch.cat([y.reshape(-1), torch.einsum("eksq,eks->q", o["jac_theta"], v[:, 1:])])

    def rhs(self, o, lam, bar):
        """The Newton right-hand side -[grad phi_mu + J^T lambda; c]."""
        g = o["grad"] + self.jt(o, lam)
        g[g.numel() - self.inst.p:] += self.f(bar)
        return -torch.cat([g, o["c"]])

    def solve(self, o, sigma, dw, dc, rhs):
        """K^-1 rhs by block elimination along the elements (dense blocks with partial
        pivoting), the parameters last, refined once; order of an element's unknowns:
        states [K + 1][n], multipliers [K + 1][n]."""
        i = self.inst
        n, p, K, E = i.n, i.p, i.K, self.E
        half = (K + 1) * n
        m = 2 * half
        M = torch.zeros(E, m, m, dtype=rhs.dtype, device=self.dev)
        eye = torch.eye(n, dtype=rhs.dtype, device=self.dev)
        st = lambda j: slice(j * n, (j + 1) * n)
        du = lambda j: slice(half + j * n, half + (j + 1) * n)
        s = torch.arange(n, device=self.dev)
        for j in range(K + 1):
            for l in range(K + 1):
                M[:, j * n + s, l * n + s] += o["hess_obj"][:, :, j, l]
                if j:
                    M[:, du(j), st(l)] += self.D[j, l] * eye
            if j:
                M[:, st(j), st(j)] += o["hess_zz"][:, j - 1]
                M[:, du(j), st(j)] += o["jac_z"][:, j - 1]
            else:
                M[:, du(0), st(0)] += eye
        M[:, :half, half:] = M[:, half:, :half].transpose(1, 2)
        d = torch.arange(half, device=self.dev)
        M[:, d, d] += sigma[:E * half].reshape(E, half) + dw
        M[:, half + d, half + d] -= dc
        B = torch.zeros(E, m, p, dtype=rhs.dtype, device=self.dev)
        for j in range(1, K + 1):
            B[:, st(j)], B[:, du(j)] = o["hess_ztheta"][:, j - 1], o["jac_theta"][:, j - 1]
        # row c0 of element e on the states of element e - 1: -b_j
        C = torch.zeros(n, m, dtype=rhs.dtype, device=self.dev)
        for j in range(K + 1):
            C[:, st(j)] = -self.b[j] * eye
        nx = E * half + p
        Th = torch.diag(o["hess_thth"] + sigma[E * half:] + dw)
        linked = [e % i.N != 0 for e in range(E)]   # e is coupled to e - 1

        def split(v):
            return torch.cat([v[:E * half].reshape(E, half), v[nx:].reshape(E, half)], 1)

        # forward: A_e = M_e - C X_(e-1) C^T on the c0 rows, X_e = A_e^-1 [C^T | B_e]
        fac, X, R = [], [], []
        S, Bc = Th.clone(), None
        for e in range(E):
            A, b = M[e].clone(), B[e].clone()
            if linked[e]:
                k = C @ X[-1]
                A[du(0), du(0)] -= k[:, :n]
                b[du(0)] -= k[:, n:]
            lu = torch.linalg.lu_factor(A)
            fac.append(lu)
            R.append(b)
            X.append(torch.linalg.lu_solve(*lu, torch.cat([C.T, b], 1)))
            S -= b.T @ X[-1][:, n:]
        Slu = torch.linalg.lu_factor(S)

        def apply(v):
            w, t = split(v), v[E * half:nx].clone()
            ys, y = [], None
            for e in range(E):
                u = w[e].clone()
                if linked[e]:
                    u[du(0)] -= C @ y
                y = torch.linalg.lu_solve(*fac[e], u[:, None])[:, 0]
                ys.append(y)
                t -= R[e].T @ y
            th = torch.linalg.lu_solve(*Slu, t[:, None])[:, 0]
            out = torch.empty(E, m, dtype=v.dtype, device=self.dev)
            for e in range(E - 1, -1, -1):
                q = ys[e] - X[e][:, n:] @ th
                if e + 1 < E and linked[e + 1]:
                    q -= X[e][:, :n] @ out[e + 1, du(0)]
                out[e] = q
            return torch.cat([out[:, :half].reshape(-1), th, out[:, half:].reshape(-1)])

        def mul(v):
            w, th = split(v), v[E * half:nx]
            y = torch.einsum("eab,eb->ea", M, w) + torch.einsum("eaq,q->ea", B, th)
            for e in range(1, E):
                if linked[e]:
                    y[e, du(0)] += C @ w[e - 1]
                    y[e - 1] += C.T @ w[e, du(0)]
            t = Th @ th + torch.einsum("eaq,ea->q", B, w)
            return torch.cat([y[:, :half].reshape(-1), t, y[:, half:].reshape(-1)])

        v = apply(rhs)
        return v + apply(rhs - mul(v))


# ---- prepare / run ----------------------------------------------------------------------



_stream = None


def _eval_stream():
    """One stream for every evaluation without allocation: they share a scratch array."""
    global _stream
    if _stream is None:
        _stream = torch.cuda.Stream()
    return _stream.cuda_stream


def _cuda(a):
    return torch.as_tensor(np.ascontiguousarray(a, dtype=np.float64), device="cuda")


def prepare(case, seed):
    kind = case["kind"]
    if kind == "solve":
        g = np.random.default_rng([int(seed), case["net"], case["starts"]])
        if case.get("uneven"):
            # sizes over the case's range, every batch the same sizes
            q = np.random.default_rng([case["net"], case["starts"], case["n"]])
            insts = []
            for j in range(case["starts"]):
                n = int(q.integers(5, case["n"] + 1))
                N = int(round(math.exp(q.uniform(math.log(100), math.log(case["N"])))))
                insts.append(_instance(case, n=n, N=N, net=case["net"] + 17 * j))
        else:
            insts = [_instance(case)] * case["starts"]
        probs = [collo.Problem(i) for i in insts]
        starts = [i.theta_true + g.uniform(-0.02, 0.02, i.p) for i in insts]
        return dict(case=case, probs=probs, starts=starts)
    inst = _instance(case)
    prob = collo.Problem(inst)
    if kind == "sweep":
        g = np.random.default_rng([int(seed), case["net"]])
        th = inst.theta_true + g.uniform(-0.1, 0.1, inst.p)
        return dict(case=case, prob=prob, theta=th)
    x, lam, sigma, bar, mu = _iterate(inst, seed)
    x, lam, sigma = _cuda(x), _cuda(lam), _cuda(sigma)
    if kind == "eval":
        n, p, E, K = inst.n, inst.p, prob.N, inst.K
        shapes = dict(phi=(1,), c=(prob.n_c,), grad=(prob.n_x,), jac_z=(E, K, n, n),
                      jac_theta=(E, K, n, p), hess_zz=(E, K, n, n), hess_ztheta=(E, K, n, p),
                      hess_thth=(p,), hess_obj=(E, n, K + 1, K + 1))
        out = {k: torch.empty(s, dtype=torch.float64, device="cuda") for k, s in shapes.items()}
        return dict(case=case, prob=prob, x=x, lam=lam, out=out,
                    ptr={k: v.data_ptr() for k, v in out.items()})
    model = _Model(inst, "cuda")
    rhs = model.rhs(model(x, lam), lam, bar)
    sol = torch.empty(prob.n_x + prob.n_c, dtype=torch.float64, device="cuda")
    torch.cuda.synchronize()
    return dict(case=case, prob=prob, x=x, lam=lam, sigma=sigma, rhs=rhs, sol=sol,
                dc=1e-8 * mu ** 0.25)


def run(s):
    case = s["case"]
    kind = case["kind"]
    if kind == "step":
        prob = s["prob"]
        prob.eval_raw(s["x"].data_ptr(), s["lam"].data_ptr())
        inertia = prob.kkt_factor(s["sigma"], DELTA_W, s["dc"], precision=PREC[case["prec"]])
        sol, _ = prob.kkt_solve(s["rhs"], out=s["sol"])
        return dict(sol=sol, inertia=list(inertia))
    if kind == "eval":
        s["prob"].eval_noalloc(s["x"].data_ptr(), s["lam"].data_ptr(), s["ptr"],
                               stream=_eval_stream())
        return s["out"]
    if kind == "sweep":
        x, failures = s["prob"].initial_states(s["theta"])
        return dict(x=x, failures=failures)
    res = collo.batch_solve(s["probs"], s["starts"], want_x=True, precision=PREC[case["prec"]],
                            max_iter=case["iters"], tol=1e-8, refine_tol=1e-13, refine_max=20)
    return dict(x=np.concatenate([r["x"] for r in res]),
                lam=np.concatenate([r["lam"] for r in res]),
                phi=np.array([r["phi"] for r in res]),
                iterations=np.array([r["iterations"] for r in res]))


# ---- what a pass cannot do without --------------------------------------------------------

def _sizes(case):
    if case["kind"] == "solve" and case.get("uneven"):
        q = np.random.default_rng([case["net"], case["starts"], case["n"]])
        got = []
        for _ in range(case["starts"]):
            n = int(q.integers(5, case["n"] + 1))
            got.append((n, int(round(math.exp(q.uniform(math.log(100), math.log(case["N"])))))))
        return got
    return [(case["n"], case["N"] * case.get("conditions", 1))] * case.get("starts", 1)


def _pairs(t0, q):
    """Multiply-adds of eliminating q pairs from a symmetric block of t0 rows, as flops."""
    return sum(2.0 * t * (t + 1) + 8.0 * t for t in (t0 - 2 * j - 2 for j in range(q)))


def work(case):
    """Each input read and each output written once; the flops of the element and chain
    eliminations, the substitutions and, for a sweep, one LU factorization per element."""
    K = 4 if case["scheme"] == "gauss" else 3
    byt = flops = 0.0
    for n, N in _sizes(case):
        p = 2 if n == 2 else 2 * n
        half = (K + 1) * n
        ext, bext = 2 * half + p, 4 * n + p
        fac = N * (_pairs(ext, K * n) + _pairs(bext, n))
        sub = N * 4.0 * (2 * K * n * ext + 2 * n * bext)
        blocks = N * (2 * K * n * (n + p) + half * (K + 1))
        vec = N * half * 8.0
        if case["kind"] == "step":
            byt, flops = byt + 8 * vec, flops + fac + sub
        elif case["kind"] == "eval":
            byt, flops = byt + 8.0 * blocks + 4 * vec, flops + 4.0 * N * K * 2 * n * 20
        elif case["kind"] == "sweep":
            byt, flops = byt + vec, flops + N * 2 / 3 * (K * n) ** 3
        else:
            byt += 3 * vec
            flops += N * 2 / 3 * (K * n) ** 3 + case["iters"] * (fac + sub)
    return {"bytes": byt, "flops": flops}


# ---- exact values ---------------------------------------------------------------------

def _sweep_exact(inst, th):
    """Newton's method on each element's collocation equations in turn, from the state at
    its start, float64 on the host."""
    m = _Model(inst, "cpu")
    nu, ra, rb, two = (a.numpy() for a in (m.nu, m.ra, m.rb, m.two))
    D, b, K, n, h = m.D.numpy(), m.b.numpy(), inst.K, inst.n, m.h
    t = m.Q.numpy() @ th
    k = np.where(inst.pidx >= 0, 10.0 ** t if inst.logscale else t, inst.kfix)
    z0, out = inst.x0.copy(), []
    lin = np.kron(D[1:, 1:], np.eye(n))
    for _ in range(inst.N):
        Z = np.tile(z0, (K, 1))
        for _ in range(30):
            za, zb = Z @ ra.T, Z @ rb.T
            da, db = np.where(two > 0, zb, 1.0), za * two
            G = np.outer(D[1:, 0], z0) + D[1:, 1:] @ Z - h * (za * da * k) @ nu.T
            J = lin.copy()
            for q in range(K):
                sl = slice(q * n, (q + 1) * n)
                J[sl, sl] -= h * (nu * k) @ (da[q][:, None] * ra + db[q][:, None] * rb)
            dZ = np.linalg.solve(J, G.reshape(-1)).reshape(K, n)
            Z = Z - dZ
            if np.abs(dZ).max() <= 1e-14 * max(1.0, np.abs(Z).max()):
                break
        out.append(np.concatenate([z0[None], Z]))
        z0 = Z[-1].copy() if inst.scheme != "gauss" else b[0] * z0 + b[1:] @ Z
    return np.concatenate([np.array(out).reshape(-1), th])


def exact(case, seed):
    kind = case["kind"]
    if kind == "solve":
        return None   # a filter line search over several systems: minutes in numpy
    inst = _instance(case)
    if kind == "sweep":
        g = np.random.default_rng([int(seed), case["net"]])
        return dict(x=_sweep_exact(inst, inst.theta_true + g.uniform(-0.1, 0.1, inst.p)),
                    failures=None)
    x, lam, sigma, bar, mu = _iterate(inst, seed)
    x, lam, sigma = _cuda(x), _cuda(lam), _cuda(sigma)
    model = _Model(inst, "cuda")
    o = model(x, lam)
    if kind == "eval":
        return o
    half = (inst.K + 1) * inst.n
    if float(2 * half) ** 3 * model.E > 3e10:
        return None   # over 20 s of dense blocks one after another
    rhs = model.rhs(o, lam, bar)
    return dict(sol=model.solve(o, sigma, DELTA_W, 1e-8 * mu ** 0.25, rhs), inertia=None)
