"""The work that users of the library have it do, as timed cases.

Every case goes through the public entry points of ``paper_2012_12419_gb300``: whole solves
(implicit, stored and user-supplied matrices, batches), policy evaluation, the differentiable
objective, the end-to-end host call and one sweep of a control loop.  Sizes are those of
``inputs.WORKLOADS``, the tests and the bench; model rates come from the seed.

``exact`` recomputes each result in FP64 with plain torch operations: value iteration with
every self-transition solved (the same fixed point) run down to rounding, a fixed-point
adjoint, and torch's own differentiation of the rates.
"""
from __future__ import annotations

import math

import torch

from paper_2012_12419_gb300 import autograd, inputs, native

GAMMAS = (0.9, 0.95, 0.99)


def _solve(name, H, C, Q, gamma=0.95, fmt="implicit", padded=False, sliced=False, self_loop=False, accurate=False):
    return dict(name=name, kind="solve", H=H, C=C, Q=Q, gamma=gamma, fmt=fmt, padded=padded, sliced=sliced,
                self_loop=self_loop, accurate=accurate)


def listed():
    return [
        # a road-side unit re-solving its own small cell: latency and launches count
        _solve("solve_tiny", 3, 3, 4),
        # a large cell, successors generated in registers: the fastest way to one solve
        _solve("solve_large", 7, 4, 15),
        # long horizon, error certificate and exact self-transitions; 22 states per host state
        _solve("solve_accurate_self", 6, 4, 10, gamma=0.99, self_loop=True, accurate=True),
        # the bench's headline: the large cell as a stored (padded) matrix with its sliced copy
        _solve("solve_large_matrix", 7, 4, 15, fmt="csr_f32", padded=True, sliced=True),
        # the largest stored matrix, BF16 probabilities with FP64 refinement
        _solve("solve_bf16_matrix", 8, 4, 15, fmt="csr_bf16", padded=True, sliced=True),
        # an explicit MDP of the user's own, ragged rows and scattered successors
        dict(name="solve_user_matrix", kind="user", S=200003, A=5, succ=12, gamma=0.95, bf16=False),
        # hundreds of uneven cells solved together
        dict(name="batch_512", kind="batch", n=512, sizes=2, self_loop=False),
        # the cells of one road, self-transitions solved
        dict(name="batch_48_self", kind="batch", n=48, sizes=7, self_loop=True),
        # one step of fitting rates: objective forward, gradient backward
        dict(name="train_step", kind="train", H=6, C=4, Q=10, gamma=0.95),
        # the greedy heuristic's values, for comparison with the optimum
        dict(name="evaluate_greedy", kind="evaluate", H=7, C=3, Q=15, gamma=0.95),
        # host parameters in, host values and policy out, instance built on the way
        dict(name="end_to_end", kind="end_to_end", H=5, C=4, Q=15, gamma=0.95, fmt="csr_f32", padded=True),
        # one sweep of a control loop that may not allocate
        dict(name="sweep_noalloc", kind="sweep", H=4, C=4, Q=6, gamma=0.95),
    ]


def _sizes(rng, lo, hi, hosts):
    """H, C, Q with the number of states spread over the logarithm of [lo, hi]."""
    want = math.exp(rng.uniform(math.log(lo), math.log(hi)))
    while True:
        H, C, Q = rng.randint(*hosts), rng.randint(2, 6), rng.randint(3, 15)
        if want / 1.6 <= inputs.num_states(H, C, Q) <= min(hi, want * 1.6):
            return dict(H=H, C=C, Q=Q)


def draw(rng):
    kind = rng.choice(["solve", "solve", "solve", "matrix", "matrix", "user", "batch", "train", "evaluate",
                       "end_to_end", "sweep"])
    gamma = rng.choice(GAMMAS)
    if kind == "solve":
        z = _sizes(rng, 600, 2_500_000, (2, 7))
        return dict(kind="solve", gamma=gamma, fmt="implicit", padded=False, sliced=False,
                    self_loop=rng.random() < 0.4, accurate=rng.random() < 0.3, **z)
    if kind == "matrix":
        z = _sizes(rng, 5_000, 2_500_000, (3, 7))
        return dict(kind="solve", gamma=gamma, fmt=rng.choice(["csr_f32", "csr_f32", "csr_bf16"]),
                    padded=rng.random() < 0.5, sliced=rng.random() < 0.7, self_loop=rng.random() < 0.3,
                    accurate=False, **z)
    if kind == "user":
        return dict(kind="user", S=int(math.exp(rng.uniform(math.log(900), math.log(300_000)))), A=rng.randint(2, 9),
                    succ=rng.randint(4, 16), gamma=gamma, bf16=rng.random() < 0.3)
    if kind == "batch":
        return dict(kind="batch", n=int(math.exp(rng.uniform(math.log(8), math.log(512)))), sizes=rng.randint(0, 999),
                    self_loop=rng.random() < 0.5)
    if kind == "train":
        return dict(kind="train", gamma=rng.choice((0.9, 0.95)), **_sizes(rng, 600, 345_000, (2, 6)))
    if kind == "evaluate":
        return dict(kind="evaluate", gamma=gamma, **_sizes(rng, 600, 2_500_000, (2, 7)))
    if kind == "end_to_end":
        fmt = rng.choice(["implicit", "csr_f32"])
        return dict(kind="end_to_end", gamma=gamma, fmt=fmt, padded=fmt != "implicit" and rng.random() < 0.5,
                    **_sizes(rng, 600, 500_000, (2, 6)))
    return dict(kind="sweep", gamma=gamma, **_sizes(rng, 600, 1_000_000, (2, 7)))


# ------------------------------------------------------------------------------- inputs
def _params(case, seed):
    return inputs.make_params(case["H"], case["C"], case["Q"], case["gamma"], seed)


def _batch_params(case, seed):
    """The case's uneven sizes (the batched workload's recipe), rates from the seed."""
    return [inputs.make_params(p["H"], p["C"], p["Q"], p["gamma"], 100_003 * seed + i)
            for i, p in enumerate(inputs.batch_params(case["n"], case["sizes"]))]


def _user_rows(case, seed):
    """A random explicit MDP on the device: ragged rows of 1..succ successors (column order),
    a fifth of the rows infeasible, action 0 always feasible.  Dense [S*A, succ] arrays."""
    g = torch.Generator(device="cuda").manual_seed(seed)
    S, A, K = case["S"], case["A"], case["succ"]
    rows = S * A
    n = torch.randint(1, K + 1, (rows,), generator=g, device="cuda")
    bad = torch.rand(rows, generator=g, device="cuda") < 0.2
    bad[::A] = False
    n[bad] = 0
    col = torch.randint(0, S, (rows, K), generator=g, device="cuda").sort(1).values
    w = torch.rand((rows, K), generator=g, device="cuda", dtype=torch.float64) + 0.05
    live = torch.arange(K, device="cuda") < n[:, None]
    w = torch.where(live, w, 0.0)
    val = (w / w.sum(1, keepdim=True).clamp_min(1e-300)).to(torch.bfloat16 if case["bf16"] else torch.float32)
    R = torch.rand(rows, generator=g, device="cuda") * 2 - 1
    R[bad] = -math.inf
    return n, live, col, val, R


def _policy_start(case):
    """Weights of the objective: uniform over the states with every host empty."""
    S, n = inputs.num_states(case["H"], case["C"], case["Q"]), 2 * (case["Q"] + 1)
    rho = torch.zeros(S, dtype=torch.float64, device="cuda")
    rho[:n] = 1.0 / n
    return rho


def prepare(case, seed):
    native.load()
    kind = case["kind"]
    if kind == "solve":
        m = native.MDP.build(_params(case, seed), fmt=case["fmt"], padded=case["padded"], sliced=case["sliced"])
        return dict(case=case, m=m)
    if kind == "user":
        n, live, col, val, R = _user_rows(case, seed)
        row_ptr = torch.zeros(n.numel() + 1, dtype=torch.int64, device="cuda")
        torch.cumsum(n, 0, out=row_ptr[1:])
        m = native.MDP.from_csr(case["S"], case["A"], row_ptr, col[live].to(torch.int32), val[live], R, case["gamma"])
        return dict(case=case, m=m)
    if kind == "batch":
        return dict(case=case, m=native.Batch(_batch_params(case, seed)))
    if kind == "train":
        p = _params(case, seed)
        theta = torch.tensor(autograd.theta_of(p), dtype=torch.float64, requires_grad=True)
        return dict(case=case, theta=theta, base=p, rho=_policy_start(case))
    if kind == "evaluate":
        return dict(case=case, m=native.MDP.build(_params(case, seed), fmt="implicit"))
    if kind == "end_to_end":
        return dict(case=case, params=_params(case, seed))
    p = _params(case, seed)
    S = inputs.num_states(case["H"], case["C"], case["Q"])
    V = _sweep_values(S, seed)
    return dict(case=case, params=p, V=V, V_out=torch.empty_like(V),
                pi=torch.empty(S, dtype=torch.int32, device="cuda"), residual=torch.empty(1, device="cuda"))


def _sweep_values(S, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    return torch.rand(S, generator=g, device="cuda") * 40 + 20


def run(state):
    case, kind = state["case"], state["case"]["kind"]
    if kind == "solve":
        V, V64, pi, _ = state["m"].value_iterate(tol=1e-6, self_loop=case["self_loop"], accurate=case["accurate"])
        return V, V64, pi
    if kind == "user":
        V, V64, pi, _ = state["m"].value_iterate(tol=1e-6)
        return V, V64, pi
    if kind == "batch":
        V, V64, pi, _, _ = state["m"].value_iterate(tol=1e-6, self_loop=case["self_loop"])
        return V, V64, pi
    if kind == "train":
        theta = state["theta"]
        theta.grad = None
        J = autograd.VCValueFn.apply(theta, state["base"], state["rho"])
        J.backward()
        return J, theta.grad
    if kind == "evaluate":
        pi = state["m"].greedy_policy()
        V, _ = state["m"].evaluate_policy(pi)
        return pi, V
    if kind == "end_to_end":
        V64, pi, _ = native.solve(state["params"], fmt=case["fmt"], padded=case["padded"])
        return V64, pi
    native.bellman32_noalloc(state["params"], state["V"], state["V_out"], state["pi"], state["residual"])
    return state["V_out"], state["pi"], state["residual"]


# --------------------------------------------------------------------------------- work
def _sweeps(gamma, scale):
    """Sweeps of Algorithm 3 from V = 0 to a 1e-6 residual (float32 values of this scale stop at
    four units in the last place of the largest value)."""
    tol = max(1e-6, 4 * 2.0 ** (math.ceil(math.log2(scale / (1 - gamma))) - 24))
    return math.ceil(math.log(tol / scale) / math.log(gamma))


def _model_sizes(H, C, Q):
    """States, non-zero successors of one state's row, feasible actions of a state (means)."""
    S = inputs.num_states(H, C, Q)
    row = H * (2 * C - 1) / (C + 1) + 2 + Q / (Q + 1)
    feasible = 1 + Q / (Q + 1) * C / (C + 1) * (0.5 * (H - 1) + 1)
    return S, row, feasible


def _model_flops(H, C, Q, sweeps):
    """Post-decision form: a multiply-add per successor of a state, a comparison per action."""
    S, row, feasible = _model_sizes(H, C, Q)
    return sweeps * S * (2 * row + feasible)


def work(case):
    """Bytes: inputs once and outputs once (a stored matrix counts as an input).  Flops: those of
    the sweeps to the residual from zero."""
    kind, gamma = case["kind"], case.get("gamma", 0.95)
    if kind == "user":
        rows = case["S"] * case["A"]
        nnz = rows * (0.2 / case["A"] + 0.8) * (case["succ"] + 1) / 2
        return dict(bytes=nnz * (6 if case["bf16"] else 8) + rows * 12 + case["S"] * 20,
                    flops=2 * nnz * _sweeps(gamma, 1.0))
    if kind == "batch":
        ps = inputs.batch_params(case["n"], case["sizes"])
        return dict(bytes=sum(20 * inputs.num_states(p["H"], p["C"], p["Q"]) for p in ps),
                    flops=sum(_model_flops(p["H"], p["C"], p["Q"], _sweeps(p["gamma"], p["H"] * p["C"] / 2))
                              for p in ps))
    H, C, Q = case["H"], case["C"], case["Q"]
    S, row, feasible = _model_sizes(H, C, Q)
    n = _sweeps(gamma, H * C / 2)
    if kind == "sweep":
        return dict(bytes=12 * S, flops=_model_flops(H, C, Q, 1))
    if kind == "solve" and case["fmt"] != "implicit":
        nnz = S * feasible * row
        return dict(bytes=nnz * (6 if case["fmt"] == "csr_bf16" else 8) + S * (H + 1) * 12 + 20 * S, flops=2 * nnz * n)
    if kind == "train":
        # the forward solve, then as many products by the transposed rows as a tenth of its sweeps
        return dict(bytes=16 * S, flops=_model_flops(H, C, Q, 1.1 * n))
    if kind == "evaluate":
        return dict(bytes=12 * S, flops=2 * S * row * n / 10)
    return dict(bytes=20 * S if kind == "solve" else 12 * S, flops=_model_flops(H, C, Q, n))


# -------------------------------------------------------------------------------- exact
class _Model:
    """The uniformised model of one or more instances, concatenated, as FP64 gather lists:
    events (target, probability) of every state read as a post-decision state, its reward, and
    for each action the post-decision state it leads to (-1: infeasible)."""

    def __init__(self, ps, theta=None):
        parts, off = [], 0
        hosts = max(p["H"] for p in ps)
        for p in ps:
            parts.append(self._one(p, off, hosts, theta))
            off += inputs.num_states(p["H"], p["C"], p["Q"])
        cat = lambda f: torch.cat([f(x) for x in parts]) if len(parts) > 1 else f(parts[0])  # noqa: E731
        n = len(parts[0]["events"])
        self.S = off
        self.events = [(cat(lambda x, e=e: x["events"][e][0]), cat(lambda x, e=e: x["events"][e][1])) for e in range(n)]
        self.reward, self.gamma = cat(lambda x: x["reward"]), cat(lambda x: x["gamma"])
        self.post = [cat(lambda x, a=a: x["post"][a]) for a in range(hosts)]
        self.occ = parts[0]["occ"]
        self.local = [cat(lambda x, a=a: x["local"][a]) for a in range(hosts)]
        self.defer = cat(lambda x: x["defer"])

    @staticmethod
    def _one(p, off, hosts, theta):
        H, C, Q = p["H"], p["C"], p["Q"]
        if theta is None:
            theta = [torch.tensor(v, dtype=torch.float64, device="cuda") for v in autograd.theta_of(p)]
        lam, mu, delta, f = theta[0], theta[1:1 + H], theta[1 + H:1 + 2 * H], theta[1 + 2 * H]
        w_occ, w_loss, w_q = theta[2 + 2 * H:5 + 2 * H]
        Lam = lam + C * sum(mu) + sum(delta) + 1
        S = inputs.num_states(H, C, Q)
        s = torch.arange(S, device="cuda", dtype=torch.int32)
        ph, q = s & 1, (s >> 1) % (Q + 1)
        code = (s >> 1) // (Q + 1)
        stride, occ = [2 * (Q + 1) * (C + 1) ** k for k in range(H)], []
        for k in range(H):
            occ.append(code % (C + 1))
            code = code // (C + 1)
        zero = torch.zeros(S, dtype=torch.float64, device="cuda")
        events, post, local = [], [], []
        loss = torch.where(q == Q, lam, zero)
        for k in range(hosts):
            if k >= H:
                events += [(s + off, zero), (s + off, zero)]
                post.append(torch.full_like(s, -1))
                local.append(torch.full_like(s, -1))
                continue
            o = occ[k].to(torch.float64)
            events.append((torch.where(occ[k] > 0, s - stride[k], s) + off, mu[k] * o / Lam))
            events.append((s - occ[k] * stride[k] + off, torch.where(occ[k] > 0, delta[k] / Lam, zero)))
            loss = loss + delta[k] * o
            ok = (q >= 1) & (occ[k] < C)
            if k < H - 1:
                ok = ok & (ph == 1)
            post.append(torch.where(ok, s + stride[k] - 2 + off, -1))
            local.append(torch.full_like(s, k))
        events.append((torch.where(q < Q, s + 2, s) + off, torch.where(q < Q, lam / Lam, zero)))
        events.append(((s ^ 1) + off, torch.where(ph == 1, (1 - f) / Lam, f / Lam)))
        reward = w_occ * sum(occ).to(torch.float64) + w_q * q.to(torch.float64) + w_loss * loss / Lam
        return dict(events=events, reward=reward, post=post, occ=occ, local=local, defer=torch.full_like(s, H),
                    gamma=torch.full((S,), float(p["gamma"]), dtype=torch.float64, device="cuda"))

    def bf16(self):
        """The same model with each row's merged probabilities rounded to BF16 and renormalised."""
        events, stay = [], 1 - sum(p for _, p in self.events)
        for k, o in enumerate(self.occ):
            (yc, pc), (yd, pd) = self.events[2 * k], self.events[2 * k + 1]
            events += [(yc, torch.where(o == 1, pc + pd, pc)), (yd, torch.where(o == 1, 0.0, pd))]
        events += self.events[-2:]
        r = lambda p: p.to(torch.bfloat16).to(torch.float64)  # noqa: E731
        events, stay = [(y, r(p)) for y, p in events], r(stay)
        total = stay + sum(p for _, p in events)
        scale = (1 / total).to(torch.float32).to(torch.float64)
        self.events, self.stay = [(y, p * scale) for y, p in events], stay * scale
        return self

    def parts(self, V):
        """Sum over the moves of every post-decision state, and the probability of staying."""
        acc, moved = torch.zeros_like(V), torch.zeros_like(V)
        for y, p in self.events:
            acc += p * V.index_select(0, y)
            moved += p
        return acc, getattr(self, "stay", 1 - moved)

    def sweep(self, V, solved=True):
        """The Bellman backup (solved: defer's self-transition solved) and its argmax."""
        acc, stay = self.parts(V)
        U = self.reward + self.gamma * (acc + stay * V)
        best = torch.full_like(V, -math.inf)
        arg = torch.zeros_like(self.defer)
        for x, a in zip(self.post, self.local):
            u = torch.where(x >= 0, U.index_select(0, x.clamp_min(0)), -math.inf)
            arg = torch.where(u > best, a, arg)
            best = torch.maximum(best, u)
        d = (self.reward + self.gamma * acc) / (1 - self.gamma * stay) if solved else U
        return torch.maximum(best, d), torch.where(d > best, self.defer, arg)

    def policy_sweep(self, V, x):
        """One evaluation sweep, x the post-decision states of a policy; staying solved."""
        acc, stay = self.parts(V)
        U = self.reward + self.gamma * (acc + stay * V)
        here = x == torch.arange(self.S, device="cuda", dtype=x.dtype)
        return torch.where(here, (self.reward + self.gamma * acc) / (1 - self.gamma * stay), U.index_select(0, x))

    def post_of(self, pi):
        x = torch.arange(self.S, device="cuda", dtype=torch.int32)
        for k, y in enumerate(self.post):
            x = torch.where((pi == k) & (y >= 0), y, x)
        return x


def _fixed_point(step, V, most=8000):
    for k in range(most):
        W = step(V)
        if k % 16 == 15 and float((W - V).abs().max()) < 1e-13 * max(1.0, float(W.abs().max())):
            return W
        V = W
    return V


def _optimum(model):
    return _fixed_point(lambda V: model.sweep(V)[0], torch.zeros(model.S, dtype=torch.float64, device="cuda"))


def _exact_user(case, seed):
    _, _, col, val, R = _user_rows(case, seed)
    S, A = case["S"], case["A"]
    p, idx = val.to(torch.float64), col.reshape(-1)
    if case["bf16"]:
        p = p * (1 / p.sum(1, keepdim=True).clamp_min(1e-300)).to(torch.float32).to(torch.float64)
    R = R.to(torch.float64)

    def step(V):
        return (R + case["gamma"] * (p * V.index_select(0, idx).reshape(p.shape)).sum(1)).reshape(S, A).max(1).values

    V = _fixed_point(step, torch.zeros(S, dtype=torch.float64, device="cuda"))
    return V, V, None


def _exact_train(case, seed):
    p = _params(case, seed)
    model = _Model([p])
    V = _optimum(model)
    x = model.post_of(model.sweep(V, solved=False)[1])
    rho, gamma = _policy_start(case), case["gamma"]
    stay = 1 - sum(q for _, q in model.events)

    def step(lam):
        mass = torch.zeros_like(lam).index_add_(0, x, lam)
        out = rho + gamma * stay * mass
        for y, q in model.events:
            out.index_add_(0, y, gamma * q * mass)
        return out

    lam = _fixed_point(step, rho.clone())
    theta = torch.tensor(autograd.theta_of(p), dtype=torch.float64, device="cuda", requires_grad=True)
    diff = _Model([p], theta=list(theta.unbind()))
    F = diff.reward
    for y, q in diff.events:
        F = F + gamma * q * (V.index_select(0, y) - V)
    (lam * F.index_select(0, x)).sum().backward()
    return (rho * V).sum(), theta.grad.cpu()


def exact(case, seed):
    kind = case["kind"]
    if kind == "user":
        return _exact_user(case, seed)
    if kind == "batch":
        V = _optimum(_Model(_batch_params(case, seed)))
        return V, V, None
    if kind == "train":
        return _exact_train(case, seed)
    model = _Model([_params(case, seed)])
    if kind == "solve":
        V64 = _optimum(model)
        return (_optimum(model.bf16()) if case["fmt"] == "csr_bf16" else V64), V64, None
    if kind == "evaluate":
        mu = _params(case, seed)["mu"]
        pi = model.defer.clone()
        for k in sorted(range(case["H"]), key=lambda k: (mu[k], -k)):
            pi = torch.where(model.post[k] >= 0, k, pi)
        x = model.post_of(pi)
        return None, _fixed_point(lambda V: model.policy_sweep(V, x), torch.zeros_like(model.reward))
    if kind == "end_to_end":
        return _optimum(model), None
    V = _sweep_values(model.S, seed).to(torch.float64)
    W = model.sweep(V, solved=False)[0]
    return W, None, (W - V).abs().max().reshape(1)
