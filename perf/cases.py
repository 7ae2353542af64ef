"""What a user of this solver has it do, as cases that can be timed and compared.

Sizes and distributions follow the repository's own workloads: rows of a
truncated lognormal degree (mean 25, at most 500) over items of Zipf(0.8)
popularity, c = -LogNormal(0, 0.5), a = U(0.5, 1.5), capacities 5 % of the
items' total use; App. A's short rows for the appendix case.  Everything is
drawn on the GPU from the seed alone.  The starting dual of an instance is the
optimum of a user sample of it, found here in plain torch: what a recurring
solve has in hand before a call.
"""
import math

import numpy as np
import torch

import paper_2606_07777_gb300 as dlm

LE, EQ, BOX, BOX_CUT = dlm.DLM_SIMPLEX_LE, dlm.DLM_SIMPLEX_EQ, dlm.DLM_BOX, dlm.DLM_BOX_CUT
KINDS = {"le": LE, "eq": EQ, "box": BOX}
SAMPLE = 32768  # users of the sample solved for the starting dual


def listed():
    return [
        # a small campaign solved in a request: 100k edges, all launches and latency
        {"name": "tiny_f32", "path": "step", "users": 10_000, "items": 100, "degrees": "poisson", "dtype": "f32",
         "kind": "le", "gamma": 1e-2, "iters": 50},
        # a daily instance between two gap checks of a solve (row normalization, adaptive restart)
        {"name": "daily_check_f32", "path": "check", "users": 1_000_000, "items": 1_000, "degrees": "lognormal",
         "dtype": "f32", "kind": "le", "gamma": 1e-3, "iters": 25},
        # the production form: FP32 values, 2,000 items
        {"name": "production_f32", "path": "step", "users": 8_000_000, "items": 2_000, "degrees": "lognormal",
         "dtype": "f32", "kind": "le", "gamma": 1e-3, "iters": 10},
        # the precision form: BF16 values, 5,000 items, the largest
        {"name": "precision_bf16", "path": "step", "users": 16_000_000, "items": 5_000, "degrees": "lognormal",
         "dtype": "bf16", "kind": "le", "gamma": 1e-3, "iters": 10},
        # many independent instances of very different sizes iterated as one batch
        {"name": "batch_bf16", "path": "batch", "members": 16, "users": 1_200_000, "items": 2_000,
         "degrees": "lognormal", "dtype": "bf16", "kind": "le", "iters": 10},
        # two capacity families
        {"name": "families_bf16", "path": "families", "families": 2, "users": 2_000_000, "items": 2_000,
         "degrees": "lognormal", "dtype": "bf16", "kind": "le", "gamma": 1e-3, "iters": 10},
        # the box cut by a budget
        {"name": "boxcut_bf16", "path": "boxcut", "users": 2_000_000, "items": 2_000, "degrees": "lognormal",
         "dtype": "bf16", "kind": "le", "gamma": 1e-3, "iters": 10},
        # the paper's appendix construction: about ten edges a request, 10,000 resources, the short-row sweep
        {"name": "appendix_f32", "path": "short", "users": 2_500_000, "items": 10_000, "dtype": "f32", "kind": "le",
         "gamma": 1e-2, "iters": 10},
        # one evaluation of the dual with its gradient and the whole primal (ObjectiveFunction.calculate)
        {"name": "evaluate_f32", "path": "evaluate", "users": 1_000_000, "items": 1_000, "degrees": "lognormal",
         "dtype": "f32", "kind": "le", "gamma": 1e-3},
        # a new day: handle from arrays on the device, a few warm-started iterations, the dual
        {"name": "recreate_bf16", "path": "recreate", "users": 2_000_000, "items": 1_000, "degrees": "lognormal",
         "dtype": "bf16", "kind": "le", "gamma": 1e-3, "iters": 10},
        # one evaluation for a caller that cannot allocate device memory
        {"name": "evaluate_static_f32", "path": "static", "users": 500_000, "items": 1_000, "degrees": "lognormal",
         "dtype": "f32", "kind": "le", "gamma": 1e-3},
        # the learned warm start: loss and gradient on 17 days of 1,000 items, the prediction of one day
        {"name": "predictor_h128", "path": "predictor", "rows": 17_000, "items": 1_000, "width": 128},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    path = rng.choice(["step", "step", "step", "check", "batch", "families", "boxcut", "short", "evaluate",
                       "recreate", "static", "predictor"])
    if path == "predictor":
        return {"path": path, "rows": _log(rng, 1_000, 40_000), "items": _log(rng, 50, 5_000),
                "width": 8 * rng.randint(4, 32)}
    case = {"path": path, "degrees": "lognormal", "dtype": rng.choice(["f32", "bf16"]), "kind": "le",
            "gamma": rng.choice([1e-1, 1e-2, 1e-3, 1e-3])}
    if path == "step":
        case.update(users=_log(rng, 5_000, 8_000_000), items=_log(rng, 50, 5_000), iters=rng.randint(5, 20),
                    kind=rng.choice(["le", "le", "eq", "box"]))
        if rng.random() < 0.25 and case["kind"] != "eq":
            case["degrees"] = "poisson"
    elif path == "check":
        case.update(users=_log(rng, 20_000, 4_000_000), items=_log(rng, 100, 2_000), iters=rng.randint(10, 40),
                    gamma=1e-3)
    elif path == "batch":
        case.update(members=rng.randint(3, 20), users=_log(rng, 60_000, 1_200_000), items=_log(rng, 200, 2_000),
                    iters=rng.randint(5, 15))
        del case["gamma"]
    elif path == "families":
        case.update(families=rng.randint(2, 3), users=_log(rng, 20_000, 2_000_000), items=_log(rng, 100, 2_000),
                    iters=rng.randint(5, 15))
    elif path == "boxcut":
        case.update(users=_log(rng, 20_000, 2_000_000), items=_log(rng, 100, 2_000), iters=rng.randint(5, 15))
    elif path == "short":
        case.update(users=_log(rng, 20_000, 4_000_000), items=_log(rng, 500, 10_000), iters=rng.randint(5, 15),
                    gamma=1e-2)
        del case["degrees"]
    elif path == "evaluate":
        case.update(users=_log(rng, 5_000, 2_000_000), items=_log(rng, 50, 5_000),
                    kind=rng.choice(["le", "le", "eq", "box"]))
    elif path == "recreate":
        case.update(users=_log(rng, 20_000, 3_000_000), items=_log(rng, 100, 5_000), iters=rng.randint(5, 30),
                    gamma=1e-3)
    else:
        case.update(users=_log(rng, 5_000, 1_000_000), items=_log(rng, 50, 5_000), dtype="f32",
                    kind=rng.choice(["le", "le", "eq", "box"]))
    return case


# ---------------------------------------------------------------------------
# Instances
# ---------------------------------------------------------------------------

DEV = "cuda"


def _gen(seed, salt=0):
    return torch.Generator(device=DEV).manual_seed((seed * 1000003 + salt * 7919 + 17) % (1 << 62))


def _degrees(case, n, J):
    """Degrees of n rows: the same list for every seed (evenly spaced quantiles)."""
    q = (np.arange(n) + 0.5) / n
    if case["path"] == "short" or case["degrees"] == "poisson":  # 1 + Poisson(9)
        k = np.arange(60)
        pmf = np.exp(-9.0 + k * math.log(9.0) - np.cumsum(np.log(np.maximum(k, 1))))
        d = 1 + np.searchsorted(np.cumsum(pmf), q)
    else:  # lognormal of mean 25, the part above 500 drawn again
        x = np.linspace(-6.0, (math.log(500.0) - math.log(25.0) + 0.5), 200_001)
        cdf = np.cumsum(np.exp(-0.5 * x * x))
        d = np.floor(np.exp(math.log(25.0) - 0.5 + np.interp(q, cdf / cdf[-1], x)) + 0.5)
    return np.clip(d, 1, min(500, J)).astype(np.int64)


def _rows(case, n, J, g, popularity):
    """row_ptr and items of n rows: one item drawn in each of d equal shares of
    the popularity, moved on to the next free one where it is taken; the row
    starts at a random share."""
    deg = torch.from_numpy(_degrees(case, n, J)).to(DEV)[torch.randperm(n, device=DEV, generator=g)]
    start = torch.zeros(n + 1, dtype=torch.int64, device=DEV)
    torch.cumsum(deg, 0, out=start[1:])
    nnz = int(start[-1])
    row = torch.repeat_interleave(torch.arange(n, device=DEV, dtype=torch.int32), deg, output_size=nnz)
    d = deg.to(torch.int32)[row]
    k = (torch.arange(nnz, device=DEV) - start[:-1][row]).to(torch.int32)
    at = (k + torch.rand(nnz, device=DEV, generator=g)) / d
    cdf = torch.cumsum(popularity.double(), 0)
    rank = torch.searchsorted((cdf / cdf[-1]).float(), at, out_int32=True).clamp_(max=J - 1)
    del at
    base = row.long() * (4 * J)  # the next free item: a running maximum within the row
    rank = (torch.cummax(base + (rank - k + J), 0).values - base).to(torch.int32) - J + k
    rank = torch.minimum(rank, J - d + k)
    del base
    turn = (torch.rand(n, device=DEV, generator=g) * deg).to(torch.int32)[row]
    place = start[:-1][row] + (k + turn) % d
    item = torch.empty(nnz, dtype=torch.int32, device=DEV)
    item[place] = torch.randperm(J, device=DEV, generator=g).to(torch.int32)[rank]
    return start, item, row


def _sums(item, v, J):
    """Per-item sums, the same from run to run (whole numbers of 2^-30)."""
    s = torch.zeros(J, dtype=torch.int64, device=DEV)
    s.index_add_(0, item.long(), (v.double() * float(1 << 30)).round().long())
    return s.double() / float(1 << 30)


def _stored(v, case):
    return v.bfloat16() if case["dtype"] == "bf16" else v.float()


def _instance(case, seed, users=None, items=None):
    """The arrays of one instance: row_ptr, item, c, a (per family), b."""
    g = _gen(seed)
    n, J = users or case["users"], items or case["items"]
    if case["path"] == "short":  # App. A: distinct requests per resource, value = v_j u_i e_ij, a = s_j value
        pop = torch.exp(torch.randn(J, device=DEV, generator=g))
        rp, col, row = _rows(case, n, J, g, pop)
        normal = lambda size, sd: torch.exp(sd * torch.randn(size, device=DEV, generator=g))  # noqa: E731
        value = (normal(J, 0.5)[col.long()] * normal(n, 0.5)[row.long()] * normal(len(col), 0.25)).clamp(max=5.0)
        c, a = _stored(-value, case), [_stored(normal(J, 1.5)[col.long()] * value, case)]
        best = torch.segment_reduce(a[0].float(), "max", offsets=rp, initial=0.0, axis=0)
        load = _sums(col, torch.where(a[0].float() == best[row.long()], a[0].float(), 0.0), J)
        b = [(0.5 + 0.5 * torch.rand(J, device=DEV, generator=g).double()) * (load + 1e-3)]
        return rp, col, c, a, b
    pop = torch.arange(1, J + 1, device=DEV, dtype=torch.float64) ** -0.8
    rp, col, _ = _rows(case, n, J, g, pop)
    nnz = len(col)
    if case["degrees"] == "poisson":  # the small recipe: c = -U(0, 1), a = 1
        c = _stored(-torch.rand(nnz, device=DEV, generator=g), case)
        a = [_stored(torch.ones(nnz, device=DEV), case)]
    else:
        c = _stored(-torch.exp(0.5 * torch.randn(nnz, device=DEV, generator=g)), case)
        a = [_stored(0.5 + torch.rand(nnz, device=DEV, generator=g), case)]
    for _ in range(1, case.get("families", 1)):
        a.append(_stored(0.1 + 1.9 * torch.rand(nnz, device=DEV, generator=g), case))
    return rp, col, c, a, [0.05 * _sums(col, f, J) for f in a]


def _member_sizes(case):
    r = np.random.RandomState(case["members"])
    out = []
    for k in range(case["members"]):
        out.append((int(round(math.exp(r.uniform(math.log(1e4), math.log(case["users"]))))),
                    int(round(math.exp(r.uniform(math.log(50), math.log(case["items"]))))), (1e-1, 1e-2, 1e-3)[k % 3]))
    return out


# ---------------------------------------------------------------------------
# The method in plain torch, 64 bits
# ---------------------------------------------------------------------------

WIDTHS = (1, 2, 3, 4, 6, 8, 12, 16, 20, 24, 32, 40, 48, 64, 96, 128, 192, 256, 384, 512, 1 << 20)
CHUNK = 1 << 25


class _Exact:
    """Dual evaluations and accelerated iterations of one instance."""

    def __init__(self, inst, case, gamma, users=None, share=1.0, whole=True):
        rp, col, c, a, b = inst
        self.n = users or len(rp) - 1
        nnz = int(rp[self.n])
        self.col, self.c = col[:nnz].long(), c[:nnz].double()
        self.a = [f[:nnz].double() for f in a]
        self.b = [f * share for f in b]
        self.J, self.gamma, self.whole, self.case = len(b[0]), gamma, whole, case
        self.kind = case["kind"]
        self.z = 0.5 if case["path"] == "boxcut" else 1.0
        deg = rp[1:self.n + 1] - rp[:self.n]
        self.groups, lo = [], 0  # rows of similar degree side by side, filled up with an edge of value -inf
        for w in WIDTHS if whole else WIDTHS[::4] + WIDTHS[-1:]:
            rows = torch.nonzero((deg > lo) & (deg <= w)).flatten()
            lo = w
            w = min(w, int(deg[rows].max())) if len(rows) else w
            for part in rows.split(max(1, CHUNK // w)):
                if len(part):
                    k = torch.arange(w, device=DEV)
                    self.groups.append(torch.where(k < deg[part][:, None], rp[part][:, None] + k, nnz))
        # curvature bounds of the items, by family (rows of the families' products)
        self.curv = []
        for f in self.a:
            h = torch.zeros(self.J, dtype=torch.float64, device=DEV)
            for o in self.a:
                h += self.item_sums(f * o).abs()
            self.curv.append(h)
        self.precondition = case["path"] != "step" or case["degrees"] != "poisson"
        self.top = max(float(h.max()) for h in self.curv)

    def item_sums(self, v):
        if not self.whole:
            return _sums(self.col, v, self.J)
        on = torch.nonzero(v).flatten()
        return torch.zeros(self.J, dtype=torch.float64, device=DEV).index_add_(0, self.col[on], v[on])

    def steps(self):
        if self.precondition:
            return [torch.where(h > 0, self.gamma / h.clamp(min=1e-300), 0.0) for h in self.curv]
        return [torch.full_like(h, self.gamma / self.top) for h in self.curv]

    def x(self, y):
        u = torch.full((len(self.c) + 1,), -math.inf, dtype=torch.float64, device=DEV)
        u[:-1] = -self.c
        for f, v in zip(self.a, y):
            u[:-1] -= f * v[self.col]
        out = torch.zeros_like(u)
        gz = self.gamma * self.z
        for at in self.groups:
            U = u[at]
            if self.case["path"] == "boxcut":
                X = ((U - self.budget(U)) / self.gamma).clamp(0, self.z)
            elif self.kind == "box":
                X = (U / self.gamma).clamp(0, self.z)
            else:  # the threshold from the sorted row (Sec. 4.3)
                v = U.sort(1, descending=True).values
                tau = (v.cumsum(1) - gz) / torch.arange(1, v.shape[1] + 1, device=DEV)
                tau = tau.gather(1, (v > tau).sum(1, keepdim=True) - 1)
                X = ((U - (tau.clamp(min=0.0) if self.kind == "le" else tau)) / self.gamma).clamp(min=0.0)
            out[at] = X
        return out[:-1]

    def budget(self, U, cut=1.0):
        total = lambda t: ((U - t) / self.gamma).clamp(0, self.z).sum(1, keepdim=True)  # noqa: E731
        lo = torch.zeros(len(U), 1, dtype=torch.float64, device=DEV)
        hi = U.max(1, keepdim=True).values.clamp(min=0.0)
        over = total(lo) > cut
        for _ in range(56 if self.whole else 24):
            mid = 0.5 * (lo + hi)
            up = total(mid) > cut
            lo, hi = torch.where(up, mid, lo), torch.where(up, hi, mid)
        return torch.where(over, 0.5 * (lo + hi), 0.0)

    def grad(self, x):
        return [self.item_sums(f * x) - b for f, b in zip(self.a, self.b)]

    def iterate(self, lam, iters, restart=False):
        lam = [v.clamp(min=0.0) for v in lam]
        y, theta = lam, 1.0
        for _ in range(iters):
            G, S = self.grad(self.x(y)), self.steps()
            new = [(v + s * q).clamp(min=0.0) for v, s, q in zip(y, S, G)]
            up = 0.5 * (1 + math.sqrt(1 + 4 * theta * theta))
            against = restart and sum(float(torch.where(s > 0, (p - v) * (p - o) / s.clamp(min=1e-300), 0.0).sum())
                                      for p, v, o, s in zip(new, y, lam, S)) < 0
            if against:
                y, theta = new, 1.0
            else:
                y = [p + (theta - 1) / up * (p - o) for p, o in zip(new, lam)]
                theta = up
            lam = new
        return lam

    def evaluate(self, lam):
        """(dual value, gradient, x, value of the point scaled into the capacities)"""
        x = self.x(lam)
        G = self.grad(x)
        g = float((self.c * x).sum() + 0.5 * self.gamma * (x * x).sum() + sum((v * q).sum() for v, q in zip(lam, G)))
        s = torch.ones(self.J, dtype=torch.float64, device=DEV)
        for q, b in zip(G, self.b):
            s = torch.minimum(s, torch.where(q > 0, b / (q + b).clamp(min=1e-300), 1.0))
        P = float((s * self.item_sums(self.c * x)).sum() + 0.5 * self.gamma * (s * s * self.item_sums(x * x)).sum())
        return g, G, x, P


def _start(inst, case, gamma):
    """A dual near the optimum: the solution of a sample of the users, gamma
    brought down from 0.1 as the solver's schedules do."""
    n = len(inst[0]) - 1
    users = min(n, SAMPLE)
    E = _Exact(inst, case, max(gamma, 0.1), users, users / n, whole=False)
    E.precondition = True
    lam = [torch.zeros(E.J, dtype=torch.float64, device=DEV) for _ in inst[3]]
    while True:
        lam = E.iterate(lam, 12)
        if E.gamma <= gamma:
            return torch.cat(lam).float()
        E.gamma = max(gamma, 0.4 * E.gamma)


# ---------------------------------------------------------------------------
# The passes
# ---------------------------------------------------------------------------

def _solver(inst, case, gamma):
    rp, col, c, a, b = inst
    kw = {"kind": KINDS[case["kind"]]}
    if case["path"] == "boxcut":
        kw = {"kind": BOX_CUT, "z": 0.5, "cut": 1.0}
    many = len(a) > 1
    s = dlm.Solver(rp, col, c, torch.stack(a, 1).contiguous() if many else a[0], torch.stack(b) if many else b[0],
                   len(b[0]), **kw)
    s.set_schedule(gamma)
    s.set_options(precondition=case["path"] != "step" or case["degrees"] != "poisson",
                  restart=case["path"] == "check", short_rows=case["path"] == "short")
    return s


def _predictor_inputs(case, seed):
    r = np.random.RandomState(seed % (1 << 31))
    n = case["rows"]
    X = np.empty((n + case["items"], 7), dtype=np.float32)
    m = len(X)
    X[:, 0], X[:, 1], X[:, 2] = r.uniform(2, 9, m), r.uniform(3, 11, m), r.uniform(0.5, 2, m)
    X[:, 3] = X[:, 2] + r.uniform(0, 3, m)
    X[:, 4] = np.where(r.uniform(size=m) < 0.2, 0.0, r.uniform(0, 1.5, m))
    X[:, 5] = math.log(1e-3)
    X[:, 6] = r.normal(0, 0.05, m)
    y = np.maximum(X[:, 4] * (1 + 2 * X[:, 6]) + 0.05 * np.tanh(X[:, 0] - 5), 0).astype(np.float32)
    H = case["width"]
    W = [r.uniform(-1, 1, (7, H)) * math.sqrt(6 / 7), r.normal(0, 0.1, H), r.uniform(-1, 1, (H, H)) * math.sqrt(6 / H),
         r.normal(0, 0.1, H), r.normal(0, 0.3, H), np.array([0.05])]
    mu, sd = X[:n].mean(0).astype(np.float32), X[:n].std(0).astype(np.float32)
    return X, y[:n], [w.astype(np.float32) for w in W], mu, np.where(sd < 1e-6, 1, sd).astype(np.float32)


def prepare(case, seed):
    path = case["path"]
    if path == "predictor":
        X, y, W, mu, sd = _predictor_inputs(case, seed)
        ws = dlm.WarmStart(case["width"], 1)
        ws.set_params(np.concatenate([w.ravel() for w in W]), mu, sd)
        n = case["rows"]
        return {"path": path, "ws": ws, "X": torch.from_numpy(X[:n]).to(DEV), "y": torch.from_numpy(y).to(DEV),
                "new": torch.from_numpy(X[n:]).to(DEV)}
    if path == "batch":
        members, lams = [], []
        for k, (users, items, gamma) in enumerate(_member_sizes(case)):
            inst = _instance(case, seed * 101 + k, users, items)
            lams.append(_start(inst, case, gamma))
            members.append(_solver(inst, case, gamma))
        return {"path": path, "batch": dlm.Batch(members), "members": members, "lams": lams, "iters": case["iters"]}
    inst = _instance(case, seed)
    lam = _start(inst, case, case["gamma"])
    state = {"path": path, "lam": lam, "gamma": case["gamma"], "iters": case.get("iters", 0)}
    if path in ("recreate", "static"):
        state.update(inst=inst, case=case)
        if path == "static":
            state.update(g=torch.empty(1, dtype=torch.float64, device=DEV), x=torch.empty_like(inst[2]),
                         grad=torch.empty(case["items"], dtype=torch.float32, device=DEV))
    else:
        state["solver"] = _solver(inst, case, case["gamma"])
    return state


def run(state):
    path = state["path"]
    if path == "predictor":
        loss, grad = state["ws"].loss_grad(state["X"], state["y"])
        return loss, grad, state["ws"].predict(state["new"])
    if path == "batch":
        for s, lam in zip(state["members"], state["lams"]):
            s.set_lambda(lam)
        state["batch"].step(state["iters"])
        return [s.lam() for s in state["members"]]
    if path == "static":
        rp, col, c, a, b = state["inst"]
        dlm.dlm_calculate_static(len(rp) - 1, len(b[0]), len(col), rp, col, c, a[0], b[0],
                                 KINDS[state["case"]["kind"]], 1.0, state["lam"], state["gamma"], state["g"],
                                 state["grad"], state["x"])
        return state["g"].float(), state["grad"], state["x"]
    if path == "recreate":
        s = _solver(state["inst"], state["case"], state["gamma"])
        s.set_lambda(state["lam"])
        s.step(state["iters"])
        lam = s.lam()
        s.close()
        return lam
    s = state["solver"]
    if path == "evaluate":
        return s.calculate(state["lam"], state["gamma"])
    s.set_lambda(state["lam"])
    s.step(state["iters"])
    if path == "check":
        st = s.stats()
        return s.lam(), st.dual_obj, st.primal_obj
    return s.lam()


def work(case):
    path = case["path"]
    if path == "predictor":
        H, n, m = case["width"], case["rows"], case["items"]
        P = 7 * H + H + H * H + H + H + 1
        # forward on n + m rows, two backward products per layer behind it (one for the first)
        return {"bytes": 4.0 * (8 * n + 8 * m + 2 * P), "flops": 2.0 * ((n + m) * (7 * H + H * H + H)
                                                                       + n * (7 * H + 2 * H * H + H))}
    vs = 2 if case["dtype"] == "bf16" else 4
    if path == "batch":
        edges = sum(int(_degrees(case, u, j).sum()) for u, j, _ in _member_sizes(case))
        m = 1
    else:
        edges = int(_degrees(case, case["users"], case["items"]).sum())
        m = case.get("families", 1)
    # per iteration each edge's item (16 bits hold it) and values; an evaluation also writes x, a new
    # handle reads its input arrays once more, a gap check takes one more pass
    sweep = edges * (2 + vs * (1 + m))
    flops = edges * (2 * m + 2)
    if path == "evaluate":
        return {"bytes": sweep + 4 * edges, "flops": flops}
    if path == "static":  # the caller's arrays: 32-bit items, 64-bit row pointers
        return {"bytes": sweep + 6 * edges + 8 * case["users"], "flops": flops}
    passes = case["iters"] + (1 if path == "check" else 0)
    extra = edges * (4 + 2 * vs) + 8 * case["users"] + sweep if path == "recreate" else 0
    return {"bytes": passes * sweep + extra, "flops": passes * flops}


def _predictor_exact(case, seed):
    X, y, W, mu, sd = _predictor_inputs(case, seed)
    t = lambda v: torch.from_numpy(v).to(DEV).double()  # noqa: E731
    W1, b1, W2, b2, w3, b3 = [t(w).requires_grad_() for w in W]

    def forward(X):
        h = torch.relu((X - t(mu)) / t(sd) @ W1 + b1)
        h = torch.relu(h @ W2 + b2)
        prev = X[:, 4].clamp(min=1e-6)
        return torch.nn.functional.softplus(h @ w3 + b3 + prev + torch.log(-torch.expm1(-prev)), threshold=1e9)

    n = case["rows"]
    loss = ((forward(t(X[:n])) - t(y)) ** 2).mean()
    loss.backward()
    grad = torch.cat([w.grad.flatten() for w in (W1, b1, W2, b2, w3, b3)]).cpu().numpy()
    with torch.no_grad():
        return float(loss), grad, forward(t(X[n:]))


def exact(case, seed):
    path = case["path"]
    if path == "predictor":
        return _predictor_exact(case, seed)
    if path == "batch":
        out = []
        for k, (users, items, gamma) in enumerate(_member_sizes(case)):
            inst = _instance(case, seed * 101 + k, users, items)
            lam = _start(inst, case, gamma).double()
            out.append(_Exact(inst, case, gamma).iterate([lam], case["iters"])[0])
        return out
    inst = _instance(case, seed)
    lam = list(_start(inst, case, case["gamma"]).double().chunk(len(inst[3])))
    E = _Exact(inst, case, case["gamma"])
    if path in ("evaluate", "static"):
        g, G, x, _ = E.evaluate(lam)
        return (g if path == "evaluate" else torch.tensor([g], dtype=torch.float64, device=DEV)), G[0], x
    lam = E.iterate(lam, case["iters"], restart=path == "check")
    if path == "check":
        g, _, _, P = E.evaluate(lam)
        return lam[0], g, P
    return torch.cat(lam)
