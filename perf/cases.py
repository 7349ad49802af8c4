"""The calls whose speed matters to a user of the stale-synchronous table.

Every case is one pass through `paper_1410_8043_gb300.esspt.Table`, the
framework's Python entry points, as a training program makes it:

  clock        one clock of matrix-factorisation SGD (`mf_sgd_clock`): the
               training step, forward (residuals) and backward (both factors'
               updates) in one call; returns the new table version and the
               running squared loss
  sequential   the same with per-entry SGD inside each worker
               (`mf_sgd_clock_sequential`)
  rows         the parameter-server interface: every worker GETs its rows and
               INCs its updates, then CLOCK; returns the rows and the version
  objective    the training objective over all entries at the newest version,
               which a program reads to follow convergence, whole or by worker

A case's state is warmed by s + 2 passes, so that the ring holds s + 2
different versions, as it does in all but a run's first clocks.
"""
import math

import numpy as np
import torch

from paper_1410_8043_gb300 import esspt

SCHED_SEED = 8043
ESSP_P = 0.7
ESSP_MAX_DELAY = 3
LAM = 0.05


def _clock(name, N, M, K, P, F, s, n, model="ssp", user_a=0.0, item_a=0.0, cap=20, eta=0.005, v0=0.0, kind="clock"):
    """An MF case: N users x M items, rank K, P workers, F minibatches of n
    entries (one per clock), staleness s.  user_a / item_a: Zipf exponent of
    the popularity of users / items (0 = uniform)."""
    c = dict(kind=kind, N=N, M=M, K=K, P=P, F=F, s=s, n=n, model=model, user_a=user_a, item_a=item_a, cap=cap,
             eta=eta, v0=v0)
    return dict(c, name=name) if name else c


def _rows(name, rows, K, P, s, n, model="ssp"):
    """A GET / INC / CLOCK case: P workers with n rows each of a rows x K table."""
    c = dict(kind="rows", rows=rows, K=K, P=P, s=s, n=n, model=model)
    return dict(c, name=name) if name else c


def listed():
    return [
        # The smallest training step (the repository's tiny workload): 10k
        # entries per clock, where launches and latency are all there is.
        _clock("tiny_ssp_k16", 2000, 1000, 16, 4, 10, 2, 10_000, cap=0, eta=0.01),
        # Narrow rows under eager push, ragged sizes: the low ranks that a
        # first model or a quick sweep uses.
        _clock("narrow_essp_k32", 200_003, 30_011, 32, 64, 3, 3, 2_000_003, model="essp", item_a=0.8),
        # A mid-sized catalogue with popular items, rank 48, eager push.
        _clock("store_essp_k48", 300_007, 40_009, 48, 64, 3, 2, 1_500_007, model="essp", item_a=1.0),
        # The Netflix-shaped matrix of the paper's experiment (mid workload).
        _clock("mid_ssp_k100", 480_000, 18_000, 100, 32, 4, 3, 5_000_000, item_a=1.0),
        # The same under the value bound and under the row-granular cache.
        _clock("mid_vap_k100", 480_000, 18_000, 100, 32, 4, 3, 5_000_000, model="vap", item_a=1.0, v0=0.3),
        _clock("mid_row_k100", 480_000, 18_000, 100, 32, 4, 3, 5_000_000, model="ssp_row", item_a=1.0),
        # High rank, as wide models use it.
        _clock("wide_ssp_k256", 100_003, 20_011, 256, 8, 3, 1, 1_000_003, item_a=0.7),
        # The largest clock (large workload: 10M x 1M, 40M entries per clock),
        # very active users and items beside millions with a few entries.
        _clock("large_ssp_k64", 10_000_000, 1_000_000, 64, 128, 2, 4, 40_000_000, user_a=1.1, item_a=1.1),
        # Per-entry SGD inside each worker.
        _clock("sequential_k64", 20_000, 2000, 64, 16, 4, 2, 64_000, item_a=0.8, kind="sequential"),
        # A program that uses the table itself: GET, INC, CLOCK.
        _rows("rows_k64", 100_003, 64, 16, 2, 2001),
        # The objective over the mid data, read after a clock.
        _clock("objective_k100", 480_000, 18_000, 100, 32, 4, 3, 5_000_000, item_a=1.0, kind="objective"),
        # The objective by worker, with popular users, rank 64.
        _clock("worker_objective_k64", 100_003, 20_011, 64, 37, 3, 2, 500_009, model="essp", user_a=0.8, item_a=0.8,
               kind="worker_objective"),
    ]


def draw(rng):
    def logu(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(["clock"] * 7 + ["rows", "sequential", "objective", "worker_objective"])
    K = 4 * logu(1, 128)
    P = logu(1, 512)
    s = rng.randint(0, 8)
    if kind == "rows":
        rows = logu(500, 2_000_000)
        return _rows(None, rows, K, min(P, 32), s, logu(1, 20_000), rng.choice(["ssp", "essp", "ssp_row"]))
    N = logu(300, 3_000_000)
    M = logu(50, 300_000)
    while (N + M) * K * (s + 2) > 3 << 30:  # at most 12 GB of versions
        N, M = N // 2 + 1, M // 2 + 1
    if kind == "sequential":
        n = logu(500, 40_000)
        N, M, P = min(N, 50_000), min(M, 5000), rng.randint(max(1, n // 6000), max(2, n // 100))
        P = min(P, 512)
        model = rng.choice(["ssp", "essp"])
    else:
        n = logu(2000, min(8_000_000, 600_000_000 // K))
        model = rng.choice(["ssp", "ssp", "essp", "essp", "vap", "ssp_row"])
    if model == "ssp_row" and P * (N + M) > 1 << 28:
        P = 32
    user_a = rng.choice([0.0, 0.0, round(rng.uniform(0.6, 1.2), 2)])
    item_a = rng.choice([0.0, round(rng.uniform(0.6, 1.2), 2), round(rng.uniform(0.6, 1.2), 2)])
    return _clock(None, N, M, K, P, rng.randint(2, 4), s, n, model=model, user_a=user_a, item_a=item_a, cap=20,
                  eta=0.005 if s <= 3 else 0.002, v0=0.3 if model == "vap" else 0.0, kind=kind)


# -- inputs -------------------------------------------------------------------
def _ids(g, n, size, a):
    """n ids in [0, size): uniform, or Zipf(a) with the ranks scattered over the ids."""
    if a == 0.0:
        return torch.randint(size, (n,), generator=g, device="cuda", dtype=torch.int32)
    # whole-number weights, so that the running sums are the same on every run
    weight = (torch.arange(1, size + 1, device="cuda", dtype=torch.float64).pow_(-a) * (1 << 40)).long()
    cdf = weight.cumsum(0)
    total = int(cdf[-1])
    perm = torch.randperm(size, generator=g, device="cuda").to(torch.int32)
    out = torch.empty(n, device="cuda", dtype=torch.int32)
    for lo in range(0, n, 1 << 24):
        hi = min(n, lo + (1 << 24))
        u = torch.randint(total, (hi - lo,), generator=g, device="cuda")
        out[lo:hi] = perm[torch.searchsorted(cdf, u, right=True)]
    return out


def _mf_inputs(c, seed):
    """Observed entries (ratings 1..5 around a low-rank truth), their partition
    over workers and minibatches, and the initial factors."""
    g = torch.Generator(device="cuda").manual_seed(seed)
    N, M, K, n_obs = c["N"], c["M"], c["K"], c["n"] * c["F"]
    i, j = _ids(g, n_obs, N, c["user_a"]), _ids(g, n_obs, M, c["item_a"])
    r = 4
    U = torch.randn(N, r, generator=g, device="cuda") * r ** -0.25
    V = torch.randn(M, r, generator=g, device="cuda") * r ** -0.25
    D = torch.randn(n_obs, generator=g, device="cuda").mul_(0.9).add_(3.6)
    for lo in range(0, n_obs, 1 << 24):
        hi = min(n_obs, lo + (1 << 24))
        D[lo:hi] += (U[i[lo:hi]] * V[j[lo:hi]]).sum(1)
    D = D.round_().clamp_(1.0, 5.0)
    mb = torch.randint(c["F"], (n_obs,), generator=g, device="cuda", dtype=torch.uint8)
    worker = torch.randint(c["P"], (N,), generator=g, device="cuda", dtype=torch.int32)
    rows = torch.randn(N + M, K, generator=g, device="cuda").mul_(K ** -0.5)
    return i, j, D, mb, worker, rows


def _rows_inputs(c, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    rows = torch.randn(c["rows"], c["K"], generator=g, device="cuda")
    ids = torch.randint(c["rows"], (c["P"], c["n"]), generator=g, device="cuda", dtype=torch.int32)
    inc = torch.randn(c["P"], c["n"], c["K"], generator=g, device="cuda").mul_(0.01)
    return rows, ids, inc


class _State:
    """A table and what a training loop keeps beside it."""

    def __init__(self, c, n_rows):
        self.c = c
        self.done = 0  # clocks completed: the newest version
        self.t = esspt.Table(n_rows, c["K"], c["P"], c["s"], model=c["model"], seed=SCHED_SEED, essp_p=ESSP_P,
                             essp_max_delay=ESSP_MAX_DELAY, vap_v0=c.get("v0", 0.0))
        words = (c["s"] + 2) * n_rows * c["K"]
        # version v of the table sits in slot v mod (s + 2) of the workspace
        self.ring = self.t.workspace[: 4 * words].view(torch.float32).view(c["s"] + 2, n_rows, c["K"])
        self.loss = torch.zeros(1, dtype=torch.float64, device="cuda")

    def newest(self):
        return self.ring[self.done % (self.c["s"] + 2)]


def prepare(case, seed):
    c = case
    if c["kind"] == "rows":
        rows, ids, inc = _rows_inputs(c, seed)
        st = _State(c, c["rows"])
        st.t.table_init(rows)
        st.ids, st.inc = list(ids), list(inc)
        st.out = torch.empty(c["P"], c["n"], c["K"], device="cuda")
        st.outs = list(st.out)
        for _ in range(c["s"] + 2):
            _rows_pass(st)
        return st
    i, j, D, mb, worker, rows = _mf_inputs(c, seed)
    st = _State(c, c["N"] + c["M"])
    st.t.mf_load(i, j, D, mb, worker, c["N"], c["F"])
    st.t.table_init(rows)
    for _ in range(c["s"] + 2):
        _mf_pass(st, None)
    return st


def _mf_pass(st, loss):
    c = st.c
    if c["kind"] == "sequential":
        st.t.mf_sgd_clock_sequential(c["eta"], LAM, c["cap"], loss)
    else:
        st.t.mf_sgd_clock(c["eta"], LAM, c["cap"], loss)
    st.done += 1


def _rows_pass(st):
    for p in range(st.c["P"]):
        st.t.get(p, st.ids[p], out=st.outs[p])
        st.t.inc(p, st.ids[p], st.inc[p])
    st.t.clock()
    st.done += 1


def run(state):
    kind = state.c["kind"]
    if kind == "rows":
        _rows_pass(state)
        return {"rows": state.out, "version": state.newest()}
    if kind == "objective":
        return np.array(state.t.mf_objective(state.done, LAM))
    if kind == "worker_objective":
        sq, pen = state.t.mf_worker_objective_noalloc(state.done, LAM)
        return {"sq": sq, "pen": pen}
    _mf_pass(state, state.loss)
    return {"version": state.newest(), "loss": state.loss}


# -- what a pass cannot do without ---------------------------------------------
def _touched(n, size, a):
    """Expected number of distinct ids among n draws."""
    if a == 0.0:
        return size * -math.expm1(-n / size)
    p = np.arange(1, size + 1, dtype=np.float64) ** -a
    return float(-np.expm1(-n * (p / p.sum())).sum())


def work(case):
    c = case
    K = c["K"]
    if c["kind"] == "rows":  # the version read and written, the rows fetched, the updates read
        n = c["P"] * c["n"]
        return {"bytes": 8 * K * c["rows"] + 12 * K * n + 8 * n, "flops": K * n}
    if c["kind"] in ("objective", "worker_objective"):
        n = c["n"] * c["F"]
        return {"bytes": 12 * n + 4 * K * (_touched(n, c["N"], c["user_a"]) + _touched(n, c["M"], c["item_a"])),
                "flops": 2 * K * n}
    # each entry, and each row that changes: read once, written once
    rows = _touched(c["n"], c["N"], c["user_a"]) + _touched(c["n"], c["M"], c["item_a"])
    return {"bytes": 12 * c["n"] + 8 * K * rows, "flops": 10 * K * c["n"]}


def tolerance(case):
    if case["kind"] in ("objective", "worker_objective"):
        # fp32 residuals of random sign, summed in 64 bits (6e-10 off the 64-bit value)
        return {"rel": 1e-8, "max": 1e-7}
    # fp32 tables after a few clocks of fp32 sums in another order: within 2e-7
    # of the 64-bit ones, single values of two runs within 6e-7
    return {"rel": 1e-6, "max": 2e-6}


# -- the same in 64 bits ------------------------------------------------------
_MASK = (1 << 64) - 1


def _mix(z):
    z = ((z ^ (z >> 30)) * 0xBF58476D1CE4E5B9) & _MASK
    z = ((z ^ (z >> 27)) * 0x94D049BB133111EB) & _MASK
    return z ^ (z >> 31)


def _draw64(stream, index):
    """Draw `index` of a SplitMix64 stream of the schedule's seed."""
    return _mix(((_mix(SCHED_SEED) ^ _mix(stream)) + (index + 1) * 0x9E3779B97F4A7C15) & _MASK)


def _read_versions(c, clk, prev, X):
    """v_p(clk) of every worker (list), from those of the clock before."""
    s = c["s"]
    if c["model"] == "ssp":
        return [max(0, clk - 1 - (clk - 1 + (((_draw64(101, p) >> 32) * (s + 1)) >> 32)) % (s + 1))
                for p in range(c["P"])]
    if c["model"] == "essp":
        thr = [math.floor((1.0 - ESSP_P) ** k * 4294967296.0) for k in range(1, min(ESSP_MAX_DELAY, s) + 1)]
        out = []
        for p in range(c["P"]):
            u = _draw64(102, (clk << 32) | p) >> 32
            out.append(max(prev[p], clk - 1 - sum(u < t for t in thr), 0))
        return out
    if c["model"] == "vap":
        cur = X[(clk - 1) % (s + 2)]
        for k in range(min(s, clk - 1), 0, -1):
            if float((cur - X[(clk - 1 - k) % (s + 2)]).abs().max()) <= c["v0"] / math.sqrt(clk):
                return [clk - 1 - k] * c["P"]
    return [clk - 1] * c["P"]  # vap: the newest; ssp_row: versions are per row


def _f32(x):
    return float(np.float32(x))


class _Ring64:
    def __init__(self, c, rows):
        self.c, self.n_rows = c, rows.shape[0]
        self.X = torch.zeros(c["s"] + 2, *rows.shape, dtype=torch.float64, device="cuda")
        self.X[0] = rows
        self.clk, self.v = 1, [0] * c["P"]
        if c["model"] == "ssp_row":
            self.V = torch.full((c["P"] * self.n_rows,), -1, dtype=torch.int32, device="cuda")

    def start(self):
        if self.clk > 1 or self.c["model"] == "vap":
            self.v = _read_versions(self.c, self.clk, self.v, self.X)

    def finish(self, delta):
        ns = self.c["s"] + 2
        torch.add(self.X[(self.clk - 1) % ns], delta, out=self.X[self.clk % ns])
        self.clk += 1
        return self.X[(self.clk - 1) % ns]

    def row_versions(self, p, r):
        """Row-granular cache: the version at which worker p (tensor or int) reads row r, refreshed first."""
        at = p * self.n_rows + r
        v = self.V[at]
        self.V[at] = torch.where((v < 0) | (v < self.clk - 1 - self.c["s"]), self.clk - 1, v).to(torch.int32)
        return self.V[at].long()


def _clock64(ring, c, data, acc_loss):
    i, j, D, mb, worker = data
    N, ns, K = c["N"], c["s"] + 2, c["K"]
    ring.start()
    sel = torch.nonzero(mb == (ring.clk - 1) % c["F"]).view(-1)
    delta = torch.zeros(ring.n_rows, K, dtype=torch.float64, device="cuda")
    X = ring.X.view(-1, K)
    vw = torch.tensor(ring.v, device="cuda")
    step = max(1 << 12, (1 << 27) // K)
    lam = _f32(LAM)
    for lo in range(0, sel.numel(), step):
        e = sel[lo:lo + step]
        u, r, p = i[e].long(), j[e].long() + N, worker[i[e].long()].long()
        if c["model"] == "ssp_row":
            vu, vr = ring.row_versions(p, u) % ns, ring.row_versions(p, r) % ns
        else:
            vu = vr = vw[p] % ns
        L, R = X[vu * ring.n_rows + u], X[vr * ring.n_rows + r]
        res = D[e].double() - (L * R).sum(1)
        acc_loss += (res * res).sum()
        res = res[:, None]
        delta.index_add_(0, u, res * R - lam * L)
        delta.index_add_(0, r, res * L - lam * R)
    delta *= _f32(c["eta"])
    if c["cap"] > 0:
        n = torch.bincount(i[sel].long(), minlength=N).double()
        m = torch.bincount(j[sel].long(), minlength=c["M"]).double()
        delta *= (c["cap"] / torch.cat([n, m]).clamp_(min=1.0)).clamp_(max=1.0)[:, None]
    return ring.finish(delta)


def _sequential64(ring, c, data, acc_loss):
    i, j, D, mb, worker = data
    N, M, P, ns, K = c["N"], c["M"], c["P"], c["s"] + 2, c["K"]
    ring.start()
    eta, lam = _f32(c["eta"]), _f32(LAM)
    sel = np.nonzero(mb == (ring.clk - 1) % c["F"])[0]
    sel = sel[np.argsort(i[sel], kind="stable")]
    own = worker[i[sel]]
    sel = sel[np.argsort(own, kind="stable")]
    own = np.sort(own, kind="stable")
    first = np.searchsorted(own, np.arange(P + 1))
    X = ring.X.cpu().numpy()
    dL, mine = np.zeros((N, K)), np.zeros((P, M, K))
    slot = np.array(ring.v) % ns
    order = np.argsort(-np.diff(first), kind="stable")  # the longest chains first
    cnt = np.diff(first)[order]
    for t in range(int(cnt[0]) if P else 0):
        p = order[: np.searchsorted(-cnt, -t, side="left")]  # workers with more than t entries
        e = sel[first[p] + t]
        u, r = i[e], j[e]
        L, R = X[slot[p], u] + dL[u], X[slot[p], N + r] + mine[p, r]
        res = D[e] - (L * R).sum(1)
        acc_loss += float((res * res).sum())
        dL[u] += eta * (res[:, None] * R - lam * L)
        mine[p, r] += eta * (res[:, None] * L - lam * R)
    delta = np.concatenate([dL, mine.sum(0)])
    if c["cap"] > 0:
        n = np.concatenate([np.bincount(i[sel], minlength=N), np.bincount(j[sel], minlength=M)])
        delta *= np.minimum(1.0, c["cap"] / np.maximum(n, 1))[:, None]
    return ring.finish(torch.from_numpy(delta).cuda())


def exact(case, seed):
    c = case
    if c["kind"] == "rows":
        rows, ids, inc = _rows_inputs(c, seed)
        ring = _Ring64(c, rows)
        ns = c["s"] + 2
        for _ in range(c["s"] + 3):
            ring.start()
            out, delta = [], torch.zeros_like(ring.X[0])
            for p in range(c["P"]):
                r = ids[p].long()
                v = ring.row_versions(p, r) % ns if c["model"] == "ssp_row" else ring.v[p] % ns
                out.append(ring.X[v, r])
                delta.index_add_(0, r, inc[p].double())
            version = ring.finish(delta)
        return {"rows": torch.stack(out), "version": version}
    i, j, D, mb, worker, rows = _mf_inputs(c, seed)
    ring = _Ring64(c, rows)
    del rows
    loss = torch.zeros(1, dtype=torch.float64, device="cuda")
    host = tuple(x.cpu().numpy() for x in (i, j, D.double(), mb, worker)) if c["kind"] == "sequential" else None
    objective = c["kind"] in ("objective", "worker_objective")
    for _ in range(c["s"] + (2 if objective else 3)):
        loss.zero_()
        if c["kind"] == "sequential":
            version = _sequential64(ring, c, host, loss)
        else:
            version = _clock64(ring, c, (i, j, D, mb, worker), loss)
    if not objective:
        return {"version": version, "loss": loss}
    sq, pen = (torch.zeros(c["P"], dtype=torch.float64, device="cuda") for _ in range(2))
    for lo in range(0, i.numel(), 1 << 20):
        u, r = i[lo:lo + (1 << 20)].long(), j[lo:lo + (1 << 20)].long() + c["N"]
        L, R, p = version[u], version[r], worker[u].long()
        e2 = (D[lo:lo + (1 << 20)].double() - (L * R).sum(1)) ** 2
        sq.index_add_(0, p, e2)
        pen.index_add_(0, p, e2 + _f32(LAM) * ((L * L).sum(1) + (R * R).sum(1)))
    if c["kind"] == "objective":
        return np.array([float(sq.sum()), float(pen.sum())])
    return {"sq": sq.cpu().numpy(), "pen": pen.cpu().numpy()}
