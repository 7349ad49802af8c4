"""GPU parity at the edges of the objective, VAP scan, sequential and GET / INC
kernels: row widths at the ends of every lane shape, lists around a part, a
segment and a ring, tables on both sides of the VAP rule."""
import numpy as np
import pytest
import torch

from gen import make_mf_data, minibatch_labels, shard_users
from oracle import Oracle, OracleConfig

pytestmark = pytest.mark.gpu

TOL = 1e-4  # the bar of every parameter after every clock (test_gpu_parity.py)
EPS = 2.0**-24


def _esspt():
    from paper_1410_8043_gb300 import esspt

    return esspt


def _mf(N, M, K, n, P, F, seed, **kw):
    d = make_mf_data(n_users=N, n_items=M, n_obs=n, K=K, seed=seed, truth_rank=4, truth_var=0.5, noise_var=0.1,
                     init_var=1.0 / K, **kw)
    return d, shard_users(N, P, seed + 1), minibatch_labels(n, F, seed + 2)


# (users, entries): items taken in parts (few items); users of one entry to
# several chunks; and more items than the GPU holds groups (taken whole).
@pytest.mark.parametrize("N,n", [(3, 40), (50, 3000), (400_000, 800_000)])
@pytest.mark.parametrize("K", [4, 16, 20, 32, 36, 64, 68, 96, 100, 128, 132, 192, 196, 256, 260, 384, 388, 512])
def test_objective_shapes(K, N, n):
    """Whole and by worker, against 64-bit sums over the same fp32 table.  A
    residual of K products differs by at most d = (K + 2) eps (|D| + sum |L R|),
    its square by 2 |e| d + d^2; a row's |.|^2 by (K + 2) eps of itself; the sums
    add (8 + 4) eps of the total."""
    if N > 1000 and K not in (4, 64, 100, 132):
        pytest.skip("large lists at one width of each group size")
    P, F, lam = 5, 2, 0.05
    d, wp, mb = _mf(N, 60, K, n, P, F, 300 + K)
    t = _esspt().Table(N + 60, K, P, 1, model="ssp")
    t.mf_load(d.i, d.j, d.D, mb, wp, N, F)
    t.table_init(np.concatenate([d.L0, d.R0]))
    sq, pen, sq_b, pen_b = (np.zeros(P) for _ in range(4))
    for a in range(0, n, 100_000):
        b = slice(a, a + 100_000)
        L, R = d.L0[d.i[b]].astype(np.float64), d.R0[d.j[b]].astype(np.float64)
        e = d.D[b].astype(np.float64) - (L * R).sum(1)
        dl = (K + 2) * EPS * (np.abs(d.D[b]) + np.abs(L * R).sum(1))
        rows = (L * L).sum(1) + (R * R).sum(1)
        eb = 2 * np.abs(e) * dl + dl * dl + 12 * EPS * e * e
        p = np.asarray(wp)[d.i[b]]
        sq += np.bincount(p, e * e, P)
        pen += np.bincount(p, e * e + lam * rows, P)
        sq_b += np.bincount(p, eb, P)
        pen_b += np.bincount(p, eb + lam * (K + 14) * EPS * rows, P)
    gs, gp = t.mf_objective(0, lam)
    assert abs(gs - sq.sum()) <= sq_b.sum() and abs(gp - pen.sum()) <= pen_b.sum()
    ws, wpen = t.mf_worker_objective_noalloc(0, lam)
    assert (np.abs(ws - sq) <= sq_b).all() and (np.abs(wpen - pen) <= pen_b).all()
    t.close()


def _constant_objective(K, N, n, D, element, P=3, long=0):
    """Objective inputs: every entry's value D (or an array of them); L's first and R's last value `element`, the rest
    0, so that the residual is the value and every row's square is one product.  The first `long` entries are of two
    users.  Returns whole and by-worker sums."""
    M, F = 7, 2
    i = torch.arange(n, dtype=torch.int32, device="cuda") % N
    i[:long] %= 2
    rows = torch.zeros((N + M, K), device="cuda")
    rows[:N, 0] = element
    rows[N:, K - 1] = element
    t = _esspt().Table(N + M, K, P, 1, model="ssp")
    t.mf_load(i, (torch.arange(n, dtype=torch.int32, device="cuda") * 5) % M,
              torch.as_tensor(D, dtype=torch.float32, device="cuda").expand(n).contiguous(),
              (torch.arange(n, device="cuda") % F).to(torch.uint8),
              torch.arange(N, dtype=torch.int32, device="cuda") % P, N, F)
    t.table_init(rows)
    out = t.mf_objective(0, 0.5), t.mf_worker_objective_noalloc(0, 0.5)
    t.close()
    return out, np.bincount(i.cpu().numpy() % P, minlength=P)


# Items taken in parts (few items, of 2, 8 and 96 entries), whole, and in parts as some are far longer than the others.
@pytest.mark.parametrize("N,n,long", [(40, 120, 0), (700, 40_000, 0), (3, 3000, 0), (200_000, 4_000_000, 0), (30_000, 40_000, 700)])
@pytest.mark.parametrize("K", [8, 32, 64, 96, 128, 256, 512])
def test_objective_sums_are_exact(K, N, n, long):
    """The value's square has 27 bits (24 in its high fp32 part, one in its low one), a row's |.|^2 24, and both
    sums keep every bit: each is a multiple of 2^-26 below 2^27, with fewer than 24 bits lost per lane."""
    x = 1 + 2.0**-11 + 2.0**-13
    norm = float(np.float32(x) * np.float32(x))
    assert norm != x * x and norm + 2.0**-26 == x * x
    ((sq, pen), (wsq, wpen)), cnt = _constant_objective(K, N, n, x, x, long=long)
    assert (sq, pen) == (n * x * x, n * (x * x + norm))
    assert (wsq == cnt * (x * x)).all() and (wpen == cnt * (x * x + norm)).all()


@pytest.mark.parametrize("K", [4, 64, 100])
@pytest.mark.parametrize("value,element", [(9e17, 0.0), (3e14, 0.0), (1e25, 0.0), (0.0, 9e17), (0.0, 1.5e19),
                                           (3.0, 3e14), (1e-20, 0.0)])
def test_objective_beyond_fp32_sums(K, value, element):
    """Squares whose sum, or themselves, pass what fp32 holds: finite wherever a sum in 64 bits is, to 1e-12."""
    n, v, a = 2_000_000, float(np.float32(value)), np.float32(element)
    ((sq, pen), (wsq, wpen)), cnt = _constant_objective(K, 5000, n, value, element)
    norm = float(a * a)
    assert np.isfinite(norm)
    np.testing.assert_allclose([sq, pen], [n * (v * v), n * (v * v + norm)], rtol=1e-12)
    np.testing.assert_allclose(wsq, cnt * (v * v), rtol=1e-12)
    np.testing.assert_allclose(wpen, cnt * (v * v + norm), rtol=1e-12)


@pytest.mark.parametrize("K", [4, 64, 100])
@pytest.mark.parametrize("bad", [float("nan"), float("inf"), -float("inf")])
def test_objective_not_finite(K, bad):
    """One such value reaches the whole sums and its worker's, and no other worker's."""
    n, N = 3000, 300
    D = torch.ones(n)
    D[7] = bad  # user 7, worker 1 of 3
    ((sq, pen), (wsq, wpen)), cnt = _constant_objective(K, N, n, D, 0.0)
    same = np.isnan if np.isnan(bad) else np.isposinf
    assert same([sq, pen, wsq[1], wpen[1]]).all()
    assert (wsq[[0, 2]] == cnt[[0, 2]]).all() and (wpen[[0, 2]] == cnt[[0, 2]]).all()


# 100 x 4: all norms at once; 120 001 x 100 (48 MB a version, kmax = 4 and 9): the scan, in one launch and two.
@pytest.mark.parametrize("rows,K,s", [(100, 4, 3), (120_001, 100, 4), (120_001, 100, 9)])
@pytest.mark.parametrize("seed", [0, 1])
def test_vap_versions_by_inc(rows, K, s, seed):
    """One element of a random row grows by a power of two per clock, so every
    norm is exact: the read version is the stalest whose norms are within v0 /
    sqrt(c), computed here in whole numbers."""
    rng = np.random.default_rng(seed)
    t = _esspt().Table(rows, K, 2, s, model="vap", vap_v0=1.9)
    t.table_init(torch.zeros((rows, K), device="cuda"))
    hist = [{}]
    for c in range(1, 16):
        bound, want = 1.9 / np.sqrt(c), c - 1
        for k in range(min(s, c - 1), 0, -1):
            a, b = hist[c - 1], hist[c - 1 - k]
            norm = max([abs(a.get(r, 0.0) - b.get(r, 0.0)) for r in set(a) | set(b)], default=0.0)
            assert abs(norm - bound) > 1e-6 * bound
            if norm <= bound:
                want = c - 1 - k
                break
        v, clk = t.read_schedule()
        assert clk == c and list(v) == [want] * 2, (c, list(v), want)
        r, x = int(rng.choice([0, rows // 2, rows - 1])), float(2.0 ** rng.integers(-6, 2))
        dl = torch.zeros((1, K), device="cuda")
        dl[0, K - 1] = x
        t.inc(0, torch.tensor([r], dtype=torch.int32, device="cuda"), dl)
        t.clock()
        new = dict(hist[-1])
        new[r] = new.get(r, 0.0) + x
        hist.append(new)
    t.poll()
    t.close()


@pytest.mark.parametrize("n", [2, 127, 128, 129, 700])  # entries per worker about a segment of 128
@pytest.mark.parametrize("K", [4, 20, 64, 68, 128, 132, 256, 388, 512])
def test_sequential_segments_and_repeats(K, n):
    """Three items only, so that the next entries repeat an item; a worker with no user."""
    P, F, N = 3, 1, 9
    d, wp, mb = _mf(N, 3, K, 2 * n, P, F, 700 + K)
    wp = (np.arange(N) % 2).astype(np.int32)
    t = _esspt().Table(N + 3, K, P, 1, model="ssp")
    t.mf_load(d.i, d.j, d.D, mb, wp, N, F)
    t.table_init(np.concatenate([d.L0, d.R0]))
    o = Oracle(OracleConfig(n_users=N, n_items=3, K=K, P=P, s=1, F=F, model="ssp", eta=0.005, lam=0.05, cap=20,
                            sequential=True), d.i, d.j, d.D, mb, wp, d.L0, d.R0)
    for c in range(1, 4):
        t.mf_sgd_clock_sequential(0.005, 0.05, 20)
        o.clock()
        g, x = t.read_table(c).cpu().numpy().astype(np.float64), o.table()
        assert float((np.abs(g - x) - TOL * (1 + np.abs(x))).max()) <= 0.0, f"clock {c}: {np.abs(g - x).max():.3e}"
    t.close()


@pytest.mark.parametrize("model", ["ssp", "ssp_row"])
@pytest.mark.parametrize("K,n", [(4, 1), (4, 1025), (12, 33), (36, 257), (64, 2001), (100, 77), (132, 5), (512, 300)])
def test_get_inc_row_lanes(K, n, model):
    """GET copies bits at any row width and count; distinct rows' INC is one fp32 addition.  The
    version is left out of every other call."""
    rng, rows, s = np.random.default_rng(K + n), 3001, 1
    t = _esspt().Table(rows, K, 2, s, model=model)
    hist = [rng.normal(size=(rows, K)).astype(np.float32)]
    t.table_init(hist[0])
    cached = -np.ones((2, rows), np.int64)
    for c in range(1, 6):
        v, _ = t.read_schedule()
        for p in range(2):
            ids = rng.integers(0, rows, n).astype(np.int32)
            ver = np.full(n, v[p])
            if model == "ssp_row":
                old = cached[p, ids]
                ver = np.where((old < 0) | (old < c - 1 - s), c - 1, old)
                cached[p, ids] = ver
            got, oldest = t.get(p, ids, want_version=(c + p) % 2 == 0)
            assert oldest is None or oldest == ver.min()
            want = np.stack([hist[a][r] for a, r in zip(ver, ids)])
            np.testing.assert_array_equal(got.cpu().numpy(), want)
        ids = rng.permutation(rows)[:n].astype(np.int32)
        dl = rng.normal(size=(n, K)).astype(np.float32)
        t.inc(0, ids, dl)
        t.clock()
        x = hist[-1].copy()
        x[ids] += dl
        hist.append(x)
        np.testing.assert_array_equal(t.read_table(c).cpu().numpy(), x)
    t.poll()
    t.close()


def test_costs_past_31_bits():
    """380M users' entries, whose costs (6 each, in the order of the work list) pass 2^31 in
    the second of two minibatches: one entry per user and minibatch, every row of L and R a
    constant, so every user row of versions 1 and 2 has the same value, computed here.  The
    gradient's few fp32 roundings are within 1e-6 of values of order 1."""
    N, M, K, eta, lam = 190_000_000, 1000, 4, 0.01, 0.05
    if torch.cuda.mem_get_info()[0] < 120 << 30:
        pytest.skip("needs 120 GB")
    dev = "cuda"
    ids = torch.arange(N, dtype=torch.int32, device=dev)
    i = torch.cat([ids, ids])
    j = i % M
    D = torch.full((2 * N,), 3.0, device=dev)
    mb = torch.cat([torch.zeros(N, dtype=torch.uint8, device=dev), torch.ones(N, dtype=torch.uint8, device=dev)])
    t = _esspt().Table(N + M, K, 2, 0, model="ssp")
    t.mf_load(i, j, D, mb, ids % 2, N, 2)
    del i, j, D, mb, ids
    rows = torch.full((N + M, K), 0.5, device=dev)
    t.table_init(rows)
    L, R = 0.5, 0.5
    for c in (1, 2):
        t.mf_sgd_clock(eta, lam, 1)  # cap 1: an item takes the mean of its 190 000 updates
        e = 3.0 - K * L * R
        L, R = L + eta * (e * R - lam * L), R + eta * (e * L - lam * R)
        got = t.read_table(c, out=rows)
        lo, hi = float(got[:N].min()), float(got[:N].max())
        assert abs(lo - L) <= 1e-6 and abs(hi - L) <= 1e-6, (c, lo, hi, L)
        # item rows: 190 000 fp32 additions over replicas of at least 2048 each (test_gpu_parity.py's bar)
        assert float((got[N:] - R).abs().max()) <= TOL, (c, R)
    t.poll()
    t.close()


@pytest.mark.parametrize("K", [4, 64, 100, 256])
def test_loss_is_exact_over_long_ranges(K):
    """Rows of zeros, so that every residual is the value 1 + 2^-8, whose square has 17
    bits: up to 96 of them are exact in fp32, so the clock's loss is exactly n times it,
    while one fp32 sum per lane would round from its 128th on (8M entries give a lane
    hundreds)."""
    N, M, n = 50_000, 1000, 8_000_000
    i = torch.arange(n, dtype=torch.int32, device="cuda") % N
    j = (torch.arange(n, dtype=torch.int32, device="cuda") * 7) % M
    t = _esspt().Table(N + M, K, 4, 1, model="ssp")
    t.mf_load(i, j, torch.full((n,), 1 + 2.0**-8, device="cuda"), torch.zeros(n, dtype=torch.uint8, device="cuda"),
              torch.arange(N, dtype=torch.int32, device="cuda") % 4, N, 1)
    t.table_init(torch.zeros((N + M, K), device="cuda"))
    loss = torch.zeros(1, dtype=torch.float64, device="cuda")
    t.mf_sgd_clock(0.01, 0.05, 20, loss)
    assert float(loss) == n * (1 + 2.0**-8) ** 2
    t.close()
