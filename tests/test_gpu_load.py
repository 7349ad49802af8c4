"""The load's layout where its bounds are tightest, and what device memory it asks for."""
import ctypes

import numpy as np
import pytest
import torch

from gen import make_mf_data
from oracle import Oracle, OracleConfig

pytestmark = pytest.mark.gpu

TOL = 1e-4  # the bar of every parameter after every clock (test_gpu_parity.py)


# Entries per user within a tile of 4096 users: the lists fall from 96 to 1 once per tile, so that a
# round of eight items mixes both at every edge of a tile; one list per user; chunks of 64 beside them.
LENGTHS = {
    "one long, others short": lambda u: np.where(u % 4096 == 7, 96, 1),
    "seven long, others one": lambda u: np.where(u % 4096 < 7, 95, 1),
    "one each": lambda u: np.ones_like(u),
    "odd lengths, most idle": lambda u: np.where(u % 5 == 0, 2 * (u % 40) + 1, 0),
    "a heavy user per tile": lambda u: np.where(u % 4096 == 4095, 300, u % 2),
}


@pytest.mark.parametrize("name", list(LENGTHS))
@pytest.mark.parametrize("K", [4, 12, 32, 64, 100, 132, 388])
def test_layout_of_uneven_tiles(K, name):
    """Every place is reserved and filled: two clocks against the oracle."""
    N, M, P, F = 3 * 4096 + 5, 29, 3, 2
    lens = LENGTHS[name](np.arange(N))
    i = np.repeat(np.arange(N), lens).astype(np.int32)
    d = make_mf_data(n_users=N, n_items=M, n_obs=2 * i.size, K=K, seed=K, truth_rank=4, truth_var=0.5, noise_var=0.1,
                     init_var=1.0 / K)
    d.i, mb = np.concatenate([i, i]), np.repeat(np.arange(F), i.size).astype(np.uint8)
    wp = (np.arange(N) % P).astype(np.int32)
    from paper_1410_8043_gb300 import esspt

    t = esspt.Table(N + M, K, P, 1, model="ssp")
    t.mf_load(d.i, d.j, d.D, mb, wp, N, F)
    t.table_init(np.concatenate([d.L0, d.R0]))
    o = Oracle(OracleConfig(n_users=N, n_items=M, K=K, P=P, s=1, F=F, model="ssp", eta=0.01, lam=0.05, cap=12),
               d.i, d.j, d.D, mb, wp, d.L0, d.R0)
    for c in (1, 2):
        t.mf_sgd_clock(0.01, 0.05, 12)
        o.clock()
        g, x = t.read_table(c).cpu().numpy().astype(np.float64), o.table()
        assert float((np.abs(g - x) - TOL * (1 + np.abs(x))).max()) <= 0.0, f"clock {c}: {np.abs(g - x).max():.3e}"
    t.poll()
    t.close()


# Workspace and scratch that the load may ask for, GB.  Per entry: 12 bytes of entries and 12 of
# stream words, a place more for each user's odd entry at two entries per step (K <= 64), 20 bytes
# per work item (a user with entries in a minibatch); per user and minibatch 4 bytes, and 40 of
# scratch beside 4 per entry.
@pytest.mark.parametrize("n,N,M,F,K,workspace,scratch", [
    (100_000, 2000, 1000, 10, 16, 0.007, 0.003),
    (100_000_000, 480_000, 18_000, 20, 100, 3.1, 0.9),
    (1_000_000_000, 8_000_000, 1_000_000, 100, 16, 59.0, 37.0),
])
def test_memory_of_the_load(n, N, M, F, K, workspace, scratch):
    from paper_1410_8043_gb300 import esspt

    t = esspt.Table(N + M, K, 4, 0, model="ssp")
    L = esspt.lib()
    ws = L.esspt_mf_workspace_bytes(t._h, ctypes.c_int64(n), ctypes.c_int64(N), ctypes.c_int32(F)) / 1e9
    sc = L.esspt_mf_scratch_bytes(t._h, ctypes.c_int64(n), ctypes.c_int64(N), ctypes.c_int32(F)) / 1e9
    assert 0 < ws <= workspace and 0 < sc <= scratch, (ws, sc)
    t.close()
    del t
    torch.cuda.empty_cache()
