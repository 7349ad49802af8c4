"""GPU parity of the SGD clock at the edges of its work list and row shapes:
row widths at both ends of every shape, users at the edges of the entry
windows and of the chunks, rounds with empty places, against the oracle."""
import numpy as np
import pytest

from gen import make_mf_data
from oracle import Oracle, OracleConfig

pytestmark = pytest.mark.gpu

TOL = 1e-4  # the bar of every parameter after every clock (test_gpu_parity.py)

# entries per user in one minibatch: windows hold 4 or 8 entries, a user with
# more than 96 is split in chunks of 64
LENGTHS = [0, 1, 3, 4, 5, 7, 8, 9, 15, 16, 17, 24, 25, 63, 64, 65, 95, 96, 97, 127, 128, 129, 193, 400]


def _data(K, lengths, F, M, seed):
    """Users with the given numbers of entries in every minibatch."""
    rng = np.random.default_rng(seed)
    lens = np.concatenate([rng.permutation(lengths) for _ in range(F)]).astype(np.int64)
    N = len(lengths)
    i = np.repeat(np.tile(np.arange(N), F), lens).astype(np.int32)
    mb = np.repeat(np.repeat(np.arange(F), N), lens).astype(np.uint8)
    d = make_mf_data(n_users=N, n_items=M, n_obs=i.size, K=K, seed=seed, truth_rank=4, truth_var=0.5, noise_var=0.1,
                     init_var=1.0 / K)
    order = rng.permutation(i.size)
    d.i, mb = i[order], mb[order]
    # item 0 in a third of the entries: an item of two and more replica rows
    d.j[rng.random(i.size) < 0.35] = 0
    return d, mb


def _check(K, lengths, model, s, clocks, F=2, M=37, P=3, cap=12):
    from paper_1410_8043_gb300 import esspt

    d, mb = _data(K, lengths, F, M, 100 + K)
    wp = (np.arange(d.n_users) % P).astype(np.int32)
    t = esspt.Table(d.n_users + M, K, P, s, model=model)
    t.mf_load(d.i, d.j, d.D, mb, wp, d.n_users, F)
    t.table_init(np.concatenate([d.L0, d.R0]))
    o = Oracle(OracleConfig(n_users=d.n_users, n_items=M, K=K, P=P, s=s, F=F, model=model, eta=0.01, lam=0.05,
                            cap=cap), d.i, d.j, d.D, mb, wp, d.L0, d.R0)
    for c in range(1, clocks + 1):
        t.mf_sgd_clock(0.01, 0.05, cap)
        o.clock()
        g, x = t.read_table(c).cpu().numpy().astype(np.float64), o.table()
        assert float((np.abs(g - x) - TOL * (1 + np.abs(x))).max()) <= 0.0, f"clock {c}: {np.abs(g - x).max():.3e}"
    t.poll()
    t.close()


@pytest.mark.parametrize("model", ["ssp", "ssp_row"])
@pytest.mark.parametrize("K", [4, 16, 20, 32, 36, 64, 68, 96, 100, 128, 132, 192, 196, 256, 260, 384, 388, 512])
def test_row_shapes_and_user_lengths(K, model):
    _check(K, LENGTHS * 3, model, s=1, clocks=5)


@pytest.mark.parametrize("lengths", [[1], [97], [0] * 70 + [2], [1] * 300, list(range(1, 260)) + [0] * 300])
@pytest.mark.parametrize("K", [8, 64, 100])
def test_list_lengths(K, lengths):
    """Work lists of one item, of fewer items than a round holds, and over several tiles of users."""
    _check(K, lengths, "ssp", s=0, clocks=3)
