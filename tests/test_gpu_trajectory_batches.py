"""The trajectory walker's batches of 32 trial moves where they can go wrong (Sec. 4.2, Eq. 4): interval
lengths around a batch, lattices on which most moves touch another one, conflict tables that sites share,
moves that go many bins, and ln g whose sums of ln f are exact, round, or are too large for the quick
decisions.  The walk must be the FP64 oracle's bit for bit."""
import numpy as np
import pytest

from rewl_pairs import assert_same_state, make_pair

pytestmark = pytest.mark.gpu

J = (1.0, 0.5, -0.05, 0.1)
B = 300


def _start(name):
    ragged = np.random.default_rng(4).normal(0.0, 3.0, B)
    return {"exact": (np.zeros(B), 1.0), "negative": (np.floor(ragged) * 2.0**-20 - 7.0, 2.0**-20),
            "rounding": (20.0 + ragged, 0.37), "huge": (3.0e9 + ragged, 1.0)}[name]


@pytest.mark.parametrize("start", ["exact", "negative", "rounding", "huge"])
@pytest.mark.parametrize("L,shells,moves", [(4, 1, 31), (4, 4, 32), (4, 2, 1000), (5, 3, 33), (9, 2, 700), (14, 4, 95),
                                            (14, 2, 1)])
def test_batches_match_the_oracle(L, shells, moves, start):
    gpu, orc = make_pair(L=L, J=J[:shells], n_bins=B, n_windows=2, walkers_per_window=2, overlap=0.75, flatness=0.8,
                         lnf_final=1e-9, seed=L + moves, exchange_interval=moves)
    assert gpu.info()["pipelined"] == 1
    gpu.init_walkers()
    orc.init_walkers()
    lng, lnf0 = _start(start)
    gpu.set_initial_lng(lng, lnf0)
    orc.set_lng(lng, lnf0)
    gpu.run_intervals(6)
    orc.run_intervals(6)
    assert_same_state(gpu, orc)
    gpu.close()


def test_narrow_bins_match_the_oracle():
    """12000 bins of bcc L = 4: most moves go more than the 64 bins that a quick decision covers."""
    gpu, orc = make_pair(L=4, J=J[:2], n_bins=12000, n_windows=1, walkers_per_window=2, overlap=0.0, flatness=0.8,
                         lnf_final=1e-9, seed=8, exchange_interval=500)
    gpu.init_walkers()
    orc.init_walkers()
    gpu.run_intervals(4)
    orc.run_intervals(4)
    assert_same_state(gpu, orc)
    gpu.close()
