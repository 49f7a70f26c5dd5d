"""The production walker with several lanes per move (Sec. 4.2, Eq. 4): a batch of 32 / G moves is evaluated
at once and its accepted moves are found one by one.  Walked one move per call no move can touch another of
its batch, so any other split of the same moves over calls must give the same state, bit for bit (the energy
recomputation goes by the number of calls: none here)."""
import numpy as np
import pytest

import paper_1411_4212_gb300 as rw

pytestmark = pytest.mark.gpu

J = (1.0, 0.5, -0.05, 0.1)
MOVES = 198
RING = np.array([[(i + d) % 60 for i in range(60)] for d in (1, 2, 59, 58)], dtype=np.int32)
SPECS = [dict(kind=rw.BCC, L=L, J=J[:shells], group_size=G)
         for L, shells, G in ((3, 1, 16), (4, 1, 8), (4, 2, 8), (5, 3, 8), (4, 4, 16), (6, 4, 8), (6, 2, 4), (6, 3, 4), (7, 2, 2),
                              (4, 2, 32), (30, 2, 4))]
SPECS += [dict(kind=rw.CHAIN, L=40, J=(1.0,), group_size=2),
          dict(kind=rw.TABLE, nbr=RING, Jt=np.full((4, 60), 0.7), e_min=-80.0, e_max=0.0, group_size=4)]


@pytest.mark.parametrize("spec", SPECS, ids=lambda s: f"kind{s['kind']}-L{s.get('L')}-G{s['group_size']}-{len(s.get('J', ()))}")
def test_any_split_of_the_moves_over_calls_gives_the_same_walk(spec):
    states = []
    for moves in (1, 6, 33, 66, MOVES):
        g = rw.REWL(n_bins=120, n_windows=2, walkers_per_window=3, overlap=0.75, flatness=0.8, lnf_final=1e-8, seed=5, recompute_every=1000,
                    exchange_interval=moves, **spec)
        assert g.info()["pipelined"] == 0
        g.init_walkers()
        for _ in range(MOVES // moves):
            g.walk()
        w = g.walkers()
        state = {k: np.array(w[k]).view(np.int64) if w[k].dtype == np.float64 else np.array(w[k]) for k in w}
        state["spins"] = g.spins().view(np.int64)
        assert (state["steps"] == MOVES).all() and state["accepts"].max() > 0
        states.append((moves, state))
        g.close()
    for moves, s in states[1:]:
        for k in s:
            assert np.array_equal(s[k], states[0][1][k]), f"{moves} moves per call: {k}"
