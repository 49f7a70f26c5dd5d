"""Batches of 32 trial moves on lattices of so few sites that moves of one batch follow each other on the same
site all the time (bcc L = 2: 16 sites, L = 3: 54): the change that an accepted move makes to its site, which a
later move of the batch has replaced by then, is what the moves after that one are corrected with."""
import numpy as np
import pytest

import paper_1411_4212_gb300 as rw

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("L,J", [(2, (1.0,)), (3, (1.0,)), (3, (1.0, 0.5))])
@pytest.mark.parametrize("moves", [33, 1000])
def test_moves_that_follow_each_other_on_a_site(L, J, moves):
    n_int, per_site = 12, sum(z * j for z, j in zip((8, 6), J))
    N = 2 * L ** 3
    states = []
    for resolver in (rw.RESOLVER_AUTO, rw.RESOLVER_SCAN, rw.RESOLVER_BLOCKS, rw.RESOLVER_SEQUENTIAL):
        with rw.REWL(kind=rw.BCC, L=L, J=J, n_bins=24, n_windows=2, walkers_per_window=2, lnf_final=1e-8, seed=L + moves,
                     exchange_interval=moves, recompute_every=1000, group_size=1, resolver=resolver) as g:
            assert g.info()["pipelined"] == 1
            g.run_intervals(n_int, stats=False)
            w = g.walkers()
            exact = g.replica_energies()[w["replica"]]
            # an accepted move's dE: at most 15 FP32 roundings of sums below 2 per_site, and half a 2^-24 bin
            bound = n_int * moves * (15 * 2.0 ** -24 * 2 * per_site + 2.0 ** -25 * 0.5 * per_site * N / 24)
            assert np.abs(w["E"] - exact).max() < bound + 1e-6
            states.append([np.array(w[k]) for k in sorted(w)] + [g.spins()])
    assert len(states) == 4
    for s in states[1:]:
        for a, b in zip(states[0], s):
            assert np.array_equal(a, b)
