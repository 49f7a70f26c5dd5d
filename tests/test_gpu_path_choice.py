"""Which way through a batch the production resolver takes where it may choose (rewl_counters): the first moves of a
run that starts in wide bins are nearly all accepted, with a few bin changes per batch, and belong to the warp scan;
where bins are as narrow as the moves are long, hardly any batch does."""
import pytest

import paper_1411_4212_gb300 as rw

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("L,J,bins", [(16, (1.0,), 500), (24, (1.0, 0.6), 2000)])
def test_the_first_moves_of_a_run_are_scanned(L, J, bins):
    N = 2 * L ** 3
    egs = -0.5 * sum(z * j for z, j in zip((8, 6), J)) * N
    with rw.REWL(kind=rw.BCC, L=L, J=J, n_bins=bins, n_windows=8, walkers_per_window=4, e_min=egs, e_max=0.0,
                 lnf_final=1e-8, exchange_interval=1000, recompute_every=1000, group_size=1, seed=1) as g:
        g.run_intervals(3, stats=False)
        c = g.counters()
        assert c["accepts"] > 0.85 * c["moves"]
        assert c["batches_scan"] > 4 * c["batches_sequential"]


def test_moves_across_narrow_bins_are_not():
    with rw.REWL(kind=rw.BCC, L=8, J=(1.0, 0.4, 0.05), n_bins=1024, n_windows=16, walkers_per_window=2, e_min=-3.3 * 1024,
                 e_max=0.0, lnf_final=1e-8, lnf_initial=2.0 ** -10, exchange_interval=4000, recompute_every=1000,
                 group_size=1, seed=1) as g:
        g.run_intervals(4, stats=False)
        c = g.counters()
        assert c["batches_sequential"] > 4 * (c["batches_scan"] + c["batches_blocks"])
