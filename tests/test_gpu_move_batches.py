"""The production walker's batches of 32 trial moves where they can go wrong (Sec. 4.2, Eq. 4): interval
lengths around a batch, dense conflicts on the smallest lattices, and conflict tables smaller than a
lattice in shared memory.  Every resolver path, and every placement of the lattice and the table, must
leave the walk in the same state, bit for bit."""
import numpy as np
import pytest

import paper_1411_4212_gb300 as rw

pytestmark = pytest.mark.gpu

J = (1.0, 0.5, -0.05, 0.1)


def _state(g):
    w = g.walkers()
    out = {k: np.array(v).view(np.int64) if v.dtype == np.float64 else np.array(v) for k, v in w.items()}
    out["spins"] = g.spins().view(np.int64)
    return out


def _assert_same(a, b, what):
    for k in a:
        assert np.array_equal(a[k], b[k]), f"{what}: {k}"


@pytest.mark.parametrize("shells", [1, 2, 3, 4])
@pytest.mark.parametrize("moves", [1, 31, 32, 33, 95, 1000])
def test_paths_agree_around_a_batch_on_the_smallest_lattice(shells, moves):
    """bcc L = 4: most moves of a batch touch another one; narrow and wide bins."""
    for bins, windows in ((24, 2), (400, 3)):
        states = []
        for resolver in (rw.RESOLVER_AUTO, rw.RESOLVER_SCAN, rw.RESOLVER_BLOCKS, rw.RESOLVER_SEQUENTIAL):
            g = rw.REWL(kind=rw.BCC, L=4, J=J[:shells], n_bins=bins, n_windows=windows, walkers_per_window=2,
                        lnf_final=1e-8, seed=3 + moves, exchange_interval=moves, group_size=1, resolver=resolver)
            if not g.info()["pipelined"]:
                g.close()
                break
            g.run_intervals(12, stats=False)
            states.append(_state(g))
            g.close()
        for i, s in enumerate(states[1:]):
            _assert_same(states[0], s, f"{shells} shells, {moves} moves, {bins} bins, path {i + 1}")


def test_a_small_table_beside_a_shared_lattice_changes_nothing():
    """bcc L = 15 in a batch of three walkers per block: the lattice (54 KB) leaves room for a table of
    fewer entries than sites, so sites share entries; alone the table has an entry per site."""
    spec = dict(kind=rw.BCC, L=15, J=J[:3], n_bins=400, n_windows=4, walkers_per_window=2, lnf_final=1e-8, seed=5,
                exchange_interval=3000, recompute_every=1000, group_size=1)
    alone, batched = rw.REWL(**spec), rw.REWL(**spec)
    assert alone.info()["conflict_entries"] >= alone.N and alone.info()["lattice_in_shared"] == 1
    alone.init_walkers()
    alone.run_intervals(3, stats=False)
    with rw.Batch([batched]) as b:
        b.set_tuning(3, batched.N)
        info = b.info()
        assert info["n_smem_lattice_jobs"] == 1 and info["arena_bytes"] < 8 * batched.N + 8 * 4096
        b.run_intervals(3)
    _assert_same(_state(alone), _state(batched), "shared lattice, small table")
    alone.close()
    batched.close()


@pytest.mark.parametrize("bins,pipelined", [(17000, 1), (17330, 1), (17500, 0)])
def test_window_tables_up_to_the_shared_memory_limit(bins, pipelined):
    """bcc L = 24 with one window so wide that its tables fill the shared memory: the widest ones leave the
    conflict table less room than the rule that admits them counts.  The walk goes by neither."""
    spec = dict(kind=rw.BCC, L=24, J=J[:2], n_bins=bins, n_windows=1, walkers_per_window=2, overlap=0.0, seed=6,
                lnf_final=1e-8, exchange_interval=2000, recompute_every=1000, group_size=1)
    states = []
    for resolver in (rw.RESOLVER_AUTO, rw.RESOLVER_SEQUENTIAL):
        g = rw.REWL(resolver=resolver, **spec)
        assert g.info()["pipelined"] == pipelined
        g.init_walkers()
        g.run_intervals(2, stats=False)
        states.append(_state(g))
        assert (states[-1]["steps"] == 4000).all()
        g.close()
    _assert_same(states[0], states[1], f"{bins} bins")
