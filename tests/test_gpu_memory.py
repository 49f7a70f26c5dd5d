"""The library's device memory: handles and handle-less calls from several threads, each on its own stream,
give what they give one after the other, and what the library keeps once they are gone is bounded."""
import threading

import numpy as np
import pytest

import paper_1411_4212_gb300 as rw

pytestmark = pytest.mark.gpu

SPEC = dict(kind=rw.BCC, L=6, J=(1.0, 0.5), n_bins=108, n_windows=4, walkers_per_window=2, lnf_final=1e-8,
            exchange_interval=700, group_size=1)


def _work(seed, stream):
    out = []
    for rep in range(3):
        with rw.REWL(seed=seed + rep, stream=stream, **SPEC) as g:
            g.run_intervals(3)
            w = g.walkers()
            lng, cen = g.merge()
            U, C, Z = rw.thermo(lng, cen, g.N, np.linspace(0.5, 4.0, 40), stream=stream)
            out += [w["lng"], w["H"], w["E"], lng, U, C, Z]
    return out


def test_threads_on_their_own_streams_match_serial_calls():
    import torch
    seeds = [11, 23, 37, 51]
    serial = [_work(s, None) for s in seeds]
    got = [None] * len(seeds)

    def body(i):
        torch.cuda.set_device(0)
        got[i] = _work(seeds[i], torch.cuda.Stream())

    threads = [threading.Thread(target=body, args=(i,)) for i in range(len(seeds))]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    for a, b in zip(serial, got):
        assert b is not None
        for x, y in zip(a, b):
            assert np.array_equal(x, y)


def test_memory_is_given_back():
    import torch
    _work(5, None)
    torch.cuda.synchronize()
    free0 = torch.cuda.mem_get_info()[0]
    for rep in range(3):
        jobs = [rw.REWL(kind=rw.BCC, L=16, J=(1.0, 0.5), n_bins=2000, n_windows=16, walkers_per_window=4, seed=s,
                        lnf_final=1e-8, exchange_interval=100) for s in range(64)]   # 4 MB of lattices each
        for j in jobs:
            j.close()
    torch.cuda.synchronize()
    # idle, the library keeps 4 MiB and the allocator's granularity
    assert free0 - torch.cuda.mem_get_info()[0] < 64 << 20
