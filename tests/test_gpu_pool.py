"""What the library's memory pool keeps on the GPU when nobody uses it any more."""
import gc

import pytest

import paper_1411_4212_gb300 as rw

pytestmark = pytest.mark.gpu


def test_the_last_run_to_be_closed_gives_its_memory_back():
    """The driver reserves memory in pieces of 32 MiB.  Idle the library keeps 4 MiB, that is one piece; a run of
    52 MB of lattices needs a second one, which would be below the 64 MiB that the pool keeps while anyone uses it.
    Closed as the last one, the run leaves no more than there was before."""
    import torch
    gc.collect()
    spec = dict(kind=rw.BCC, L=16, J=(1.0, 0.5), n_bins=400, n_windows=8, lnf_final=1e-8, exchange_interval=100)
    rw.REWL(seed=1, walkers_per_window=1, **spec).close()
    torch.cuda.synchronize()
    free0 = torch.cuda.mem_get_info()[0]
    g = rw.REWL(seed=2, walkers_per_window=100, **spec)
    torch.cuda.synchronize()
    assert free0 - torch.cuda.mem_get_info()[0] > 16 << 20
    g.close()
    assert free0 - torch.cuda.mem_get_info()[0] <= 4 << 20
