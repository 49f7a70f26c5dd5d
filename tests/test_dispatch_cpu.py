"""Which walker a run gets, decided on the host (on a CUDA runtime without a GPU): the GPU tests that compare the
pipelined walker's paths stop where a run is not pipelined, so that it is has to be seen elsewhere."""
import pytest

import fake_runtime


@pytest.mark.parametrize("shells", [1, 2, 3, 4])
def test_the_smallest_lattices_with_one_lane_per_move_are_pipelined(shells):
    """The shapes of test_gpu_move_batches.py: narrow and wide bins, every resolver."""
    fake_runtime.run(f"""
n = 0
for bins, windows in ((24, 2), (400, 3)):
    for resolver in (rw.RESOLVER_AUTO, rw.RESOLVER_SCAN, rw.RESOLVER_BLOCKS, rw.RESOLVER_SEQUENTIAL):
        g = rw.REWL(kind=rw.BCC, L=4, J=(1.0, 0.5, -0.05, 0.1)[:{shells}], n_bins=bins, n_windows=windows,
                    walkers_per_window=2, lnf_final=1e-8, exchange_interval=1000, group_size=1, resolver=resolver,
                    stream=0)
        n += g.info()["pipelined"]
        g.close()
assert n == 8
""")
