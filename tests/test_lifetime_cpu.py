"""What the library's host code does with device memory and streams where a call fails or a run is closed early,
on a CUDA runtime without a GPU that keeps account of it (tests/cuda/fake_runtime.cpp)."""
import pytest

import fake_runtime

JOBS = """
def job(seed, **kw):
    return rw.REWL(kind=rw.BCC, L=8, J=(1.0, 0.5), n_bins=200, n_windows=4, walkers_per_window=2, seed=seed,
                   group_size=1, exchange_interval=100, stream=0, **kw)

def refused(f, *a):
    try:
        f(*a)
    except rw.RewlError as e:
        return e.status
    raise AssertionError("the call went through")
"""


@pytest.mark.parametrize("call,skip,run", [
    ("cudaGraphInstantiate", 1, "b.run_intervals, 9"),          # the graph of eight intervals runs, that of one fails
    ("cudaGraphLaunch", 1, "b.run_intervals, 9"),
    ("cudaStreamBeginCapture", 1, "b.run_intervals, 9"),
    ("cudaEventSynchronize", 1, "b.autotune, 100"),
    ("cudaMemcpyAsync", 0, "b.run_to_convergence, 8, 8"),
])
def test_a_batch_call_that_fails_leaves_its_jobs_ordered_after_it(call, skip, run):
    fake_runtime.run(JOBS + f"""
jobs = [job(1), job(2)]
b = rw.Batch(jobs, stream=0)
lib.fake_fail(b"{call}", {skip}, 719)
assert refused({run}) == rw.ECUDA and lib.fake_failed()
lib.cudaStreamSynchronize(None)        # the jobs' stream
assert lib.fake_unfinished() == 0
for j in jobs:
    j.close()
b.close()
assert lib.fake_bad_frees() == 0
""")


def test_a_run_that_is_closed_waits_for_work_on_other_streams():
    """Work that the caller has captured or ordered onto a stream of its own may still use the run's arrays."""
    fake_runtime.run(JOBS + """
g = job(1)
other = lib.fake_stream(1)             # does not wait for the legacy stream, nor that one for it
lib.fake_work(other)
g.close()
assert lib.fake_bad_frees() == 0
""")


LARGE = """
def large(seed):
    return rw.REWL(kind=rw.BCC, L=16, J=(1.0, 0.5), n_bins=400, n_windows=8, walkers_per_window=100, group_size=1,
                   stream=0, seed=seed)
"""


def test_what_the_pool_keeps_once_nobody_uses_it():
    """Runs of 52 MB of lattices: while another one lives the pool keeps them (it keeps up to 64 MiB), once the last
    one is gone 4 MiB are left, whatever its size.  A model's scratch counts too."""
    fake_runtime.run(JOBS + LARGE + """
a, b = large(1), job(2)
a.close()
assert lib.fake_pool_reserved() > 50 << 20
a = large(3)
b.close()
assert lib.fake_pool_reserved() > 50 << 20
a.close()
assert lib.fake_pool_reserved() <= 4 << 20
m = rw.Mlp(np.zeros(6, np.float32), np.ones(6, np.float32), stream=0)
m.forward(np.zeros((1 << 20, 6), np.float32))
assert lib.fake_pool_reserved() > 25 << 20
m.close()
assert lib.fake_pool_reserved() <= 4 << 20
""")


def test_scratch_that_a_stream_refuses_to_free_is_not_lost():
    fake_runtime.run("""
m = rw.Mlp(np.zeros(6, np.float32), np.ones(6, np.float32), stream=0)
lib.fake_fail(b"cudaFreeAsync", 0, 719)
m.forward(np.zeros((1 << 20, 6), np.float32))
assert lib.fake_failed()
m.close()
assert lib.fake_pool_reserved() <= 4 << 20 and lib.fake_bad_frees() == 0
""")


def test_training_that_runs_out_of_memory_can_be_tried_again():
    """The first gradient allocates; where that fails the model stays usable, the retry's first step is Adam's first
    one, and no error is left for the next call to find."""
    fake_runtime.run(JOBS + """
m = rw.Mlp(np.zeros(6, np.float32), np.ones(6, np.float32), stream=0)
args = (np.zeros((10, 6), np.float32), np.zeros(10, np.float32), np.array([0, 10], np.int32))
lib.fake_fail(b"cudaMallocFromPoolAsync", 7, 2)     # after the corpus, six arrays, and the loss history
assert refused(m.train, *args, 3, 1e-3) == rw.ENOMEM and lib.fake_failed()
lib.fake_watch(b"mlp_reduce_kernel", 11, 24)
m.train(*args, 2, 1e-3)
adam = (ctypes.c_float * 6)()
for i in range(2):
    assert lib.fake_seen(i, adam) == 2
    assert abs(adam[4] - (1 - 0.9 ** (i + 1))) < 1e-6, list(adam)
m.close()
""")


@pytest.mark.parametrize("call", ["cudaMallocFromPoolAsync", "cudaMalloc"])
def test_creating_something_without_memory_leaves_no_error_behind(call):
    fake_runtime.run(JOBS + f"""
make = (lambda: job(1)) if "{call}" == "cudaMallocFromPoolAsync" else (lambda: rw.Batch([g], stream=0))
g = job(2)
g.init_walkers()
lib.fake_fail(b"{call}", 0, 2)
assert refused(make) == rw.ENOMEM and lib.fake_failed()
g.run_intervals(1)
make().close()
g.close()
""")


def test_a_model_holds_no_more_scratch_than_its_samples_need():
    """2.5 KB per sample for the backward pass, at most two rounds of all CTAs (38912 samples); it grows with the
    largest gradient so far, by half at least, and is freed with the model."""
    fake_runtime.run(JOBS + """
m = rw.Mlp(np.zeros(6, np.float32), np.ones(6, np.float32), stream=0)
row, full = 5 * 128 * 4, 2 * 152 * 8 * 16
held = []
for n in (10, 7, 1000, 1001, 5, full + 1, 3 * full):
    m.gradient(np.zeros((n, 6), np.float32), np.zeros(n, np.float32), np.array([0, n], np.int32))
    held.append(lib.fake_pool_used() // row)
assert held == [10, 10, 1000, 1500, 1500, full, full], held
m.close()
assert lib.fake_plain_bytes() == 0 and lib.fake_pool_used() == 0 and lib.fake_bad_frees() == 0
""")


@pytest.mark.parametrize("call", [
    "rw.thermo(np.zeros(100), np.linspace(-1, 0, 100), 10, np.linspace(1, 2, 100000), stream=0)",
    "traj.walkers()",
    "traj.run_intervals(1)",
    "traj.exchange()",
    "m.train(np.zeros((10, 6), np.float32), np.zeros(10, np.float32), np.array([0, 10], np.int32), 200000, 1e-3)",
])
def test_host_memory_that_is_refused_is_a_status(call):
    """Read-backs go through host memory of the library's: without it a call returns REWL_ENOMEM (an exception would
    not get past the C interface) and leaves the run or the model as it was."""
    fake_runtime.run(JOBS + f"""
traj = rw.REWL(kind=rw.BCC, L=4, J=(1.0,), n_bins=80, n_windows=4, walkers_per_window=6000, mode=rw.TRAJECTORY,
               stream=0, seed=1)
traj.run_intervals(1, stats=False)
m = rw.Mlp(np.zeros(6, np.float32), np.ones(6, np.float32), stream=0)
lib.fake_refuse_from(1 << 20)
assert refused(lambda: {call}) == rw.ENOMEM
lib.fake_refuse_from(1 << 62)
{call}
traj.close()
m.close()
""")
