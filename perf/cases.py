"""The work that users of this package have it do, as cases that can be timed and compared.

A case goes through the package's public entry points (the REWL, Batch and Mlp classes, stitch_device,
thermo, peak_temperature).  Sizes are those of the package's own workloads, tests and benchmark; draw()
gives more of the same ranges.  Kinds of case:
  walk    -- exchange intervals of one run, then the walkers' state read back;
  batch   -- exchange intervals of many runs in one persistent launch, then every run's state;
  start   -- a run created and driven from the aligned state into its windows;
  results -- fragments joined into ln g(E), thermodynamics on a temperature grid, the peak of C(T);
  train   -- full-batch Adam steps of the warm-start network;
  infer   -- its prediction of ln g/N.
The walk is deterministic for given arguments, so the states of two builds can be compared bit by bit.
"""
import math

import numpy as np
import torch

import paper_1411_4212_gb300 as rw
from paper_1411_4212_gb300 import warmstart, workloads

Z = (8, 6, 12, 24)      # neighbours per bcc shell
HIDDEN = 128            # units of each of the network's three hidden layers


def listed():
    return [
        # the smallest run of the package (bcc L = 4 on its restricted range, as its statistics tests and
        # quick looks use it): latency of one walker's chain, one interval at a time
        dict(name="walk small L4", kind="walk", L=4, J1=1.0, J2=0.5, J3=0.0, J4=0.0, shells=2, mode="production",
             lo=-400.0 / 128, hi=0.0, bins=120, windows=4, walkers=2, moves=10000, intervals=1, lnf=0.0, warm=2,
             window_sync=False, group=0, merge=True),
        # the single-run benchmark geometry: bcc L = 16, two shells, the whole range [E_gs, 0], early stages
        dict(name="walk L16 full range", kind="walk", L=16, J1=1.0, J2=0.5, J3=0.0, J4=0.0, shells=2,
             mode="production", lo=-5.5, hi=0.0, bins=2000, windows=16, walkers=4, moves=10000, intervals=8, lnf=0.0,
             warm=4, window_sync=False, group=0, merge=False),
        # the same geometry in the FP64 trajectory mode that reproduces the reference walk bit for bit
        dict(name="walk L16 trajectory", kind="walk", L=16, J1=1.0, J2=0.5, J3=0.0, J4=0.0, shells=2,
             mode="trajectory", lo=-5.5, hi=0.0, bins=2000, windows=16, walkers=4, moves=10000, intervals=1, lnf=0.0,
             warm=1, window_sync=False, group=0, merge=False),
        # a run on the way to convergence (what most of a run's time goes into): bcc L = 8 on
        # [0.6 E_gs, 0], one bin per spin, small ln f, one lane per move as the warm-start workflow has it
        dict(name="walk L8 converging", kind="walk", L=8, J1=1.0, J2=0.4, J3=0.05, J4=0.0, shells=3,
             mode="production", lo=-3.3, hi=0.0, bins=1024, windows=16, walkers=2, moves=4000, intervals=16,
             lnf=2.0 ** -10, warm=16, window_sync=False, group=1, merge=True),
        # the large benchmark geometry: bcc L = 32, four shells, 64 windows x 8 walkers over [E_gs, 0]
        dict(name="walk L32 full range", kind="walk", L=32, J1=1.0, J2=0.6, J3=-0.05, J4=-0.1, shells=4,
             mode="production", lo=-4.3, hi=0.0, bins=8000, windows=64, walkers=8, moves=10000, intervals=4, lnf=0.0,
             warm=2, window_sync=False, group=0, merge=False),
        # the converged large run: the same lattice on its range around the specific-heat peak, bins of
        # 1.6 J1, 300 windows x 2 walkers, small ln f
        dict(name="walk L32 converging", kind="walk", L=32, J1=1.0, J2=0.6, J3=-0.05, J4=-0.1, shells=4,
             mode="production", lo=-2.5, hi=-2.1, bins=16384, windows=300, walkers=2, moves=4000, intervals=8,
             lnf=2.0 ** -7, warm=8, window_sync=False, group=0, merge=False),
        # 64 unlike runs together, every lattice in global memory and 1024-entry tables (what the batch's
        # autotuner picks for them)
        dict(name="batch 64 runs", kind="batch", sizes="8,12,16,20", per_size=16, shells=3, full_range=True,
             moves=10000, intervals=4, lnf=0.0, warm=1, walkers=4, workers=2, smem_n=0, entries=1024),
        # the runs that make the network's training corpus: small lattices of three sizes converging
        # together, the batch's default launch shape
        dict(name="batch corpus", kind="batch", sizes="4,5,6", per_size=16, shells=3, full_range=False, moves=4000,
             intervals=16, lnf=2.0 ** -7, warm=8, walkers=2, workers=0, smem_n=0, entries=0),
        # starting a run: creation, ground state of the default range, initial drive into the windows
        dict(name="start L12", kind="start", L=12, shells=2, bins=864, windows=16, walkers=4),
        # finishing one: 300 windows x 2 walkers joined over 16384 bins, C(T) on the grid T in [0.2, 3]
        dict(name="results 16384 bins", kind="results", L=32, bins=16384, windows=300, walkers=2, temps=281),
        # training on the corpus of 192 runs at L = 4, 5, 6 (51840 samples): eight full-batch steps, as
        # the last ones of a training, at a small learning rate
        dict(name="train 51840 samples", kind="train", sizes="4,5,6", per_size=64, steps=8),
        # predicting the large converged run's ln g at its bins
        dict(name="infer 16384 bins", kind="infer", n=16384),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["walk", "walk", "walk", "batch", "start", "results", "train", "infer"])
    if kind == "walk":
        L, shells = rng.randint(4, 24), rng.randint(1, 4)
        mode = "trajectory" if L <= 12 and rng.random() < 0.25 else "production"
        J = [1.0, rng.uniform(0.2, 0.6), rng.uniform(-0.1, 0.1), rng.uniform(-0.1, 0.1)]
        J = [j if s < shells else 0.0 for s, j in enumerate(J)]
        egs = -0.5 * sum(z * j for z, j in zip(Z, J))
        N = 2 * L ** 3
        converging = rng.random() < 0.6
        bins = N if converging else max(100, N // 4 + rng.randint(0, 7))
        # windows of at least 24 bins, and narrow enough for a walker's tables to fit beside its lattice
        windows = min(max(_log_int(rng, 2, 40), math.ceil(bins / 1000)), max(2, bins // 24))
        if mode == "trajectory":
            windows = min(windows, 16)
        return dict(kind="walk", L=L, J1=J[0], J2=J[1], J3=J[2], J4=J[3], shells=shells, mode=mode,
                    lo=(0.6 if converging else 1.0) * egs, hi=0.0, bins=bins, windows=windows,
                    walkers=rng.randint(1, 8), moves=_log_int(rng, 500, 10000),
                    intervals=1 if mode == "trajectory" else rng.randint(1, 8),
                    lnf=2.0 ** -rng.randint(4, 12) if converging else 0.0, warm=rng.randint(1, 4),
                    window_sync=rng.random() < 0.2, group=rng.choice([0, 1]), merge=rng.random() < 0.5)
    if kind == "batch":
        sizes = sorted(rng.sample(range(4, 17), rng.randint(1, 4)))
        return dict(kind="batch", sizes=",".join(map(str, sizes)), per_size=rng.randint(1, 6),
                    shells=rng.choice([3, 4]), full_range=rng.random() < 0.3, moves=_log_int(rng, 500, 8000),
                    intervals=rng.randint(1, 4), lnf=2.0 ** -rng.randint(2, 10), warm=rng.randint(1, 2),
                    walkers=rng.randint(1, 2), workers=rng.randint(0, 3), smem_n=rng.choice([0, 500, 2000]),
                    entries=rng.choice([512, 1024, 4096]))
    if kind == "start":
        L = rng.randint(4, 14)
        bins = L ** 3 + rng.randint(0, 9)
        return dict(kind="start", L=L, shells=rng.randint(1, 4), bins=bins,
                    windows=min(rng.randint(2, 16), max(2, bins // 16)), walkers=rng.randint(1, 4))
    if kind == "results":
        bins = _log_int(rng, 200, 20000)
        return dict(kind="results", L=rng.randint(4, 32), bins=bins,
                    windows=min(_log_int(rng, 1, 400), max(1, bins // 16)), walkers=rng.randint(1, 8),
                    temps=_log_int(rng, 8, 400))
    if kind == "train":
        return dict(kind="train", sizes=rng.choice(["4", "5", "4,5", "5,6,7", "4,5,6"]), per_size=_log_int(rng, 1, 40),
                    steps=rng.randint(1, 8))
    return dict(kind="infer", n=_log_int(rng, 50, 60000))


# ---- inputs ------------------------------------------------------------------------------------------


def _slope(u, J):
    """A plausible d ln g / dE of the model at energy per spin u <= 0: -u / <u^2> near 0, a plateau near
    the transition, 1 / (u - u_gs) towards the ground state."""
    zj, zj2 = sum(z * j for z, j in zip(Z, J)), sum(z * j * j for z, j in zip(Z, J))
    top = 0.36 * 11.0 / zj
    return np.maximum(top * (1.0 - np.exp(u / (top * zj2 / 6.0))), 1.0 / np.maximum(u + 0.5 * zj, 1e-3))


def _ln_g_per_spin(u, J):
    """Integral of _slope over u (a trapezoid sum over the given increasing grid), 0 at its top."""
    b = _slope(u, J)
    s = np.concatenate([[0.0], np.cumsum(0.5 * (b[1:] + b[:-1]) * np.diff(u))])
    return s - s[-1]


def _sim(J, L, seed, lo, hi, bins, windows, walkers, moves, mode=rw.PRODUCTION, group=0, sync=False, lnf=0.0):
    N = 2 * L ** 3
    s = rw.REWL(kind=rw.BCC, L=L, J=J, e_min=lo * N, e_max=hi * N, n_bins=bins, n_windows=windows,
                walkers_per_window=walkers, overlap=0.75 if windows > 1 else 0.0, flatness=0.8, lnf_final=1e-8,
                seed=seed, mode=mode, exchange_interval=moves, group_size=group,
                iteration=rw.ITERATION_WINDOW if sync else rw.ITERATION_WALKER)
    s.init_walkers()
    if lnf > 0.0:
        u = lo + (np.arange(bins) + 0.5) * (hi - lo) / bins
        s.set_initial_lng(N * _ln_g_per_spin(u, list(J) + [0.0] * (4 - len(J))), lnf)
    return s


def _network(seed):
    """Parameters as a fresh network has them: uniform in +-1/sqrt(inputs of the layer), biases 0."""
    g = np.random.Generator(np.random.Philox(key=seed))
    parts = []
    for n_in, n_out in ((6, HIDDEN), (HIDDEN, HIDDEN), (HIDDEN, HIDDEN), (HIDDEN, 1)):
        parts += [g.uniform(-1.0, 1.0, n_in * n_out) / math.sqrt(n_in), np.zeros(n_out)]
    return np.concatenate(parts).astype(np.float32)


def _corpus(c, seed):
    """Samples of converged runs: per run one coupling set and one bin per spin over [0.6 E_gs, 0]."""
    xs, ts, off = [], [], [0]
    k = 0
    for L in map(int, c["sizes"].split(",")):
        N = 2 * L ** 3
        for _ in range(c["per_size"]):
            J = workloads.random_couplings(1000 * seed + k) + (0.0,)
            k += 1
            lo = -0.3 * sum(z * j for z, j in zip(Z, J))
            u = lo * (1.0 - (np.arange(N) + 0.5) / N)
            xs.append(np.column_stack([u] + [np.full(N, v) for v in (1.0 / L,) + J]))
            ts.append(_ln_g_per_spin(u, J))
            off.append(off[-1] + N)
    return np.concatenate(xs).astype(np.float32), np.concatenate(ts).astype(np.float32), np.array(off, dtype=np.int32)


def _bins_input(c, seed):
    """The network's inputs at the bins of one run, as mlp_features gives them."""
    J = workloads.random_couplings4(seed)
    u = np.linspace(-2.5, -0.01, c["n"])
    return np.column_stack([u] + [np.full(c["n"], v) for v in (1.0 / 32,) + J]).astype(np.float32)


def _layout(c):
    """Window width and starts of `windows` windows over `bins` bins at 75 % overlap."""
    B, h = c["bins"], c["windows"]
    W = min(B, math.ceil(B / (1 + (h - 1) * 0.25)))
    return W, [0 if h == 1 else int(math.floor(k * (B - W) / (h - 1) + 0.5)) for k in range(h)]


def _fragments(c, seed):
    """(fragments [h][m][W], starts, bin centres, temperatures): every walker's ln g is the run's curve
    on its window, up to a constant and the noise that a converged walk leaves."""
    g = np.random.Generator(np.random.Philox(key=seed))
    J = workloads.random_couplings4(seed)
    N = 2 * c["L"] ** 3
    B, h, m = c["bins"], c["windows"], c["walkers"]
    W, starts = _layout(c)
    zj = sum(z * j for z, j in zip(Z, J))
    u = -0.45 * zj * (1.0 - (np.arange(B) + 0.5) / B)
    lng = N * _ln_g_per_spin(u, J)
    frag = np.empty((h, m, W))
    for k in range(h):
        frag[k] = lng[starts[k]:starts[k] + W] + 0.05 * g.standard_normal((m, W)).cumsum(1) / math.sqrt(W)
        frag[k] += g.uniform(0.0, 1e3, (m, 1))
    return frag, starts, N * u, N, np.linspace(0.2, 3.0, c["temps"])


# ---- the four functions ------------------------------------------------------------------------------


def prepare(case, seed):
    c, kind = case, case["kind"]
    if kind == "walk":
        J = (c["J1"], c["J2"], c["J3"], c["J4"])[:c["shells"]]
        s = _sim(J, c["L"], seed, c["lo"], c["hi"], c["bins"], c["windows"], c["walkers"], c["moves"],
                 mode=rw.TRAJECTORY if c["mode"] == "trajectory" else rw.PRODUCTION, group=c["group"],
                 sync=c["window_sync"], lnf=c["lnf"])
        s.run_intervals(c["warm"])
        return dict(kind=kind, sim=s, intervals=c["intervals"], merge=c["merge"])
    if kind == "batch":
        jobs = []
        pick = workloads.random_couplings4 if c["shells"] == 4 else workloads.random_couplings
        for L in map(int, c["sizes"].split(",")):
            N = 2 * L ** 3
            for _ in range(c["per_size"]):
                k = len(jobs)
                J = pick(1000 * seed + k)
                egs = -0.5 * sum(z * j for z, j in zip(Z, J))
                bins = N // 4 if c["full_range"] else N
                h = workloads.BATCH_WINDOWS.get(L, 8) if c["full_range"] else min(warmstart.windows_for(L), 64)
                if c["full_range"] and L < 8:
                    h = 4
                jobs.append(_sim(J, L, seed + k, egs if c["full_range"] else 0.6 * egs, 0.0, bins, h, c["walkers"],
                                 c["moves"], group=1, lnf=c["lnf"]))
        b = rw.Batch(jobs)
        if c["workers"]:
            b.set_tuning(c["workers"], c["smem_n"], c["entries"])
        b.run_intervals(c["warm"])
        return dict(kind=kind, intervals=c["intervals"], batch=b)
    if kind == "start":
        J = workloads.random_couplings4(seed)[:c["shells"]]
        return dict(kind=kind, args=dict(kind=rw.BCC, L=c["L"], J=J, n_bins=c["bins"], n_windows=c["windows"],
                                         walkers_per_window=c["walkers"], lnf_final=1e-8, seed=seed))
    if kind == "results":
        frag, starts, E, N, T = _fragments(c, seed)
        return dict(kind=kind, frag=torch.from_numpy(frag).cuda(), starts=np.array(starts, dtype=np.int32), E=E, N=N,
                    T=T, out=torch.empty(c["bins"], dtype=torch.float64, device="cuda"))
    net = rw.Mlp(warmstart.SHIFT, warmstart.SCALE, seed=0)
    net.set_params(_network(seed))
    if kind == "train":
        return dict(kind=kind, net=net, corpus=_corpus(c, seed), steps=c["steps"])
    return dict(kind=kind, net=net, x=_bins_input(c, seed))


STATE = ("lng", "H", "E", "bin", "lnf", "replica", "stage", "accepts", "steps")


def run(state):
    kind = state["kind"]
    if kind == "walk":
        s = state["sim"]
        s.run_intervals(state["intervals"])
        w = s.walkers()
        out = {k: w[k] for k in STATE}
        if state["merge"]:
            out["merged"] = s.merge()[0]
        return out
    if kind == "batch":
        state["batch"].run_intervals(state["intervals"])
        w = [j.walkers() for j in state["batch"].jobs]
        return {k: np.concatenate([x[k].reshape(-1) for x in w]) for k in STATE}
    if kind == "start":
        s = rw.REWL(**state["args"])
        s.init_walkers()
        w = s.walkers()
        out = {k: w[k] for k in ("E", "bin", "replica", "init_moves")}
        s.close()
        return out
    if kind == "results":
        lng = rw.stitch_device(state["frag"], state["starts"], state["E"].size, state["out"]).cpu().numpy()
        U, C, lnZ = rw.thermo(lng, state["E"], state["N"], state["T"])
        return dict(lng=lng, U=U, C=C, lnZ=lnZ, T_peak=rw.peak_temperature(state["T"], C))
    if kind == "train":
        x, t, off = state["corpus"]
        loss = state["net"].train(x, t, off, steps=state["steps"], lr=1e-5)
        return dict(loss=loss, params=state["net"].params())
    return state["net"].forward(state["x"])


def _walk_work(slots, N, W, z, moves, intervals, traj):
    """Every configuration and window table in and out once per call; per move the field of z
    neighbours (three sums each) and about 60 operations for the draw, the increment and the decision."""
    state = slots * (N * (24 if traj else 8) + W * 12)
    return dict(bytes=2 * state, flops=slots * moves * intervals * (6 * z + 60))


def work(case):
    c, kind = case, case["kind"]
    if kind == "walk":
        W, _ = _layout(c)
        return _walk_work(c["windows"] * c["walkers"], 2 * c["L"] ** 3, W, sum(Z[:c["shells"]]), c["moves"],
                          c["intervals"], c["mode"] == "trajectory")
    if kind == "batch":
        tot = dict(bytes=0, flops=0)
        for L in map(int, c["sizes"].split(",")):
            N = 2 * L ** 3
            h = workloads.BATCH_WINDOWS.get(L, 8 if L >= 8 else 4) if c["full_range"] else \
                min(warmstart.windows_for(L), 64)
            W, _ = _layout(dict(bins=N // 4 if c["full_range"] else N, windows=h))
            w = _walk_work(c["per_size"] * h * c["walkers"], N, W, sum(Z[:c["shells"]]), c["moves"], c["intervals"],
                           False)
            tot = {k: tot[k] + w[k] for k in tot}
        return tot
    if kind == "start":   # about one trial move per spin and walker is the shortest drive
        N, S = 2 * c["L"] ** 3, c["windows"] * c["walkers"]
        return dict(bytes=S * N * 8, flops=S * N * (6 * sum(Z[:c["shells"]]) + 60))
    if kind == "results":
        W, _ = _layout(c)
        return dict(bytes=8 * (c["windows"] * c["walkers"] * W + 2 * c["bins"] + 4 * c["temps"]),
                    flops=c["bins"] * c["temps"] * 40 + 4 * c["windows"] * c["walkers"] * W)
    layers = 6 * HIDDEN + 2 * HIDDEN * HIDDEN + HIDDEN
    params = layers + 3 * HIDDEN + 1
    if kind == "train":
        M = sum(2 * int(L) ** 3 for L in c["sizes"].split(",")) * c["per_size"]
        return dict(bytes=M * 28 + c["steps"] * params * 28, flops=c["steps"] * M * 6 * layers)
    return dict(bytes=c["n"] * 28 + params * 2, flops=c["n"] * 2 * layers)


# ---- 64-bit values -----------------------------------------------------------------------------------


def _layers(p):
    """The network's weights and biases [(W [in][out], b [out])] out of a flat vector."""
    out, at = [], 0
    for n_in, n_out in ((6, HIDDEN), (HIDDEN, HIDDEN), (HIDDEN, HIDDEN), (HIDDEN, 1)):
        W = p[at:at + n_in * n_out].reshape(n_in, n_out)
        at += n_in * n_out
        out.append((W, p[at:at + n_out]))
        at += n_out
    return out


def _forward64(p, x):
    shift, scale = (torch.from_numpy(np.asarray(v, dtype=np.float64)).to(x) for v in (warmstart.SHIFT, warmstart.SCALE))
    a = (x - shift) * scale
    ls = _layers(p)
    for W, b in ls[:-1]:
        z = a @ W + b
        a = z * torch.sigmoid(z)
    return (a @ ls[-1][0] + ls[-1][1])[:, 0]


def _train64(c, seed):
    x, t, off = _corpus(c, seed)
    dev = "cuda" if torch.cuda.is_available() else "cpu"
    x, t = (torch.from_numpy(v).to(dev, torch.float64) for v in (x, t))
    run_of = torch.from_numpy(np.repeat(np.arange(off.size - 1), np.diff(off))).to(dev)
    count = torch.from_numpy(np.diff(off).astype(np.float64)).to(dev)
    w = torch.from_numpy(_network(seed)).to(dev, torch.float64)
    m, v = torch.zeros_like(w), torch.zeros_like(w)
    loss = []
    for it in range(1, c["steps"] + 1):
        p = w.to(torch.bfloat16).double().requires_grad_(True)
        r = _forward64(p, x) - t
        mean = torch.zeros_like(count).index_add(0, run_of, r) / count
        L = ((r - mean[run_of]) ** 2).mean()
        g, = torch.autograd.grad(L, p)
        loss.append(float(L))
        m = 0.9 * m + 0.1 * g
        v = 0.999 * v + 0.001 * g * g
        w = w - 1e-5 * (m / (1 - 0.9 ** it)) / (torch.sqrt(v / (1 - 0.999 ** it)) + 1e-8)
    return dict(loss=np.array(loss), params=w.cpu().numpy())


def _results64(c, seed):
    frag, starts, E, N, T = _fragments(c, seed)
    W, h, B = frag.shape[2], c["windows"], c["bins"]
    A = (frag - frag.mean(2, keepdims=True)).mean(1)
    shift, join = [0.0], []
    for k in range(h - 1):
        b = np.arange(starts[k + 1] + 1, starts[k] + W - 1)
        i, j = b - starts[k], b - starts[k + 1]
        at = int(b[np.argmin(np.abs((A[k][i + 1] - A[k][i - 1]) - (A[k + 1][j + 1] - A[k + 1][j - 1])))]) if b.size \
            else starts[k + 1]
        join.append(at)
        shift.append(shift[-1] + A[k][at - starts[k]] - A[k + 1][at - starts[k + 1]])
    lng = np.empty(B)
    k = 0
    for b in range(B):
        while k + 1 < h and b >= join[k]:
            k += 1
        lng[b] = A[k][b - starts[k]] + shift[k]
    lng -= lng.mean()
    x = lng[None, :] - E[None, :] / T[:, None]
    mx = x.max(1)
    p = np.exp(x - mx[:, None])
    z = p.sum(1)
    U = (p * E).sum(1) / z
    C = (p * (E[None, :] - U[:, None]) ** 2).sum(1) / z / (N * T * T)
    return dict(lng=lng, U=U, C=C, lnZ=mx + np.log(z), T_peak=None)


def exact(case, seed):
    if case["kind"] == "results":
        return _results64(case, seed)
    if case["kind"] == "train":
        return _train64(case, seed)
    if case["kind"] == "infer":
        p = torch.from_numpy(_network(seed)).to(torch.bfloat16).double()
        return _forward64(p, torch.from_numpy(_bins_input(case, seed)).double()).numpy()
    return None
