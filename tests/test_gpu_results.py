"""Joining fragments (Sec. 4.3) and thermodynamics (Sec. 4.1, Eq. 2-3) where their kernels change form:
curves that do and do not fit in shared memory, join bins out of order, bins per thread kept in registers
or not, and the integer exponential at the ends of its range."""
import numpy as np
import pytest

import oracle
import paper_1411_4212_gb300 as rw

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("B,h,m", [(3, 1, 2), (40, 2, 1), (700, 30, 3), (1031, 64, 2), (9000, 33, 1), (24999, 100, 2),
                                   (25601, 90, 1), (40000, 300, 1)])
def test_join_is_bit_exact(B, h, m):
    import torch
    W, starts = oracle.window_layout(B, h, 0.75) if h > 1 else (B, [0])
    rng = np.random.default_rng(B)
    base = np.cumsum(rng.normal(0.1, 1.0, B))
    frag = np.empty((h, m, W))
    for k in range(h):
        # noise large enough that the join bins of neighbouring windows come out of order
        frag[k] = base[starts[k]:starts[k] + W] + rng.normal(0, 2.0, (m, W)) + rng.normal(0, 50, (m, 1))
    out = torch.empty(B, dtype=torch.float64, device="cuda")
    rw.stitch_device(torch.from_numpy(frag).cuda(), starts, B, out)
    ref = oracle.merge_fragments(frag, starts, B)
    ref = ref[0] if isinstance(ref, tuple) else ref
    assert np.array_equal(out.cpu().numpy().view(np.int64), np.asarray(ref).view(np.int64))


def _thermo64(lng, E, n, T):
    """Plain FP64, sums in extended precision."""
    U, C, Z = np.empty(T.size), np.empty(T.size), np.empty(T.size)
    for i, t in enumerate(T):
        x = lng - E / t
        mx = x.max()
        w = np.exp(np.longdouble(x - mx))
        z = w.sum()
        u = (w * E).sum() / z
        U[i], C[i], Z[i] = u, (w * (E - u) ** 2).sum() / z / (n * t * t), mx + np.log(z)
    return U, C, Z


@pytest.mark.parametrize("B", [1, 31, 4095, 4096, 4097, 16384, 16385, 30000])
def test_thermo_over_register_and_memory_forms(B):
    """Tolerance: exponents reach 1e5, whose rounding is 1e-11; each weight carries it, so 1e-10 relative on
    ln Z and U, and 1e-9 on C, which is a variance far below E^2."""
    n = 1000.0
    E = np.linspace(-4.0 * n, 0.0, B) if B > 1 else np.array([-2.0 * n])
    lng = n * (1.3 * E / n - 0.2 * (E / n) ** 2)
    lng -= lng.mean()
    T = np.array([0.05, 0.2, 0.7, 1.0, 2.5, 100.0])
    U, C, Z = rw.thermo(lng, E, n, T)
    U0, C0, Z0 = _thermo64(lng, E, n, T)
    assert np.allclose(U, U0, rtol=1e-10, atol=1e-12) and np.allclose(Z, Z0, rtol=1e-10)
    assert np.allclose(C, C0, rtol=1e-9, atol=1e-12)


def test_thermo_with_empty_bins_and_extremes():
    """Bins of ln g = -inf count nothing; weights down to e^-708 and below; NaN anywhere gives NaN."""
    E = np.array([-10.0, -5.0, 0.0, 1.0])
    T = np.array([0.01, 1.0, 1e6])
    lng = np.array([0.0, -np.inf, 3.0, -2000.0])
    U, C, Z = rw.thermo(lng, E, 4.0, T)
    keep = np.isfinite(lng)
    U0, C0, Z0 = _thermo64(lng[keep], E[keep], 4.0, T)
    assert np.allclose(U, U0, rtol=1e-12) and np.allclose(Z, Z0, rtol=1e-12) and np.allclose(C, C0, rtol=1e-9, atol=1e-300)
    for bad in (np.nan, -np.nan):
        U, C, Z = rw.thermo(np.array([0.0, bad, 1.0, 2.0]), E, 4.0, T)
        assert np.isnan(U).all() and np.isnan(C).all() and np.isnan(Z).all()
    U, C, Z = rw.thermo(np.full(4, -np.inf), E, 4.0, T)
    assert np.isnan(U).all()
