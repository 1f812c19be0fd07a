"""The join's kernels at the sizes where their split changes, on tables set on
both sides, against the oracle: windows of one chunk and of several, few and
many walkers, holes, all three formats, and a caller's unaligned tables."""
import ctypes

import numpy as np
import pytest

import oracle
from oracle import OracleConfig, OracleREWL

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def P():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1508_02748_gb300 as P
    from paper_1508_02748_gb300 import build
    build.build()
    return P


def _set(o, runs, seed):
    """A smooth surface plus noise per bin and an offset per walker, multiples
    of 1/64 below 2^12 (exact in every format), visits with holes."""
    N = o.cfg.L ** 2
    win, (lng, H, toff) = o.windows(), o.tables()
    rng = np.random.default_rng(seed)
    for k in range(toff.size - 1):
        e0, e1, m0, m1, _ = win[k // o.cfg.walkers_per_window]
        e, m = np.meshgrid(np.arange(e0, e1 + 1), np.arange(m0, m1 + 1), indexing="ij")
        x = m / N
        can = e <= 2 * N * np.minimum(x, 1 - x) + 1e-9
        v = 4.0 * N * x * (1 - x) - (e - 2 * N * x * (1 - x)) ** 2 / (0.5 * N) + rng.normal(0, 0.3, e.shape) + rng.uniform(0, 900)
        seen = can & (rng.random(e.shape) < 0.97)
        lng[toff[k]:toff[k + 1]] = np.where(seen, np.round(v * 64) / 64, 0.0).ravel()
        H[toff[k]:toff[k + 1]] = np.where(seen, rng.integers(0, 60, e.shape), -1).ravel()
    o.set_tables(lng, H)
    for r in runs:
        r.set_tables(lng, H)
    return lng, H


def _near(got, ref):
    fin = np.isfinite(ref)
    assert np.array_equal(np.isfinite(got), fin)
    np.testing.assert_allclose(got[fin], ref[fin], rtol=1e-12, atol=1e-9)


@pytest.mark.parametrize("L,nE,nM,W", [(6, 3, 2, 1), (6, 3, 2, 2), (6, 3, 2, 3), (7, 2, 2, 5), (8, 1, 1, 2), (8, 1, 1, 9),
                                       (8, 1, 2, 130), (11, 2, 1, 3), (4, 1, 1, 40)])
def test_join_splits(P, L, nE, nM, W):
    kw = dict(L=L, n_win_E=nE, n_win_M=nM, overlap_E=0.5, overlap_M=0.5, walkers_per_window=W, seed=6, drive_budget=10**8)
    o = OracleREWL(OracleConfig(**kw))
    runs = [P.REWL(P.Config(precision=p, **kw)) for p in (P.FP64, P.F32X2, P.F32)]
    _set(o, runs, L + W)
    for ro, rg in ((oracle.JOIN_MARGINAL, P.JOIN_MARGINAL), (oracle.JOIN_PER_SLICE, P.JOIN_PER_SLICE)):
        Jo, em, mm = o.join(ro)
        for r in runs:
            Jg, emg, mmg = r.lng(matches=True, rule=rg)
            np.testing.assert_array_equal(emg, em)
            np.testing.assert_array_equal(mmg, mm)
            _near(Jg, Jo)
            assert np.array_equal(Jg, r.lng(rule=rg), equal_nan=True)       # the same bits each time
    if 2 <= W <= 9:
        mo, eo = oracle.jackknife(o)
        for r in runs:
            mg, eg = r.jackknife()
            _near(mg, np.asarray(mo).reshape(mg.shape))
            fin = np.isfinite(mg)
            np.testing.assert_allclose(eg[fin], np.asarray(eo).reshape(eg.shape)[fin], rtol=1e-6, atol=1e-9)


def test_jackknife_names_the_failing_replicate(P):
    """Two walkers that share no bin: every replicate has one walker and
    succeeds.  Three, of which the first two share none: leaving out the third
    (replicate 2) fails."""
    kw = dict(L=5, walkers_per_window=3, seed=2)
    r = P.REWL(P.Config(**kw))
    lng, H = r.tables()
    n = H.size // 3
    H[:] = 1
    H[:n][n // 2:] = -1
    H[n:2 * n][:n // 2] = -1
    lng[:] = 1.0
    r.set_tables(lng, H)
    with pytest.raises(P.REWLError, match="replicate 2: join failed .code 1"):
        r.jackknife()


def test_noalloc_join_of_unaligned_tables(P):
    import torch
    kw = dict(L=7, n_win_E=2, overlap_E=0.5, walkers_per_window=3, seed=6)
    o, g = OracleREWL(OracleConfig(**kw)), P.REWL(P.Config(**kw))
    lng, H = _set(o, [g], 9)
    d_lng = torch.zeros(lng.size + 1, dtype=torch.float64, device="cuda")[1:].copy_(torch.from_numpy(lng))
    d_H = torch.zeros(H.size + 1, dtype=torch.int32, device="cuda")[1:].copy_(torch.from_numpy(H.astype(np.int32)))
    out = torch.empty(g.N + 1, g.N + 1, dtype=torch.float64, device="cuda")
    torch.cuda.synchronize()
    c = g.cfg.to_c()
    assert P.load_library().rewl_join_noalloc(ctypes.byref(c), ctypes.c_void_p(d_lng.data_ptr()), ctypes.c_void_p(d_H.data_ptr()),
                                              ctypes.c_void_p(out.data_ptr()), None) == 0
    _near(out.cpu().numpy(), o.join()[0])


# Eq. 5 either side of the series' end at 1/8, empty bins, non-finite ones, odd
# counts and tables that start at an odd entry
@pytest.mark.parametrize("n,shift", [(1, 0), (2, 0), (4097, 0), (4096, 1), (100_001, 1)])
def test_relative_difference_forms(P, n, shift):
    import torch
    rng = np.random.default_rng(n)
    a = rng.normal(0, 300, n)
    b = a + np.where(rng.random(n) < 0.5, 1, -1) * 10.0 ** rng.uniform(-13, 2, n)
    for i, (x, y) in enumerate([(0.0, 0.125), (0.125, 0.0), (0.0, np.nextafter(0.125, 0)), (-np.inf, 1.0), (1.0, -np.inf),
                                (-np.inf, -np.inf), (np.inf, 1.0), (np.nan, 1.0), (5.0, 5.0)][:n]):
        a[-1 - i], b[-1 - i] = x, y
    da, db = (torch.zeros(n + shift, dtype=torch.float64, device="cuda")[shift:].copy_(torch.from_numpy(v)) for v in (a, b))
    got = P.relative_difference(da, db).cpu().numpy()
    with np.errstate(invalid="ignore"):
        ref = 2.0 * np.tanh(0.5 * np.abs(a - b))
    ea, eb = np.isneginf(a), np.isneginf(b)
    ref = np.where(ea & eb, np.nan, np.where(ea | eb, 2.0, ref))
    np.testing.assert_allclose(got, ref, rtol=2e-15, atol=0)
