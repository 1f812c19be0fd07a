"""The join over the whole range of what it takes: ln g of large magnitude
against the oracle, and grids of more windows than one grid axis has blocks."""
import ctypes

import numpy as np
import pytest

import oracle
from oracle import OracleConfig, OracleREWL
from test_gpu_join_shapes import _set

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


# ln g is free up to a constant.  Beside +-2^30 a double's upper word stands for
# 1024: all values just above such a step, and just below one.  Each side makes
# at most some 20 roundings of 2^-53 |offset| between a table's entry and the
# normalised one: the merge's differences, sum and quotient (6), for each of
# three matching points two marginals and the shift (9), the entry's two shifts
# and the normalisation's three.
@pytest.mark.parametrize("nE,nM", [(1, 1), (3, 2)])
@pytest.mark.parametrize("offset", [2**30 + 1000, -2**30 - 1100, 2 * 10**9, -10**9, -10**8])
def test_join_of_large_tables(P, offset, nE, nM):
    kw = dict(L=6, n_win_E=nE, n_win_M=nM, overlap_E=0.5, overlap_M=0.5, walkers_per_window=3, seed=6, drive_budget=10**8)
    o = OracleREWL(OracleConfig(**kw))
    lng, H = _set(o, [], 17)
    lng = np.where(H >= 0, lng + offset, 0.0)
    o.set_tables(lng, H)
    tol = 2 * 20 * 2.0**-53 * abs(offset)
    for precision in (P.FP64, P.F32X2):
        r = P.REWL(P.Config(precision=precision, **kw))
        r.set_tables(lng, H)
        for ro, rg in ((oracle.JOIN_MARGINAL, P.JOIN_MARGINAL), (oracle.JOIN_PER_SLICE, P.JOIN_PER_SLICE)):
            Jo, em, mm = o.join(ro)
            Jg, emg, mmg = r.lng(matches=True, rule=rg)
            np.testing.assert_array_equal(emg, em)
            np.testing.assert_array_equal(mmg, mm)
            fin = np.isfinite(Jo)
            assert np.array_equal(np.isfinite(Jg), fin)
            np.testing.assert_allclose(Jg[fin], Jo[fin], rtol=0, atol=tol)


# Tables with entries that are no number or infinite, in one walker or in all:
# what the oracle's join makes of them, or refuses, this one does too.
@pytest.mark.parametrize("L,nE,nM,W,seen", [(6, 2, 1, 3, 0.99), (8, 3, 2, 1, 0.9), (12, 4, 1, 3, 0.5), (9, 2, 2, 8, 0.9), (5, 1, 1, 2, 1.0)])
@pytest.mark.parametrize("bad", [(np.inf, np.inf), (-np.inf, -np.inf), (np.nan, -np.nan), (np.inf, np.nan)])
def test_join_of_tables_that_are_not_finite(P, L, nE, nM, W, seen, bad):
    kw = dict(L=L, n_win_E=nE, n_win_M=nM, overlap_E=0.5, overlap_M=0.5, walkers_per_window=W, seed=6, drive_budget=10**8)
    o, r = OracleREWL(OracleConfig(**kw)), P.REWL(P.Config(**kw))
    rng = np.random.default_rng(L)
    for everywhere in (False, True):
        lng, H = _set(o, [], 11)
        H = np.where((H >= 0) & (rng.random(H.size) < seen), H, -1).astype(np.int32)
        n = H.size // (W * nE * nM)
        for w in range(0, H.size // n, 1 if everywhere else H.size // n):
            at = w * n + rng.choice(np.flatnonzero(H[w * n:(w + 1) * n] >= 0), 2, replace=False)
            lng[at] = bad
        for x in (o, r):
            x.set_tables(lng, H)
        for ro, rg in ((oracle.JOIN_MARGINAL, P.JOIN_MARGINAL), (oracle.JOIN_PER_SLICE, P.JOIN_PER_SLICE)):
            try:
                Jo, em, mm = o.join(ro)
            except RuntimeError:
                with pytest.raises(P.REWLError, match="join failed"):
                    r.lng(rule=rg)
                continue
            Jg, emg, mmg = r.lng(matches=True, rule=rg)
            np.testing.assert_array_equal(emg, em)
            np.testing.assert_array_equal(mmg, mm)
            np.testing.assert_allclose(Jg, Jo, rtol=1e-12, atol=1e-9)


def test_join_of_more_windows_than_a_grid_axis(P):
    """257 x 257 windows of 2 x 2 bins cut out of one table, each with an offset
    of its own: joined again, the table comes back up to a constant.  It falls
    off by 50 a bin beside a ridge that all windows of an m range hold with its
    neighbours, so that rows of different length agree on their marginals."""
    import torch
    L, n = 16, 257
    cfg = P.Config(L=L, n_win_E=n, n_win_M=n, overlap_E=0.5, overlap_M=0.5)
    lo = (2 * np.arange(n) * (n - 2) + n - 1) // (2 * (n - 1))              # window starts, rounded half up
    can = np.array([[oracle.lib().orc_bin_possible(L, e, m) for m in range(n)] for e in range(n)]) != 0
    e = np.arange(n)[:, None]
    ridge = np.array([np.flatnonzero(can[:, m]).mean().round() for m in range(n)])
    G = -50.0 * np.abs(e - ridge[None, :])
    rng = np.random.default_rng(4)
    two = np.arange(2)
    rows, cols = lo[None, :, None, None] + two[:, None], lo[:, None, None, None] + two[None, :]
    tab = G[rows, cols] + np.round(rng.uniform(0, 900, (n, n, 1, 1)) * 64) / 64
    d = torch.from_numpy(np.ascontiguousarray(tab).ravel()).cuda()
    H = torch.ones(d.numel(), dtype=torch.int32, device="cuda")
    out = torch.empty(n, n, dtype=torch.float64, device="cuda")
    torch.cuda.synchronize()
    lib, c = P.load_library(), cfg.to_c()
    rc = lib.rewl_join_noalloc(ctypes.byref(c), d.data_ptr(), H.data_ptr(), out.data_ptr(), None)
    assert rc == 0, lib.rewl_noalloc_last_error()
    J = out.cpu().numpy()
    fin = np.isfinite(J)
    assert fin[can].all()
    diff = (J - G)[fin]
    # 512 matching points, at each two marginals, their difference and a shift, of at most 2^14 in magnitude
    assert np.ptp(diff) < 2 * 512 * 4 * 2.0**-53 * 2**14
    top = J[fin].max()
    np.testing.assert_allclose(top + np.log(np.exp(J[fin] - top).sum()), L * L * np.log(2.0), rtol=0, atol=1e-9)
