"""Kernels that split their work by size, at splits that the other tests' sizes
do not reach: clusters of 4 and 8 blocks in the flatness check, chunks of more
bins than a pass holds in the join's offsets."""
import numpy as np
import pytest

import oracle
from oracle import OracleConfig, OracleREWL
from test_gpu_join_shapes import _near, _set

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


# one window of 66,049 bins: 8 blocks a walker below 152 walkers, 4 below 304.
# Every bin 100 visits but a single one just above or below the line of 80%,
# which lies in each block's share (and in the odd last bin) in turn
@pytest.mark.parametrize("W,parts", [(20, 8), (160, 4)])
def test_flatness_split_over_a_cluster(P, W, parts):
    r = P.REWL(P.Config(L=16, walkers_per_window=W, seed=3))
    n = 257 * 257
    rng = np.random.default_rng(W)
    H = np.where(rng.random((W, n)) < 0.9, 100, -1).astype(np.int32)
    for w in range(W):
        rank = w // 2 % (parts + 1)
        turn = rng.integers(0, 66048 // (parts * 1024) - 1)
        at = n - 1 if rank == parts else 4 * ((turn * parts + rank) * 256 + rng.integers(0, 256)) + rng.integers(0, 4)
        H[w, at] = 79 + 2 * (w % 2)
    r.set_tables(np.zeros(H.size), H.ravel())
    r.check()
    seen = H >= 0
    flat = np.where(seen, H, 10**6).min(1).astype(np.int64) * seen.sum(1) * 10**6 >= 800000 * np.where(seen, H, 0).sum(1)
    assert flat.any() and not flat.all()
    np.testing.assert_array_equal(r.walkers(spins=False)[0][:, 3], flat.astype(np.int64))


# 600 walkers and 4225 bins: two chunks of 4096 and 129 bins, the first in two
# passes; every third bin is visited by all
def test_join_of_many_walkers(P):
    kw = dict(L=8, walkers_per_window=600, seed=6, drive_budget=10**8)
    o = OracleREWL(OracleConfig(**kw))
    lng, H = _set(o, [], 5)
    H = H.reshape(600, -1)
    H[:, ::3] = np.maximum(H[:, ::3], 0)
    H = H.ravel()
    o.set_tables(lng, H)
    ref = o.join()[0]
    for precision in (P.FP64, P.F32X2, P.F32):
        r = P.REWL(P.Config(precision=precision, **kw))
        r.set_tables(lng, H)
        _near(r.lng(), ref)


def test_jackknife_of_two_walkers_that_share_no_bin(P):
    """Each replicate has one walker and joins; the walkers together do not."""
    kw = dict(L=5, walkers_per_window=2, seed=2)
    o, r = OracleREWL(OracleConfig(**kw)), P.REWL(P.Config(**kw))
    lng, H = r.tables()
    half = H.size // 2
    H[:] = 1
    H[:half][half // 2:] = -1
    H[half:][:half // 2] = -1
    lng[:] = np.where(H >= 0, 1.0, 0.0)
    for x in (o, r):
        x.set_tables(lng, H)
    with pytest.raises(P.REWLError, match="join failed .code 1"):
        r.lng()
    mean, err = r.jackknife()
    mo, _ = oracle.jackknife(o)
    assert np.array_equal(mean, np.asarray(mo).reshape(mean.shape)) and np.isneginf(mean).all() and np.isnan(err).all()


# Eq. 5 either side of the count from which a thread takes two bins
@pytest.mark.parametrize("n,shift", [(77_823, 0), (77_824, 0), (77_825, 0), (77_824, 1), (200_001, 0)])
def test_relative_difference_by_pairs(P, n, shift):
    import torch
    rng = np.random.default_rng(n + shift)
    a = rng.normal(0, 300, n)
    b = a + np.where(rng.random(n) < 0.5, 1, -1) * 10.0 ** rng.uniform(-13, 2, n)
    a[rng.integers(0, n, 50)] = -np.inf
    b[rng.integers(0, n, 50)] = -np.inf
    a[-1], b[-1] = 0.0, 0.125
    da, db = (torch.zeros(n + shift, dtype=torch.float64, device="cuda")[shift:].copy_(torch.from_numpy(v)) for v in (a, b))
    with np.errstate(invalid="ignore"):
        ref = 2.0 * np.tanh(0.5 * np.abs(a - b))
    ea, eb = np.isneginf(a), np.isneginf(b)
    ref = np.where(ea & eb, np.nan, np.where(ea | eb, 2.0, ref))
    np.testing.assert_allclose(P.relative_difference(da, db).cpu().numpy(), ref, rtol=2e-15, atol=0)
