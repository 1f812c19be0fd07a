"""The warp sampler at the edges of its lattice blocks, groups and table
placements, bit for bit against the oracle."""
import numpy as np
import pytest

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


def _same(P, steps, tile, **kw):
    o = OracleREWL(OracleConfig(**kw))
    g = P.REWL(P.Config(**kw, **tile))
    for n in steps:
        o.sweep(n)
        g.sweep(n)
        so, spo = o.walkers()
        sg, spg = g.walkers()
        np.testing.assert_array_equal(sg[:, :3], so[:, :3])
        np.testing.assert_array_equal(spg, spo)
        lo, Ho, _ = o.tables()
        lg, Hg = g.tables()
        np.testing.assert_array_equal(Hg, Ho)
        np.testing.assert_array_equal(lg, lo)
    g.close()
    o.close()


# rows of one block (L <= 30 and L = 32), of two (31, 33-60) and of three
# (61-64); 5 walkers: groups of 8 and 16 lanes leave idle ones in a warp;
# launches shorter than a step, and ones that end in the middle of one
@pytest.mark.parametrize("lanes", [32, 16, 8])
@pytest.mark.parametrize("L", [7, 9, 29, 30, 31, 32, 34, 60, 61, 62])
def test_lattice_blocks_and_idle_groups(P, L, lanes):
    _same(P, (1, 2, 3, 4, 5, 6, 1500), dict(lanes_per_walker=lanes), L=L, walkers_per_window=5, seed=300 + L)


# a grid with empty windows: their walkers' groups share warps with live ones
@pytest.mark.parametrize("lanes,tables", [(16, 1), (16, 2), (8, 1), (8, 2)])
def test_empty_windows_beside_live_ones(P, lanes, tables):
    kw = dict(L=8, n_win_E=6, n_win_M=6, overlap_E=0.5, overlap_M=0.5, walkers_per_window=3, seed=17,
              drive_budget=10**8)
    _same(P, (7, 2000), dict(lanes_per_walker=lanes, table_mode=tables, walkers_per_block=2), **kw)


def test_staged_window_at_the_shared_memory_limit(P):
    """28,390 bins fit in a block's shared memory, their staged rows with the
    entries around them do not: the run still goes, from global memory."""
    kw = dict(L=13, n_win_E=2, overlap_E=0.98, walkers_per_window=1, seed=5)
    _same(P, (3, 1200), dict(lanes_per_walker=32, table_mode=P.TABLES_STAGED), **kw)


# narrow windows: staged rows are padded to 16 entries
@pytest.mark.parametrize("lattice", [1, 2])
def test_staged_narrow_rows(P, lattice):
    kw = dict(L=4, n_win_M=4, overlap_M=0.5, walkers_per_window=3, seed=23, drive_budget=10**8)
    _same(P, (5, 1700), dict(lanes_per_walker=32, table_mode=P.TABLES_STAGED, lattice_mode=lattice), **kw)


# either side of each line of the automatic tiling (staged or global tables,
# 32, 16 or 8 lanes, lattice in a register or not), against the thread sampler
@pytest.mark.parametrize("L,nE,nM,W", [(4, 1, 1, 608), (4, 1, 1, 609), (4, 2, 1, 608), (4, 2, 1, 609), (8, 3, 3, 185),
                                       (8, 3, 3, 186), (8, 3, 3, 271), (8, 3, 3, 304), (8, 3, 3, 305), (6, 3, 2, 912),
                                       (6, 3, 2, 913), (12, 2, 1, 76), (12, 2, 1, 77)])
def test_automatic_tiling(P, L, nE, nM, W):
    kw = dict(L=L, n_win_E=nE, n_win_M=nM, walkers_per_window=W, seed=40 + L, exchange_interval=700)
    a, b = P.REWL(P.Config(**kw)), P.REWL(P.Config(sampler=P.SAMPLER_THREAD, **kw))
    sa, sb = a.run_cycles(3), b.run_cycles(3)
    assert sa == sb and a.digest() == b.digest()
    np.testing.assert_array_equal(a.walkers()[1], b.walkers()[1])


# in a batch the runs' walkers share the GPU, so the tiling goes by their sum
def test_batch_tiling_keeps_the_chains(P):
    kws = [dict(L=L, n_win_E=3, n_win_M=2, walkers_per_window=w, seed=s, exchange_interval=900)
           for L, w, s in ((8, 300, 1), (8, 200, 2), (16, 70, 3))]
    alone, together = [[P.REWL(P.Config(**kw)) for kw in kws] for _ in range(2)]
    P.Batch(together).run_cycles(4)
    for a, t in zip(alone, together):
        a.run_cycles(4)
        assert a.digest() == t.digest()
        np.testing.assert_array_equal(a.walkers()[0], t.walkers()[0])
        a.run_cycles(2), t.run_cycles(2)                 # and each goes on alone
        assert a.digest() == t.digest()


# the digest's chunks and vector tails, and a flatness check split over a
# cluster's blocks (windows of 30,276 bins and few walkers) or not: the digest
# from its definition on the host, the verdicts from the 80% rule
@pytest.mark.parametrize("L,nE,W,prec", [(4, 1, 2, 0), (13, 1, 3, 0), (13, 1, 3, 1), (13, 1, 700, 1), (6, 3, 5, 0),
                                         (13, 1, 2, 2)])
def test_digest_and_flatness(P, L, nE, W, prec):
    r = P.REWL(P.Config(L=L, n_win_E=nE, walkers_per_window=W, seed=3, precision=prec, exchange_interval=500))
    r.run_cycles(2)
    lng, H = r.tables()
    rng = np.random.default_rng(L + W)
    n = H.size // r.n_walkers
    for w in range(r.n_walkers):       # either side of the line
        H[w * n:(w + 1) * n] = np.where(rng.random(n) < 0.7, rng.integers(66 + w % 2, 101, n), -1)
    lng = np.round(lng * 256) / 256
    r.set_tables(lng, H)
    lng, H = r.tables()

    def mix(z):
        z = (z ^ (z >> np.uint64(30))) * np.uint64(0xBF58476D1CE4E5B9)
        z = (z ^ (z >> np.uint64(27))) * np.uint64(0x94D049BB133111EB)
        return z ^ (z >> np.uint64(31))

    with np.errstate(over="ignore"):
        i = np.arange(H.size, dtype=np.uint64)
        h = H.astype(np.uint32).astype(np.uint64)
        want = int((mix(lng.view(np.uint64) ^ mix(i)) + mix(h + np.uint64(0x9E3779B97F4A7C15) * i)).sum(dtype=np.uint64))
    assert r.digest() == want
    r.check()
    Hw = H.reshape(r.n_walkers, n)
    flat = [int(x[x >= 0].min()) * (x >= 0).sum() * 10**6 >= 800000 * int(x[x >= 0].sum()) for x in Hw]
    np.testing.assert_array_equal(r.walkers(spins=False)[0][:, 3], np.array(flat, dtype=np.int64))
