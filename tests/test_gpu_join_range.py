"""The join over the whole range of what it takes: ln g of large magnitude
against the oracle, and grids of more windows than one grid axis has blocks."""
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
