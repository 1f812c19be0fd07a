"""What the autotuner times and keeps (host logic, no GPU): placements that the
automatic modes pass over, and no result of other kernels."""
import pytest

import paper_1508_02748_gb300 as P
from paper_1508_02748_gb300 import autotune, workloads


# L = 8, 3 x 3 windows: both placements of tables and lattice; one L = 12 window
# of 21,025 bins: 168 KB, staged for one walker a warp; L = 32: neither
@pytest.mark.parametrize("cfg,lanes,tables,lattices", [
    (P.Config.from_workload(workloads.REWL_L8), 8, {P.TABLES_STAGED, P.TABLES_GLOBAL}, {P.LATTICE_REGISTER, P.LATTICE_SHARED}),
    (P.Config(L=12), 32, {P.TABLES_STAGED, P.TABLES_GLOBAL}, {P.LATTICE_AUTO}),
    (P.Config(L=12), 16, {P.TABLES_AUTO}, {P.LATTICE_AUTO}),
    (P.Config.from_workload(workloads.REWL_L32), 32, {P.TABLES_AUTO}, {P.LATTICE_AUTO})])
def test_every_placement_has_its_name(cfg, lanes, tables, lattices):
    offered = autotune.candidates(cfg, samplers=(P.SAMPLER_WARP,))
    names = [autotune.named(c, offered) for c in offered]
    assert len(set(names)) == len(offered)
    assert {(x[3], x[4]) for x in names if x[1] == lanes} == {(t, m) for t in tables for m in lattices}


def test_staged_tables_are_found_where_the_automatic_mode_passes_over_them():
    """AUTO is the global launch here, 5% apart by chance; staged 30% faster."""
    def time(c):
        return 7.0 if c[3] == P.TABLES_STAGED else 10.0 if c[3] == P.TABLES_GLOBAL else 9.5
    ms, c = autotune.fastest(autotune.candidates(P.Config(L=9), samplers=(P.SAMPLER_WARP,)), time)
    assert c[3] == P.TABLES_STAGED and ms == 7.0


def test_the_automatic_mode_stays_where_it_is_the_same_launch():
    """One slow sample of AUTO beside the named placement changes nothing; what
    cannot be launched is passed by."""
    seen = []

    def time(c):
        seen.append(c)
        if c[1] != 32 or c[2] != 1:
            return None
        return 1.3 if c[3] == P.TABLES_AUTO and seen.count(c) == 1 else 1.0 if c[3] != P.TABLES_GLOBAL else 2.0
    ms, c = autotune.fastest(autotune.candidates(P.Config(L=8), samplers=(P.SAMPLER_WARP,)), time)
    assert c[:4] == (P.SAMPLER_WARP, 32, 1, P.TABLES_AUTO) and ms == 1.0


def test_results_of_other_kernels_are_not_kept(tmp_path, monkeypatch):
    cfg = P.Config(L=8)
    a = autotune._key(cfg, "gpu", (0,))
    assert a == autotune._key(cfg, "gpu", (0,))
    changed = tmp_path / "kernel.cu"
    changed.write_text("another kernel")
    monkeypatch.setattr(autotune, "SOURCES", autotune.SOURCES[1:] + [str(changed)])
    assert autotune._key(cfg, "gpu", (0,)) != a
