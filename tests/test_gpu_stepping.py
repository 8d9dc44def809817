"""Ways of stepping at the edges of their ranges: the largest cluster, long graphs, and ensembles whose
members have different kinds of rain."""
import numpy as np
import pytest

from paper_2307_14302_gb300 import dgswe as D
from paper_2307_14302_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2307_14302_gb300 import build as B

    B.build()
    D.lib()


@pytest.mark.parametrize("prec,p,nx,ny,cluster", [
    (D.MIXED, 1, 64, 63, True),    # 252 tiles in 16 CTAs of 16 warps
    (D.MIXED, 1, 64, 64, True),    # 256: every warp has a tile
    (D.MIXED, 1, 65, 63, True),    # 256, the last of 30 elements
    (D.MIXED, 1, 64, 65, False),   # 260: stage by stage
    (D.FP64, 1, 48, 32, True),     # 96: six tiles to a CTA
    (D.FP64, 1, 48, 33, False),
    (D.FP64, 2, 32, 32, True),     # 64: four
    (D.FP64, 2, 32, 33, False),
])
def test_the_largest_clusters(prec, p, nx, ny, cluster):
    w = W.basin_c1(nx=nx, ny=ny)
    w.p = p
    a = D.from_workload(w, precision=prec)
    b = D.from_workload(w, precision=prec, block=64, waves=1, split=2)
    a.step(1)
    n0 = a.launch_count()
    a.step(5)
    assert (a.launch_count() - n0 == 1) == cluster
    b.step(6)
    a.sync()
    b.sync()
    if a.launch()[2] == 2:  # the same form: the same bits
        assert np.array_equal(a.state(), b.state())


@pytest.mark.parametrize("limiter", [False, True])
@pytest.mark.parametrize("prec", [D.FP64, D.MIXED])
def test_every_graph_length_equals_direct_launches(prec, limiter):
    """63 steps are one graph each of 32, 16, 8, 4, 2 and 1 steps."""
    w = W.coastal_c2(12_000, seed=23, fast_mesh=True)
    w.cfl = 0.1
    a, b = (D.from_workload(w, precision=prec, block=128, waves=1, split=2, limiter=limiter) for _ in range(2))
    b.set_graphs(False)
    for s in (a, b):
        n0 = s.launch_count()
        s.step(63)
        assert s.launch_count() - n0 == 63 * 2 * (2 if limiter else 1)
        s.sync()
    assert np.array_equal(a.state(), b.state()) and a.ledger() == b.ledger()


def _gridded(nx, ny, nt, seed):
    w = W.basin_c1(nx=nx, ny=ny, seed=seed)
    w.rain_nodal = None
    f = np.random.default_rng(seed).uniform(0, 100, (nt, 3, 4)).astype(np.float32)
    w.rain_grid = W.RainGrid(4, 3, nt, 0.0, 0.0, 3e3, 2e3, 0.0, 7.0, f)
    return w


@pytest.mark.parametrize("k", [1, 6])
def test_an_ensemble_of_different_rains(k):
    """Gridded (two grids), storm, nodal and no rain side by side, in a cluster and stage by stage: in FP64,
    where one instantiation serves every run, the bits of the members' solo runs."""
    coastal = W.coastal_c2(500 * k * k, seed=23, fast_mesh=True)
    coastal.cfl = 0.1
    dry = W.basin_c1(nx=5 * k, ny=3 * k)
    dry.rain_nodal = None
    ws = [_gridded(6 * k, 4 * k, 5, 1), coastal, W.basin_c1(nx=7 * k, ny=3 * k), _gridded(5 * k, 5 * k, 2, 2), dry]
    solo = [D.from_workload(w, precision=D.FP64, block=64, waves=1, split=2) for w in ws]
    ens = D.Ensemble([D.from_workload(w, precision=D.FP64) for w in ws])
    ens.step(1)
    n0 = ens.launch_count()
    ens.step(6)
    assert (ens.launch_count() - n0 == 1) == (k == 1)
    ens.sync()
    same = ens.launch()[2] == 2
    for i, s in enumerate(solo):
        s.step(7)
        s.sync()
        want = s.state()
        assert np.array_equal(ens.state(i), want) if same else np.abs(ens.state(i) - want).max() <= 1e-11 * np.abs(want).max()
        assert ens.ledger(i)["rel_err"] < 1e-12
