"""Gridded rain keeps the accuracy of its records: after the last one, and in the node kernel."""
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


def _area(m):
    a, b, c = (m.xy[m.tri[:, k]] for k in range(3))
    return 0.5 * ((b - a)[:, 0] * (c - a)[:, 1] - (c - a)[:, 0] * (b - a)[:, 1])


@pytest.mark.parametrize("launch", [{}, {"block": 64, "split": 0}, {"block": 64, "split": 2}])
@pytest.mark.parametrize("prec,bound", [(D.FP64, 1e-13), (D.MIXED, 2 * 2.0**-24)])
def test_after_a_storm_the_last_record_holds(prec, bound, launch):
    """A drizzle after a downpour: the volume of the last record alone.  Mixed: the record is held in FP32
    (2^-24), twice that with the area's product; FP64: the sums."""
    w = W.basin_c1(nx=13, ny=7)
    w.rain_nodal = None
    f = np.stack([np.full((2, 2), 100.0), np.full((2, 2), 0.003)]).astype(np.float32)
    w.rain_grid = W.RainGrid(2, 2, 2, 0.0, 0.0, 1e4, 5e3, -1e4, 40.0, f)
    s = D.from_workload(w, precision=prec, dt=0.5, **launch)
    s.step(20)
    s.sync()
    want = 20 * 0.5 * _area(w.mesh).sum() * float(f[1, 0, 0]) * W.MMH
    assert abs(s.ledger()["rain_in"] / want - 1) <= bound


def test_the_node_kernel_agrees_to_rounding():
    """4,400 records on 500k triangles (8.8 GB of element means) go through the node kernel; the two around
    the run's time, as a grid of their own, through records.  250,000 s into 60 s records, 10 and 90 mm/h in
    turn.  Both hold FP32 values: a blend and a mean of four roundings each, and the stored rates."""
    w = W.coastal_c2(500_000, seed=3, fast_mesh=True)
    w.storm = None
    f = np.empty((4400, 1, 1), np.float32)
    f[0::2], f[1::2] = 10.0, 90.0
    t0 = 250_000.3
    k = int(t0 // 60.0)
    rain = []
    for first, rec in ((0, f), (k, f[k:k + 2])):
        w.rain_grid = W.RainGrid(1, 1, len(rec), 0.0, 0.0, 1.0, 1.0, 60.0 * first, 60.0, rec)
        dev = D.from_workload(w, dt=0.2, block=64, waves=1, split=2)
        dev.set_state(w.zeta0, t0=t0)
        n0 = dev.launch_count()
        dev.step(1)
        assert dev.launch_count() - n0 == (4 if first == 0 else 2)
        dev.sync()
        rain.append(dev.ledger()["rain_in"])
        dev.close()
    assert abs(rain[0] / rain[1] - 1) <= 10 * 2.0**-24


@pytest.mark.parametrize("prec", [D.FP64, D.MIXED])
def test_members_of_an_ensemble_keep_their_own_grids_in_the_node_kernel(prec):
    """Two small gridded members beside one whose records are beyond 8 GiB: nodes of different scenarios
    share blocks.  Their rain is that of their solo runs, which go through records."""
    big = W.coastal_c2(500_000, seed=3, fast_mesh=True)
    big.storm = None
    nt = 4400 if prec == D.MIXED else 2200
    big.rain_grid = W.RainGrid(1, 1, nt, 0.0, 0.0, 1.0, 1.0, 0.0, 60.0, np.full((nt, 1, 1), 5.0, np.float32))
    ws = []
    for k in (2, 3):
        w = W.basin_c1(nx=5 * k, ny=4)
        w.rain_nodal = None
        f = np.random.default_rng(k).uniform(0, 100, (k, 3, 4)).astype(np.float32)
        w.rain_grid = W.RainGrid(4, 3, k, 0.0, 0.0, 3e3, 2e3, 0.0, 0.7 * k, f)
        ws.append(w)
    ens = D.Ensemble([D.from_workload(w, precision=prec, dt=0.2, block=64, split=2) for w in [ws[0], big, ws[1]]])
    ens.set_launch(64, 1, 2)
    n0 = ens.launch_count()
    ens.step(5)
    assert ens.launch_count() - n0 == 20  # a node launch per stage
    ens.sync()
    for i, w in ((0, ws[0]), (2, ws[1])):
        s = D.from_workload(w, precision=prec, dt=0.2, block=64, waves=1, split=2)
        s.step(5)
        s.sync()
        assert abs(ens.ledger(i)["rain_in"] / s.ledger()["rain_in"] - 1) <= (10 * 2.0**-24 if prec == D.MIXED else 1e-13)
        s.close()
    ens.close()
