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
