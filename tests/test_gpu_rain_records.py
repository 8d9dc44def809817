"""Gridded rain: the element records that a stage blends in time, at the edges of the grid and of its
records, and the node kernel that serves grids whose records would not fit in memory."""
import numpy as np
import pytest

import oracle as O
from paper_2307_14302_gb300 import dgswe as D
from paper_2307_14302_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2307_14302_gb300 import build as B

    B.build()
    D.lib()


def _basin(nx, ny, nt, t0):
    w = W.basin_c1(nx=13, ny=7)
    w.rain_nodal = None
    rng = np.random.default_rng(5)
    # the grid covers the middle of the basin only: nodes outside take its edge cells
    w.rain_grid = W.RainGrid(nx, ny, nt, 2000.0, 1000.0, 6000.0 / max(nx - 1, 1), 3000.0 / max(ny - 1, 1), t0, 40.0,
                             rng.uniform(0, 100, (nt, ny, nx)).astype(np.float32))
    return w


@pytest.mark.parametrize("form", [0, 1, 2])
@pytest.mark.parametrize("nx,ny,nt,t0", [(2, 2, 2, 0.0), (5, 4, 3, -60.0), (3, 2, 2, 1e4), (4, 3, 2, -1e4), (7, 5, 6, 5.0)])
def test_records_match_the_oracle(nx, ny, nt, t0, form):
    """FP64 within the FP64 bar of the oracle: inside the records, before the first, after the last."""
    w = _basin(nx, ny, nt, t0)
    ref = O.from_workload(w)
    dt = ref.cfl_dt(w.cfl)
    ref.set_dt(dt)
    ref.step(40)
    dev = D.from_workload(w, precision=D.FP64, dt=dt, block=64, waves=1, split=form)
    dev.step(40)
    dev.sync()
    want, got = ref.state(), dev.state()
    assert max(np.abs(got[:, v] - want[:, v]).max() / max(1.0, np.abs(want[:, v]).max()) for v in range(3)) <= 1e-11
    assert abs(dev.ledger()["rain_in"] / ref.ledger()["rain_in"] - 1) <= 1e-12


@pytest.mark.parametrize("nx,ny,nt", [(1, 1, 1), (2, 1, 1), (1, 3, 2)])
def test_degenerate_grids(nx, ny, nt):
    """One column, row or record: the volume that falls in is the closed form of the held field."""
    w = _basin(nx, ny, nt, 1e4)  # before the first record: the first field throughout
    dev = D.from_workload(w, precision=D.FP64, dt=1.0, block=64, waves=1, split=2)
    dev.step(10)
    dev.sync()
    g, xy, tri = w.rain_grid, w.mesh.xy, w.mesh.tri
    x = np.clip((xy[:, 0] - g.x0) / g.dx, 0, nx - 1)
    y = np.clip((xy[:, 1] - g.y0) / g.dy, 0, ny - 1)
    f = g.mm_per_h[0].astype(float)
    fx = f[:, 0] + (f[:, -1] - f[:, 0]) * x[:, None] if nx > 1 else np.repeat(f[:, :1].T, len(x), 0)
    fx = fx.reshape(len(x), ny)
    iy = np.minimum(y.astype(int), max(ny - 2, 0))
    node = fx[np.arange(len(x)), iy] * (1 - (y - iy)) + fx[np.arange(len(x)), np.minimum(iy + 1, ny - 1)] * (y - iy)
    a, b, c = (xy[tri[:, k]] for k in range(3))
    area = 0.5 * ((b - a)[:, 0] * (c - a)[:, 1] - (c - a)[:, 0] * (b - a)[:, 1])
    assert abs(dev.ledger()["rain_in"] / (10.0 * (area * node[tri].mean(1)).sum() * W.MMH) - 1) <= 1e-12


def test_node_kernel_serves_records_that_do_not_fit():
    """4,400 records on 500k triangles (8.8 GB of element means) go through the node kernel; the same
    run with the records it meets goes through them.  The node path forms a cell position in FP32
    (6e-8 of up to 1,000 cells): rain agrees to 1e-4; the state to FP32 rounding of its slopes."""
    w = W.coastal_c2(500_000, seed=3, fast_mesh=True)
    w.storm = None
    f = np.random.default_rng(1).uniform(0, 100, (4400, 3, 4)).astype(np.float32)
    out = []
    for nt in (4400, 3):
        w.rain_grid = W.RainGrid(4, 3, nt, 0.0, 0.0, 133_000.0, 149_000.0, 0.0, 60.0, f[:nt])
        dev = D.from_workload(w, dt=0.2, block=64, waves=1, split=2)
        n0 = dev.launch_count()
        dev.step(3)
        dev.sync()
        out.append((dev.state(), dev.ledger(), dev.launch_count() - n0))
        dev.close()
    (a, la, na), (b, lb, nb) = out
    assert na > nb  # a node launch per stage
    assert abs(la["rain_in"] / lb["rain_in"] - 1) <= 1e-4
    assert np.abs(a - b).max() <= 1e-5 * max(1.0, np.abs(b).max())
