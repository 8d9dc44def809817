"""Tile plans: tiles whose edges and neighbours exceed the inline part of the plan, and ragged tails.

A triangle far away makes the space-filling curve's cells so large that all other elements share one,
so the library keeps their given order; shuffled, nearly every neighbour of a tile is in another tile
(up to 96 edges and 96 neighbours per tile, against about 60 and 23 in curve order)."""
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


def scattered(nx, ny, p=1, ocean=False):
    w = W.basin_c1(nx=nx, ny=ny, seed=3)
    m = w.mesh
    if ocean:  # tide on the x = 0 side
        mid = 0.5 * (m.xy[m.bedge[:, 0]] + m.xy[m.bedge[:, 1]])
        m.btype[mid[:, 0] < 1e-6] = W.OCEAN
        w.tide = W.Tide(np.array([0.4]), np.array([600.0]), np.array([0.3]))
    tri = m.tri[np.random.default_rng(11).permutation(m.n_tri)]
    n = m.n_nodes
    far = np.array([[1e9, 1e9], [1e9 + 2e3, 1e9], [1e9, 1e9 + 2e3]])
    w.mesh = W.Mesh(np.concatenate([m.xy, far]), np.concatenate([tri, [[n, n + 1, n + 2]]]).astype(np.int32),
                    m.bedge, m.btype, m.bseg)
    w.hb = np.concatenate([w.hb, [9.0] * 3])
    w.zeta0 = np.concatenate([w.zeta0, [0.0] * 3])
    w.rain_nodal = np.concatenate([w.rain_nodal, [0.0] * 3])
    w.manning = np.full(w.mesh.n_tri, 0.025)
    w.p = p
    return w


@pytest.mark.parametrize("prec", [D.FP64, D.MIXED])
@pytest.mark.parametrize("nx,ny,p,ocean", [(20, 10, 1, True), (13, 7, 2, False), (3, 5, 1, False), (4, 4, 1, True), (1, 1, 2, False)])
def test_scattered_tiles_match_the_oracle(nx, ny, p, ocean, prec):
    """The bars of the other parity tests; the tile form stage by stage and in the library's own choice."""
    w = scattered(nx, ny, p, ocean)
    ref = O.from_workload(w)
    dt = ref.cfl_dt(w.cfl)
    ref.set_dt(dt)
    ref.step(60)
    want = ref.state()
    for launch in ({"block": 64, "waves": 1, "split": 2}, {}):
        dev = D.from_workload(w, precision=prec, dt=dt, **launch)
        dev.step(60)
        dev.sync()
        got = dev.state()
        if prec == D.FP64:
            assert max(np.abs(got[:, v] - want[:, v]).max() / max(1.0, np.abs(want[:, v]).max()) for v in range(3)) <= 1e-11
        else:
            assert np.abs(got - want).max() <= 1e-4
        assert dev.ledger()["rel_err"] < 1e-12
