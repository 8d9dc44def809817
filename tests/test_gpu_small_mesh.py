"""Small meshes: whole steps in one cluster launch give the bits of the tile form launched stage by
stage, over tile counts from one to the largest cluster, schemes, degrees, precisions and forcings."""
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


def _basin(nx, ny, p=1):
    w = W.basin_c1(nx=nx, ny=ny)
    w.p = p
    return w


def _coastal(n, p=1):
    w = W.coastal_c2(n, seed=23, fast_mesh=True)
    w.p = p
    w.cfl = 0.1
    return w


def _hurricane():
    w = W.hurricane_c5(3000)
    w.cfl = 0.04  # explicit friction on films needs dt tau < 1: at 0.3 the oracle itself diverges on this mesh
    return w


CASES = {
    "one_tile": (lambda: _basin(1, 1), {}),
    "four_tiles": (lambda: _basin(8, 8), {}),
    "five_tiles": (lambda: _basin(13, 5), {"ssp_stages": 3}),
    "basin_p2": (lambda: _basin(20, 10, 2), {}),
    "basin_llf5": (lambda: _basin(20, 10), {"flux": D.FLUX_LLF, "ssp_stages": 5}),
    "quadratic": (lambda: _basin(17, 11), {"friction": D.QUADRATIC, "cf": 0.002}),
    "river": (lambda: W.river_basin(q=(2.0, 0.5, 1.5), internal=True), {}),
    "flume": (lambda: W.inclined_plane("A", sim_s=1.0), {"dt": 1e-3}),
    "coastal": (lambda: _coastal(2000), {}),
    "graded_p2": (lambda: W.graded_c3(2000), {}),
    "hurricane": (_hurricane, {}),
    "sixteen_ctas": (lambda: _coastal(4500), {}),
}


@pytest.mark.parametrize("prec", [D.FP64, D.MIXED])
@pytest.mark.parametrize("case", list(CASES))
def test_cluster_steps_equal_the_tile_form(case, prec):
    make, opt = CASES[case]
    w = make()
    a = D.from_workload(w, precision=prec, **opt)
    b = D.from_workload(w, precision=prec, block=64, waves=1, split=2, **opt)
    n0 = a.launch_count()
    for n in (1, 2, 30):
        a.step(n)
        b.step(n)
        a.sync()
        b.sync()
        assert np.array_equal(a.state(), b.state()), (case, n)
    assert a.launch_count() - n0 <= 6 or case == "sixteen_ctas"  # 3 launches and 3 state copies
    la, lb = a.ledger(), b.ledger()
    assert la["steps"] == lb["steps"] == 33 and la["V"] == lb["V"]
    scale = max(abs(lb["VH0"]), abs(lb["V0"]))
    for k in ("rain_in", "bdry_in"):
        assert abs(la[k] - lb[k]) <= 1e-13 * scale, (case, k, la[k], lb[k])
    # the other ways of stepping go on from the same state: stage by stage, then the cluster again
    a.set_graphs(False)
    a.step(2)
    a.set_graphs(True)
    a.step(1)
    b.step(3)
    assert np.array_equal(a.state(), b.state())


def test_long_runs_are_split_into_launches():
    """1030 steps: two launches; the state goes on as in single steps."""
    w = _basin(5, 5)
    a, b = (D.from_workload(w) for _ in range(2))
    a.step(1)
    n0 = a.launch_count()
    a.step(1030)
    assert a.launch_count() - n0 == 2
    for n in (31, 1000):
        b.step(n)
    a.sync()
    b.sync()
    assert np.array_equal(a.state(), b.state()) and a.ledger()["steps"] == 1031


def test_ensemble_of_small_meshes_and_bound_records():
    """Several scenarios in one cluster equal their solo runs; records in caller memory are stepped."""
    import torch

    ws = [_coastal(500), _basin(6, 4), W.river_basin(nx=8, ny=4)]
    solo = [D.from_workload(w) for w in ws]
    ens = D.Ensemble([D.from_workload(w) for w in ws])
    mem = torch.empty(solo[0].record_bytes(), dtype=torch.uint8, device="cuda")
    solo[0].bind_device(mem.data_ptr(), mem.numel())
    ens.step(7)
    ens.sync()
    for i, s in enumerate(solo):
        s.set_launch(64, 1, 2) if i else None
        s.step(7)
        s.sync()
    # the members' feature union selects the ensemble's kernel: equal to rounding
    for i, s in enumerate(solo):
        assert np.abs(ens.state(i) - s.state()).max() <= 1e-5 * max(1.0, np.abs(s.state()).max())
        assert ens.ledger(i)["rel_err"] < 1e-12


def test_a_larger_mesh_in_the_same_context():
    """A context that ran a small mesh takes another one; the choice is made again."""
    w, big = _basin(6, 4), _coastal(20_000)
    s = D.from_workload(w)
    s.step(3)
    s.set_mesh(big.mesh)
    s.set_fields(big.hb, big.manning)
    s.set_storm(big.storm)
    s.set_tide(big.tide)
    s.set_state(big.zeta0)
    s.step(3)
    s.sync()
    t = D.from_workload(big, dt=s.dt())
    t.set_launch(*s.launch())
    t.step(3)
    t.sync()
    assert np.array_equal(s.state(), t.state())


@pytest.mark.parametrize("prec", [D.FP64, D.MIXED])
def test_single_steps_equal_a_longer_call(prec):
    """Steps taken one by one (replayed from a graph) give the bits of one call, also after the records
    have moved to other memory and after a new state."""
    import torch

    w = _basin(9, 5)
    a, b = (D.from_workload(w, precision=prec) for _ in range(2))
    for s in (a, b):
        s.step(1)
    mem = torch.empty(a.record_bytes(), dtype=torch.uint8, device="cuda")
    a.bind_device(mem.data_ptr(), mem.numel())
    for _ in range(4):
        a.step(1)
    b.step(4)
    for s in (a, b):
        s.sync()
    assert np.array_equal(a.state(), b.state()) and a.ledger()["steps"] == b.ledger()["steps"] == 5
    for s in (a, b):
        s.set_state(w.zeta0)
    a.step(1)
    a.step(1)
    b.step(2)
    for s in (a, b):
        s.sync()
    assert np.array_equal(a.state(), b.state())
