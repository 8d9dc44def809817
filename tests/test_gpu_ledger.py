"""The mass ledger over changes of launch shape and over long calls."""
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


@pytest.mark.parametrize("nx,ny", [(9, 5), (60, 40)])
def test_a_new_shape_keeps_what_steps_in_flight_book(nx, ny):
    """Steps enqueued in a fixed shape, then the library's own choice at once: the volumes of a run that
    waits in between.  FP64 sums of 1,001 bookings in another order: 1,001 half ulps at most."""
    w = W.basin_c1(nx=nx, ny=ny)
    led = []
    for wait in (True, False):
        s = D.from_workload(w, precision=D.FP64, dt=0.05, block=256, waves=1, split=0)
        s.step(500)
        if wait:
            s.sync()
        s.set_launch(0)
        s.step(1)
        s.sync()
        led.append(s.ledger())
    a, b = led
    assert a["steps"] == b["steps"] == 501
    assert abs(a["rain_in"] - b["rain_in"]) <= 1001 * 1.2e-16 * a["rain_in"]


@pytest.mark.parametrize("nx,ny,rate,stages", [(1, 1, 1e-5, 2), (8, 8, 3.3e-6, 5), (20, 10, 1.2345e-5, 5), (20, 10, 1e-5, 3)])
def test_a_long_call_books_what_its_stages_book(nx, ny, rate, stages):
    """1,000 steps of steady rain on a small mesh in one call against stage by stage.  Both add a lane's
    pairs of floats (2^-47 an addition, at most): a product, five stages and five levels of a warp, twelve
    with the weight; beyond that FP64."""
    w = W.basin_c1(nx=nx, ny=ny)
    w.rain_nodal = np.full_like(w.rain_nodal, rate)
    led = []
    for launch in ({}, {"block": 64, "waves": 1, "split": 2}):
        s = D.from_workload(w, dt=0.01, ssp_stages=stages, **launch)
        s.step(1000)
        s.sync()
        led.append(s.ledger())
    a, b = led
    assert a["steps"] == b["steps"] == 1000
    assert abs(a["rain_in"] / b["rain_in"] - 1) <= 12 * 2.0**-47
