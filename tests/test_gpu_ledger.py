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
