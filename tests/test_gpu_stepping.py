"""Ways of stepping at the edges of their ranges."""
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
