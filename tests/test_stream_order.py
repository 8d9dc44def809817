"""Order between the default stream and the library's own stream, on the CPU.

The library's stream is non-blocking, so nothing orders it against uploads on the default stream but a
synchronisation.  A stand-in for the CUDA runtime (order_cudart.cpp, loaded before the real one in a child
process) follows the calls of a few programs and reports every order that CUDA does not promise."""
import os
import re
import subprocess
import sys

import pytest

from paper_2307_14302_gb300 import build as B

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)

PRELUDE = """
import ctypes, sys
import numpy as np
from paper_2307_14302_gb300 import dgswe as D
from paper_2307_14302_gb300 import workloads as W

def basin(nx, ny, grid=False):
    w = W.basin_c1(nx=nx, ny=ny)
    if grid:
        w.rain_nodal = None
        w.rain_grid = W.RainGrid(3, 2, 4, 0.0, 0.0, 5e3, 5e3, 0.0, 600.0, np.ones((4, 2, 3), np.float32))
    return w
"""
EPILOGUE = """
r = ctypes.CDLL(None).{}
r.restype = ctypes.c_char_p
sys.stdout.write(r().decode())
"""

PROGRAMS = {
    "gridded_rain": """
s = D.from_workload(basin(9, 5, grid=True), dt=1.0, precision=PREC, block=64, split=2)
s.sync()
""",
    # the time step's upload, then the first step at once in a shape that is not timed
    "fixed_shape": """
s = D.from_workload(basin(9, 5), precision=PREC, block=64, split=2)
s.step(3)
s.sync()
""",
    # the ledger of the shape before is folded, then the first launch books into it
    "cluster": """
s = D.from_workload(basin(9, 5), precision=PREC)
s.step(3)
s.sync()
""",
    # a choice of shape asked for while steps are in flight
    "retuned": """
s = D.from_workload(basin(9, 5), precision=PREC, block=256, split=1)
s.step(50)
s.set_launch(0)
s.step(1)
s.sync()
""",
    "retuned_large": """
s = D.from_workload(basin(90, 50), precision=PREC, block=256, split=1)
s.step(50)
s.set_launch(0)
s.step(1)
s.sync()
""",
    # a new state, and a new mesh, while steps are in flight
    "new_state": """
w, v = basin(9, 5), basin(13, 7, grid=True)
s = D.from_workload(w, precision=PREC)
s.step(50)
s.set_state(w.zeta0)
s.step(50)
s.set_mesh(v.mesh)
s.set_fields(v.hb, v.manning)
s.set_rain_grid(v.rain_grid)
s.set_state(v.zeta0)
s.step(1)
s.sync()
""",
    "read_outs": """
s = D.from_workload(basin(90, 50), precision=PREC, dt=1.0)
s.step(50)
s.ledger()
s.step(1)
s.volume()
s.step(1)
s.dry()
s.step(1)
a = s.state_arrays()
s.step(1)
s.load_state(*a)
s.step(1)
s.exchange(*a)
e = D.Ensemble([s, D.from_workload(basin(9, 5), precision=PREC)])
e.step(3)
e.ledger(1)
e.step(1)
e.state(0)
e.sync()
""",
}


@pytest.fixture(scope="module")
def runtime(tmp_path_factory):
    B.build()
    so = tmp_path_factory.mktemp("order") / "order_cudart.so"
    inc = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(B._nvcc()))), "include")
    subprocess.run(["g++", "-std=c++17", "-O1", "-shared", "-fPIC", f"-I{inc}", "-o", str(so),
                    os.path.join(HERE, "order_cudart.cpp")], check=True)
    return so


def _run(runtime, program, what):
    code = PRELUDE + program + EPILOGUE.format(what)
    env = dict(os.environ, LD_PRELOAD=str(runtime), PYTHONPATH=ROOT)
    r = subprocess.run([sys.executable, "-c", code], env=env, capture_output=True, text=True, timeout=600)
    assert r.returncode == 0, r.stderr[-2000:]
    return r.stdout


@pytest.mark.parametrize("prec", ["D.FP64", "D.MIXED"])
@pytest.mark.parametrize("program", list(PROGRAMS))
def test_no_unordered_work(program, prec, runtime):
    assert _run(runtime, f"PREC = {prec}\n" + PROGRAMS[program], "order_report") == ""


# kernel, grid and block of a call of several steps on nx x ny x 2 triangles; None: stage by stage
@pytest.mark.parametrize("prec,p,nx,ny,want", [
    ("D.FP64", 1, 20, 10, ("steps_kernel", 13, 32)),     # FP64: one tile per SM while there are 16 or fewer
    ("D.FP64", 1, 32, 32, ("steps_kernel", 16, 128)),
    ("D.FP64", 1, 48, 32, ("steps_kernel", 16, 192)),    # the last that keep the cluster
    ("D.FP64", 1, 48, 33, None),
    ("D.FP64", 2, 32, 32, ("steps_kernel", 16, 128)),
    ("D.FP64", 2, 32, 33, None),
    ("D.MIXED", 1, 20, 10, ("steps_kernel", 4, 128)),
    ("D.MIXED", 1, 64, 64, ("steps_kernel", 16, 512)),   # as many tiles as the largest cluster has warps
    ("D.MIXED", 1, 64, 65, None),
])
def test_form_of_small_meshes(runtime, prec, p, nx, ny, want):
    out = _run(runtime, f"""
w = basin({nx}, {ny})
w.p = {p}
s = D.from_workload(w, precision={prec}, dt=1.0)
s.step(2)
""", "order_launches").split("\n")[-2].split()
    assert ((want[0] in out[0] and (int(out[1]), int(out[2])) == want[1:]) if want else "steps_kernel" not in out[0])


@pytest.mark.parametrize("free,node", [(200 << 30, False), (1 << 30, False), (100 << 20, True)])
def test_rain_path_follows_the_size(runtime, free, node, monkeypatch):
    """360 MB of rain records: element records whatever else the device holds, the node kernel only where
    they do not fit."""
    monkeypatch.setenv("ORDER_FREE", str(free))
    out = _run(runtime, """
w = basin(9, 5)
w.rain_nodal = None
w.rain_grid = W.RainGrid(2, 1, 1_000_000, 0.0, 0.0, 1e4, 1e4, 0.0, 60.0, np.ones((1_000_000, 1, 2), np.float32))
s = D.from_workload(w, dt=1.0, block=64, split=2)
s.step(1)
""", "order_launches")
    assert ("node_rain_kernel" in out) == node and ("rain_record_kernel" in out) != node


@pytest.mark.parametrize("workload,options", [
    ("basin(9, 5)", ""), ("basin(9, 5)", "ssp_stages=3"), ("W.coastal_c2(800, seed=1, fast_mesh=True)", ""),
    ("W.coastal_c2(800, seed=1, fast_mesh=True)", "ssp_stages=5, flux=D.FLUX_LLF"), ("W.inclined_plane('A', sim_s=1.0)", ""),
    ("W.inclined_plane('A', sim_s=1.0)", "ssp_stages=3"), ("W.graded_c3(800)", ""), ("W.river_basin(nx=8, ny=4)", ""),
])
def test_both_kernels_take_the_same_instantiation(runtime, workload, options):
    """The small-mesh kernel and the tile kernel of a run: equal template arguments."""
    out = [_run(runtime, f"""
s = D.from_workload({workload}, dt=1.0{launch}{options and ", " + options})
s.step(2)
""", "order_launches").split("\n")[-2] for launch in ("", ", block=64, split=2")]
    args = [re.search(kernel + r"(I.*?5MixedE.*?E)Ev", o) for kernel, o in zip(("steps_kernel", "tile_kernel"), out)]
    assert args[0] and args[1] and args[0].group(1) == args[1].group(1)
