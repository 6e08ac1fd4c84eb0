"""What the library's host code asks of the CUDA runtime, seen on the CPU: the calls run
in a process of their own over a stand-in for the runtime (fake_cudart.cpp), which
launches nothing but checks and records every launch."""
import json
import os
import subprocess
import sys
from pathlib import Path

import pytest

from paper_1109_6672_gb300 import build

ROOT = Path(__file__).resolve().parents[1]
PROLOGUE = """
import ctypes, json
import numpy as np
from paper_1109_6672_gb300 import inputs, lbm, lbm3d

fake = ctypes.CDLL(None)
fake.fake_graphs.restype = ctypes.c_longlong


def counts():
    a = (ctypes.c_longlong * 5)()
    fake.fake_counts(a)
    return dict(zip(("launches", "stale", "refused", "no_attr", "replayed"), a))


def last():  # grid x, y, z, threads, dynamic shared memory of the last launch
    a = (ctypes.c_longlong * 5)()
    fake.fake_last(a)
    return list(a)


def rest(p):
    shape = [p[k] for k in ("nz", "ny", "nx") if k in p]
    one, zero = np.ones(shape), np.zeros(shape)
    return [one] + [zero] * len(shape) + [one]


def status(call):
    try:
        call()
        return 0
    except lbm.LbmError as e:
        return e.status
"""


@pytest.fixture(scope="module")
def run(tmp_path_factory):
    """run(code) -> the JSON value that the code prints."""
    build.build()
    so = tmp_path_factory.mktemp("fake") / "fake_cudart.so"
    include = Path(build.nvcc()).resolve().parents[1] / "include"
    subprocess.run(["g++", "-std=c++17", "-O1", "-shared", "-fPIC", f"-I{include}",
                    str(ROOT / "tests" / "fake_cudart.cpp"), "-o", str(so)], check=True)

    def go(code):
        env = dict(os.environ, LD_PRELOAD=str(so), PYTHONPATH=str(ROOT))
        r = subprocess.run([sys.executable, "-c", PROLOGUE + code], env=env, capture_output=True,
                           text=True, timeout=600)
        assert r.returncode == 0, (r.returncode, r.stderr[-2000:])
        return json.loads(r.stdout)

    return go


def test_replayed_batch_graph_uses_the_current_work_list(run):
    """A batch that outgrows its work list between two runs of the same length: the
    second run replays no launch that holds the freed list."""
    got = run("""
fake.fake_pointers(1)
b = lbm.Batch(lbm.LBM_P_FP32, 8, 1 << 28)
b.set_schedule(1, 1)  # an item a row: 1024 are allocated at first
p, f = inputs.cavity(n=300, precision=lbm.LBM_P_FP32)
b.add(p, f, 100)
b.run(10)
for _ in range(3):
    b.add(p, f, 100)
b.run(10)
print(json.dumps(counts()))
""")
    assert got["replayed"] == 20 and got["stale"] == 0


def test_every_tile_request_gets_tiles_that_cover_the_grid(run):
    """FP64 grids from one column on, any requested height: a tile that fits its limits
    (96 nodes, two halo warps with the correction) and tiles that cover the grid."""
    got = run("""
bad = []
for nx in (1, 2, 3, 4, 9, 33, 70):
    for ny in (1, 2, 31, 32, 33, 64, 100):
        for corr in (0, 1):
            p = inputs.base_params(nx, ny, correction=corr)
            g = lbm.Lbm(p).init(*rest(p))
            for rows in (0, 1, 2, 30, 31, 32, 33, 50, 96, 1000):
                g.set_launch(0, rows).step(1)
                a = (ctypes.c_int * 4)()
                fake.fake_second(a)
                lw, r, tx, ghosts = a
                W, (blocks, _, _, threads, _) = 1 << lw, last()
                halo = -(-(2 * W + 2 * r) // 32) if corr else 0
                ok = (0 < r <= (rows or 32) and W * r <= 96 and halo <= 2 and tx == -(-nx // W)
                      and blocks - ghosts == tx * -(-ny // r)
                      and threads == 32 * (-(-W * r // 32) + halo))
                if not ok:
                    bad.append((nx, ny, corr, rows, lw, r))
            g.close()
print(json.dumps(bad))
""")
    assert got == []


@pytest.mark.parametrize("step", ["lbm.Lbm(inputs.base_params(9, 9))",
                                  "lbm.Lbm(inputs.base_params(9, 9, precision=1))",
                                  "lbm3d.Lbm3d(inputs.base_params3d(5, 5, 5, bc_z=[1, 1], "
                                  "T_wall_z=[1.0, 1.0]))"])
def test_a_refused_step_leaves_no_error_for_the_next_call(run, step):
    got = run(f"""
g, h = {step}, {step}
f = rest(dict(zip(("nx", "ny", "nz"), g.shape[::-1])))
g.init(*f)
fake.fake_fail_in(ctypes.c_longlong(1 if len(f) == 5 else 0))  # 3-D: the walls' launch
print(json.dumps([status(lambda: g.step(1)), status(lambda: h.init(*f)),
                  status(lambda: h.step(1))]))
""")
    assert got == [-3, 0, 0]


def test_tall_grids_stay_within_the_launch_limits(run):
    """A launch has at most 65535 blocks along y; grids have up to 2^20 rows."""
    got = run("""
out = []
for precision in range(4):
    p = inputs.base_params(4, 400000, precision=precision)
    g = lbm.Lbm(p).init(*rest(p))
    for variant, rows in ((0, 0), (0, 1), (2, 0), (2, 1), (128, 0), (128, 1)):
        g.set_launch(variant, rows)
        out.append(status(lambda: g.step(1)))
    g.close()
print(json.dumps([out, counts()["refused"]]))
""")
    assert got == [[0] * 24, 0]


def test_3d_grids_wide_along_y_stay_within_the_launch_limits(run):
    got = run("""
out = []
for precision, shapes in ((0, ((0, 0), (8, 0))), (1, ((0, 0), (8, 0), (16, 0), (8, 1)))):
    p = inputs.base_params3d(2, 1100000, 1, precision=precision)
    g = lbm3d.Lbm3d(p).init(*rest(p))
    for shape in shapes:
        g.set_launch(*shape)
        out.append(status(lambda: g.step(1)))
    g.close()
print(json.dumps([out, counts()["refused"]]))
""")
    assert got == [[0] * 6, 0]


def test_each_device_gets_the_kernels_shared_memory(run):
    """The limit of dynamic shared memory is raised per kernel and device."""
    got = run("""
out = []
for device in (0, 1, 0):
    fake.fake_device(device)
    for precision in (0, 1):
        p = inputs.base_params(64, 64, precision=precision)
        b = lbm.Batch(precision, 1, 1 << 26)
        b.add(p, rest(p), 9)
        out.append(status(lambda: b.run(1)))
        g = lbm.Lbm(p).set_launch(2, 0).init(*rest(p))
        out.append(status(lambda: g.step(1)))
        p = inputs.base_params3d(8, 8, 8, precision=precision)
        g = lbm3d.Lbm3d(p).init(*rest(p))
        out.append(status(lambda: g.step(1)))
print(json.dumps([out, counts()["no_attr"]]))
""")
    assert got == [[0] * 18, 0]


def test_a_failed_capture_leaves_no_graph_behind(run):
    got = run("""
p = inputs.base_params(64, 64, precision=1)
b = lbm.Batch(1, 2, 1 << 26)
b.add(p, rest(p), 9)
fake.fake_fail_in(ctypes.c_longlong(1))
print(json.dumps([status(lambda: b.run(3)), fake.fake_graphs(), status(lambda: b.run(3)),
                  fake.fake_graphs()]))
""")
    assert got == [-3, 0, 0, 0]


@pytest.mark.parametrize("reps", [1, 20, 257, 5000])
def test_autotune_times_the_launches_asked_for(run, reps):
    """12 candidates (6 heights, 2 ways to hand out items), each at least `reps` times."""
    got = run(f"""
p = inputs.base_params(64, 64, precision=1)
b = lbm.Batch(1, 2, 1 << 26)
b.add(p, rest(p), 9)
b.autotune({reps})
print(json.dumps(counts()["replayed"]))
""")
    assert 12 * reps <= got <= 13 * (reps + reps // 256 + 1)
