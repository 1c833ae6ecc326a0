"""The builder's range tables (one quantisation per plane, input and coordinate)
against the general path: the recompute-mode export runs the RK4 scheme for
every (cell, input) pair, and importing the exported boxes walks every box for
the predecessor index.  Boxes, records and predecessor boxes are integers and
must be identical.
"""
import math

import numpy as np
import pytest

import paper_2001_06231_gb300 as bf
from paper_2001_06231_gb300 import workloads as wl

pytestmark = pytest.mark.gpu


def _with(w, **kw):
    for k, v in kw.items():
        setattr(w, k, v)
    return w


def _periodic(w, p):
    w.grid = wl.Grid(w.grid.n, w.grid.lo, w.grid.hi, p)
    return w


CASES = {
    "unicycle": lambda: wl.unicycle3d(n=(37, 41, 13), n_obstacles=2),
    "unicycle one plane": lambda: wl.unicycle3d(n=(33, 20, 1), n_obstacles=2),
    "unicycle theta open": lambda: _periodic(wl.unicycle3d(n=(30, 31, 9), n_obstacles=2), (False, False, False)),
    "unicycle x periodic": lambda: _periodic(wl.unicycle3d(n=(24, 21, 8), n_obstacles=2), (True, False, True)),
    "unicycle wide records": lambda: _with(wl.unicycle3d(n=(300, 6, 5), n_obstacles=2), tau=5.0),
    "unicycle 11 substeps": lambda: _with(wl.unicycle3d(n=(21, 19, 8), n_obstacles=2), substeps=11),
    "fire": lambda: wl.fire4d(n=(25, 23, 10, 3), n_blobs=1, n_nofly=1, tau=2.0),
    "fire V periodic": lambda: _periodic(wl.fire4d(n=(21, 20, 9, 4), n_blobs=1, n_nofly=1, tau=1.0),
                                         (False, False, True, True)),
    "fire 2 substeps": lambda: _with(wl.fire4d(n=(26, 17, 12, 2), n_blobs=1, n_nofly=1, tau=1.5), substeps=2),
}


@pytest.mark.parametrize("name", sorted(CASES))
def test_range_tables_equal_the_general_path(name):
    w = CASES[name]()
    A = bf.abs_build_workload(w)
    boxes = A.export_boxes()
    R = bf.abs_build_workload(w, mode=bf.MODE_RECOMPUTE)
    assert np.array_equal(boxes, R.export_boxes())
    B = bf.abs_from_boxes(w.grid, boxes)
    pred = B.export_pred()
    assert np.array_equal(A.export_pred(), pred)
    assert np.array_equal(R.export_pred(), pred)
    assert A.box_record_bytes == B.box_record_bytes
    assert (A.shape_planes, A.shape_mismatch) == (B.shape_planes, B.shape_mismatch)
    K = max(1, w.ninputs // 3)
    H = bf.abs_build_workload(w, box_budget=8 * w.ncells * K)
    assert np.array_equal(H.export_boxes(), boxes) and np.array_equal(H.export_pred(), pred)


@pytest.mark.parametrize("n,held", [((6, 6, 300), False), ((10, 10, 200), False), ((20, 20, 60), True),
                                    ((40, 40, 20), True)])
def test_recompute_handles_stay_small(n, held):
    """What a recompute handle holds beside the inputs, the predecessor index and the
    shared RK4 parts is at most a quarter of the compact records it avoids: on
    planes of few cells nothing, and its solves regenerate the boxes."""
    w = wl.unicycle3d(n=n, n_obstacles=1)
    S, R = bf.abs_build_workload(w), bf.abs_build_workload(w, mode=bf.MODE_RECOMPUTE)
    C, U, planes = w.ncells, w.ninputs, n[2]
    base = 16 * U + 4 * 3 * C + 22 * 8 * planes * U
    extra = R.device_bytes - base
    assert 0 <= extra <= 8 * C * U // 4 and (extra > 0) == held
    r, s = (bf.bf_solve(A, w.G, target=w.target, avoid=w.avoid) for A in (R, S))
    assert (r["stats"]["kernel_launches"] == 2) == held
    assert np.array_equal(r["V"], s["V"]) and np.array_equal(r["mu"], s["mu"]) and r["iters"] == s["iters"]


MANY_PLANES = r'''
import sys
import numpy as np
sys.path.insert(0, sys.argv[1])
import paper_2001_06231_gb300 as bf
from paper_2001_06231_gb300 import workloads as wl
def held():                                # most host memory the process held, MB
    return int(next(l for l in open("/proc/self/status") if l.startswith("VmHWM")).split()[1]) / 1024
w = wl.unicycle3d(n=(20, 18, 8), n_obstacles=2)
bf.abs_build_workload(w)                   # the context is up
g = bf.make_grid([3, 3, 16383], w.grid.lo, w.grid.hi, w.grid.periodic)
before = held()
A = [bf.abs_build(w.kind, [0.5] + list(w.params[1:]), w.substeps, g, w.inputs[:2], w.tau, m)
     for m in (bf.MODE_STORED, bf.MODE_RECOMPUTE)]
print("grew", held() - before)
boxes = A[0].export_boxes()
assert (boxes[:, :, 0, 0] != bf.BLOCKED).any() and np.array_equal(boxes, A[1].export_boxes())
pred = bf.abs_from_boxes(g, boxes).export_pred()
assert np.array_equal(A[0].export_pred(), pred) and np.array_equal(A[1].export_pred(), pred)
assert A[0].box_record_bytes == 12
'''


def test_ranges_over_many_planes_take_the_general_path():
    """A grid of 9 cells a plane whose boxes span 784 of 16,383 planes: the lists of
    target planes would hold 26 M entries (411 MB on the host and on the device
    each); the build takes the general path, with the same boxes and predecessor
    boxes in either mode, and holds little host memory.  In a process of its own."""
    import os
    import subprocess
    import sys
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    r = subprocess.run([sys.executable, "-c", MANY_PLANES, root], capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stdout + r.stderr
    assert float(r.stdout.split()[1]) < 150, r.stdout
