"""The word engine (single solves on abstractions whose every box is its
plane's entry) against the CPU oracle and against the list form on the same
handle, at the sizes where its bitmaps can go wrong: planes of 31 to 33 and
1023 to 1025 cells (word and unit edges), rows of 31, 63 and 95 cells (windows
that need a third word), one plane, one cell wide planes, periodic and not on
dims 2 and 3, 1 and 32 inputs.  Values are compared bit for bit: no tolerance.
"""
import numpy as np
import pytest

import oracle
import paper_2001_06231_gb300 as bf
from test_gpu_solve import plane_instance, same

pytestmark = pytest.mark.gpu
INF = float("inf")


def handle(n, periodic, boxes):
    D = len(n)
    return bf.abs_from_boxes(bf.make_grid(n, [0.0] * D, [float(k) for k in n], periodic), boxes)


def list_form(A):
    bf.bf_set_schedule(A, slice_target=2, fuse_mark=1, window33=0, plane_lists=1, cell_masks=0)


@pytest.mark.parametrize("n,periodic,U,wmax,seed", [
    ([31, 1, 5], [False, False, True], 3, (5, 1, 3, 1), 1),
    ([8, 4, 6], [False, False, False], 4, (4, 3, 3, 1), 2),
    ([11, 3, 7], [False, False, True], 5, (5, 2, 4, 1), 3),
    ([33, 31, 4], [False, False, True], 4, (5, 5, 3, 1), 4),
    ([32, 32, 3], [False, False, False], 4, (6, 6, 3, 1), 5),
    ([41, 25, 5], [False, False, True], 1, (3, 3, 2, 1), 6),
    ([63, 17, 6], [False, False, True], 6, (5, 5, 4, 1), 7),
    ([95, 23, 3, 4], [False, False, True, True], 5, (4, 4, 3, 3), 8),
    ([19, 18, 4, 3], [False, False, False, True], 32, (4, 4, 2, 2), 9),
    ([70, 40], [False, False], 7, (6, 6, 1, 1), 10),
    ([1, 50, 9], [False, False, True], 3, (1, 4, 3, 1), 11),
    ([26, 90, 2, 2], [False, False, True, False], 6, (5, 4, 2, 2), 12),
])
def test_words_match_oracle_and_list_form(n, periodic, U, wmax, seed):
    rng = np.random.default_rng(4000 + seed)
    boxes, G, target, avoid = plane_instance(rng, n, periodic, U, wmax=wmax, p_differ=0.0)
    A = handle(n, periodic, boxes)
    assert A.shape_mismatch == 0
    T = np.where(target.astype(bool), 0.0, INF)
    ref = oracle.solve(n, periodic, boxes, G, T, avoid)
    k = ref["iters"]
    word = [bf.bf_solve(A, G, target=target, avoid=avoid, trace_cap=4096, host_loop=hl) for hl in (False, True, False)]
    assert word[0]["stats"]["kernel_launches"] == 2            # set-up and one launch for all passes
    list_form(A)
    word.append(bf.bf_solve(A, G, target=target, avoid=avoid, trace_cap=4096))
    for r in word:
        assert r["iters"] == k and r["status"] == ref["status"]
        assert same(r["V"], ref["V"]) and same(r["mu"], ref["mu"])
        assert same(r["trace"][:k, 1], ref["changed"][:k])
    # the frontier of the word engine is Algorithm 1's exactly
    assert same(word[0]["trace"][:k, 0], ref["f1"][:k])
    assert word[0]["stats"]["relaxed_cells"] == int(ref["f1"][:k].sum())


@pytest.mark.parametrize("cap", [1, 2, 5, 0])
def test_words_cap_terminal_and_negative_cycle(cap):
    """A pass cap, a terminal cost that is finite everywhere and costs below
    zero (the loop then runs into the cap, or into |X| passes without one)."""
    n, periodic, U = [9, 7, 4], [False, False, True], 3
    rng = np.random.default_rng(77)
    boxes, G, target, avoid = plane_instance(rng, n, periodic, U, wmax=(3, 3, 2, 1), p_differ=0.0)
    G = G - 0.75
    T = rng.integers(0, 40, size=boxes.shape[0]) * 0.25
    A = handle(n, periodic, boxes)
    for t in (T, np.where(target.astype(bool), 0.0, INF)):
        ref = oracle.solve(n, periodic, boxes, G, t, avoid, max_iters=cap)
        for hl in (False, True):
            r = bf.bf_solve(A, G, terminal=t, avoid=avoid, max_iters=cap, host_loop=hl)
            assert r["iters"] == ref["iters"] and r["status"] == ref["status"]
            assert same(r["V"], ref["V"]) and same(r["mu"], ref["mu"])


def test_words_check_every_cost():
    """One bad cost anywhere (the first, the last, an unaligned array's ends)
    is an error, and the handle solves again afterwards; device costs that
    start 8 bytes past a 16-byte boundary give the same result."""
    import torch
    n, periodic, U = [13, 9, 5], [False, False, True], 3
    rng = np.random.default_rng(5)
    boxes, G, target, avoid = plane_instance(rng, n, periodic, U, wmax=(3, 3, 2, 1), p_differ=0.0)
    A = handle(n, periodic, boxes)
    good = bf.bf_solve(A, G, target=target, avoid=avoid)
    N = G.size
    for shift in (0, 1):
        buf = torch.zeros(N + 2, dtype=torch.float64, device="cuda")
        g = buf[shift:shift + N]
        for at in (0, 1, N // 2, N - 2, N - 1):
            for bad in (float("nan"), -INF, 1e300):
                g.copy_(torch.from_numpy(G.reshape(-1)))
                g[at] = bad
                with pytest.raises(bf.BfError):
                    bf.bf_solve(A, g, target=target, avoid=avoid)
        g.copy_(torch.from_numpy(G.reshape(-1)))
        r = bf.bf_solve(A, g, target=target, avoid=avoid)
        assert same(r["V"], good["V"]) and same(r["mu"], good["mu"]) and r["iters"] == good["iters"]


@pytest.mark.parametrize("n,periodic,U,wmax,seed", [
    ([33, 17, 5], [False, False, True], 4, (5, 4, 3, 1), 21),
    ([12, 31, 4, 3], [False, False, True, False], 5, (4, 4, 3, 2), 22),
    ([63, 9, 3], [False, False, False], 3, (2, 3, 2, 1), 23),
    ([40, 30], [False, False], 6, (1, 4, 1, 1), 24),
])
@pytest.mark.parametrize("share", [0.0, 0.3, 1.0])
def test_words_successor_class(n, periodic, U, wmax, seed, share):
    """The class form (two value tables, the cost by the successor's class):
    no cell, some cells, every cell in the class; finite terminal cost and
    negative class costs included."""
    rng = np.random.default_rng(4000 + seed)
    boxes, G, target, avoid = plane_instance(rng, n, periodic, U, wmax=wmax, p_differ=0.0)
    C = boxes.shape[0]
    cls = (rng.random(C) < share).astype(np.uint8)
    Gc = rng.integers(-2, 5, size=(C, U)) * 0.25
    Gc[rng.random((C, U)) < 0.02] = INF
    A = handle(n, periodic, boxes)
    for T in (np.where(target.astype(bool), 0.0, INF), rng.integers(0, 30, size=C) * 0.5):
        ref = oracle.solve(n, periodic, boxes, G, T, avoid, succ_class=cls, G_class=Gc, max_iters=200)
        k = ref["iters"]
        for hl in (False, True):
            r = bf.bf_solve(A, G, terminal=T, avoid=avoid, succ_class=cls, G_class=Gc, max_iters=200, trace_cap=4096,
                            host_loop=hl)
            assert r["iters"] == k and r["status"] == ref["status"]
            assert same(r["V"], ref["V"]) and same(r["mu"], ref["mu"])
            assert same(r["trace"][:k, 1], ref["changed"][:k])
    plain = bf.bf_solve(A, G, target=target, avoid=avoid)      # the same handle without a class again
    ref = oracle.solve(n, periodic, boxes, G, np.where(target.astype(bool), 0.0, INF), avoid)
    assert same(plain["V"], ref["V"]) and same(plain["mu"], ref["mu"])


@pytest.mark.parametrize("n,periodic,U,reach,width,seed", [
    ([31], [False], 3, 3, 4, 31), ([33], [True], 2, 5, 33, 32), ([1], [False], 2, 0, 1, 33),
    ([32, 33], [True, True], 4, 4, 9, 34), ([64, 16], [False, True], 32, 2, 5, 35),
    ([41, 25], [False, False], 3, 40, 12, 36), ([7, 5, 31], [True, False, True], 5, 3, 6, 37),
    ([95, 11, 3], [False, False, True], 4, 2, 7, 38), ([6, 7, 5, 9], [True, True, True, True], 3, 2, 5, 39),
    ([300, 3, 2], [False, False, False], 6, 130, 2, 40),
])
def test_box_form_matches_oracle_and_list_form(n, periodic, U, reach, width, seed):
    """Boxes that differ from cell to cell (the engine's box form): wrapping any
    dim, whole circles, boxes that read 3 x 3 windows or rows of any length,
    records too far for the compact form, one cell, 32 inputs."""
    from test_gpu_solve import random_instance
    rng = np.random.default_rng(4000 + seed)
    boxes, G, target, avoid = random_instance(rng, n, periodic, U, reach=reach, width=width, neg=False)
    target[rng.integers(0, boxes.shape[0])] = 1
    A = handle(n, periodic, boxes)
    T = np.where(target.astype(bool), 0.0, INF)
    ref = oracle.solve(n, periodic, boxes, G, T, avoid)
    k = ref["iters"]
    res = [bf.bf_solve(A, G, target=target, avoid=avoid, trace_cap=4096, host_loop=hl) for hl in (False, True)]
    list_form(A)
    res.append(bf.bf_solve(A, G, target=target, avoid=avoid, trace_cap=4096))
    for r in res:
        assert r["iters"] == k and r["status"] == ref["status"]
        assert same(r["V"], ref["V"]) and same(r["mu"], ref["mu"])
        assert same(r["trace"][:k, 1], ref["changed"][:k])
    assert same(res[0]["trace"][:k, 0], ref["f1"][:k])


def one_launch(r):
    """Did a solve run as its set-up and one launch for all passes?"""
    return r["stats"]["kernel_launches"] == 2


def schedule_of(t):
    """The settings of a bf_tune result (what bf_set_schedule reads)."""
    return {k: v for k, v in t.items() if k not in ("candidates", "best_ms", "default_ms")}


def form_instance(kind):
    """A grid with more than 128 units of work for a single block: 160 planes of
    63 cells (every box its plane's entry), 141 words of boxes that differ."""
    from test_gpu_solve import random_instance
    rng = np.random.default_rng(4100)
    if kind == "entries":
        n, periodic, U = [9, 7, 40, 4], [False, False, True, False], 5
        boxes, G, target, avoid = plane_instance(rng, n, periodic, U, wmax=(3, 3, 2, 2), p_differ=0.0)
    else:
        n, periodic, U = [75, 60], [True, False], 4
        boxes, G, target, avoid = random_instance(rng, n, periodic, U, reach=3, width=4, neg=False)
        target[rng.integers(0, boxes.shape[0])] = 1
    ref = oracle.solve(n, periodic, boxes, G, np.where(target.astype(bool), 0.0, INF), avoid)
    return n, periodic, boxes, G, target, avoid, ref


@pytest.mark.parametrize("kind", ["entries", "boxes"])
def test_schedule_names_its_form(kind):
    """one_launch says which form a solve takes, whatever the list form's fields
    say, at every width (one block then relaxes more units than it tests at a
    time); the list form's own fields are in force when it is 0."""
    n, periodic, boxes, G, target, avoid, ref = form_instance(kind)
    A = handle(n, periodic, boxes)
    pair_queue = dict(slice_target=0, fuse_mark=0, window33=1, plane_lists=1, templates=1, pair_inputs=1, cell_masks=2,
                      input_frontier=1)
    plain = dict(slice_target=2, fuse_mark=1, window33=0, plane_lists=0, templates=0)
    for fields in (pair_queue, plain):
        for form, width in ((1, 0), (1, 1), (0, 0), (1, 2), (1, 151), (0, 1), (1, 100000)):
            bf.bf_set_schedule(A, one_launch=form, relax_blocks=width, **fields)
            r = bf.bf_solve(A, G, target=target, avoid=avoid)
            assert one_launch(r) == (form == 1), (fields, form, width)
            assert r["iters"] == ref["iters"] and r["status"] == ref["status"]
            assert same(r["V"], ref["V"]) and same(r["mu"], ref["mu"]), (fields, form, width)
            bf.bf_set_schedule(A, one_launch=-1, **fields)           # leaves the form as it is
            assert one_launch(bf.bf_solve(A, G, target=target, avoid=avoid)) == (form == 1)


@pytest.mark.parametrize("kind", ["entries", "boxes"])
def test_tuned_schedule_replays_on_another_handle(kind):
    """What bf_tune reports, put in force on another handle of the same system,
    takes the same form; so does what it reports when the handle starts from a
    list schedule."""
    n, periodic, boxes, G, target, avoid, ref = form_instance(kind)
    for start in (None, dict(slice_target=2, fuse_mark=1)):
        A, B = handle(n, periodic, boxes), handle(n, periodic, boxes)
        if start:
            bf.bf_set_schedule(A, **start)
        t = bf.bf_tune(A, G, target=target, avoid=avoid)
        bf.bf_set_schedule(B, **schedule_of(t))
        a, b = (bf.bf_solve(H, G, target=target, avoid=avoid) for H in (A, B))
        assert one_launch(a) == one_launch(b) == (t["one_launch"] == 1)
        assert same(a["V"], ref["V"]) and same(b["V"], ref["V"]) and same(a["mu"], ref["mu"]) and same(b["mu"], ref["mu"])


def tune_inplace(A, G, target, avoid):
    """bf_tune on solves with the in-place schedule, through the C interface."""
    import ctypes
    opts, res = bf.SolveOpts(), bf.TuneResult()
    opts.schedule = bf.SCHED_INPLACE
    rc = bf.lib().bf_tune(A.handle, G.ctypes.data, target.ctypes.data, avoid.ctypes.data, ctypes.byref(opts),
                          ctypes.byref(res), None)
    assert rc == 0
    return {k: getattr(res, k) for k, _ in res._fields_}


def test_tuner_leaves_the_form_to_the_solves_it_timed():
    """Tuned for solves that the one-launch form does not take (in place; boxes
    that differ with a successor class), a handle keeps its form, and the list
    form's settings are searched, whether or not it was solved before."""
    n, periodic, boxes, G, target, avoid, ref = form_instance("boxes")
    cls = (np.random.default_rng(3).random(boxes.shape[0]) < 0.3).astype(np.uint8)
    for solved in (False, True):
        for tune in (lambda A: bf.bf_tune(A, G, target=target, avoid=avoid, succ_class=cls, G_class=G),
                     lambda A: tune_inplace(A, G, target, avoid)):
            A = handle(n, periodic, boxes)
            if solved:
                assert one_launch(bf.bf_solve(A, G, target=target, avoid=avoid))
            t = tune(A)
            assert t["one_launch"] == -1 and t["candidates"] > 5
            r = bf.bf_solve(A, G, target=target, avoid=avoid)
            assert one_launch(r) and same(r["V"], ref["V"]) and same(r["mu"], ref["mu"])


def test_tuner_times_the_one_launch_form_from_a_list_schedule():
    """A handle with a list schedule in force is tuned to the one-launch form
    (on this unicycle 2.5 times as fast)."""
    from paper_2001_06231_gb300 import workloads as wl
    w = wl.unicycle3d(n=(40, 40, 100), n_obstacles=3)
    A = bf.abs_build_workload(w)
    bf.bf_set_schedule(A)
    before = bf.bf_solve(A, w.G, target=w.target, avoid=w.avoid)
    assert not one_launch(before)
    t = bf.bf_tune(A, w.G, target=w.target, avoid=w.avoid)
    after = bf.bf_solve(A, w.G, target=w.target, avoid=w.avoid)
    assert t["one_launch"] == 1 and one_launch(after)
    assert same(after["V"], before["V"]) and same(after["mu"], before["mu"])


@pytest.mark.parametrize("n,U,scattered,one", [
    ([9000], 32, False, True), ([320, 320], 8, False, True),
    ([340, 340], 8, False, False), ([340, 340], 8, True, True), ([500, 500], 5, True, False),
    ([64, 64, 65], 8, False, True), ([70, 70, 70], 8, False, False), ([70, 70, 70], 8, True, True),
    ([90, 90, 86], 8, True, False), ([24, 24, 24, 24], 16, False, True),
    ([30, 30, 30, 30], 8, False, False), ([30, 30, 30, 30], 8, True, True),
])
def test_box_form_by_pairs_and_breadth_of_the_frontier(n, U, scattered, one):
    """Boxes that differ from cell to cell, on both sides of the lines between
    the one-launch form and the list form: the form a solve takes by itself, host
    and device inputs, and the same V, mu and passes from either (40 passes)."""
    import torch
    rng = np.random.default_rng(4300)
    C, D = int(np.prod(n)), len(n)
    coords = np.stack(np.unravel_index(np.arange(C), tuple(reversed(n)))[::-1], axis=1)
    boxes = np.empty((C, U, 2, D), dtype=np.int16)
    for u in range(U):
        lo = coords + rng.integers(-2, 3, size=(1, D)) * (np.arange(D) == u % D)
        hi = lo + rng.integers(0, 2, size=(C, 1))
        ok = np.all((lo >= 0) & (hi < np.array(n)), axis=1)
        boxes[:, u, 0], boxes[:, u, 1] = np.where(ok[:, None], lo, 0), np.where(ok[:, None], hi, 0)
        boxes[~ok, u, 0, 0] = bf.BLOCKED
    G = rng.integers(1, 6, size=(C, U)) * 0.25
    target = (rng.random(C) < 0.004 if scattered else np.all(np.abs(coords - np.array(n) // 2) <= 1, axis=1)).astype(np.uint8)
    avoid = (rng.random(C) < 0.02).astype(np.uint8)
    A = handle(n, [False] * D, boxes)
    dev = [torch.from_numpy(x).cuda() for x in (G, target, avoid)]
    r = bf.bf_solve(A, dev[0], target=dev[1], avoid=dev[2], max_iters=40)
    assert one_launch(r) == one
    T = np.where(target.astype(bool), 0.0, INF)
    assert one_launch(bf.bf_solve(A, G, terminal=T, avoid=avoid, max_iters=40)) == one
    for form in (0, 1):
        bf.bf_set_schedule(A, one_launch=form)
        q = bf.bf_solve(A, G, target=target, avoid=avoid, max_iters=40)
        assert one_launch(q) == (form == 1)
        assert same(q["V"], r["V"]) and same(q["mu"], r["mu"]) and (q["iters"], q["status"]) == (r["iters"], r["status"])


def test_solves_of_several_threads_share_the_device():
    """Solves of four threads, a handle and a stream each, overlap (they took
    four times a lone solve one after the other, 1.4 times when they share the
    SMs) and give what a lone solve gives, beside a batched call too."""
    import threading
    import time

    import torch
    from paper_2001_06231_gb300 import workloads as wl
    w = wl.unicycle3d(n=(100, 100, 32), n_obstacles=10)
    ins = [torch.from_numpy(x).cuda() for x in (w.G, w.target, w.avoid)]

    def job():
        A, s = bf.abs_build_workload(w), torch.cuda.Stream()
        V = torch.empty(w.ncells, dtype=torch.float64, device="cuda")
        mu = torch.empty(w.ncells, dtype=torch.uint8, device="cuda")
        return A, lambda: bf.bf_solve(A, ins[0], target=ins[1], avoid=ins[2], V=V, mu=mu, stream=s.cuda_stream)

    jobs = [job() for _ in range(4)]
    torch.cuda.synchronize()

    def timed(fs, reps=12):
        def go(f):
            f()
            gate.wait()
            for _ in range(reps):
                f()
            gate.wait()
        gate = threading.Barrier(len(fs) + 1)
        th = [threading.Thread(target=go, args=(f,)) for f in fs]
        for t in th:
            t.start()
        gate.wait()
        t0 = time.perf_counter()
        gate.wait()
        dt = time.perf_counter() - t0
        for t in th:
            t.join()
        return dt

    lone = jobs[0][1]()
    lone = (lone["V"].clone(), lone["mu"].clone(), lone["iters"])
    one = min(timed([jobs[0][1]]) for _ in range(3))
    four = min(timed([f for _, f in jobs]) for _ in range(3))
    assert four < 2.5 * one, (one, four)
    As, batch = [bf.abs_build_workload(w) for _ in range(3)], []
    timed([f for _, f in jobs] + [lambda: batch.append(bf.bf_solve_batch(
        As, [w.G] * 3, targets=[w.target] * 3, avoids=[w.avoid] * 3))], reps=3)
    for r in [f() for _, f in jobs]:
        assert torch.equal(r["V"], lone[0]) and torch.equal(r["mu"], lone[1]) and r["iters"] == lone[2]
    for rs in batch:
        for r in rs:
            assert same(r["V"], lone[0].cpu().numpy()) and same(r["mu"], lone[1].cpu().numpy()) and r["iters"] == lone[2]


@pytest.mark.parametrize("gate", [0, 1])
def test_a_wait_that_runs_out_sets_its_flag_and_leaves(tmp_path, gate):
    """A block whose partner never arrives gives up after its polls, sets the fault
    flag and returns; the device goes on (a solve afterwards)."""
    import ctypes
    from test_host_cpu import build_word_wait
    lib = build_word_wait(tmp_path)
    passed, fault = ctypes.c_int(-2), ctypes.c_int(-2)
    assert lib.wait_runs_out(gate, ctypes.byref(passed), ctypes.byref(fault)) == 0
    assert passed.value == 0 and fault.value == 1
    n, periodic, boxes, G, target, avoid, ref = form_instance("entries")
    r = bf.bf_solve(handle(n, periodic, boxes), G, target=target, avoid=avoid)
    assert one_launch(r) and same(r["V"], ref["V"])


FULL_DEVICE = r'''
import sys
sys.path.insert(0, sys.argv[1])
import torch
import paper_2001_06231_gb300 as bf
from paper_2001_06231_gb300 import workloads as wl
w = wl.unicycle3d()
A = bf.abs_build_workload(w)
a = [torch.from_numpy(x).cuda() for x in (w.G, w.target, w.avoid)]
V = torch.empty(w.ncells, dtype=torch.float64, device="cuda")
mu = torch.empty(w.ncells, dtype=torch.uint8, device="cuda")
solve = lambda **k: bf.bf_solve(A, a[0], target=a[1], avoid=a[2], V=V, mu=mu, **k)
solve(schedule=bf.SCHED_INPLACE)           # the list form's workspace
hog, step = [], 1 << 34
while step >= 1 << 21:                     # the rest of the memory
    try:
        hog.append(torch.empty(step, dtype=torch.uint8, device="cuda"))
    except torch.OutOfMemoryError:
        step >>= 1
full = solve()
got = V.cpu()
hog = None
torch.cuda.empty_cache()
again = solve()
assert again["stats"]["kernel_launches"] == 2 and full["iters"] == again["iters"] and torch.equal(got, V.cpu())
print("solved")
'''


def test_without_memory_for_the_one_launch_form_the_list_form_solves():
    """A handle with the list form's workspace solves on a full device (the 40 MB of
    the one-launch form cannot be had), and takes the one-launch form when there
    is memory again.  In a process of its own."""
    import os
    import subprocess
    import sys
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    r = subprocess.run([sys.executable, "-c", FULL_DEVICE, root], capture_output=True, text=True, timeout=300)
    assert r.returncode == 0 and "solved" in r.stdout, r.stdout + r.stderr


def test_mu_may_be_written_over_an_input():
    """A device buffer given as the class or the avoid mask and as mu too: read as
    the input to the end, then written, as in the list form."""
    import torch
    n, periodic, U = [33, 17, 5], [False, False, True], 4
    rng = np.random.default_rng(4400)
    boxes, G, target, avoid = plane_instance(rng, n, periodic, U, wmax=(5, 4, 3, 1), p_differ=0.0)
    C = boxes.shape[0]
    cls = (rng.random(C) < 0.3).astype(np.uint8)
    Gc = rng.integers(-2, 5, size=(C, U)) * 0.25
    T = rng.integers(0, 30, size=C) * 0.5
    A = handle(n, periodic, boxes)
    ref = oracle.solve(n, periodic, boxes, G, T, avoid, succ_class=cls, G_class=Gc, max_iters=200)
    assert ref["iters"] > 3
    for over in ("cls", "avoid"):
        for form in (1, 0):
            bf.bf_set_schedule(A, one_launch=form)
            d = {k: torch.from_numpy(x.copy()).cuda() for k, x in
                 (("G", G), ("T", T), ("avoid", avoid), ("cls", cls), ("Gc", Gc))}
            V = torch.empty(C, dtype=torch.float64, device="cuda")
            r = bf.bf_solve(A, d["G"], terminal=d["T"], avoid=d["avoid"], succ_class=d["cls"], G_class=d["Gc"], V=V,
                            mu=d[over], max_iters=200)
            assert one_launch(r) == (form == 1) and r["iters"] == ref["iters"], (over, form)
            assert same(V.cpu().numpy(), ref["V"]) and same(d[over].cpu().numpy(), ref["mu"]), (over, form)
