"""Host-side checks that need no GPU: the C ABI library and its exports, the
input generators, and the multi-rank aggregation of bench.py (gloo ranks)."""
import ctypes
import os
import re
import socket

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def header_functions():
    txt = open(os.path.join(ROOT, "include", "bfgpu.h")).read()
    return sorted(set(re.findall(r"BF_API\s+[\w\s\*]+?\b(\w+)\s*\(", txt)))


def test_library_loads_and_exports_every_declared_function():
    from paper_2001_06231_gb300 import _build
    path = _build.build()
    lib = ctypes.CDLL(path)
    names = header_functions()
    assert len(names) >= 14
    missing = [n for n in names if not hasattr(lib, n)]
    assert not missing, missing
    # the binding lists the same functions
    import paper_2001_06231_gb300 as bf
    assert sorted(bf.EXPORTED) == names


def test_workload_generators_are_deterministic():
    from paper_2001_06231_gb300 import workloads as wl
    a, b = wl.unicycle3d(n=(40, 30, 16)), wl.unicycle3d(n=(40, 30, 16))
    assert np.array_equal(a.avoid, b.avoid) and np.array_equal(a.target, b.target)
    assert np.array_equal(a.G, b.G)
    c = wl.unicycle3d(n=(40, 30, 16), seed=99)
    assert not np.array_equal(a.avoid, c.avoid)
    d = wl.di2d()
    assert d.target.sum() == 36 and d.ncells == 4096
    f = wl.fire4d(n=(20, 20, 12, 4), target=((0, 400), (0, 400), (-1.0, 1.0), (10, 15)))
    assert f.G.min() < 0 < f.G.max()          # negative costs over fire


def _rank_main(rank, world, port, out):
    import torch.distributed as dist
    os.environ["MASTER_ADDR"] = "127.0.0.1"
    os.environ["MASTER_PORT"] = str(port)
    dist.init_process_group("gloo", rank=rank, world_size=world)
    import sys
    sys.path.insert(0, ROOT)
    import bench
    units = 1000.0 * (rank + 1)          # ranks solve different amounts of work
    seconds = 0.5 + 0.25 * rank          # and take different times
    v, u, t = bench.whole_job(units, seconds, dist, "cpu")
    out.put((rank, v, u, t))
    dist.destroy_process_group()


def test_bench_whole_job_aggregation_over_gloo_ranks():
    import torch.multiprocessing as mp
    with socket.socket() as s:
        s.bind(("127.0.0.1", 0))
        port = s.getsockname()[1]
    ctx = mp.get_context("spawn")
    q = ctx.Queue()
    ps = [ctx.Process(target=_rank_main, args=(r, 2, port, q)) for r in range(2)]
    for p in ps:
        p.start()
    res = sorted(q.get(timeout=120) for _ in ps)
    for p in ps:
        p.join(timeout=60)
        assert p.exitcode == 0
    for rank, v, u, t in res:
        assert u == 3000.0 and t == 0.75 and abs(v - 4000.0) < 1e-9


def test_grid_division_by_multiply_high_is_exact():
    """Cell coordinates divide by the grid extents with a multiply-high and a
    shift (division by invariant integers, Granlund & Montgomery 1994):
    l = ceil(log2 n), m = floor(2^32 (2^l - n) / n) + 1, x // n = (mulhi(m, x) + x) >> l
    for every extent 1..16383 and every cell index below 2^31."""
    import numpy as np
    rng = np.random.default_rng(7)
    xs = np.concatenate([np.arange(0, 70000, dtype=np.uint64),
                         np.array([2**31 - 1, 2**31 - 2, 2**30, 2**31 - 64], dtype=np.uint64),
                         rng.integers(0, 2**31, 20000, dtype=np.uint64)])
    for n in range(1, 16384):
        l = (n - 1).bit_length()
        m = ((1 << 32) * ((1 << l) - n)) // n + 1
        assert 0 < m < (1 << 32)
        q = (((xs * np.uint64(m)) >> np.uint64(32)) + xs) >> np.uint64(l)
        assert np.array_equal(q, xs // np.uint64(n)), n
        # near multiples of n, where an off-by-one would show
        k = np.arange(1, 2**31 // n, max(1, (2**31 // n) // 500), dtype=np.uint64) * np.uint64(n)
        for x in (k - np.uint64(1), k):
            q = (((x * np.uint64(m)) >> np.uint64(32)) + x) >> np.uint64(l)
            assert np.array_equal(q, x // np.uint64(n)), n


def test_box_extent_division_by_multiply_high_is_exact():
    """Gather and marking split a lookup or row index t by box extents d with
    m = ceil(2^31 / d) and t // d = mulhi(2t, m) for 1 <= d <= 255 and
    t < 2^23: checked for every d on every t near a multiple of d (where an
    off-by-one would show) up to 2^23, and on every t below 2^16."""
    import numpy as np
    top = np.uint64(1 << 23)
    small = np.arange(0, 1 << 16, dtype=np.uint64)
    for d in range(1, 256):
        m = np.uint64(((1 << 31) + d - 1) // d)
        k = np.arange(1, (1 << 23) // d + 2, dtype=np.uint64) * np.uint64(d)
        ts = np.concatenate([small, k - np.uint64(1), k, top - np.uint64(1 + np.arange(4, dtype=np.uint64))])
        ts = ts[ts < top]
        q = ((ts << np.uint64(1)) * m) >> np.uint64(32)
        assert np.array_equal(q, ts // np.uint64(d)), d


def test_bench_kernel_hash_ignores_comments_and_profiles_parse(tmp_path, monkeypatch):
    """bench.py matches a committed ncu summary to the relax code it was taken
    on by a hash of the sources without comments: a comment edit keeps the
    hash, a code edit changes it; every summary bench.py names carries the
    keys it reads (kernel hash, relax form)."""
    import sys
    sys.path.insert(0, ROOT)
    import bench
    src = tmp_path / "k.cuh"
    src.write_text("// header\nint f(int x) { return x + 1; }  /* note */\n")
    monkeypatch.setattr(bench, "KERNEL_SOURCES", [str(src)])
    h0 = bench.kernel_hash()
    src.write_text("// another header\n\nint f(int x) {   return x + 1; }\n")
    assert bench.kernel_hash() == h0
    src.write_text("int f(int x) { return x + 2; }\n")
    assert bench.kernel_hash() != h0
    for path in bench.PROFILES.values():
        kv = {k.strip(): v.strip() for k, v in (l.split(":", 1) for l in open(path)
                                                  if ":" in l and not l.startswith("#"))}
        assert re.fullmatch(r"[0-9a-f]{16}", kv["kernel_hash"]), path
        form = dict(x.split("=") for x in kv["relax_form"].split())
        assert {"plane_lists", "cell_masks", "input_frontier"} <= set(form), path


SERVE_CLIENT = r'''
import ctypes, sys, time
import numpy as np
sys.path.insert(0, sys.argv[2])
import paper_2001_06231_gb300 as bf
L = ctypes.CDLL(sys.argv[1])
P = ctypes.c_void_p
L.fake_abstraction.restype = P
L.fake_abstraction.argtypes = [ctypes.c_int64, ctypes.c_int32]
L.bf_serve_open.argtypes = [ctypes.c_size_t, ctypes.c_int32, ctypes.c_int32, P]
L.bf_serve_submit.argtypes = [P, P, P]
L.bf_serve_poll.argtypes = [P, ctypes.c_uint64, ctypes.c_int32, P]
L.bf_serve_close.argtypes = [P]
A, C, U, N = L.fake_abstraction(64, 2), 64, 2, 6
G, tg = np.ones((C, U)), np.ones(C, dtype=np.uint8)
srv = P()
assert L.bf_serve_open(100 * (N - 1) + 50, 64, 8, ctypes.byref(srv)) == 0    # room for N - 1 requests' state

def wave(n=N):
    """n requests: the first is a plain solve, the others wait for it and go to
    the engine together."""
    out, ids = [(np.zeros(C), np.zeros(C, dtype=np.uint8)) for _ in range(n)], []
    for V, mu in out:
        q, rid = bf.Request(), ctypes.c_uint64()
        q.abs, q.G, q.target, q.V, q.mu = A, G.ctypes.data, tg.ctypes.data, V.ctypes.data, mu.ctypes.data
        assert L.bf_serve_submit(srv, ctypes.byref(q), ctypes.byref(rid)) == 0
        ids.append(rid.value)
        if len(ids) == 1:
            time.sleep(0.1)                    # it is running (0.3 s)
    res = [bf.Result() for _ in ids]
    for i, r in zip(ids, res):
        assert L.bf_serve_poll(srv, i, 1, ctypes.byref(r)) == 0
    return [(r.error, r.iters) for r in res], [V[0] for V, _ in out]

TIMEOUT = -4
for code in (TIMEOUT, -3, 0):
    L.fake_fail(1 if code else 0, code)
    before = L.fake_added()
    res, V = wave()
    want = [(0, 7)] + ([(code, 0)] if code else [(0, 7)]) * (N - 1)
    assert res == want, (code, res)
    assert V == [1.0] + [0.0 if code else 1.0] * (N - 1), V
    # every one of them was on the engine, and none is left there
    assert L.fake_added() - before == N - 1 and L.fake_removed() == L.fake_added()
L.bf_serve_close(srv)
print("served")
'''


def test_server_survives_a_step_that_times_out(tmp_path):
    """A wait that runs out on the device fails the requests of that step, with its
    code, and nothing else: their state leaves the engine, their bytes go back
    to the budget, their buffers are not written later, and requests that
    follow are served.  The server's own source over an engine that only
    counts (serve_fake.cu), in a process of its own."""
    import shutil
    import subprocess
    import sys
    from paper_2001_06231_gb300 import _build
    so = str(tmp_path / "libserve_fake.so")
    flags = ["-std=c++17", "-Xcompiler", "-fPIC", "-I", _build.INCLUDE, "-I", _build.CSRC]
    cuda = tmp_path / "cuda_calls.c"
    cuda.write_text("int cudaSetDevice(int d) { return 0; }\n"
                    "int cudaGetDevice(int *d) { *d = 0; return 0; }\n"
                    "int cudaStreamCreateWithFlags(void **s, unsigned f) { *s = 0; return 0; }\n"
                    "int cudaStreamSynchronize(void *s) { return 0; }\n"
                    "int cudaStreamDestroy(void *s) { return 0; }\n")
    src = [os.path.join(_build.CSRC, "serve.cu"), os.path.join(ROOT, "tests", "serve_fake.cu"), str(cuda)]
    subprocess.run([shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"] + _build.ARCH + flags +
                   ["-shared", "-cudart", "shared", "-o", so] + src + ["-lpthread"], check=True)
    r = subprocess.run([sys.executable, "-c", SERVE_CLIENT, so, ROOT], capture_output=True, text=True, timeout=120,
                       env=dict(os.environ, LD_LIBRARY_PATH="/usr/local/cuda/lib64"))
    assert r.returncode == 0 and "served" in r.stdout, r.stdout + r.stderr


def build_word_wait(tmp_path):
    """tests/word_wait.cu as a library: the word engine's waits."""
    import shutil
    import subprocess
    from paper_2001_06231_gb300 import _build
    so = str(tmp_path / "libword_wait.so")
    subprocess.run([shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"] + _build.ARCH +
                   ["-std=c++17", "-Xcompiler", "-fPIC", "-I", _build.INCLUDE, "-I", _build.CSRC, "-shared", "-o", so,
                    os.path.join(ROOT, "tests", "word_wait.cu")], check=True)
    lib = ctypes.CDLL(so)
    lib.spin_limit.restype = ctypes.c_double
    return lib


def test_barrier_waits_outlast_the_work_of_a_block(tmp_path):
    """A block may work between two barriers while the others wait for it: the polls
    of a wait (0.15 us at least) last longer than that at a rate no SM is below
    (1e9 table lookups a second), on the most pairs that fit the memory with the
    most lookups of a list, and on boxes that differ and hold the whole grid."""
    polls = build_word_wait(tmp_path).spin_limit()
    seconds = 0.15e-6 * polls
    # 60 lookups a pair, costs of 8 bytes in 280 GB, all SMs
    assert seconds > 60 * 280e9 / 8 / 152 / 1e9
    # units of 1024 cells, windows of 3 cells (rows that wrap), most pairs of the box form
    for cells, pairs in ((170e3, 0.85e6), (1 << 20, 5.5e6)):
        units = -(-cells // 1024)
        assert seconds > -(-units // 152) * (pairs / units) * (cells / 3) / 1e9
