"""Host code of the library against a fake CUDA runtime (no GPU).

fake_cudart.cpp holds device memory in host memory, carries copies out only when
their stream is waited for, and runs no kernel; it refuses chosen allocations and
counts memory given back while work on it is still queued.  The library is
compiled a second time, unoptimised, against it.
"""
import ctypes
import os
import shutil
import subprocess

import numpy as np
import pytest

import paper_1205_3809_gb300 as gc

HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    out = str(tmp_path_factory.mktemp("fake") / "libgc_fake.so")
    if shutil.which("nvcc") is None:
        pytest.skip("no nvcc here")
    subprocess.run(["nvcc", "-gencode", "arch=compute_103a,code=compute_103a", "-O0", "-Xcicc", "-O0", "-std=c++17",
                    "-Xcompiler", "-fPIC", "-shared", "-cudart", "none", "-Xlinker", "-Bsymbolic", "--threads", "2", "-I", gc._INCLUDE,
                    "-o", out, os.path.join(gc._CSRC, "gc.cu"), os.path.join(gc._CSRC, "gc_mlp.cu"), os.path.join(HERE, "fake_cudart.cpp")], check=True)
    h = ctypes.CDLL(out)
    vp, i32 = ctypes.c_void_p, ctypes.c_int32
    h.gc_batch_create.argtypes = [vp, vp, vp, vp, i32, vp, vp, vp, vp, ctypes.POINTER(gc.Options), vp,
                                  ctypes.POINTER(vp)]
    h.gc_batch_destroy.argtypes = [vp]
    h.gc_color_ex.argtypes = [vp, vp, i32, vp, vp, vp, vp, vp, ctypes.POINTER(gc.Options), vp, i32]
    h.gc_validate_csr.argtypes = [vp, vp, i32, vp]
    h.gc_last_phase_ms.argtypes = [vp, i32]
    h.gc_batch_mode.argtypes = [vp]
    h.gc_color_host.argtypes = [vp, vp, i32, vp, vp, vp, vp, vp, vp]
    h.fake_result.argtypes = [ctypes.c_char_p, ctypes.c_int, ctypes.c_size_t, ctypes.c_uint32]
    h.gc_batch_status.argtypes = [vp, vp, vp, vp]
    h.gc_batch_round_stats.argtypes = [vp, vp, vp, i32, vp, vp]
    h.gc_batch_workspace_bytes.argtypes = [vp]
    h.gc_batch_workspace_bytes.restype = ctypes.c_size_t
    h.fake_bytes_live.restype = ctypes.c_size_t
    h.fake_bytes_taken.restype = ctypes.c_size_t
    h.fake_pool_bytes.restype = ctypes.c_size_t
    h.fake_capacity.argtypes = [ctypes.c_size_t]
    h.fake_grid.argtypes = [ctypes.c_char_p]
    h.fake_kernel_cost.argtypes = [ctypes.c_char_p, ctypes.c_double]
    yield h
    h.gc_release()


def _p(a):
    return ctypes.c_void_p(a.ctypes.data)


class EdgelessBatch:
    """A plan of graphs without entries: sizes alone decide how a batch is split."""

    def __init__(self, lib, sizes, keys=False, **options):
        self.lib = lib
        n, g = int(sum(sizes)), len(sizes)
        self.voff = np.concatenate([[0], np.cumsum(sizes)]).astype(np.int64)
        self.eoff = np.zeros(g + 1, np.int64)
        self.rowptr = np.zeros(n + g, np.int32)
        self.colors, self.nc, self.rd = (np.zeros(max(k, 1), np.int32) for k in (n, g, g))
        self.prio = np.zeros(max(n, 1), np.uint32) if keys else None
        self.plan = ctypes.c_void_p()
        self.rc = lib.gc_batch_create(_p(self.rowptr), None, _p(self.voff), _p(self.eoff), g,
                                      _p(self.prio) if keys else None, _p(self.colors), _p(self.nc), _p(self.rd),
                                      ctypes.byref(gc._options(options)), None, ctypes.byref(self.plan))

    def close(self):
        self.lib.gc_batch_destroy(self.plan)


SPLIT = [400000] + [500] * 199   # the first graph alone outlasts the others' share: colored apart


def test_plan_of_a_split_batch_at_every_refused_allocation(lib):
    """An allocation refused at any point gives a plan without the split or
    GC_ERR_OOM, gives back no memory that queued work still uses, and leaves none
    behind."""
    b = EdgelessBatch(lib, SPLIT, keys=True)
    assert b.rc == gc.GC_OK
    whole = lib.gc_batch_workspace_bytes(b.plan)
    b.close()
    b = EdgelessBatch(lib, SPLIT, keys=True, batch_mode=2)
    unsplit = lib.gc_batch_workspace_bytes(b.plan)
    b.close()
    assert whole > unsplit and lib.fake_misuse() == 0
    start = lib.fake_bytes_live()
    seen = []
    for which in range(1, 20):
        lib.fake_refuse_allocation(which)
        b = EdgelessBatch(lib, SPLIT, keys=True)
        lib.fake_refuse_allocation(0)
        assert b.rc in (gc.GC_OK, gc.GC_ERR_OOM)
        seen.append((b.rc, lib.gc_batch_workspace_bytes(b.plan) if b.rc == gc.GC_OK else 0))
        if b.rc == gc.GC_OK:
            b.close()
        assert lib.fake_misuse() == 0, f"refused allocation {which}: memory given back in use"
        assert lib.fake_bytes_live() == start
        if seen[-1] == (gc.GC_OK, whole):
            break
    assert seen[-1] == (gc.GC_OK, whole)                 # past the last allocation
    assert (gc.GC_ERR_OOM, 0) in seen and (gc.GC_OK, unsplit) in seen


@pytest.mark.parametrize("options", [{}, {"batch_mode": 1}, {"batch_mode": 2}], ids=["split", "shared-grid", "block-per-graph"])
def test_status_of_a_plan_that_has_not_run(lib, options):
    """The plan's memory may hold what an earlier plan left there: until a run
    writes them, the status and the per-round record must not come from it."""
    b = EdgelessBatch(lib, SPLIT, **options)
    assert b.rc == gc.GC_OK
    rounds, colors, bits = (ctypes.c_int32(-1) for _ in range(3))
    assert lib.gc_batch_status(b.plan, None, ctypes.byref(rounds), ctypes.byref(colors)) == gc.GC_OK
    assert (rounds.value, colors.value) == (0, 0)
    sizes, volumes = np.full(8, -1, np.int32), np.full(8, -1, np.int64)
    assert lib.gc_batch_round_stats(b.plan, _p(sizes), _p(volumes), 8, ctypes.byref(bits), None) == 0
    b.close()


def _phases(lib, **options):
    n = 1000
    rowptr, colors = np.zeros(n + 1, np.int32), np.zeros(n, np.int32)
    nc, rd = ctypes.c_int32(), ctypes.c_int32()
    rc = lib.gc_color_ex(_p(rowptr), None, n, None, _p(colors), ctypes.byref(nc), ctypes.byref(rd), None,
                         ctypes.byref(gc._options(dict(options, telemetry=1))), None, 0)
    assert rc == gc.GC_OK
    ms = (ctypes.c_float * 4)()
    assert lib.gc_last_phase_ms(ms, 4) == 4
    return list(ms)


def test_phase_times_leave_the_entry_checks_out(lib):
    """One unit of time a kernel, a thousand for the entry checks: setup scan,
    round 1, later rounds and their sum, with and without the checks."""
    lib.fake_kernel_cost(b"validate_kernel", 1000.0)
    try:
        assert _phases(lib) == [1.0, 1.0, 1.0, 3.0]
        assert _phases(lib, validate=1) == [1.0, 1.0, 1.0, 3.0]
    finally:
        lib.fake_kernel_cost(b"validate_kernel", 1.0)


def test_memory_kept_from_plans_does_not_refuse_a_later_call(lib):
    """The pool keeps freed plan memory; a workspace that only fits without it is
    still allocated."""
    lib.gc_release()
    b = EdgelessBatch(lib, [3000000])
    assert b.rc == gc.GC_OK
    b.close()
    kept = lib.fake_bytes_taken() - lib.fake_bytes_live()
    assert 100 << 20 < kept <= 256 << 20
    n = 1000000                                          # about 36 bytes a vertex
    rowptr, colors = np.zeros(n + 1, np.int32), np.zeros(n, np.int32)
    nc, rd = ctypes.c_int32(), ctypes.c_int32()
    lib.fake_capacity(lib.fake_bytes_taken() + (16 << 20))
    try:
        assert lib.gc_color_ex(_p(rowptr), None, n, None, _p(colors), ctypes.byref(nc), ctypes.byref(rd), None, None,
                               None, 0) == gc.GC_OK
    finally:
        lib.fake_capacity(ctypes.c_size_t(-1).value)
        lib.gc_release()


def test_large_plans_do_not_go_through_the_pool(lib):
    """Memory that the pool would unmap when it is freed comes from cudaMalloc."""
    lib.gc_release()
    for n, pooled in ((3000000, True), (10000000, False)):
        b = EdgelessBatch(lib, [n])
        assert b.rc == gc.GC_OK
        ws = lib.gc_batch_workspace_bytes(b.plan)
        assert (ws <= 384 << 20) == pooled
        assert (lib.fake_pool_bytes() >= ws) == pooled and lib.fake_bytes_live() >= ws
        b.close()
        assert lib.fake_pool_bytes() == 0 and lib.fake_misuse() == 0
    lib.gc_release()


@pytest.mark.parametrize("n", [1, 9, 1500, 4000, 9728, 10000, 3000000])
def test_entry_checks_have_a_warp_for_every_row_of_a_small_graph(lib, n):
    """Blocks of eight warps, a warp a row as far as the GPU holds them (152 SMs, eight blocks each)."""
    rowptr = np.zeros(n + 1, np.int32)
    assert lib.gc_validate_csr(_p(rowptr), None, n, None) == gc.GC_OK
    assert lib.fake_grid(b"validate_kernel") == min((n + 7) // 8, 152 * 8)


STATS_ARG, STATS_CAP, STATS_OVER = 5, 16, 28   # stats_kernel's record: cap[0..1], over2, over8, over16 (bytes)


@pytest.mark.parametrize("sizes, skewed, keyed, mode", [
    ([48000], False, False, 2), ([50000], False, False, 1),   # one graph: a block up to about 49,200
    ([60000] * 2, False, False, 2), ([65000] * 2, False, False, 1), ([85000] * 8, False, False, 2),
    ([90000] * 32, False, False, 2), ([150000] * 32, False, False, 2),
    ([150000] * 8, False, False, 1), ([150000] * 64, False, False, 2),
    ([62500] * 4, False, False, 2), ([62500] * 4, True, False, 1), ([62500] * 64, True, False, 2),
    ([19000], True, False, 2), ([21000], True, False, 1), ([128000] * 16, True, False, 1), ([128000] * 64, True, False, 2),
    ([32000], False, True, 2), ([34000], False, True, 1),     # keys: up to about 32,700
    ([67000] * 4, False, True, 1), ([67000] * 32, False, True, 2), ([147000] * 32, False, True, 1),
    ([30000] * 4, True, True, 1), ([12000], True, True, 2),
])
def test_split_of_a_batch_of_equal_graphs(lib, sizes, skewed, keyed, mode):
    """Where the library's choice between a block a graph and one union changes, for even graphs, for
    batches with one row in 200 longer than 121, and with keys (measured on both sides; the graphs
    here have no entries, so their sizes stand for vertices and entries together)."""
    lib.fake_no_results()
    try:
        if skewed:
            for off in (STATS_CAP, STATS_CAP + 4, STATS_OVER, STATS_OVER + 4, STATS_OVER + 8):
                lib.fake_result(b"stats_kernel", STATS_ARG, off, sum(sizes) // 200 + 1)
        b = EdgelessBatch(lib, sizes, keys=keyed)
        assert b.rc == gc.GC_OK
        assert lib.gc_batch_mode(b.plan) == mode
        b.close()
    finally:
        lib.fake_no_results()
        lib.gc_release()


def test_rejected_host_graph_leaves_no_copy_of_it_queued(lib):
    """After gc_color_host returns, with whatever status, the caller may free its arrays."""
    n, nnz = 64, 3 << 20                                 # three chunks
    rowptr = np.linspace(0, nnz, n + 1).astype(np.int32)
    colidx, colors = np.zeros(nnz, np.int32), np.zeros(n, np.int32)
    nc, rd = ctypes.c_int32(), ctypes.c_int32()
    lib.fake_no_results()
    try:
        lib.fake_result(b"stats_kernel", STATS_ARG, 4, 1)   # the setup scan finds the row starts unusable
        assert lib.gc_color_host(_p(rowptr), _p(colidx), n, None, _p(colors), ctypes.byref(nc), ctypes.byref(rd),
                                 None, None) == gc.GC_ERR_BAD_GRAPH
        assert lib.fake_pending() == 0
    finally:
        lib.fake_no_results()
        lib.gc_release()
