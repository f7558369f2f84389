"""What a handle keeps between calls: the run's workspace, the memory behind it, what stream capture may see of it.

A run inside a stream capture is also the test for "makes no allocating or synchronising call": in the global capture
mode such a call is refused by CUDA, so a run that is captured into kernel nodes only has made none.
"""
import numpy as np
import pytest

from paper_2604_17834_b200 import workloads as wl

from helpers import assert_close, captured_run, reference, run_gpu, to_device

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def lib():
    from paper_2604_17834_b200 import binding
    return binding


def _long_rows(dtype, m=512, k=60000, n=900, seed=3):
    """Rows of n entries whose columns neighbouring rows share almost never: the row kernel's, several parts a row."""
    rng = np.random.default_rng(seed)
    step = k // n
    col = (np.arange(n, dtype=np.int64)[None, :] * step + rng.integers(0, step, (m, 1))).astype(np.int32)
    return {"m": m, "k": k, "row_ptr": np.arange(m + 1, dtype=np.int64) * n, "col_idx": col.ravel(),
            "vals": wl.dense(seed, 1, m * n, ("normal", 0.0, 1.0), dtype).ravel()}


@pytest.mark.parametrize("kind", ["rows", "window"])
def test_a_run_under_capture_never_takes_its_workspace_from_the_graph(lib, kind):
    """Without spmm_prepare a captured run has no workspace: it is refused and launches nothing, and the handle then
    works as if it had not been tried.  After spmm_prepare the same run is captured, and its replay and ordinary
    runs agree.  (The workspace must never be an allocation node: its memory would be the graph's.)"""
    import torch
    dtype, N = "fp16", 128
    a = _long_rows(dtype) if kind == "rows" else wl.random_csr(51, 1000, 900, 0.3, dtype)
    h = lib.spmm_wcsr_create_csr(a["m"], a["k"], a["row_ptr"], a["col_idx"], a["vals"], dtype, 16,
                                 **({} if kind == "rows" else dict(split_cols=64)))
    try:
        Bs = wl.dense(8, a["k"], N, ("normal", 0.0, 1.0), dtype)
        B = to_device(Bs)
        C = torch.zeros((a["m"], N), dtype=torch.float32, device="cuda")
        code, nodes = captured_run(lib, h, B, C, N)
        assert code == lib.SPMM_ERR_ALLOC and nodes is None
        want = run_gpu(lib, h, Bs, a["m"], N)
        Cr, S = reference(a, Bs, dtype)
        assert_close(want, Cr, S, dtype, "after a refused capture")
        code, nodes = captured_run(lib, h, B, C, N, replay=True)
        assert code == lib.SPMM_OK and nodes and set(nodes) == {"kernel"}
        assert np.array_equal(C.cpu().numpy(), want)
        assert np.array_equal(run_gpu(lib, h, Bs, a["m"], N), want)
    finally:
        lib.spmm_destroy(h)


@pytest.mark.parametrize("kind", ["rows", "window", "bcsr", "bcsr_ksplit"])
def test_a_relaxed_capture_allocates_outside_the_graph(lib, kind):
    """cudaStreamCaptureModeRelaxed allows allocations: workspaces and schedules are then ordinary memory that
    outlives the graph."""
    import torch
    dtype, N = "fp16", 96
    if kind.startswith("bcsr"):
        a = wl.bcsr_sweep(97, m=1024, k=1024, b=64, density=0.05, dtype=dtype)
        h = lib.spmm_bcsr_create_csr(1024, 1024, a["row_ptr"], a["col_idx"], a["vals"], dtype, 64, k_split=1 if kind == "bcsr_ksplit" else 0)
    else:
        a = _long_rows(dtype, seed=4) if kind == "rows" else wl.random_csr(52, 1000, 900, 0.3, dtype)
        h = lib.spmm_wcsr_create_csr(a["m"], a["k"], a["row_ptr"], a["col_idx"], a["vals"], dtype, 16,
                                     **({} if kind == "rows" else dict(split_cols=64)))
    try:
        Bs = wl.dense(9, a["k"], N, ("normal", 0.0, 1.0), dtype)
        B = to_device(Bs)
        C = torch.zeros((a["m"], N), dtype=torch.float32, device="cuda")
        code, nodes = captured_run(lib, h, B, C, N, relaxed=True, replay=True)
        assert code == lib.SPMM_OK and set(nodes) == {"kernel"}
        first = C.cpu().numpy().copy()
        assert np.array_equal(run_gpu(lib, h, Bs, a["m"], N), first)
        Cr, S = reference(a, Bs, dtype)
        assert_close(first, Cr, S, dtype, "relaxed capture")
    finally:
        lib.spmm_destroy(h)


@pytest.mark.parametrize("kind", ["bcsr", "wcsr"])
def test_a_handle_is_complete_when_its_creation_returns(lib, kind):
    """Built and run on a stream of its own while the default stream is busy: nothing of the handle may still wait
    behind that work.  A status word cleared late would wipe what the run reported (here a wait that runs out)."""
    import torch
    a = wl.bcsr_sweep(404, m=2048, k=2048, b=64, density=0.3, dtype="fp16") if kind == "bcsr" else wl.wcsr_irregular(seed=405, m=20000, dtype="tf32")
    dtype, size, N = ("fp16", 64, 1024) if kind == "bcsr" else ("tf32", 16, 128)
    mk = lib.spmm_bcsr_create_csr_device if kind == "bcsr" else lib.spmm_wcsr_create_csr_device
    dev = [to_device(a[x]) for x in ("row_ptr", "col_idx", "vals")]
    B = to_device(wl.dense(6, a["k"], N, ("normal", 0.0, 1.0), dtype))
    C = torch.empty((a["m"], N), dtype=torch.float32, device="cuda")
    side = torch.cuda.Stream()
    torch.cuda.synchronize()
    torch.cuda._sleep(500_000_000)                         # a quarter of a second on the default stream
    h = mk(a["m"], a["k"], *[d.data_ptr() for d in dev], dtype, size, side.cuda_stream)
    try:
        lib.spmm_set_wait_limit_ns(0)
        lib.spmm_run(h, B.data_ptr(), C.data_ptr(), N, side.cuda_stream)
        side.synchronize()
        torch.cuda.synchronize()
        with pytest.raises(lib.SpmmError) as e:
            lib.spmm_check(h)
        assert e.value.code == lib.SPMM_ERR_DEV_TIMEOUT
        lib.spmm_check(h)
    finally:
        lib.spmm_set_wait_limit_ns(2_000_000_000)
        lib.spmm_destroy(h)


def test_destroying_a_handle_gives_its_memory_back(lib):
    """What a large handle held is the device's again when spmm_destroy returns, but for the pool's 256 MB."""
    import torch
    m, n = 32768, 1024                                     # 2 M blocks of 16 x 16: 1 GB
    rp = torch.arange(m + 1, device="cuda", dtype=torch.int64) * n
    ci = (torch.arange(n, device="cuda", dtype=torch.int32) * 32).repeat(m)
    va = torch.ones(m * n, dtype=torch.float16, device="cuda")
    torch.cuda.synchronize()
    free0 = torch.cuda.mem_get_info()[0]
    h = lib.spmm_bcsr_create_csr_device(m, m, rp.data_ptr(), ci.data_ptr(), va.data_ptr(), "fp16", 16, stack_min_fill=-1)
    held = free0 - torch.cuda.mem_get_info()[0]
    lib.spmm_destroy(h)
    left = free0 - torch.cuda.mem_get_info()[0]
    assert held > 700 << 20
    assert left <= (256 << 20) + (64 << 20), "%.0f MB still held" % (left / 2 ** 20)       # (64: the pool grows in steps)


def _band_with_long_rows(dtype, m=50000, n_long=40):
    """A band that condenses 1.5 values per padded column -- the row kernel's below 64 (TF32: 128) columns, the window
    kernel's from there on -- and, far from it, rows of 1200 entries, which both kernels cut into parts."""
    rng = np.random.default_rng(3)
    band = np.sort(np.arange(m)[:, None] + rng.permuted(np.tile(np.arange(240), (m, 1)), axis=1)[:, :16], axis=1)
    k = m + 240
    cols = [band[i] for i in range(m)]
    for r in range(n_long):
        cols[r * 16] = np.sort(rng.choice(k, 1200, replace=False))
    lens = np.array([c.size for c in cols])
    rp = np.concatenate(([0], np.cumsum(lens))).astype(np.int64)
    return {"m": m, "k": k, "row_ptr": rp, "col_idx": np.concatenate(cols).astype(np.int32),
            "vals": wl.dense(5, 1, int(rp[-1]), ("normal", 0.0, 1.0), dtype).ravel()}


@pytest.mark.parametrize("matrix,dtype,N,narrower", [
    ("band", "fp16", 128, (128, 72, 64, 56, 32, 8)),       # window kernel at N, row kernel below 64
    ("band", "tf32", 256, (256, 128, 124, 36, 4)),
    ("long", "fp16", 4104, (4104, 4096, 3976, 1024, 8)),   # nine tiles of 29 lanes need less than eight of 31
    ("long", "tf32", 2052, (2052, 1988, 96)),
])
def test_after_prepare_no_narrower_run_allocates(lib, matrix, dtype, N, narrower):
    """spmm_prepare(h, N) covers every N' <= N: both kernels, and widths whose workspace is larger than N's own."""
    import torch
    a = _band_with_long_rows(dtype) if matrix == "band" else _long_rows(dtype, m=300, k=30000)
    h = lib.spmm_wcsr_create_csr(a["m"], a["k"], a["row_ptr"], a["col_idx"], a["vals"], dtype, 16)
    try:
        tdt = torch.float32 if dtype == "tf32" else torch.float16
        B = torch.zeros((a["k"], N), dtype=tdt, device="cuda")
        C = torch.empty((a["m"], N), dtype=torch.float32, device="cuda")
        lib.spmm_prepare(h, N)
        kernels = []
        for n in narrower:
            code, nodes = captured_run(lib, h, B, C, n)
            assert code == lib.SPMM_OK and nodes and set(nodes) == {"kernel"}, "N' = %d: %s %s" % (n, code, nodes)
            kernels.append(len(nodes))
        if (matrix, dtype) == ("band", "fp16"):            # windows are cut: the window kernel is two launches, the row kernel one
            assert kernels == [2, 2, 2, 1, 1, 1]
    finally:
        lib.spmm_destroy(h)


@pytest.mark.parametrize("kind", ["bcsr", "bcsr_ksplit", "wcsr"])
def test_a_refused_run_leaves_nothing_behind(lib, kind):
    """A width that was not prepared is refused under capture, whatever the handle holds already; the prepared width,
    new handles and new widths then work (no error of the refused call is found by a later one)."""
    import torch
    dtype = "fp16"

    def make():
        if kind == "wcsr":
            a = _long_rows(dtype, seed=6)
            return a, lib.spmm_wcsr_create_csr(a["m"], a["k"], a["row_ptr"], a["col_idx"], a["vals"], dtype, 16)
        a = wl.bcsr_sweep(93, m=1024, k=1024, b=64, density=0.05, dtype=dtype)
        return a, lib.spmm_bcsr_create_csr(1024, 1024, a["row_ptr"], a["col_idx"], a["vals"], dtype, 64, k_split=1 if kind == "bcsr_ksplit" else 0)

    def product(h, a, N):
        Bs = wl.dense(95, a["k"], N, ("normal", 0.0, 1.0), dtype)
        C = run_gpu(lib, h, Bs, a["m"], N)
        assert_close(C, *reference(a, Bs, dtype), dtype, "%s N=%d" % (kind, N))
        return C

    a, h = make()
    try:
        first = product(h, a, 64)
        B = torch.zeros((a["k"], 512), dtype=torch.float16, device="cuda")
        C = torch.empty((a["m"], 512), dtype=torch.float32, device="cuda")
        code, nodes = captured_run(lib, h, B, C, 512)
        assert code in (lib.SPMM_ERR_ALLOC, lib.SPMM_ERR_CUDA) and nodes is None
        a2, h2 = make()
        try:
            code, _ = captured_run(lib, h2, B, C, 512)          # a handle that holds nothing yet
            assert code in (lib.SPMM_ERR_ALLOC, lib.SPMM_ERR_CUDA)
            assert np.array_equal(product(h2, a2, 64), first)
        finally:
            lib.spmm_destroy(h2)
        assert np.array_equal(product(h, a, 64), first)
        product(h, a, 512)
    finally:
        lib.spmm_destroy(h)


_SCARCE = r"""
import sys
import numpy as np, torch
sys.path[:0] = [".", "tests"]
from paper_2604_17834_b200 import binding as lib, workloads as wl
from helpers import assert_close, reference
left = int(sys.argv[1])
m = k = 500000
n, N, dtype = 16, 8, "fp16"
step = k // n
start = np.random.default_rng(1).integers(0, step, (m, 1))
ci = (np.arange(n, dtype=np.int64)[None, :] * step + start).astype(np.int32).ravel()
rp = np.arange(m + 1, dtype=np.int64) * n
va = wl.dense(2, 1, m * n, ("normal", 0.0, 1.0), dtype).ravel()
Bs = wl.dense(3, k, N, ("normal", 0.0, 1.0), dtype)
B, C = torch.from_numpy(Bs).cuda(), torch.full((m, N), float("nan"), device="cuda")
def make(rp, ci, va, m, **opt):
    return lib.spmm_wcsr_create_csr(m, k, rp, ci, va, dtype, 16, **opt)
st = torch.cuda.current_stream().cuda_stream
small = (rp[:65], ci[:1024], va[:1024])
for opt in ({}, dict(gather=lib.GATHER_TMA)):                      # loads the kernels
    h = make(*small, 64, **opt)
    lib.spmm_run(h, B.data_ptr(), C.data_ptr(), N, st)
    torch.cuda.synchronize()
    lib.spmm_destroy(h)
free = torch.cuda.mem_get_info()[0]
if left < 0:
    h = make(rp, ci, va, m, gather=lib.GATHER_TMA)
    print("window", free - torch.cuda.mem_get_info()[0])
    h2 = make(rp, ci, va, m)
    print("both", free - torch.cuda.mem_get_info()[0])
else:
    hog = torch.empty(free - left, dtype=torch.uint8, device="cuda")
    h = make(rp, ci, va, m)
    lib.spmm_run(h, B.data_ptr(), C.data_ptr(), N, st)
    torch.cuda.synchronize()
    lib.spmm_check(h)
    Cr, S = reference(dict(row_ptr=rp, col_idx=ci, vals=va), Bs, dtype)
    assert_close(C.cpu().numpy(), Cr, S, dtype, "without a row stream")
    print("ran")
"""


def test_a_handle_does_without_its_row_stream_where_memory_is_short(lib):
    """The private copy of the nonzeros only makes runs faster: where the format's own arrays fit and it does not,
    the handle is created all the same and the window kernel serves it.  (In processes of their own, whose memory
    is filled up to the window handle's need and a little more.)"""
    import os
    import subprocess
    import sys
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

    def child(left):
        r = subprocess.run([sys.executable, "-c", _SCARCE, str(left)], cwd=root, capture_output=True, text=True, timeout=300)
        assert r.returncode == 0, r.stdout[-500:] + r.stderr[-1500:]
        return r.stdout.split()

    said = child(-1)
    window, both = int(said[1]), int(said[3])
    assert both > 2 * window + (64 << 20)
    # ... and holds every nonzero once: 6 bytes an entry, at most 3 of padding per 16 entries, 16 bytes a task (the pool
    # grows by 32 MB at a time for each of the larger arrays)
    entries = 500000 * 17
    assert both - 2 * window <= entries * (6 * (1 + 3 / 16) + 1) + (96 << 20)
    assert child(window + (56 << 20)) == ["ran"]


@pytest.mark.parametrize("matrix,opt", [("long", {}), ("long", dict(gather=2)), ("band", {}), ("short", {}), ("short", dict(split_cols=64))])
def test_workspace_bytes_is_what_a_run_allocates(lib, matrix, opt):
    """spmm_get_info tells the workspace of the kernel that runs at N: a new handle's first run takes memory
    (and is refused under capture) exactly where that is not zero."""
    import torch
    dtype = "fp16"
    a = {"long": lambda: _long_rows(dtype, m=300, k=30000), "band": lambda: _band_with_long_rows(dtype, m=20000, n_long=0),
         "short": lambda: wl.wcsr_irregular(seed=96, m=3000, dtype=dtype, max_len=200)}[matrix]()
    for N in (32, 128, 512):
        h = lib.spmm_wcsr_create_csr(a["m"], a["k"], a["row_ptr"], a["col_idx"], a["vals"], dtype, 16, **opt)
        try:
            B = torch.zeros((a["k"], N), dtype=torch.float16, device="cuda")
            C = torch.empty((a["m"], N), dtype=torch.float32, device="cuda")
            need = lib.spmm_get_info(h, N)["workspace_bytes"]
            code, _ = captured_run(lib, h, B, C, N)
            assert code == (lib.SPMM_ERR_ALLOC if need else lib.SPMM_OK), (N, need)
            assert lib.spmm_get_info(h, 0)["workspace_bytes"] == 0
        finally:
            lib.spmm_destroy(h)


def test_waits_do_not_count_the_launch_before(lib):
    """One block-row of 2048 blocks: a launch of a millisecond on a few SMs.  The next one, of a matrix of 8 blocks, starts
    beside it on the others and waits for its end; that time is no part of its bounded waits, whose limit is shorter."""
    import torch
    m, N = 128, 128
    hs, ks = [], (262144, 1024)
    try:
        for k in ks:
            rp = torch.arange(m + 1, dtype=torch.int64, device="cuda") * k
            ci = torch.arange(k, dtype=torch.int32, device="cuda").repeat(m)
            va = torch.ones(m * k, dtype=torch.bfloat16, device="cuda")
            hs.append(lib.spmm_bcsr_create_csr_device(m, k, rp.data_ptr(), ci.data_ptr(), va.data_ptr(), "bf16", 128))
        B = torch.ones((ks[0], N), dtype=torch.bfloat16, device="cuda")
        C = torch.zeros((2, m, N), dtype=torch.float32, device="cuda")
        st = torch.cuda.current_stream().cuda_stream
        ev = [torch.cuda.Event(enable_timing=True) for _ in range(2)]
        for limit in (2_000_000_000, 0, 300_000, 300_000):         # (the first pass: kernels loaded, plans made; the second: the long one alone)
            for i in range(2 if limit else 1):
                if not limit:
                    ev[0].record()
                lib.spmm_set_wait_limit_ns(limit if i else 2_000_000_000)
                lib.spmm_run(hs[i], B.data_ptr(), C[i].data_ptr(), N, st)
                if not limit:
                    ev[1].record()
        torch.cuda.synchronize()
        assert ev[0].elapsed_time(ev[1]) > 0.6                     # (twice the limit)
        for i in range(2):
            lib.spmm_check(hs[i])
            assert bool(torch.all(C[i] == ks[i]))
    finally:
        lib.spmm_set_wait_limit_ns(2_000_000_000)
        for h in hs:
            lib.spmm_destroy(h)


@pytest.mark.parametrize("kind", ["bcsr", "wcsr"])
def test_handles_built_by_several_threads_for_different_widths(lib, kind):
    """The GPU builders' shared memory grows with the matrix's width: threads that build for a narrow and for a wide one at the
    same time do not take each other's allowance away."""
    import threading
    import torch
    m, n = 16, 256                                         # (one entry per 256 columns: WCSR's bitmap kernel)
    widths = (500_000, 800_000) if kind == "wcsr" else (4_000_000, 12_000_000)
    mats = []
    for k in widths:
        rp = torch.arange(m + 1, dtype=torch.int64, device="cuda") * n
        ci = (torch.arange(n, device="cuda") * (k // n)).to(torch.int32).repeat(m)
        mats.append((k, rp, ci, torch.ones(m * n, dtype=torch.float16, device="cuda")))
    torch.cuda.synchronize()
    create = lib.spmm_bcsr_create_csr_device if kind == "bcsr" else lib.spmm_wcsr_create_csr_device
    failed = []

    def build(i):
        k, rp, ci, va = mats[i % 2]
        stream = torch.cuda.Stream()
        try:
            for _ in range(200):
                h = create(m, k, rp.data_ptr(), ci.data_ptr(), va.data_ptr(), "fp16", 16, stream.cuda_stream)
                units = lib.spmm_get_info(h, 64)["n_units"]
                lib.spmm_destroy(h)
                assert units == n
        except Exception as e:                             # for the main thread to raise
            failed.append(e)

    threads = [threading.Thread(target=build, args=(i,)) for i in range(8)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not failed, failed[0]
