"""GPU parity of the output-type and operand-layout variants: C in the input's 16-bit type
(BCSR and WCSR) and column-major operands (BCSR: X = B^T in, Y = C^T out, the layout of the
paper's BCSR kernel, Sec. 3.2, and of a sparse linear layer, Sec. 4.4).  Same oracle, same
bound as the default path: a 16-bit C adds at most 2^-9 |C| <= 2^-9 sum|a b| of rounding.
"""
import numpy as np
import pytest

from paper_2604_17834_b200 import workloads as wl

from helpers import assert_close, captured_launches, captured_run, reference, run_gpu, run_gpu_variant, to_device

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def lib():
    from paper_2604_17834_b200 import binding
    return binding


def _bcsr_variant(lib, a, dtype, b, N, c16, col_major, seed=29):
    Bs = wl.dense(seed, a["k"], N, ("uniform", -1.0, 1.0), dtype)
    h = lib.spmm_bcsr_create_csr(a["m"], a["k"], a["row_ptr"], a["col_idx"], a["vals"], dtype, b,
                                 c_type=lib.C_SAME_AS_INPUT if c16 else lib.C_FP32,
                                 layout=lib.COLMAJOR if col_major else lib.ROWMAJOR)
    try:
        C = run_gpu_variant(lib, h, Bs, a["m"], N, dtype, c16=c16, col_major=col_major)
        Cr, S = reference(a, Bs, dtype)
        worst = assert_close(C, Cr, S, dtype, "bcsr b=%d N=%d c16=%d cm=%d" % (b, N, c16, col_major))
        C2 = run_gpu_variant(lib, h, Bs, a["m"], N, dtype, c16=c16, col_major=col_major)
        assert np.array_equal(C, C2)
        return worst
    finally:
        lib.spmm_destroy(h)


@pytest.mark.parametrize("dtype", ["bf16", "fp16"])
@pytest.mark.parametrize("b", [16, 32, 64, 128])
@pytest.mark.parametrize("c16,col_major", [(True, False), (False, True), (True, True)])
def test_bcsr_variants_block_sizes(lib, dtype, b, c16, col_major):
    a = wl.bcsr_sweep(500 + b, m=1024, k=768, b=b, density=0.2, dtype=dtype)
    _bcsr_variant(lib, a, dtype, b, 640, c16, col_major)      # 640 = 512 + 128: several token tiles


@pytest.mark.parametrize("m,k,b,N", [(504, 304, 64, 200), (136, 72, 32, 136), (1000, 1000, 16, 1030),
                                      (264, 640, 128, 333), (64, 64, 64, 128)])
@pytest.mark.parametrize("c16", [False, True])
def test_bcsr_colmajor_ragged_shapes(lib, m, k, b, N, c16):
    """m, k multiples of 8 only; N arbitrary (not a multiple of 128, 64 or even 8); scattered
    entries, empty block-rows."""
    a = wl.random_csr(17 + m, m, k, 0.02, "bf16", empty_rows=tuple(range(min(b, m // 2))))
    _bcsr_variant(lib, a, "bf16", b, N, c16, True)


def test_bcsr_colmajor_matches_rowmajor_bitwise(lib):
    """Same products in the same order: the two layouts differ only in how operands are read and
    results written, so fp32 results are identical."""
    a = wl.bcsr_sweep(77, m=512, k=1024, b=64, density=0.3, dtype="fp16")
    Bs = wl.dense(5, 1024, 512, ("normal", 0.0, 1.0), "fp16")
    h0 = lib.spmm_bcsr_create_csr(512, 1024, a["row_ptr"], a["col_idx"], a["vals"], "fp16", 64)
    h1 = lib.spmm_bcsr_create_csr(512, 1024, a["row_ptr"], a["col_idx"], a["vals"], "fp16", 64, layout=lib.COLMAJOR)
    C0 = run_gpu(lib, h0, Bs, 512, 512)
    C1 = run_gpu_variant(lib, h1, Bs, 512, 512, "fp16", col_major=True)
    lib.spmm_destroy(h0)
    lib.spmm_destroy(h1)
    assert np.array_equal(C0, C1)


def test_bcsr_c16_is_the_rounded_fp32_result(lib):
    a = wl.bcsr_tiny()
    Bs = wl.dense(3, 512, 256, ("uniform", -1.0, 1.0), "bf16")
    h0 = lib.spmm_bcsr_create_csr(512, 512, a["row_ptr"], a["col_idx"], a["vals"], "bf16", 64)
    h1 = lib.spmm_bcsr_create_csr(512, 512, a["row_ptr"], a["col_idx"], a["vals"], "bf16", 64, c_type=lib.C_SAME_AS_INPUT)
    C0 = run_gpu(lib, h0, Bs, 512, 256)
    C1 = run_gpu_variant(lib, h1, Bs, 512, 256, "bf16", c16=True)
    lib.spmm_destroy(h0)
    lib.spmm_destroy(h1)
    import torch
    want = torch.from_numpy(C0).to(torch.bfloat16).float().numpy()     # round to nearest even
    assert np.array_equal(C1, want)


@pytest.mark.parametrize("dtype", ["fp16", "bf16"])
@pytest.mark.parametrize("N", [128, 72, 328])
def test_wcsr_c16(lib, dtype, N):
    a = wl.random_csr(53, 1000, 900, 0.02, dtype, empty_rows=tuple(range(32, 64)))
    Bs = wl.dense(19, 900, N, ("normal", 0.0, 1.0), dtype)
    h = lib.spmm_wcsr_create_csr(1000, 900, a["row_ptr"], a["col_idx"], a["vals"], dtype, 16, split_cols=64,
                                 c_type=lib.C_SAME_AS_INPUT)
    try:
        info = lib.spmm_get_info(h, N)
        assert info["n_split"] > 0 and info["n_empty"] >= 2        # direct, merged and zero-filled rows
        assert info["bytes_c"] == 1000 * N * 2
        C = run_gpu_variant(lib, h, Bs, 1000, N, dtype, c16=True)
        Cr, S = reference(a, Bs, dtype)
        assert_close(C, Cr, S, dtype, "wcsr c16 %s N=%d" % (dtype, N))
        assert np.array_equal(C, run_gpu_variant(lib, h, Bs, 1000, N, dtype, c16=True))
    finally:
        lib.spmm_destroy(h)


@pytest.mark.parametrize("dtype", ["tf32", "fp16", "bf16", "fp8"])
@pytest.mark.parametrize("N", [128, 80, 336])
def test_wcsr_window_height_64(lib, dtype, N):
    """The paper's own window height (Sec. 4.1): 64-row windows, MMA N = 64.  Format arrays
    bit-exact against the format oracle, result against the SpMM oracle, split + empty windows."""
    from oracle import formats as F
    a = wl.random_csr(57, 1000, 900, 0.02, dtype, empty_rows=tuple(range(64, 192)))
    Bs = wl.dense(19, 900, N, ("normal", 0.0, 1.0), dtype)
    h = lib.spmm_wcsr_create_csr(1000, 900, a["row_ptr"], a["col_idx"], a["vals"], dtype, 64, split_cols=128)
    try:
        b_col = 32 // wl.elem_size(dtype)
        f = F.wcsr_from_csr(1000, 900, a["row_ptr"], a["col_idx"], a["vals"], 64, b_col)
        bits = {4: np.uint32, 2: np.uint16, 1: np.uint8}[wl.elem_size(dtype)]
        assert np.array_equal(lib.spmm_export(h, lib.X_WCSR_WINDOW_ROW_PTR, np.int32), f["window_row_ptr"])
        assert np.array_equal(lib.spmm_export(h, lib.X_WCSR_WINDOW_COL_IDX, np.int32), f["window_col_idx"])
        assert np.array_equal(lib.spmm_export(h, lib.X_WCSR_VALUES, wl.storage_np_dtype(dtype)).view(bits),
                              f["values"].view(bits).ravel())
        info = lib.spmm_get_info(h, N)
        assert info["block"] == 64 and info["n_split"] > 0 and info["n_empty"] >= 2
        assert info["stored_values"] == 64 * f["window_col_idx"].shape[0]
        assert info["workspace_bytes"] == info["n_slots"] * 64 * N * 4
        plan = F.split_plan(f["window_row_ptr"], 128)
        assert np.array_equal(lib.spmm_export(h, lib.X_WCSR_TASKS, np.int32).reshape(-1, 4), plan)
        C = run_gpu(lib, h, Bs, 1000, N)
        Cr, S = reference(a, Bs, dtype)
        assert_close(C, Cr, S, dtype, "wcsr wh=64 %s N=%d" % (dtype, N))
        assert np.array_equal(C, run_gpu(lib, h, Bs, 1000, N))
    finally:
        lib.spmm_destroy(h)


def test_wcsr_tf32_same_as_input_is_fp32(lib):
    a = wl.wcsr_irregular(seed=6, m=3000, dtype="tf32")
    Bs = wl.dense(2, a["k"], 128, ("normal", 0.0, 1.0), "tf32")
    h0 = lib.spmm_wcsr_create_csr(a["m"], a["k"], a["row_ptr"], a["col_idx"], a["vals"], "tf32", 16)
    h1 = lib.spmm_wcsr_create_csr(a["m"], a["k"], a["row_ptr"], a["col_idx"], a["vals"], "tf32", 16, c_type=lib.C_SAME_AS_INPUT)
    C0, C1 = run_gpu(lib, h0, Bs, a["m"], 128), run_gpu(lib, h1, Bs, a["m"], 128)
    lib.spmm_destroy(h0)
    lib.spmm_destroy(h1)
    assert np.array_equal(C0, C1)


@pytest.mark.parametrize("b,N", [(16, 1024), (32, 2048), (64, 640), (128, 1032), (64, 4096)])
def test_bcsr_dynamic_schedule_matches_static_bitwise(lib, b, N):
    """Tiles handed out at run time through Cluster Launch Control (more tiles than SMs, so
    running CTAs do take over tiles of CTAs that never start): every tile is computed exactly
    once and exactly as in the static plan, whichever CTA runs it."""
    a = wl.bcsr_sweep(700 + b, m=2048, k=1024, b=b, density=0.15, dtype="fp16")
    Bs = wl.dense(31, a["k"], N, ("uniform", -1.0, 1.0), "fp16")
    args = (a["m"], a["k"], a["row_ptr"], a["col_idx"], a["vals"], "fp16", b)
    h0 = lib.spmm_bcsr_create_csr(*args)
    h1 = lib.spmm_bcsr_create_csr(*args, schedule=lib.SCHED_DYNAMIC)
    try:
        C0 = run_gpu(lib, h0, Bs, a["m"], N)
        C1 = run_gpu(lib, h1, Bs, a["m"], N)
        assert np.array_equal(C0, C1)
        assert np.array_equal(C1, run_gpu(lib, h1, Bs, a["m"], N))
        Cr, S = reference(a, Bs, "fp16")
        assert_close(C1, Cr, S, "fp16", "bcsr dynamic b=%d N=%d" % (b, N))
        # the dynamic plan is one list: every (block-row, token tile) once, slab by slab, longest first
        tp = lib.spmm_export(h1, lib.X_BCSR_TILE_PTR, np.int32)
        tiles = lib.spmm_export(h1, lib.X_BCSR_TILES, np.int32).reshape(-1, 2)
        info = lib.spmm_get_info(h1, N)
        n_tt = -(-N // info["plan_token_tile"])
        assert tp.tolist() == [0, tiles.shape[0]] and tiles.shape[0] == (2048 // b) * n_tt
        from oracle import formats as F
        f = F.bcsr_from_csr(a["m"], a["k"], a["row_ptr"], a["col_idx"], a["vals"], b)
        want_ptr, want_tiles = F.bcsr_tile_schedule(f["block_row_ptr"], n_tt, info["plan_slab_tiles"], 1)
        assert np.array_equal(tiles, want_tiles)
    finally:
        lib.spmm_destroy(h0)
        lib.spmm_destroy(h1)


@pytest.mark.parametrize("b", [32, 64, 128])
@pytest.mark.parametrize("N", [640, 333, 128])
def test_bcsr_fp8_e4m3_colmajor(lib, b, N):
    """8-bit E4M3 inputs (the next step Sec. 5 names), K-major operands: X [N][k] and the stored
    blocks as E4M3, fp32 accumulation and output.  Products of two E4M3 values are exact in
    fp32, so the 16-bit bound applies unchanged."""
    a = wl.bcsr_sweep(900 + b, m=1024, k=768, b=b, density=0.2, dtype="fp8")
    Bs = wl.dense(37, a["k"], N, ("uniform", -1.0, 1.0), "fp8")
    h = lib.spmm_bcsr_create_csr(a["m"], a["k"], a["row_ptr"], a["col_idx"], a["vals"], "fp8", b, layout=lib.COLMAJOR)
    try:
        from oracle import formats as F
        f = F.bcsr_from_csr(a["m"], a["k"], a["row_ptr"], a["col_idx"], a["vals"], b)
        assert np.array_equal(lib.spmm_export(h, lib.X_BCSR_BLOCK_COL_IDX, np.int32), f["block_col_idx"])
        assert np.array_equal(lib.spmm_export(h, lib.X_BCSR_BLOCKS, np.uint8), f["blocks"].ravel())
        C = run_gpu_variant(lib, h, Bs, a["m"], N, "fp8", col_major=True)
        Cr, S = reference(a, Bs, "fp8")
        assert_close(C, Cr, S, "fp8", "bcsr fp8 b=%d N=%d" % (b, N))
        assert np.array_equal(C, run_gpu_variant(lib, h, Bs, a["m"], N, "fp8", col_major=True))
    finally:
        lib.spmm_destroy(h)


@pytest.mark.parametrize("dtype,b,m,k", [("fp16", 64, 1024, 768), ("bf16", 16, 1000, 1000), ("fp16", 32, 130, 70),
                                          ("bf16", 128, 257, 640), ("fp16", 16, 4096, 70000)])
def test_bcsr_built_on_the_gpu_is_bit_exact(lib, dtype, b, m, k):
    """Format construction as GPU kernels from a CSR matrix in device memory: every exported
    array equals the format oracle's, and the handle runs like a host-built one."""
    import torch
    from oracle import formats as F
    a = wl.random_csr(23 + m, m, k, 0.02 if k < 5000 else 0.0005, dtype, empty_rows=tuple(range(min(b, m // 2))))
    rp = torch.from_numpy(a["row_ptr"].astype(np.int64)).cuda()
    ci = torch.from_numpy(a["col_idx"].astype(np.int32)).cuda()
    va = to_device(a["vals"])
    h = lib.spmm_bcsr_create_csr_device(m, k, rp.data_ptr(), ci.data_ptr(), va.data_ptr(), dtype, b)
    try:
        f = F.bcsr_from_csr(m, k, a["row_ptr"], a["col_idx"], a["vals"], b)
        assert np.array_equal(lib.spmm_export(h, lib.X_BCSR_BLOCK_ROW_PTR, np.int32), f["block_row_ptr"])
        assert np.array_equal(lib.spmm_export(h, lib.X_BCSR_BLOCK_COL_IDX, np.int32), f["block_col_idx"])
        assert np.array_equal(lib.spmm_export(h, lib.X_BCSR_BLOCKS, np.uint16), f["blocks"].view(np.uint16).ravel())
        assert np.array_equal(lib.spmm_export(h, lib.X_BCSR_ROW_ORDER, np.int32), F.bcsr_row_order(f["block_row_ptr"]))
        info = lib.spmm_get_info(h, 128)
        assert info["nnz"] == a["col_idx"].shape[0] and info["n_units"] == f["block_col_idx"].shape[0]
        assert info["n_empty"] == int((np.diff(f["block_row_ptr"]) == 0).sum())
        N = 200
        Bs = wl.dense(3, k, N, ("uniform", -1.0, 1.0), dtype)
        C = run_gpu(lib, h, Bs, m, N)
        Cr, S = reference(a, Bs, dtype)
        assert_close(C, Cr, S, dtype, "bcsr built on the GPU b=%d" % b)
    finally:
        lib.spmm_destroy(h)


@pytest.mark.parametrize("dtype,wh,m,k,dens", [("tf32", 16, 1000, 900, 0.02), ("fp16", 16, 333, 517, 0.05),
                                                ("bf16", 64, 1000, 4000, 0.01), ("fp16", 16, 5000, 70000, 0.0005),
                                                ("tf32", 64, 130, 70, 0.2), ("fp8", 16, 1000, 900, 0.02),
                                                ("fp8", 64, 400, 2000, 0.01)])
def test_wcsr_built_on_the_gpu_is_bit_exact(lib, dtype, wh, m, k, dens):
    """Window condensation and value packing as GPU kernels (sort / unique of (window, column)
    keys): every exported array equals the format oracle's, plan and bins included, and the
    handle runs like a host-built one."""
    import torch
    from oracle import formats as F
    a = wl.random_csr(29 + m, m, k, dens, dtype, empty_rows=tuple(range(wh, min(3 * wh, m))))
    rp = torch.from_numpy(a["row_ptr"].astype(np.int64)).cuda()
    ci = torch.from_numpy(a["col_idx"].astype(np.int32)).cuda()
    va = to_device(a["vals"])
    h = lib.spmm_wcsr_create_csr_device(m, k, rp.data_ptr(), ci.data_ptr(), va.data_ptr(), dtype, wh, split_cols=64)
    h0 = lib.spmm_wcsr_create_csr(m, k, a["row_ptr"], a["col_idx"], a["vals"], dtype, wh, split_cols=64)
    try:
        b_col = 32 // wl.elem_size(dtype)
        f = F.wcsr_from_csr(m, k, a["row_ptr"], a["col_idx"], a["vals"], wh, b_col)
        bits = {4: np.uint32, 2: np.uint16, 1: np.uint8}[wl.elem_size(dtype)]
        assert np.array_equal(lib.spmm_export(h, lib.X_WCSR_WINDOW_ROW_PTR, np.int32), f["window_row_ptr"])
        assert np.array_equal(lib.spmm_export(h, lib.X_WCSR_WINDOW_COL_IDX, np.int32), f["window_col_idx"])
        assert np.array_equal(lib.spmm_export(h, lib.X_WCSR_VALUES, wl.storage_np_dtype(dtype)).view(bits),
                              f["values"].view(bits).ravel())
        for which in (lib.X_WCSR_TASKS, lib.X_WCSR_BIN_PTR, lib.X_WCSR_BIN_TASKS):
            assert np.array_equal(lib.spmm_export(h, which, np.int32), lib.spmm_export(h0, which, np.int32))
        # the gather hints (reuse class per four padded columns): same bytes from both builders
        assert np.array_equal(lib.spmm_export(h, lib.X_WCSR_GROUP_CLASS, np.uint8), lib.spmm_export(h0, lib.X_WCSR_GROUP_CLASS, np.uint8))
        i1, i0 = lib.spmm_get_info(h, 128), lib.spmm_get_info(h0, 128)
        assert i1 == i0
        N = 144
        Bs = wl.dense(3, k, N, ("normal", 0.0, 1.0), dtype)
        C = run_gpu(lib, h, Bs, m, N)
        assert np.array_equal(C, run_gpu(lib, h0, Bs, m, N))
        Cr, S = reference(a, Bs, dtype)
        assert_close(C, Cr, S, dtype, "wcsr built on the GPU wh=%d" % wh)
    finally:
        lib.spmm_destroy(h)
        lib.spmm_destroy(h0)


@pytest.mark.parametrize("dtype,wh,k", [("fp16", 16, 30000), ("tf32", 16, 5_000_000), ("bf16", 64, 884_737), ("fp8", 64, 60000)])
def test_wcsr_gpu_builder_by_window_size(lib, dtype, wh, k):
    """Windows at the edges of the builder's kernels (up to 64, 128, 256 entries one warp; from an entry per 256 columns on,
    and above 18,432 entries, a bitmap of 884,736 columns at a time; up to 2048 and 18,432 entries merged), empty ones, rows
    that hold everything; more columns than the first reuse class has room for, with many ties: the same arrays as the
    host builder's."""
    import torch
    rng = np.random.default_rng(wh + k)
    lens = []
    for total, rows in ((64, wh), (65, 2), (128, wh), (129, 1), (256, wh), (257, wh), (2048, wh), (2049, 3), (0, wh), (1, 1), (3456, 5), (3457, wh),
                        (18432, wh), (18433, 2), (25000, wh), (200, 3), (40, wh), (5000, 1)):
        cut = np.sort(rng.integers(0, total + 1, rows - 1))
        part = np.diff(np.concatenate(([0], cut, [total])))
        lens += list(rng.permutation(np.concatenate((part, np.zeros(wh - rows, np.int64)))))
    lens = np.asarray(lens[:-(wh // 2)], np.int64)                     # a ragged last window
    m = lens.size
    rp = np.concatenate(([0], np.cumsum(lens))).astype(np.int64)
    ci = np.concatenate([np.sort(rng.choice(k, n, replace=False)) for n in lens] + [np.zeros(0, np.int64)]).astype(np.int32)
    vals = wl.to_storage(rng.uniform(-1, 1, ci.size), dtype)
    d = [torch.from_numpy(rp).cuda(), torch.from_numpy(ci).cuda(), to_device(vals)]
    h = lib.spmm_wcsr_create_csr_device(m, k, *[x.data_ptr() for x in d], dtype, wh)
    h0 = lib.spmm_wcsr_create_csr(m, k, rp, ci, vals, dtype, wh)
    try:
        bits = {4: np.uint32, 2: np.uint16, 1: np.uint8}[wl.elem_size(dtype)]
        for which, t in ((lib.X_WCSR_WINDOW_ROW_PTR, np.int32), (lib.X_WCSR_WINDOW_COL_IDX, np.int32), (lib.X_WCSR_VALUES, bits),
                         (lib.X_WCSR_GROUP_CLASS, np.uint8), (lib.X_WCSR_TASKS, np.int32), (lib.X_WCSR_BIN_PTR, np.int32), (lib.X_WCSR_BIN_TASKS, np.int32)):
            assert np.array_equal(lib.spmm_export(h, which, t), lib.spmm_export(h0, which, t)), which
        assert lib.spmm_get_info(h, 64) == lib.spmm_get_info(h0, 64)
        N = 16 // wl.elem_size(dtype)
        Bs = wl.dense(3, k, N, ("normal", 0.0, 1.0), dtype)
        assert np.array_equal(run_gpu(lib, h, Bs, m, N), run_gpu(lib, h0, Bs, m, N))
    finally:
        lib.spmm_destroy(h)
        lib.spmm_destroy(h0)


@pytest.mark.parametrize("dtype,b,dens,layout,c16", [
    ("bf16", 64, 0.7, "row", False), ("fp16", 64, 0.7, "row", True), ("bf16", 64, 0.7, "col", True), ("fp16", 64, 0.7, "col", False),
    ("tf32", 64, 0.7, "row", False), ("tf32", 64, 0.7, "col", False), ("fp8", 64, 0.7, "col", False),
    ("fp16", 128, 0.8, "row", False), ("bf16", 128, 0.8, "col", True), ("tf32", 128, 0.8, "row", False), ("fp8", 128, 0.8, "col", False),
    ("fp16", 16, 0.2, "row", False), ("bf16", 32, 0.3, "col", True), ("tf32", 16, 0.2, "col", False), ("tf32", 32, 0.3, "row", False),
    ("bf16", 16, 0.2, "row", True), ("fp8", 32, 0.3, "col", False), ("fp16", 16, 1.0, "row", False), ("bf16", 16, 1.0, "col", True),
    ("tf32", 16, 1.0, "row", False), ("bf16", 32, 1.0, "row", True), ("tf32", 32, 1.0, "row", False), ("tf32", 32, 1.0, "col", False),
    ("fp8", 32, 1.0, "col", False), ("tf32", 16, 0.2, "row", False)])
def test_bcsr_few_long_tiles_run_as_half_tiles(lib, dtype, b, dens, layout, c16):
    """Launches with at most half as many 128-token tiles as CTAs, each of 768 KB and more: two CTAs to a tile (halves of its
    tokens for plain blocks, of the stacked blocks' rows for row groups; the launches' sizes show it).  The same bits as with
    one CTA per tile (a grid too small for two), and the oracle's result; token counts around the halves of a tile, an empty
    block-row, ragged last rows."""
    import torch
    m = 328 if dens < 1 else 264
    need = (768 << 10) // ((128 + (b if dens < 1 else 128)) * b * wl.elem_size(dtype)) + 2       # blocks of the longest tile
    k = (need * b + 8) // 16 * 16
    rng = np.random.default_rng(b)
    nbr, nbc = -(-m // b), -(-k // b)
    mask = rng.random((nbr, nbc)) < dens
    mask[0, :] = True
    if dens < 1:
        mask[1, :] = False
    full = np.kron(mask, np.ones((b, b), bool))[:m, :k]
    rp = np.concatenate(([0], np.cumsum(full.sum(1)))).astype(np.int64)
    ci = np.nonzero(full)[1].astype(np.int32)
    vals = wl.to_storage(rng.uniform(-1, 1, ci.size), dtype)
    a = {"m": m, "k": k, "row_ptr": rp, "col_idx": ci, "vals": vals}
    opt = dict(layout=lib.COLMAJOR if layout == "col" else lib.ROWMAJOR, c_type=lib.C_SAME_AS_INPUT if c16 else lib.C_FP32)
    if dens < 1:
        opt["stack_min_fill"] = -1                          # plain blocks
    assert need * (128 + (b if dens < 1 else 128)) * b * wl.elem_size(dtype) >= 768 << 10
    for N in ((128, 129, 200, 321) if layout == "col" else (72, 96, 128, 136, 256)):
        # (TF32 blocks of 64 and 128: halves that fill the grid)
        fill = {"n_ctas": 2 * nbr * -(-N // 128)} if dtype == "tf32" and b >= 64 else {}
        h = lib.spmm_bcsr_create_csr(m, k, rp, ci, vals, dtype, b, **opt, **fill)
        h1 = lib.spmm_bcsr_create_csr(m, k, rp, ci, vals, dtype, b, n_ctas=3, **opt)
        try:
            Bs = wl.dense(7 + N, k, N, ("uniform", -1.0, 1.0), dtype)
            C, C1 = (run_gpu_variant(lib, x, Bs, m, N, dtype, c16=c16, col_major=layout == "col") for x in (h, h1))
            Cr, S = reference(a, Bs, dtype)
            assert_close(C, Cr, S, dtype, "half tiles b=%d N=%d" % (b, N))
            assert np.array_equal(C, C1), N
            Bd, Cd = to_device(np.ascontiguousarray(Bs.T) if layout == "col" else Bs), torch.empty((m, N), dtype=torch.float32, device="cuda")
            grouped = lib.spmm_export(h, lib.X_BCSR_STACK_TILES, np.int32).size // 2
            assert (grouped > 0) == (dens == 1)
            tiles = grouped or lib.spmm_export(h, lib.X_BCSR_TILES, np.int32).size // 2
            even = N % 32 == 0 and not (b == 64 and N % 128 >= 64)          # (TF32, row-major: whole lines, nearly whole tiles)
            whole = dtype == "tf32" and layout == "row" and b == 16 and dens < 1 and even
            assert captured_launches(lib, h, Bd, Cd, N)[0][0] == (lib.spmm_get_info(h, N)["n_ctas"] if whole else 2 * tiles), (N, tiles)
            assert captured_launches(lib, h1, Bd, Cd, N)[0][0] == 3
            if fill:                                       # and on a grid they leave half empty: by the layout, and by the width
                halves = b == 128 if layout == "col" else not even
                h2 = lib.spmm_bcsr_create_csr(m, k, rp, ci, vals, dtype, b, n_ctas=4 * tiles, **opt)
                try:
                    assert np.array_equal(run_gpu_variant(lib, h2, Bs, m, N, dtype, c16=c16, col_major=layout == "col"), C1), N
                    assert captured_launches(lib, h2, Bd, Cd, N)[0][0] == (2 * tiles if halves else 4 * tiles), N
                finally:
                    lib.spmm_destroy(h2)
        finally:
            lib.spmm_destroy(h)
            lib.spmm_destroy(h1)


@pytest.mark.parametrize("dtype,b,layout,c16", [("tf32", 64, "row", False), ("tf32", 128, "row", False), ("bf16", 64, "row", False), ("fp16", 64, "row", True),
                                                ("fp8", 64, "row", False), ("bf16", 128, "row", True), ("fp8", 128, "row", False), ("fp16", 128, "col", True)])
def test_bcsr_order_of_requests_changes_no_bit(lib, dtype, b, layout, c16):
    """Few block-rows for the grid (a fifth; TF32 blocks of 64: a third): a stage's token tiles are requested before its stored
    blocks (row-major ones, with blocks of 64 in tiles of more than 128 tokens).  Grids on either side of the line, rows of one block to several
    rings full, an empty one, a ragged last token tile: the same bits, and the oracle's result."""
    third = dtype == "tf32" and b == 64
    nbr, nbc = 3, 40
    rng = np.random.default_rng(b)
    mask = np.zeros((nbr, nbc), bool)
    mask[0] = True
    mask[2, rng.permutation(nbc)[:1]] = True
    m, k = nbr * b - 8, nbc * b - 16
    full = np.kron(mask, np.ones((b, b), bool))[:m, :k]
    rp = np.concatenate(([0], np.cumsum(full.sum(1)))).astype(np.int64)
    ci = np.nonzero(full)[1].astype(np.int32)
    vals = wl.to_storage(rng.uniform(-1, 1, ci.size), dtype)
    N = 128 * 95 + 16                                     # two token groups and more to a tile on 16 CTAs
    Bs = wl.dense(11, k, N, ("uniform", -1.0, 1.0), dtype)
    got = []
    for n_ctas in ((9, 10) if third else (15, 16)):
        h = lib.spmm_bcsr_create_csr(m, k, rp, ci, vals, dtype, b, n_ctas=n_ctas, layout=lib.COLMAJOR if layout == "col" else lib.ROWMAJOR,
                                     c_type=lib.C_SAME_AS_INPUT if c16 else lib.C_FP32)
        try:
            got.append(run_gpu_variant(lib, h, Bs, m, N, dtype, c16=c16, col_major=layout == "col"))
            assert lib.spmm_get_info(h, N)["plan_token_tile"] > 128
        finally:
            lib.spmm_destroy(h)
    assert np.array_equal(got[0], got[1])
    cols = np.arange(0, N, 37)
    Cr, S = reference({"m": m, "k": k, "row_ptr": rp, "col_idx": ci, "vals": vals}, Bs, dtype, cols=cols)
    assert_close(got[0][:, cols], Cr, S, dtype, "order of requests b=%d" % b)


def _long_window_rows(rng, kind, wh, k):
    """Columns of the rows of four windows of more than 18,432 entries (the last one ragged, one from which on it is cut where a
    bitmap holds all columns), and a short one between them."""
    rows = []
    for w in range(5):
        n = (18433, 0, 60000, 49153, 49500)[w]
        if w == 1:
            rows += [rng.choice(k, 3, replace=False) for _ in range(wh)]
        elif kind == "spread":
            rows += [rng.choice(k, n // wh + (i < n % wh), replace=False) for i in range(wh)]
        elif kind == "one row":
            rows += [rng.choice(k, n, replace=False)] + [np.zeros(0, np.int64)] * (wh - 1)
        elif kind == "same columns":
            rows += [rng.permutation(rng.choice(k, -(-n // wh), replace=False))] * wh
        elif kind == "two ends":                           # runs of neighbours at the first and the last columns
            rows += [np.concatenate((np.arange(n // wh - 7), k - 1 - rng.choice(k // 2, 9, replace=False))) for _ in range(wh)]
        else:                                              # powers: most entries among few columns
            rows += [np.unique((k * rng.random(2 * n // wh) ** 6).astype(np.int64))[:n // wh + 40] for _ in range(wh)]
    return [np.sort(np.asarray(r, np.int64)) for r in rows[:len(rows) - wh // 2]]


@pytest.mark.parametrize("dtype,wh,k", [("fp16", 16, 70_000), ("tf32", 16, 3_000_000), ("bf16", 64, 70_000), ("fp8", 64, 40_000_000)])
@pytest.mark.parametrize("kind", ["spread", "one row", "same columns", "two ends", "powers"])
def test_wcsr_gpu_builder_long_windows(lib, kind, dtype, wh, k):
    """Windows of more than 18,432 entries that a bitmap does not serve are cut into pieces by column: the same arrays as the host
    builder's."""
    import torch
    rows = _long_window_rows(np.random.default_rng(wh + k), kind, wh, k)
    m = len(rows)
    rp = np.concatenate(([0], np.cumsum([r.size for r in rows]))).astype(np.int64)
    ci = np.concatenate(rows).astype(np.int32)
    vals = wl.to_storage(np.random.default_rng(1).uniform(-1, 1, ci.size), dtype)
    d = [torch.from_numpy(rp).cuda(), torch.from_numpy(ci).cuda(), to_device(vals)]
    h = lib.spmm_wcsr_create_csr_device(m, k, *[x.data_ptr() for x in d], dtype, wh)
    h0 = lib.spmm_wcsr_create_csr(m, k, rp, ci, vals, dtype, wh)
    try:
        bits = {4: np.uint32, 2: np.uint16, 1: np.uint8}[wl.elem_size(dtype)]
        for which, t in ((lib.X_WCSR_WINDOW_ROW_PTR, np.int32), (lib.X_WCSR_WINDOW_COL_IDX, np.int32), (lib.X_WCSR_VALUES, bits),
                         (lib.X_WCSR_GROUP_CLASS, np.uint8), (lib.X_WCSR_TASKS, np.int32)):
            assert np.array_equal(lib.spmm_export(h, which, t), lib.spmm_export(h0, which, t)), which
        assert lib.spmm_get_info(h, 64) == lib.spmm_get_info(h0, 64)
    finally:
        lib.spmm_destroy(h)
        lib.spmm_destroy(h0)


@pytest.mark.parametrize("wh,k", [(16, 100_000), (64, 20_000_000)])
def test_wcsr_gpu_builder_refuses_bad_entries_of_long_windows(lib, wh, k):
    """Columns out of range, doubled, or out of order anywhere in a window that is cut into pieces: the status of the host's check
    (the cuts are looked up in the rows before anything is known of their order)."""
    import torch
    rng = np.random.default_rng(5)
    rows = _long_window_rows(rng, "spread", wh, k)
    m = len(rows)
    rp = np.concatenate(([0], np.cumsum([r.size for r in rows]))).astype(np.int64)
    good = np.concatenate(rows).astype(np.int32)
    zeros = np.zeros(good.size, np.float16)
    first, last = int(rp[2 * wh]), int(rp[2 * wh + 1]) - 1           # a row of the window of 60,000 entries

    def put(at, value):
        c = good.copy()
        c[at] = value
        return c

    def shuffled(a, b):
        c = good.copy()
        c[a:b] = rng.permutation(c[a:b])
        return c

    bad = [put(first, -1), put(last, k), put(last, 2**31 - 1), put(first + 9, good[first + 8]), put((first + last) // 2, 0), put(last, good[first]),
           put(first + 5, k - 1), shuffled(first, last + 1), shuffled(int(rp[2 * wh]), int(rp[3 * wh])), np.zeros_like(good), np.full_like(good, k), good[::-1].copy()]
    for i, ci in enumerate(bad):
        d = [torch.from_numpy(rp).cuda(), torch.from_numpy(np.ascontiguousarray(ci)).cuda(), to_device(zeros)]
        codes = []
        for create, args in ((lib.spmm_wcsr_create_csr_device, [x.data_ptr() for x in d]), (lib.spmm_wcsr_create_csr, [rp, ci, zeros])):
            with pytest.raises(lib.SpmmError) as e:
                create(m, k, *args, "fp16", wh)
            codes.append(e.value.code)
        assert codes[0] == codes[1] and codes[0] in (lib.SPMM_ERR_UNSORTED, lib.SPMM_ERR_OUT_OF_RANGE), (i, codes)


def test_wcsr_gpu_builder_takes_long_windows_in_its_stride(lib):
    """16 million entries in one window (16 full rows) cost no multiple of what they cost in 62,500 windows: 72 ms against 7
    where one CTA condensed a whole window, half a millisecond where it is cut.  Three times as much is allowed; medians of five, in turn."""
    import time
    import torch
    k = 1_000_000
    mats = []
    for m, n in ((16, k), (k, 16)):
        rp = torch.arange(m + 1, dtype=torch.int64, device="cuda") * n
        ci = (torch.arange(n, device="cuda") * (k // n)).to(torch.int32).repeat(m)
        if m > 16:                                         # (a window's rows do not share their columns)
            ci += (torch.arange(m, device="cuda", dtype=torch.int32) % (k // n)).repeat_interleave(n)
        mats.append((m, rp, ci, torch.ones(m * n, dtype=torch.float16, device="cuda")))
    took = [[], []]
    for rep in range(6):
        for i, (m, rp, ci, va) in enumerate(mats):
            torch.cuda.synchronize()
            t0 = time.perf_counter()
            h = lib.spmm_wcsr_create_csr_device(m, k, rp.data_ptr(), ci.data_ptr(), va.data_ptr(), "fp16", 16)
            took[i].append(time.perf_counter() - t0)
            if rep == 0 and i == 0:
                assert lib.spmm_get_info(h, 64)["n_units"] == k
            lib.spmm_destroy(h)
    long_windows, short_windows = (sorted(t[1:])[2] for t in took)
    assert long_windows < 3 * short_windows, (long_windows, short_windows)


@pytest.mark.parametrize("dtype", ["tf32", "fp16", "fp8"])
def test_bcsr_gpu_builder_with_many_block_columns(lib, dtype):
    """More than 196,608 block columns: the builder's bitmap takes more than 48 KB of shared memory."""
    import torch
    from oracle import formats as F
    m, k, b = 70, 7_000_000, 32
    rng = np.random.default_rng(9)
    lens = rng.integers(0, 40, m)
    rp = np.concatenate(([0], np.cumsum(lens))).astype(np.int64)
    ci = np.concatenate([np.sort(rng.choice(k, n, replace=False)) for n in lens]).astype(np.int32)
    va = wl.dense(10, 1, int(rp[-1]), ("normal", 0.0, 1.0), dtype).ravel()
    dev = [to_device(x) for x in (rp, ci, va)]
    h = lib.spmm_bcsr_create_csr_device(m, k, *[d.data_ptr() for d in dev], dtype, b, torch.cuda.current_stream().cuda_stream)
    try:
        f = F.bcsr_from_csr(m, k, rp, ci, va, b)
        assert np.array_equal(lib.spmm_export(h, lib.X_BCSR_BLOCK_COL_IDX, np.int32), f["block_col_idx"])
        bits = {4: np.uint32, 2: np.uint16, 1: np.uint8}[va.itemsize]
        assert np.array_equal(lib.spmm_export(h, lib.X_BCSR_BLOCKS, bits), f["blocks"].view(bits).ravel())
    finally:
        lib.spmm_destroy(h)


def test_bcsr_gpu_builder_rejects_malformed_csr(lib):
    import torch
    vals = to_device(wl.to_storage(np.ones(4), "fp16"))
    cases = [(np.array([0, 2, 4]), np.array([1, 0, 2, 3]), lib.SPMM_ERR_UNSORTED),         # descending columns
             (np.array([0, 2, 4]), np.array([0, 0, 2, 3]), lib.SPMM_ERR_UNSORTED),         # duplicate
             (np.array([0, 2, 4]), np.array([0, 1, 2, 9]), lib.SPMM_ERR_OUT_OF_RANGE),     # column >= k
             (np.array([0, 3, 2]), np.array([0, 1, 2, 3]), lib.SPMM_ERR_INVALID_ARG),      # row_ptr not monotone
             (np.array([1, 2, 4]), np.array([0, 1, 2, 3]), lib.SPMM_ERR_INVALID_ARG)]      # row_ptr[0] != 0
    for rp, ci, code in cases:
        rpd = torch.from_numpy(rp.astype(np.int64)).cuda()
        cid = torch.from_numpy(ci.astype(np.int32)).cuda()
        with pytest.raises(lib.SpmmError) as e:
            lib.spmm_bcsr_create_csr_device(2, 8, rpd.data_ptr(), cid.data_ptr(), vals.data_ptr(), "fp16", 16)
        assert e.value.code == code
        with pytest.raises(lib.SpmmError) as e:
            lib.spmm_wcsr_create_csr_device(2, 8, rpd.data_ptr(), cid.data_ptr(), vals.data_ptr(), "fp16", 16)
        assert e.value.code == code


def test_variant_argument_errors(lib):
    a = wl.bcsr_tiny()
    args = (512, 512, a["row_ptr"], a["col_idx"], a["vals"], "bf16")
    with pytest.raises(lib.SpmmError) as e:
        lib.spmm_wcsr_create_csr(*args, 16, layout=lib.COLMAJOR)            # BCSR only
    assert e.value.code == lib.SPMM_ERR_UNSUPPORTED
    with pytest.raises(lib.SpmmError) as e:
        lib.spmm_bcsr_create_csr(*args, 64, c_type=7)
    assert e.value.code == lib.SPMM_ERR_INVALID_ARG
    with pytest.raises(lib.SpmmError) as e:
        lib.spmm_bcsr_create_csr(*args, 64, schedule=lib.SCHED_DYNAMIC, c_type=lib.C_SAME_AS_INPUT)   # fp32 row-major only
    assert e.value.code == lib.SPMM_ERR_UNSUPPORTED
    with pytest.raises(lib.SpmmError) as e:
        lib.spmm_wcsr_create_csr(*args, 16, schedule=lib.SCHED_DYNAMIC)
    assert e.value.code == lib.SPMM_ERR_UNSUPPORTED
    a8 = wl.bcsr_sweep(5, m=256, k=256, b=32, density=0.3, dtype="fp8")
    for kw in (dict(c_type=lib.C_SAME_AS_INPUT), dict(layout=lib.COLMAJOR, c_type=lib.C_SAME_AS_INPUT),
               dict(schedule=lib.SCHED_DYNAMIC)):                                  # E4M3: fp32 C, static schedule only
        with pytest.raises(lib.SpmmError) as e:
            lib.spmm_bcsr_create_csr(256, 256, a8["row_ptr"], a8["col_idx"], a8["vals"], "fp8", 32, **kw)
        assert e.value.code == lib.SPMM_ERR_UNSUPPORTED
    with pytest.raises(lib.SpmmError) as e:
        lib.spmm_bcsr_create_csr(256, 256, a8["row_ptr"], a8["col_idx"], a8["vals"], "fp8", 16, layout=lib.COLMAJOR)
    assert e.value.code == lib.SPMM_ERR_UNSUPPORTED
    b = wl.random_csr(3, 100, 64, 0.1, "bf16")                             # m = 100: not a multiple of 8
    with pytest.raises(lib.SpmmError) as e:
        lib.spmm_bcsr_create_csr(100, 64, b["row_ptr"], b["col_idx"], b["vals"], "bf16", 32, layout=lib.COLMAJOR)
    assert e.value.code == lib.SPMM_ERR_UNSUPPORTED
    import torch
    h = lib.spmm_bcsr_create_csr(*args, 64, layout=lib.COLMAJOR)
    buf = torch.zeros(1 << 20, dtype=torch.float32, device="cuda")
    with pytest.raises(lib.SpmmError) as e:
        lib.spmm_run(h, buf.data_ptr(), buf.data_ptr(), 64)                 # fewer than 128 tokens
    assert e.value.code == lib.SPMM_ERR_UNSUPPORTED
    lib.spmm_destroy(h)


# --------------------------------------------------------------------------- row groups (stacked 128-row blocks)


def _grouped_matrix(seed, m, k, b, dtype):
    """Block pattern with what the grouping looks for: a band of dense block-rows, block-rows
    that share most of their columns, sparse ones and empty ones, in scattered positions."""
    rng = np.random.default_rng(seed)
    nbr, nbc = -(-m // b), -(-k // b)
    kind = rng.choice(4, size=nbr, p=[0.3, 0.3, 0.25, 0.15])
    shared = rng.random(nbc) < 0.5
    mask = np.zeros((nbr, nbc), dtype=bool)
    for i in range(nbr):
        if kind[i] == 0:
            mask[i] = True
        elif kind[i] == 1:
            mask[i] = shared & (rng.random(nbc) < 0.9)
        elif kind[i] == 2:
            mask[i] = rng.random(nbc) < 0.08
    D = np.zeros((nbr * b, nbc * b), dtype=np.float32)
    for i, j in zip(*np.nonzero(mask)):
        blk = rng.uniform(-1.0, 1.0, size=(b, b)).astype(np.float32)
        blk[rng.random((b, b)) < 0.3] = 0.0                           # blocks are not full either
        D[i * b:(i + 1) * b, j * b:(j + 1) * b] = blk
    D = D[:m, :k]
    rows, cols = np.nonzero(D)
    row_ptr = np.concatenate(([0], np.cumsum(np.bincount(rows, minlength=m)))).astype(np.int64)
    return dict(m=m, k=k, row_ptr=row_ptr, col_idx=cols.astype(np.int32), vals=wl.to_storage(D[rows, cols], dtype))


@pytest.mark.parametrize("b,dtype,m,k,N,c16,cm,fill", [
    (16, "fp16", 1024, 640, 384, False, False, 0),
    (16, "bf16", 1000, 520, 328, True, False, 0),        # ragged m, k and N
    (32, "fp16", 1024, 768, 256, False, True, 0),
    (32, "bf16", 1096, 512, 200, True, True, 0),         # N below one 256-token tile, Y rows of 1096 elements
    (64, "fp16", 2048, 512, 1184, False, False, 0),      # (b = 64 groups are used when they make a tile per CTA: 24 CTAs)
    (64, "bf16", 2048, 512, 1184, True, True, 0),
    (16, "fp16", 512, 512, 128, False, False, 1),        # forced: groups of sparse rows, mostly absent sub-blocks
    (32, "fp16", 640, 384, 512, False, False, 1),
    (64, "fp16", 4096, 256, 608, False, False, 1),
    (32, "fp8", 1024, 768, 328, False, True, 0),         # E4M3: column-major operands, fp32 Y
    (64, "fp8", 2048, 512, 1184, False, True, 0),
    (32, "fp8", 640, 384, 512, False, True, 1),
])
def test_bcsr_row_groups_match_the_oracle(lib, b, dtype, m, k, N, c16, cm, fill):
    from oracle import formats as F
    a = _grouped_matrix(7 * b + N, m, k, b, dtype)
    Bs = wl.dense(300 + b, k, N, ("uniform", -1.0, 1.0), dtype)
    Cr, S = reference(a, Bs, dtype)
    outs = {}
    for mode in (fill, -1):
        h = lib.spmm_bcsr_create_csr(m, k, a["row_ptr"], a["col_idx"], a["vals"], dtype, b,
                                     c_type=lib.C_SAME_AS_INPUT if c16 else lib.C_FP32,
                                     layout=lib.COLMAJOR if cm else lib.ROWMAJOR, stack_min_fill=mode,
                                     n_ctas=24 if b == 64 else 0)
        try:
            info = lib.spmm_get_info(h, N)
            if mode >= 0:
                assert info["n_stacked_rows"] >= 128 // b, "the test matrix must produce row groups"
            else:
                assert info["n_stacked_rows"] == 0
            got = run_gpu_variant(lib, h, Bs, m, N, dtype, c16=c16, col_major=cm)
            assert_close(got, Cr, S, dtype, "b=%d %s groups %s" % (b, dtype, "on" if mode >= 0 else "off"))
            if mode >= 0:
                used = lib.spmm_export(h, lib.X_BCSR_STACK_TILES, np.int32).size > 0
                assert used, "the plan must use the row groups in this case"
                # the exported format stays the canonical one
                f = F.bcsr_from_csr(m, k, a["row_ptr"], a["col_idx"], a["vals"], b)
                assert np.array_equal(lib.spmm_export(h, lib.X_BCSR_BLOCK_COL_IDX, np.int32), f["block_col_idx"])
                again = run_gpu_variant(lib, h, Bs, m, N, dtype, c16=c16, col_major=cm)
                assert np.array_equal(got, again), "run-to-run difference"
            outs[mode] = got
        finally:
            lib.spmm_destroy(h)
    # absent sub-blocks add exact zeros: the grouped and the plain launch agree to the last bit
    assert np.array_equal(outs[fill], outs[-1])


def test_bcsr_row_groups_from_the_gpu_builder(lib):
    """Same handle from a device-resident CSR: the stacked values are built from the blocks the GPU builder wrote."""
    import torch
    b, dtype, m, k, N = 16, "fp16", 768, 512, 256
    a = _grouped_matrix(5, m, k, b, dtype)
    Bs = wl.dense(77, k, N, ("uniform", -1.0, 1.0), dtype)
    Cr, S = reference(a, Bs, dtype)
    rp, ci, v = to_device(a["row_ptr"]), to_device(a["col_idx"]), to_device(a["vals"])
    h = lib.spmm_bcsr_create_csr_device(m, k, rp.data_ptr(), ci.data_ptr(), v.data_ptr(), dtype, b,
                                        stream=torch.cuda.current_stream().cuda_stream)
    try:
        assert lib.spmm_get_info(h, N)["n_stacked_rows"] > 0
        got = run_gpu_variant(lib, h, Bs, m, N, dtype)
        assert_close(got, Cr, S, dtype, "gpu-built, row groups")
    finally:
        lib.spmm_destroy(h)


@pytest.mark.parametrize("b,dtype", [(16, "fp16"), (32, "bf16")])
def test_bcsr_row_groups_find_scattered_families(lib, b, dtype):
    """Block-rows of one family are far apart in the index range and in the length order: the
    groups must still be (mostly) families, i.e. far fewer stacked blocks than R neighbours' union
    would need, and the product must match the oracle."""
    from oracle import formats as F
    m, k, N = 2048, 2048, 384
    a = wl.bcsr_families(55 + b, m=m, k=k, b=b, density=0.15, n_families=8, drop=0.1, dtype=dtype)
    Bs = wl.dense(56 + b, k, N, ("uniform", -1.0, 1.0), dtype)
    Cr, S = reference(a, Bs, dtype)
    f = F.bcsr_from_csr(m, k, a["row_ptr"], a["col_idx"], a["vals"], b)
    rows, ptr, cols = F.bcsr_row_groups(f["block_row_ptr"], f["block_col_idx"], b, {16: 30, 32: 45}[b])
    R = 128 // b
    stored = np.diff(f["block_row_ptr"].astype(np.int64))[rows].sum()
    assert rows.shape[0] >= (m // b) // R * 3 // 4, "most block-rows must end up in a group"
    # (a group of one family is ~90 % full; the leftovers of every family mix; unrelated rows at this
    # density would give ~20 %)
    assert stored >= 0.65 * R * cols.size, "groups must be made of rows of one family"
    h = lib.spmm_bcsr_create_csr(m, k, a["row_ptr"], a["col_idx"], a["vals"], dtype, b)
    try:
        info = lib.spmm_get_info(h, N)
        assert info["n_stacked_rows"] == rows.size and info["n_stack_blocks"] == cols.size
        assert np.array_equal(lib.spmm_export(h, lib.X_BCSR_STACK_ROWS, np.int32).reshape(-1, R), rows)
        got = run_gpu_variant(lib, h, Bs, m, N, dtype)
        assert_close(got, Cr, S, dtype, "families b=%d" % b)
    finally:
        lib.spmm_destroy(h)


@pytest.mark.parametrize("kind", ["bcsr", "bcsr_ksplit", "wcsr"])
def test_prepare_leaves_nothing_to_allocate_for_the_run(lib, kind):
    """After spmm_prepare(h, N) the first spmm_run at that width changes neither the free device
    memory nor the workspace the handle reports (one throw-away handle of the same kind runs first,
    so that the kernel variant's code is already loaded).  Free memory alone would not show an
    allocation that the library's pool serves, so the run is captured first: nothing but kernels."""
    import torch
    dtype, N = "fp16", 512
    st = torch.cuda.current_stream().cuda_stream

    def make():
        if kind == "wcsr":
            a = wl.wcsr_irregular(seed=91, m=6000, dtype=dtype)
            return a, lib.spmm_wcsr_create_csr(a["m"], a["k"], a["row_ptr"], a["col_idx"], a["vals"], dtype, 16, split_cols=64)
        a = wl.bcsr_sweep(93, m=2048, k=2048, b=64, density=0.05, dtype=dtype)
        return a, lib.spmm_bcsr_create_csr(a["m"], a["k"], a["row_ptr"], a["col_idx"], a["vals"], dtype, 64,
                                           k_split=1 if kind == "bcsr_ksplit" else 0)

    a, h0 = make()
    Bs = wl.dense(94, a["k"], N, ("normal", 0.0, 1.0), dtype)
    Bd = to_device(Bs)
    C = torch.empty((a["m"], N), dtype=torch.float32, device="cuda")
    lib.spmm_run(h0, Bd.data_ptr(), C.data_ptr(), N, st)                 # loads the kernels
    torch.cuda.synchronize()
    want = C.cpu().numpy().copy()
    lib.spmm_destroy(h0)
    _, h = make()
    try:
        lib.spmm_prepare(h, N)
        info = lib.spmm_get_info(h, N)
        if kind != "bcsr":
            assert info["workspace_bytes"] > 0, "the case must need a workspace"
        code, nodes = captured_run(lib, h, Bd, C, N)
        assert code == lib.SPMM_OK and nodes and set(nodes) == {"kernel"}
        C.fill_(float("nan"))
        torch.cuda.synchronize()
        free0 = torch.cuda.mem_get_info()[0]
        lib.spmm_run(h, Bd.data_ptr(), C.data_ptr(), N, st)
        free1 = torch.cuda.mem_get_info()[0]
        torch.cuda.synchronize()
        lib.spmm_check(h)
        assert free1 == free0
        assert lib.spmm_get_info(h, N)["workspace_bytes"] == info["workspace_bytes"]
        assert np.array_equal(C.cpu().numpy(), want)
        Cr, S = reference(a, Bs, dtype)
        assert_close(C.cpu().numpy(), Cr, S, dtype, "prepared run, " + kind)
    finally:
        lib.spmm_destroy(h)


# --------------------------------------------------------------------------- the paper's own gather (load/store units)


@pytest.mark.parametrize("dtype,m,k,N,T", [("tf32", 3000, 2500, 128, 0), ("tf32", 1000, 900, 328, 64), ("fp16", 4000, 3000, 256, 0),
                                           ("bf16", 777, 1300, 72, 32), ("fp16", 2048, 2048, 1000, 128)])
def test_wcsr_lsu_gather_matches_the_oracle_and_the_tma_gather(lib, dtype, m, k, N, T):
    """opts.gather = GATHER_LSU: B rows copied by the producer warps with 16-byte cp.async (the
    cooperative 128-bit gather of Sec. 3.2) to the swizzled positions the MMA reads.  Same MMAs in the
    same order as the default TMA gather, so the two results agree to the last bit."""
    a = wl.wcsr_irregular(seed=500 + N, m=m, k=k, dtype=dtype, max_len=700)
    Bs = wl.dense(501, k, N, ("normal", 0.0, 1.0), dtype)
    Cr, S = reference(a, Bs, dtype)
    outs = []
    for gather in (lib.GATHER_LSU, lib.GATHER_TMA):
        h = lib.spmm_wcsr_create_csr(m, k, a["row_ptr"], a["col_idx"], a["vals"], dtype, 16, split_cols=T, gather=gather)
        try:
            info = lib.spmm_get_info(h, N)
            if T:
                assert info["n_split"] > 0, "the case must exercise split windows"
            C = run_gpu(lib, h, Bs, m, N)
            assert_close(C, Cr, S, dtype, "wcsr %s gather=%d" % (dtype, gather))
            assert np.array_equal(C, run_gpu(lib, h, Bs, m, N))
            outs.append(C)
        finally:
            lib.spmm_destroy(h)
    assert np.array_equal(outs[0], outs[1])


def test_wcsr_lsu_gather_argument_errors(lib):
    a = wl.wcsr_irregular(seed=9, m=256, k=256, dtype="fp16")
    for kw, wh in ((dict(gather=lib.GATHER_LSU), 64), (dict(gather=lib.GATHER_LSU, c_type=lib.C_SAME_AS_INPUT), 16)):
        with pytest.raises(lib.SpmmError) as e:
            lib.spmm_wcsr_create_csr(256, 256, a["row_ptr"], a["col_idx"], a["vals"], "fp16", wh, **kw)
        assert e.value.code == lib.SPMM_ERR_UNSUPPORTED
    with pytest.raises(lib.SpmmError) as e:
        lib.spmm_wcsr_create_csr(256, 256, a["row_ptr"], a["col_idx"], a["vals"], "fp16", 16, gather=7)
    assert e.value.code == lib.SPMM_ERR_INVALID_ARG


@pytest.mark.parametrize("dtype,b,m,k,N", [("fp16", 64, 2048, 4096, 1024), ("bf16", 128, 1000, 4096, 1000),
                                           ("tf32", 64, 1536, 2048, 520), ("fp16", 32, 2048, 2048, 768)])
def test_bcsr_k_split_of_long_block_rows(lib, dtype, b, m, k, N):
    """A few full block-rows among short ones: the plan cuts them into parts whose partial tiles a
    second kernel adds in order.  Same oracle bound as the uncut plan, run-to-run identical bits, and
    (parts only regroup the fp32 sum) agreement with the uncut result to fp32 rounding."""
    a = wl.bcsr_sweep(700 + b, m=m, k=k, b=b, density=0.05, dtype=dtype)
    Bs = wl.dense(41, k, N, ("normal", 0.0, 1.0), dtype)
    h1 = lib.spmm_bcsr_create_csr(m, k, a["row_ptr"], a["col_idx"], a["vals"], dtype, b, stack_min_fill=-1, k_split=1)
    h0 = lib.spmm_bcsr_create_csr(m, k, a["row_ptr"], a["col_idx"], a["vals"], dtype, b, stack_min_fill=-1)
    try:
        C1 = run_gpu(lib, h1, Bs, m, N)
        info = lib.spmm_get_info(h1, N)
        assert info["n_slots"] > 0 and info["n_split"] > 0 and info["workspace_bytes"] == info["n_slots"] * b * N * 4
        units = lib.spmm_export(h1, lib.X_BCSR_UNITS, np.int32).reshape(-1, 4)
        assert (units[:, 2] - units[:, 1]).max() <= info["split_cols"]
        C0 = run_gpu(lib, h0, Bs, m, N)
        assert lib.spmm_get_info(h0, N)["n_slots"] == 0
        Cr, S = reference(a, Bs, dtype)
        assert_close(C1, Cr, S, dtype, "bcsr with K-split %s b=%d" % (dtype, b))
        assert_close(C0, Cr, S, dtype, "bcsr without K-split %s b=%d" % (dtype, b))
        assert np.array_equal(C1, run_gpu(lib, h1, Bs, m, N))            # fixed summation order
        assert np.max(np.abs(C1 - C0)) <= 1e-4 * max(1.0, float(S.max()))
    finally:
        lib.spmm_destroy(h0)
        lib.spmm_destroy(h1)


@pytest.mark.parametrize("b,N", [(32, 640), (64, 1024), (128, 400), (64, 128)])
def test_bcsr_fp8_e4m3_rowmajor(lib, b, N):
    """E4M3 inputs with the default row-major operands (B [k][N] as the token-major tensor-core
    operand of 1-byte elements): oracle bound, and the same bits as the column-major path (same
    products, same order)."""
    a = wl.bcsr_sweep(950 + b, m=1024, k=768, b=b, density=0.2, dtype="fp8")
    Bs = wl.dense(43, a["k"], N, ("uniform", -1.0, 1.0), "fp8")
    h0 = lib.spmm_bcsr_create_csr(a["m"], a["k"], a["row_ptr"], a["col_idx"], a["vals"], "fp8", b)
    h1 = lib.spmm_bcsr_create_csr(a["m"], a["k"], a["row_ptr"], a["col_idx"], a["vals"], "fp8", b, layout=lib.COLMAJOR,
                                  stack_min_fill=-1)
    try:
        C0 = run_gpu_variant(lib, h0, Bs, a["m"], N, "fp8")
        Cr, S = reference(a, Bs, "fp8")
        assert_close(C0, Cr, S, "fp8", "bcsr fp8 row-major b=%d N=%d" % (b, N))
        assert np.array_equal(C0, run_gpu_variant(lib, h0, Bs, a["m"], N, "fp8"))
        C1 = run_gpu_variant(lib, h1, Bs, a["m"], N, "fp8", col_major=True)
        assert np.array_equal(C0, C1)
    finally:
        lib.spmm_destroy(h0)
        lib.spmm_destroy(h1)


@pytest.mark.parametrize("kind,opt", [("bcsr", {}), ("bcsr", dict(stack_min_fill=-1)), ("wcsr", {}), ("wcsr", dict(split_cols=64))])
def test_runs_that_feed_one_another_on_a_stream(lib, kind, opt):
    """Launches overlap (each sets itself up while the one before it is running): a run whose dense operand
    is the previous run's result, and whose result overwrites what that run read, sees every value in place.
    A chain of eight unsynchronised products equals the same chain with a synchronise after every run."""
    import torch
    n, N, dtype = 1536, 192, "fp16"
    if kind == "bcsr":                     # 10 % full block-rows: row groups unless switched off
        a = wl.bcsr_sweep(611, m=n, k=n, b=16, density=0.1, dtype=dtype)
        mk, size = lib.spmm_bcsr_create_csr, 16
    else:                                  # one nonzero per window column, or (dense windows) the window kernel
        a = wl.wcsr_irregular(seed=612, m=n, dtype=dtype, max_len=400) if opt == {} else wl.random_csr(613, n, n, 0.3, dtype)
        mk, size = lib.spmm_wcsr_create_csr, 16
    vals = wl.to_storage(wl.widen(a["vals"], dtype) * (1.0 / 16), dtype)
    h = mk(n, n, a["row_ptr"], a["col_idx"], vals, dtype, size, c_type=lib.C_SAME_AS_INPUT, **opt)
    st = torch.cuda.current_stream().cuda_stream
    try:
        x0 = to_device(wl.dense(614, n, N, ("normal", 0.0, 1.0), dtype))
        outs = []
        for sync in (True, False, False):
            x, y = x0.clone(), torch.empty_like(x0)
            for _ in range(8):
                lib.spmm_run(h, x.data_ptr(), y.data_ptr(), N, st)
                if sync:
                    torch.cuda.synchronize()
                x, y = y, x
            torch.cuda.synchronize()
            lib.spmm_check(h)
            outs.append(x.clone())
        assert bool(torch.isfinite(outs[0]).all())
        assert torch.equal(outs[0], outs[1]) and torch.equal(outs[0], outs[2])
    finally:
        lib.spmm_destroy(h)


@pytest.mark.parametrize("b,col_major", [(16, False), (32, False), (32, True)])
@pytest.mark.parametrize("N", [256, 392, 2048])
def test_bcsr_tf32_row_groups_and_narrow_tiles(lib, b, col_major, N):
    """Row groups of TF32 blocks (rows of up to 128 bytes), and of any type with 128-token tiles: few groups and a
    narrow dense operand take those (N = 256, 392), many tokens the 256-token ones.  Same MMAs in the same
    order as without groups: equal to the last bit, and to the oracle within the bound."""
    for dtype in ("tf32", "fp16"):
        a = wl.bcsr_sweep(700 + b, m=2048, k=1536, b=b, density=0.05, dtype=dtype)
        Bs = wl.dense(701, 1536, N, ("uniform", -1.0, 1.0), dtype)
        outs = []
        for fill in (0, -1):
            h = lib.spmm_bcsr_create_csr(2048, 1536, a["row_ptr"], a["col_idx"], a["vals"], dtype, b, stack_min_fill=fill,
                                         layout=lib.COLMAJOR if col_major else lib.ROWMAJOR)
            try:
                assert (lib.spmm_get_info(h, N)["n_stacked_rows"] > 0) == (fill == 0)
                outs.append(run_gpu_variant(lib, h, Bs, 2048, N, dtype, col_major=col_major))
            finally:
                lib.spmm_destroy(h)
        assert np.array_equal(outs[0], outs[1])
        Cr, S = reference(a, Bs, dtype)
        assert_close(outs[0], Cr, S, dtype, "%s row groups b=%d N=%d" % (dtype, b, N))


@pytest.mark.parametrize("b,col_major,N", [(16, False, 256), (16, True, 712), (32, False, 2048), (32, True, 132)])
def test_bcsr_tf32_row_groups_keep_non_finite_operands_to_their_rows(lib, b, col_major, N):
    """Row groups multiply absent sub-blocks as zeros, and 0 x Inf is NaN: with TF32 values an Inf or NaN in B
    must reach the block-rows that store a block in its block column, and no others, as without groups.  Outputs whose
    own blocks meet only finite operands are compared with the oracle on B with the others set to zero."""
    m, k = 1992, 1528
    a = _grouped_matrix(70 + b, m, k, b, "tf32")
    Bs = wl.dense(702, k, N, ("uniform", -1.0, 1.0), "tf32")
    rng = np.random.default_rng(703)
    for value in (np.inf, -np.inf, np.nan):                # scattered entries, one whole row, one whole token
        Bs[rng.integers(0, k, 40), rng.integers(0, N, 40)] = value
    Bs[k - 1] = np.inf
    Bs[:, 5] = np.nan
    outs = []
    for fill in (0, -1):
        h = lib.spmm_bcsr_create_csr(m, k, a["row_ptr"], a["col_idx"], a["vals"], "tf32", b, stack_min_fill=fill,
                                     layout=lib.COLMAJOR if col_major else lib.ROWMAJOR)
        try:
            assert (lib.spmm_get_info(h, N)["n_stacked_rows"] > 0) == (fill == 0)
            outs.append(run_gpu_variant(lib, h, Bs, m, N, "tf32", col_major=col_major))
        finally:
            lib.spmm_destroy(h)
    finite = np.isfinite(Bs)
    nbr, nbc = -(-m // b), -(-k // b)
    stored = np.zeros((nbr, nbc), bool)
    stored[np.repeat(np.arange(m), np.diff(a["row_ptr"])) // b, a["col_idx"] // b] = True
    bad = np.zeros((nbc * b, N), bool)
    bad[:k] = ~finite
    hit = (stored.astype(np.int32) @ bad.reshape(nbc, b, N).any(1).astype(np.int32)) > 0
    hit = np.repeat(hit, b, axis=0)[:m]
    assert hit.any() and not hit.all()
    for C in outs:
        assert np.isfinite(C[~hit]).all()
        assert not np.isfinite(C[hit]).any()               # (a stored block holds a zero times Inf or an Inf of its own)
    Cr, S = reference(a, np.where(finite, Bs, 0.0).astype(np.float32), "tf32")
    for C in outs:
        assert_close(np.where(hit, 0.0, C).astype(np.float32), np.where(hit, 0.0, Cr), S, "tf32", "non-finite B b=%d" % b)


@pytest.mark.parametrize("dtype,wh,c16", [("tf32", 16, False), ("fp16", 16, False), ("bf16", 16, True), ("fp8", 16, False),
                                          ("tf32", 64, False), ("fp16", 64, True), ("bf16", 64, False), ("fp8", 64, False)])
@pytest.mark.parametrize("N,T", [(128, 0), (48, 128), (336, 128), (64, 0)])
def test_wcsr_window_kernel_on_matrices_that_condense(lib, dtype, wh, c16, N, T):
    """Windows that share columns (a third of the matrix is stored) are the window kernel's with every option at its
    default: whole, split, ragged and empty windows, both window heights, one token tile to three, both types of C;
    host- and GPU-built handles."""
    import torch
    m, k = 1003, 1500
    a = wl.random_csr(58 + wh, m, k, 0.3, dtype, empty_rows=tuple(range(64, 192)))
    Bs = wl.dense(20, k, N, ("normal", 0.0, 1.0), dtype)
    Cr, S = reference(a, Bs, dtype)
    dev = [to_device(a[x]) for x in ("row_ptr", "col_idx", "vals")]
    opt = dict(split_cols=T, c_type=lib.C_SAME_AS_INPUT if c16 else lib.C_FP32)
    outs = []
    for h in (lib.spmm_wcsr_create_csr(m, k, a["row_ptr"], a["col_idx"], a["vals"], dtype, wh, **opt),
              lib.spmm_wcsr_create_csr_device(m, k, *[d.data_ptr() for d in dev], dtype, wh, torch.cuda.current_stream().cuda_stream, **opt)):
        try:
            info = lib.spmm_get_info(h, N)
            assert info["nnz"] > 1.75 * info["n_units"] and info["n_empty"] >= 2
            assert (info["n_split"] > 0) or not T
            outs.append(run_gpu_variant(lib, h, Bs, m, N, dtype, c16=c16))
            assert_close(outs[-1], Cr, S, dtype, "window kernel %s wh=%d N=%d T=%d" % (dtype, wh, N, T))
        finally:
            lib.spmm_destroy(h)
    assert np.array_equal(outs[0], outs[1])


def test_runs_of_different_kinds_that_feed_one_another(lib):
    """The chain of the test above across kinds: the grid whose CTAs are cancelled, a plan with a merge kernel, the row
    kernel in several launches of several column tiles, the window kernel with its merge, and two handles in
    turn.  Without a synchronise the chain gives the bits it gives with one after every run."""
    import torch
    n, N = 1024, 2176                      # TF32, row kernel: 2176 columns are nine tiles, two launches
    st = torch.cuda.current_stream().cuda_stream
    scaled = lambda a, dtype, x: wl.to_storage(wl.widen(a["vals"], dtype) * x, dtype)  # noqa: E731
    b1 = wl.bcsr_sweep(621, m=n, k=n, b=64, density=0.1, dtype="fp16")
    b2 = wl.bcsr_sweep(622, m=n, k=n, b=32, density=0.02, dtype="tf32")
    w = wl.wcsr_irregular(seed=623, m=n, dtype="tf32", max_len=700)
    w2 = wl.wcsr_irregular(seed=624, m=n, dtype="tf32", max_len=300)
    hs = [lib.spmm_bcsr_create_csr(n, n, b1["row_ptr"], b1["col_idx"], scaled(b1, "fp16", 1 / 16), "fp16", 64, schedule=lib.SCHED_DYNAMIC),
          lib.spmm_bcsr_create_csr(n, n, b2["row_ptr"], b2["col_idx"], scaled(b2, "tf32", 1 / 8), "tf32", 32, stack_min_fill=-1, k_split=1),
          lib.spmm_wcsr_create_csr(n, n, w["row_ptr"], w["col_idx"], scaled(w, "tf32", 1 / 2), "tf32", 16),
          lib.spmm_wcsr_create_csr(n, n, w["row_ptr"], w["col_idx"], scaled(w, "tf32", 1 / 2), "tf32", 16, split_cols=64),
          lib.spmm_wcsr_create_csr(n, n, w2["row_ptr"], w2["col_idx"], scaled(w2, "tf32", 1 / 2), "tf32", 16)]
    try:
        x0 = to_device(wl.dense(625, n, N, ("normal", 0.0, 1.0), "fp16"))
        bufs = [torch.empty((n, N), dtype=torch.float32, device="cuda") for _ in range(2)]
        outs = []
        for sync in (True, True, False, False):
            x = x0.clone()
            for _ in range(3):
                src = x
                for i, j in enumerate((0, 1, 2, 4, 2, 3, 4)):
                    lib.spmm_run(hs[j], src.data_ptr(), bufs[i % 2].data_ptr(), N, st)
                    src = bufs[i % 2]
                    if sync:
                        torch.cuda.synchronize()
                x = (src / src.abs().max()).to(torch.float16)
                if sync:
                    torch.cuda.synchronize()
            torch.cuda.synchronize()
            for h in hs:
                lib.spmm_check(h)
            outs.append(x)
        assert lib.spmm_get_info(hs[1], N)["n_split"] > 0 and lib.spmm_get_info(hs[3], N)["n_split"] > 0
        assert bool(torch.isfinite(outs[0].float()).all()) and float(outs[0].float().abs().max()) == 1.0
        assert all(torch.equal(outs[0], x) for x in outs[1:])
    finally:
        for h in hs:
            lib.spmm_destroy(h)
