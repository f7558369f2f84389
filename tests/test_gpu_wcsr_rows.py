"""WCSR row kernel (windows that condense almost nothing): row lengths at the edges of its tasks, parts and
length classes, every task size, both vector widths, several column tiles, ragged tails, against the fp64 oracle.
Bound: that of the other WCSR tests; products are exact or rounded once, sums are fp32, a 16-bit C adds 2^-9.
"""
import numpy as np
import pytest

from paper_2604_17834_b200 import workloads as wl

from helpers import CANARY, GUARD, assert_close, captured_launches, captured_run, check_guards, reference, run_gpu_variant, to_device

pytestmark = pytest.mark.gpu

EDGES = [0, 1, 7, 8, 9, 15, 16, 17, 31, 32, 33, 63, 64, 65, 127, 128, 129, 255, 256, 257, 511, 512, 513, 1023, 1025, 2048, 2049, 5000]


@pytest.fixture(scope="module")
def lib():
    from paper_2604_17834_b200 import binding
    return binding


def _matrix(m, k, mean, dtype, seed=61):
    """EDGES, 16 rows apart and in both orders, among rows of 0 .. 2 * mean entries; a row's columns are k / length
    apart from a random start, so neighbouring rows share almost none."""
    rng = np.random.default_rng(seed)
    lens = rng.integers(0, 2 * mean + 1, m)
    lens[np.arange(len(EDGES)) * 16] = EDGES
    lens[m - 1 - np.arange(len(EDGES)) * 16] = EDGES
    rp = np.zeros(m + 1, np.int64)
    rp[1:] = np.cumsum(lens)
    step = k // np.maximum(lens, 1)
    start = (rng.random(m) * step).astype(np.int64)
    j = np.arange(rp[-1]) - np.repeat(rp[:-1], lens)
    col = (np.repeat(start, lens) + j * np.repeat(step, lens)).astype(np.int32)
    vals = wl.dense(seed + 1, 1, int(rp[-1]), ("normal", 0.0, 1.0), dtype).ravel()
    return {"m": m, "k": k, "row_ptr": rp, "col_idx": col, "vals": vals}


# rows, mean length: 4, 20, 54, 122 and 539 entries per SM and 128 groups, one for every choice of task sizes;
# N: a row of B that is one vector, 16-byte vectors (to 128 bytes, or 144 and 8400 bytes: no multiple of 32),
# 32-byte vectors with a ragged last tile, and more column tiles than one launch covers (8400 bytes)
@pytest.mark.parametrize("dtype,c16,m,mean,N", [
    ("fp16", False, 3001, 16, 8), ("tf32", False, 3001, 16, 36), ("bf16", True, 3001, 16, 64), ("fp16", False, 3001, 16, 4200),
    ("tf32", False, 3001, 16, 328), ("bf16", True, 3001, 16, 1040), ("fp16", True, 40007, 8, 80), ("tf32", False, 100003, 9, 32),
    ("bf16", False, 100003, 22, 32), ("tf32", False, 600011, 16, 8)])
def test_wcsr_row_kernel(lib, dtype, c16, m, mean, N):
    import torch
    k = max(m, 20000)
    a = _matrix(m, k, mean, dtype)
    Bs = wl.dense(63, k, N, ("uniform", -1.0, 1.0), dtype)
    Cr, S = reference(a, Bs, dtype)
    out = []
    dev = [to_device(x) for x in (a["row_ptr"], a["col_idx"], a["vals"])]
    opts = dict(c_type=lib.C_SAME_AS_INPUT if c16 else lib.C_FP32)
    for built_on_gpu in (True, False):
        if built_on_gpu:
            h = lib.spmm_wcsr_create_csr_device(m, k, *[d.data_ptr() for d in dev], dtype, 16, **opts)
        else:
            h = lib.spmm_wcsr_create_csr(m, k, a["row_ptr"], a["col_idx"], a["vals"], dtype, 16, **opts)
        try:
            info = lib.spmm_get_info(h, N)
            assert info["nnz"] * 16 <= 1.2 * info["stored_values"]          # the row kernel's at every width
            out.append(run_gpu_variant(lib, h, Bs, m, N, dtype, c16=c16))
            if built_on_gpu:
                # operands on a 16-byte boundary only: the 16-byte vectors, whatever the width; same sums
                es, cs = a["vals"].itemsize, 2 if c16 else 4
                raw = torch.empty(k * N * es + 16, dtype=torch.uint8, device="cuda")
                raw[16:] = to_device(Bs).view(torch.uint8).reshape(-1)
                cdt = {4: torch.float32, 2: torch.bfloat16 if dtype == "bf16" else torch.float16}[cs]
                buf = torch.full((2 * GUARD + m * N + 16 // cs,), CANARY, dtype=cdt, device="cuda")
                C = buf[GUARD + 16 // cs:GUARD + 16 // cs + m * N].view(m, N)
                lib.spmm_run(h, raw.data_ptr() + 16, C.data_ptr(), N, torch.cuda.current_stream().cuda_stream)
                torch.cuda.synchronize()
                check_guards(buf, "spmm_run")
                out.append(C.float().cpu().numpy())
        finally:
            lib.spmm_destroy(h)
    assert_close(out[0], Cr, S, dtype, "row kernel %s N=%d" % (dtype, N))
    assert np.array_equal(out[0], out[1]) and np.array_equal(out[0], out[2])


@pytest.mark.parametrize("dtype,N,expect", [("fp16", 32, True), ("fp16", 64, False), ("tf32", 64, True), ("tf32", 128, False)])
def test_wcsr_kernel_by_width(lib, dtype, N, expect):
    """A band that condenses 1.5 values per column: the row kernel below 64 (TF32: 128) tokens, the window kernel
    from there on (their sums differ in the last bits); a run over column chunks goes by the whole width."""
    m = 50000
    rng = np.random.default_rng(3)
    col = np.sort((np.arange(m)[:, None] + rng.permuted(np.tile(np.arange(240), (m, 1)), axis=1)[:, :16]), axis=1)
    a = {"m": m, "k": m + 240, "row_ptr": np.arange(m + 1, dtype=np.int64) * 16, "col_idx": col.astype(np.int32).ravel(),
         "vals": wl.dense(5, 1, m * 16, ("normal", 0.0, 1.0), dtype).ravel()}
    h = lib.spmm_wcsr_create_csr(m, m + 240, a["row_ptr"], a["col_idx"], a["vals"], dtype, 16)
    try:
        info = lib.spmm_get_info(h, N)
        assert 1.25 < info["nnz"] * 16 / info["stored_values"] < 1.7
        Bs = wl.dense(6, m + 240, N, ("uniform", -1.0, 1.0), dtype)
        C = run_gpu_variant(lib, h, Bs, m, N, dtype)
        Cr, S = reference(a, Bs, dtype)
        assert_close(C, Cr, S, dtype, "band N=%d" % N)
        # the row kernel adds a row of up to 32 values in their order, one rounding each
        B64 = wl.widen(Bs, dtype)
        v = wl.widen(a["vals"], dtype).reshape(m, 16)
        acc = np.zeros((64, N), np.float32)
        for j in range(16):
            acc = (acc.astype(np.float64) + v[:64, j, None] * B64[col[:64, j]]).astype(np.float32)
        assert np.array_equal(C[:64], acc) == expect
        if N == 128:
            import torch
            host = np.empty((m, N), np.float32)                            # chunks of 64 columns
            lib.spmm_run_host(h, np.ascontiguousarray(Bs), host, N, torch.cuda.current_stream().cuda_stream)
            assert np.array_equal(host, C)
    finally:
        lib.spmm_destroy(h)


def _rows_kernel_ran(a, Bs, C):
    """TF32 handles: the window kernel multiplies what the tensor core keeps of an operand (its low 13 bits dropped),
    the row kernel the whole value; a row of one entry shows which it was."""
    one = np.flatnonzero(np.diff(a["row_ptr"]) == 1)[:200]
    p = a["row_ptr"][one]
    v, b = a["vals"][p][:, None], Bs[a["col_idx"][p]]
    cut = [(x.view(np.uint32) & np.uint32(0xffffe000)).view(np.float32) for x in (np.ascontiguousarray(v), np.ascontiguousarray(b))]
    full, tf32 = np.array_equal(C[one], v * b), np.array_equal(C[one], cut[0] * cut[1])
    assert one.size > 20 and full != tf32
    return full


@pytest.mark.parametrize("on_gpu", [False, True])
def test_options_of_the_window_kernel_are_honoured(lib, on_gpu):
    """A matrix the row kernel takes by default: asking for a gather, a sub-task size or a grid size gets the window
    kernel, which they describe; the two gathers then agree to the last bit, and so does an explicit default T."""
    a = wl.wcsr_irregular(seed=31, m=5000, dtype="tf32")
    N = 128
    Bs = wl.dense(32, a["k"], N, ("normal", 0.0, 1.0), "tf32")
    Cr, S = reference(a, Bs, "tf32")
    dev = [to_device(a[x]) for x in ("row_ptr", "col_idx", "vals")]

    def run(**opt):
        if on_gpu:
            h = lib.spmm_wcsr_create_csr_device(a["m"], a["k"], *[d.data_ptr() for d in dev], "tf32", 16, **opt)
        else:
            h = lib.spmm_wcsr_create_csr(a["m"], a["k"], a["row_ptr"], a["col_idx"], a["vals"], "tf32", 16, **opt)
        try:
            C = run_gpu_variant(lib, h, Bs, a["m"], N, "tf32")
            assert_close(C, Cr, S, "tf32", str(opt))
            return C, lib.spmm_get_info(h, N)
        finally:
            lib.spmm_destroy(h)

    C0, info = run()
    assert _rows_kernel_ran(a, Bs, C0)
    outs = [run(**opt)[0] for opt in (dict(gather=lib.GATHER_TMA), dict(gather=lib.GATHER_LSU), dict(split_cols=info["split_cols"]),
                                      dict(split_cols=64), dict(n_ctas=info["n_ctas"]))]
    assert not any(_rows_kernel_ran(a, Bs, C) for C in outs)
    assert all(np.array_equal(outs[0], outs[i]) for i in (1, 2, 4))


def test_a_wait_limit_of_zero_does_not_change_the_kernel(lib):
    """The limit is process wide: set between the preparation of a handle and its run it makes the run give up, and
    must not send it to another kernel with another workspace (a captured run shows that nothing was allocated)."""
    import torch
    a = _matrix(3001, 20000, 16, "tf32")
    N = 128
    Bs = wl.dense(33, a["k"], N, ("normal", 0.0, 1.0), "tf32")
    B, C = to_device(Bs), torch.empty((a["m"], N), dtype=torch.float32, device="cuda")
    h = lib.spmm_wcsr_create_csr(a["m"], a["k"], a["row_ptr"], a["col_idx"], a["vals"], "tf32", 16)
    try:
        want = run_gpu_variant(lib, h, Bs, a["m"], N, "tf32")
        assert _rows_kernel_ran(a, Bs, want)
        lib.spmm_set_wait_limit_ns(0)
        code, nodes = captured_run(lib, h, B, C, N)
        assert code == lib.SPMM_OK and nodes == ["kernel"]                   # (the window kernel would be two)
        lib.spmm_run(h, B.data_ptr(), C.data_ptr(), N, torch.cuda.current_stream().cuda_stream)
        torch.cuda.synchronize()
        with pytest.raises(lib.SpmmError) as e:
            lib.spmm_check(h)
        assert e.value.code == lib.SPMM_ERR_DEV_TIMEOUT
        lib.spmm_set_wait_limit_ns(2_000_000_000)
        assert np.array_equal(run_gpu_variant(lib, h, Bs, a["m"], N, "tf32"), want)
    finally:
        lib.spmm_set_wait_limit_ns(2_000_000_000)
        lib.spmm_destroy(h)


def test_static_run_takes_the_kernel_of_spmm_run(lib):
    """Partial rows of more than the built-in scratch holds (14,208 of 160 columns, 9.1 MB): the static run goes
    through it in narrower column tiles instead of taking another kernel, and stays bitwise equal to spmm_run."""
    import torch
    m, n, k, N, dtype = 7104, 1100, 400000, 160, "fp16"
    g = torch.Generator(device="cuda").manual_seed(7)
    step = k // n
    start = torch.randint(0, step, (m, 1), generator=g, device="cuda")
    ci = (torch.arange(n, device="cuda")[None, :] * step + start).to(torch.int32).contiguous()
    rp = torch.arange(m + 1, device="cuda", dtype=torch.int64) * n
    va = torch.randn(m * n, generator=g, device="cuda").to(torch.float16)
    B = torch.randn((k, N), generator=g, device="cuda").to(torch.float16)
    h = lib.spmm_wcsr_create_csr_device(m, k, rp.data_ptr(), ci.data_ptr(), va.data_ptr(), dtype, 16)
    try:
        info = lib.spmm_get_info(h, N)
        assert info["n_slots"] * 16 * N * 4 <= 8 << 20 and info["nnz"] * 16 <= 1.2 * info["stored_values"]
        st = torch.cuda.current_stream().cuda_stream
        want, got = (torch.full((m, N), float("nan"), device="cuda") for _ in range(2))
        lib.spmm_run(h, B.data_ptr(), want.data_ptr(), N, st)
        for _ in range(2):
            lib.spmm_wcsr_run_static(h, B.data_ptr(), got.data_ptr(), N, st)
            torch.cuda.synchronize()
            lib.spmm_check(h)
            assert torch.equal(got, want)
        a = {"row_ptr": rp.cpu().numpy(), "col_idx": ci.cpu().numpy().ravel(), "vals": va.cpu().numpy()}
        cols = np.array([0, 7, 8, 143, 144, 159])
        Cr, S = reference(a, B.cpu().numpy(), dtype, cols=cols)
        assert_close(want[:, torch.from_numpy(cols).cuda()].cpu().numpy(), Cr, S, dtype, "long rows")
    finally:
        lib.spmm_destroy(h)


@pytest.mark.parametrize("dtype,widths", [("tf32", (36, 64, 128, 320)), ("fp16", (72, 128, 320, 520))])
def test_the_sums_do_not_depend_on_the_cta_size(lib, dtype, widths):
    """A small launch takes CTAs of 128 or 256 threads by the groups that its dense width leaves a warp (8 to 1 of them
    here; 256 with up to three, as the launches show); a column's sums are those of the widest run, bit by bit."""
    import torch
    m, k = 3001, 20000
    a = _matrix(m, k, 16, dtype)
    Bs = wl.dense(64, k, widths[-1], ("uniform", -1.0, 1.0), dtype)
    h = lib.spmm_wcsr_create_csr(m, k, a["row_ptr"], a["col_idx"], a["vals"], dtype, 16)
    try:
        want = run_gpu_variant(lib, h, Bs, m, widths[-1], dtype)
        Cr, S = reference(a, Bs, dtype)
        assert_close(want, Cr, S, dtype, "rows N=%d" % widths[-1])
        for N in (16,) + widths:
            B = np.ascontiguousarray(Bs[:, :N])
            assert np.array_equal(run_gpu_variant(lib, h, B, m, N, dtype), want[:, :N]), N
            launches = captured_launches(lib, h, to_device(B), torch.empty((m, N), dtype=torch.float32, device="cuda"), N)
            groups = {16: 8 if dtype == "tf32" else 16, 36: 3, 64: 4, 72: 3, 128: 2 if dtype == "tf32" else 4, 320: 2 if dtype == "tf32" else 1, 520: 1}[N]
            assert {t for _, t in launches} == {256 if groups < 4 else 128}, (N, launches)
    finally:
        lib.spmm_destroy(h)


@pytest.mark.parametrize("m,per_row", [(3001, 5), (30001, 5), (30001, 9), (160000, 16)])
def test_plain_sums_of_16_byte_vectors_are_the_same_bits(lib, m, per_row):
    """TF32 with rows of B that are no multiple of 32 bytes: one or two columns per instruction, and the strands of long rows
    with or without padding, by the width, the entries a row (6) and the size of the launch.  A column's sums are those of an
    aligned, wider run, which has two columns and the padding, bit by bit."""
    rng = np.random.default_rng(m + per_row)
    k = 5000
    lens = np.full(m, per_row, np.int64)
    lens[[3, 700]] = (2500, 4001)                          # long rows, one cut into parts
    rp = np.concatenate(([0], np.cumsum(lens))).astype(np.int64)
    starts = rng.integers(0, k - 20, m)
    ci = np.concatenate([starts[i] + np.arange(n) if n < 20 else np.sort(rng.choice(k, n, replace=False)) for i, n in enumerate(lens)]).astype(np.int32)
    vals = wl.to_storage(rng.uniform(-1, 1, ci.size), "tf32")
    Bs = wl.dense(12, k, 136, ("uniform", -1.0, 1.0), "tf32")
    h = lib.spmm_wcsr_create_csr(m, k, rp, ci, vals, "tf32", 16)
    try:
        want = run_gpu_variant(lib, h, Bs, m, 136, "tf32")
        Cr, S = reference({"m": m, "k": k, "row_ptr": rp, "col_idx": ci, "vals": vals}, Bs, "tf32", rows=(0, 800))
        assert_close(want[:800], Cr[:800], S[:800], "tf32", "rows N=136")
        for N in (4, 20, 32, 36, 52, 132):
            got = run_gpu_variant(lib, h, np.ascontiguousarray(Bs[:, :N]), m, N, "tf32")
            assert np.array_equal(got, want[:, :N]), N
    finally:
        lib.spmm_destroy(h)


def test_many_parts_of_long_rows_keep_small_ctas(lib):
    """900 rows of 100 entries, each a part of its own in a launch this small: CTAs of 128 threads where a warp holds two groups,
    of 256 where it holds one (by the parts that an SM takes in turn); the same bits and the oracle's result."""
    import torch
    m, k, n = 900, 6000, 100
    rng = np.random.default_rng(9)
    rp = np.arange(m + 1, dtype=np.int64) * n
    ci = np.concatenate([np.sort(rng.choice(k, n, replace=False)) for _ in range(m)]).astype(np.int32)
    vals = wl.to_storage(rng.uniform(-1, 1, ci.size), "tf32")
    Bs = wl.dense(13, k, 128, ("uniform", -1.0, 1.0), "tf32")
    h = lib.spmm_wcsr_create_csr(m, k, rp, ci, vals, "tf32", 16)
    try:
        got = {}
        for N, threads in ((128, 128), (76, 256)):
            B = np.ascontiguousarray(Bs[:, :N])
            got[N] = run_gpu_variant(lib, h, B, m, N, "tf32")
            launches = captured_launches(lib, h, to_device(B), torch.empty((m, N), dtype=torch.float32, device="cuda"), N)
            assert {t for _, t in launches} == {threads}, (N, launches)
        assert np.array_equal(got[76], got[128][:, :76])
        Cr, S = reference({"m": m, "k": k, "row_ptr": rp, "col_idx": ci, "vals": vals}, Bs, "tf32")
        assert_close(got[128], Cr, S, "tf32", "many parts")
    finally:
        lib.spmm_destroy(h)
