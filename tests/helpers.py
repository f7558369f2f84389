"""Shared pieces of the GPU parity tests: run the CUDA path through the C ABI and
compare it element by element with the fp64 oracle under the stated bound

    |C_gpu - C_ref| <= tau * sum_k |a_ik b_kj| + 1e-6,

tau = 8e-3 for bf16 / fp16 (and E4M3) inputs, 2e-3 for the TF32 path (fp32 accumulation).
"""
import numpy as np

from oracle import spmm_ref
from paper_2604_17834_b200 import workloads as wl

TAU = {"bf16": 8e-3, "fp16": 8e-3, "tf32": 2e-3, "fp8": 8e-3}


def to_device(arr):
    """numpy storage array -> torch CUDA tensor holding the same bytes."""
    import torch
    a = np.ascontiguousarray(arr)
    if a.dtype == np.uint16:
        a = a.view(np.int16)
    return torch.from_numpy(a).cuda()


GUARD = 8192          # elements of canary on either side of C
CANARY = 24576.0      # exact in fp32, fp16 and bf16


def guarded_c(shape, tdt, fill):
    """C inside a larger allocation whose margins hold a canary value: a store that lands outside C
    (a tile clipped wrongly, a row index off by one block) shows up in check_guards.
    -> (whole buffer, view of C with the requested shape)."""
    import torch
    n = int(np.prod(shape))
    buf = torch.full((n + 2 * GUARD,), CANARY, dtype=tdt, device="cuda")
    C = buf[GUARD:GUARD + n].view(*shape)
    C.fill_(fill)
    return buf, C


def check_guards(buf, what=""):
    import torch
    lo, hi = buf[:GUARD].float(), buf[-GUARD:].float()
    assert bool(torch.all(lo == CANARY)) and bool(torch.all(hi == CANARY)), "%s: a store landed outside C" % what


def run_gpu(lib, h, B_storage, m, N, fill=float("nan"), check=True):
    """One spmm_run on device buffers; C is pre-filled with NaN so unwritten elements show, and
    sits between two canary margins so that stores outside it show as well."""
    import torch
    Bd = to_device(B_storage)
    buf, C = guarded_c((m, N), torch.float32, fill)
    lib.spmm_run(h, Bd.data_ptr(), C.data_ptr(), N, torch.cuda.current_stream().cuda_stream)
    torch.cuda.synchronize()
    if check:
        lib.spmm_check(h)
    check_guards(buf, "spmm_run")
    return C.cpu().numpy()


def run_gpu_variant(lib, h, B_storage, m, N, dtype, c16=False, col_major=False, check=True):
    """spmm_run for a handle created with c_type / layout options.  B_storage is always the
    k x N operand; with col_major the device gets X = B^T (N x k) and returns Y = C^T (N x m).
    The result comes back as an m x N float32 array either way."""
    import torch
    Bs = np.ascontiguousarray(B_storage.T) if col_major else B_storage
    Bd = to_device(Bs)
    tdt = torch.float32 if not c16 else (torch.bfloat16 if dtype == "bf16" else torch.float16)
    shape = (N, m) if col_major else (m, N)
    buf, C = guarded_c(shape, tdt, float("nan"))
    lib.spmm_run(h, Bd.data_ptr(), C.data_ptr(), N, torch.cuda.current_stream().cuda_stream)
    torch.cuda.synchronize()
    if check:
        lib.spmm_check(h)
    check_guards(buf, "spmm_run")
    out = C.float().cpu().numpy()
    return np.ascontiguousarray(out.T) if col_major else out


def reference(a, B_storage, dtype, cols=None, rows=None):
    v64 = wl.widen(a["vals"], dtype)
    B64 = wl.widen(B_storage if cols is None else B_storage[:, cols], dtype)
    return spmm_ref(a["row_ptr"], a["col_idx"], v64, B64, rows=rows)


def assert_close(C_gpu, C_ref, S, dtype, what=""):
    assert C_gpu.shape == C_ref.shape
    assert np.all(np.isfinite(C_gpu)), "%s: %d non-finite / unwritten outputs" % (what, int((~np.isfinite(C_gpu)).sum()))
    err = np.abs(C_gpu.astype(np.float64) - C_ref)
    bound = TAU[dtype] * S + 1e-6
    bad = err > bound
    if bad.any():
        i, j = np.unravel_index(np.argmax(err - bound), err.shape)
        raise AssertionError("%s: %d of %d outside the bound; worst at (%d,%d): gpu %.6g ref %.6g err %.3g bound %.3g"
                             % (what, int(bad.sum()), err.size, i, j, C_gpu[i, j], C_ref[i, j], err[i, j], bound[i, j]))
    return float(np.max(err / bound))


def kernel_launch(cu, node):
    """(CTAs, threads per CTA) of a kernel node of a captured graph."""
    import ctypes

    class Params(ctypes.Structure):                                          # CUDA_KERNEL_NODE_PARAMS (v2)
        _fields_ = [("func", ctypes.c_void_p)] + [(x, ctypes.c_uint) for x in ("gx", "gy", "gz", "bx", "by", "bz", "shared")] + \
                   [(x, ctypes.c_void_p) for x in ("params", "extra", "kern", "ctx")]

    p = Params()
    assert cu.cuGraphKernelNodeGetParams_v2(ctypes.c_void_p(node), ctypes.byref(p)) == 0
    return p.gx * p.gy * p.gz, p.bx * p.by * p.bz


def captured_launches(lib, h, B, C, N):
    """(CTAs, threads per CTA) of every kernel that one spmm_run launches, in order; nothing runs."""
    found = []
    code, kinds = captured_run(lib, h, B, C, N, launches=found)
    assert code == lib.SPMM_OK and len(found) == len(kinds), (code, kinds)
    return found


def captured_run(lib, h, B, C, N, relaxed=False, replay=False, static=False, launches=None):
    """One spmm_run (static: spmm_wcsr_run_static) inside a stream capture of its own stream.  -> (status code of the run, kinds of the captured
    nodes, or None where the capture gave no graph).  replay: launch the graph once, unless the run was refused.  launches: a list
    that the kernel nodes' sizes are added to (the nodes of a graph of one stream come in its order)."""
    import ctypes
    import torch
    cu = ctypes.CDLL("libcuda.so.1")
    torch.cuda.synchronize()
    stream = torch.cuda.Stream()
    st, graph, n = ctypes.c_void_p(stream.cuda_stream), ctypes.c_void_p(), ctypes.c_size_t()
    assert cu.cuStreamBeginCapture_v2(st, 2 if relaxed else 0) == 0          # CU_STREAM_CAPTURE_MODE_RELAXED / _GLOBAL
    code = lib.SPMM_OK
    try:
        (lib.spmm_wcsr_run_static if static else lib.spmm_run)(h, B.data_ptr(), C.data_ptr(), N, stream.cuda_stream)
    except lib.SpmmError as e:
        code = e.code
    if cu.cuStreamEndCapture(st, ctypes.byref(graph)) != 0 or not graph.value:
        return code, None
    assert cu.cuGraphGetNodes(graph, None, ctypes.byref(n)) == 0
    nodes = (ctypes.c_void_p * n.value)()
    assert n.value == 0 or cu.cuGraphGetNodes(graph, nodes, ctypes.byref(n)) == 0
    kinds = []
    for x in nodes:
        t = ctypes.c_int(-1)
        assert cu.cuGraphNodeGetType(ctypes.c_void_p(x), ctypes.byref(t)) == 0
        kinds.append("kernel" if t.value == 0 else "type %d" % t.value)      # CU_GRAPH_NODE_TYPE_KERNEL
        if launches is not None and t.value == 0:
            launches.append(kernel_launch(cu, x))
    if replay and code == lib.SPMM_OK:
        ex = ctypes.c_void_p()
        assert cu.cuGraphInstantiateWithFlags(ctypes.byref(ex), graph, ctypes.c_ulonglong(0)) == 0
        assert cu.cuGraphLaunch(ex, st) == 0
        stream.synchronize()
        lib.spmm_check(h)
        cu.cuGraphExecDestroy(ex)
    cu.cuGraphDestroy(graph)
    return code, kinds
