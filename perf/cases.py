"""Performance cases of the SpMM library: what a user has it do, over the ranges it is used in.

A case is a dict of plain values.  ``listed()`` are the fixed ones, ``draw(rng)`` gives one more of
the same ranges.  Matrices, values and dense operands are drawn on the GPU from the seed; they
follow the generators of ``paper_2604_17834_b200/workloads.py`` (block-pruned weights, skewed
block-row lengths, power-law rows with a diagonal band, R-MAT graphs).  A pass is one or two
``spmm_run`` calls on device-resident operands, or (``op = create``) the construction of a handle
from a CSR matrix in device memory followed by its first product.

Keys of a case
  op      bcsr     C = A B with a block-sparse A (one spmm_run)
          ffn      the two sparse projections of a pruned feed-forward layer as linear layers:
                   H = X Wup^T and Y = G Wdown^T (column-major operands, two spmm_run)
          wcsr     C = A B with an irregular A (one spmm_run)
          create   spmm_wcsr_create_csr_device + spmm_run + spmm_destroy on a new matrix
  matrix  blocks | irregular | rmat, with the sizes and densities named as in workloads.py
  dtype   bf16 | fp16 | tf32 | fp8      c16  C in the input's 16-bit type      N  dense width
"""
from __future__ import annotations

import math

import torch

from paper_2604_17834_b200 import binding as spmm

_TORCH = {"bf16": torch.bfloat16, "fp16": torch.float16, "tf32": torch.float32, "fp8": torch.float8_e4m3fn}
_ES = {"bf16": 2, "fp16": 2, "tf32": 4, "fp8": 1}


def listed():
    return [
        # the smallest call: a 512 x 512 layer, where the launch and one pass over the pipeline count
        {"name": "bcsr_tiny", "op": "bcsr", "m": 512, "k": 512, "b": 64, "density": 0.5, "skewed": False,
         "dtype": "bf16", "c16": False, "N": 256},
        # prefill of a pruned up-projection, 64K tokens, fp32 result: the largest call
        {"name": "bcsr_prefill_64k", "op": "bcsr", "m": 18944, "k": 3584, "b": 64, "density": 0.1, "skewed": False,
         "dtype": "bf16", "c16": False, "N": 65536},
        # both projections of the pruned layer over a ragged number of prompt tokens, bf16 in and out
        {"name": "ffn_prefill", "op": "ffn", "d": 3584, "f": 18944, "b": 64, "density": 0.1, "dtype": "bf16",
         "c16": True, "N": 9001},
        # the same layer in a decode step of 128 sequences
        {"name": "ffn_decode", "op": "ffn", "d": 3584, "f": 18944, "b": 64, "density": 0.1, "dtype": "bf16",
         "c16": True, "N": 128},
        # the same layer quantised to E4M3 (fp32 result), a short prompt
        {"name": "ffn_fp8", "op": "ffn", "d": 3584, "f": 18944, "b": 64, "density": 0.1, "dtype": "fp8",
         "c16": False, "N": 2048},
        # fine-grained blocks, a few full block-rows among sparse and empty ones
        {"name": "bcsr_b16_skewed", "op": "bcsr", "m": 8192, "k": 8192, "b": 16, "density": 0.1, "skewed": True,
         "dtype": "fp16", "c16": False, "N": 4096},
        # fp32 storage with TF32 arithmetic, sizes that no tile divides
        {"name": "bcsr_b32_tf32", "op": "bcsr", "m": 6000, "k": 5000, "b": 32, "density": 0.05, "skewed": True,
         "dtype": "tf32", "c16": False, "N": 1500},
        # scientific matrix: power-law rows, half of the entries near the diagonal
        {"name": "wcsr_irregular", "op": "wcsr", "matrix": "irregular", "m": 100000, "alpha": 2.0, "dtype": "tf32",
         "c16": False, "N": 128},
        # a small one of the same kind, narrow operand: latency
        {"name": "wcsr_small", "op": "wcsr", "matrix": "irregular", "m": 4000, "alpha": 1.8, "dtype": "tf32",
         "c16": False, "N": 36},
        # aggregation over a large graph
        {"name": "wcsr_graph", "op": "wcsr", "matrix": "rmat", "scale": 21, "degree": 16, "dtype": "fp16",
         "c16": False, "N": 128},
        # a smaller graph with narrow features, 16-bit result
        {"name": "wcsr_graph_narrow", "op": "wcsr", "matrix": "rmat", "scale": 17, "degree": 24, "dtype": "bf16",
         "c16": True, "N": 40},
        # a matrix that is new in every step: built on the GPU, multiplied once, dropped
        {"name": "wcsr_new_matrix", "op": "create", "matrix": "irregular", "m": 60000, "alpha": 1.8, "dtype": "fp16",
         "c16": False, "N": 64},
    ]


def _log(rng, lo, hi):
    """An integer of [lo, hi], spread over the logarithm."""
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _up(x, q):
    return -(-int(x) // q) * q


def draw(rng):
    op = rng.choice(["bcsr", "bcsr", "ffn", "ffn", "wcsr", "wcsr", "wcsr", "create"])
    if op == "bcsr":
        dtype = rng.choice(["bf16", "fp16", "fp16", "tf32"])
        b = rng.choice([16, 32, 64, 128])
        c = {"op": op, "m": _log(rng, 512, 18944), "k": _log(rng, 512, 18944), "b": b,
             "density": round(math.exp(rng.uniform(math.log(0.01), math.log(0.5))), 4), "skewed": rng.random() < 0.5,
             "dtype": dtype, "c16": dtype != "tf32" and rng.random() < 0.4, "N": _up(_log(rng, 64, 65536), 8)}
        # no costlier than the largest listed case
        while c["m"] * c["k"] * (0.1 + c["density"]) * c["N"] > 4.5e11 or c["m"] * c["N"] > 1.0e9:
            c["N"] = _up(c["N"] // 2, 8)
        return c
    if op == "ffn":
        d = _up(_log(rng, 512, 4096), 64)
        dtype = rng.choice(["bf16", "bf16", "fp16", "fp8"])
        return {"op": op, "d": d, "f": _up(d * rng.uniform(2.5, 5.5), 64), "b": rng.choice([32, 64, 64, 128]),
                "density": round(rng.uniform(0.05, 0.3), 3), "dtype": dtype, "c16": dtype != "fp8",
                "N": _log(rng, 128, 12288)}
    dtype = rng.choice(["fp16", "bf16", "tf32", "tf32"])
    c = {"op": op, "dtype": dtype, "c16": dtype != "tf32" and rng.random() < 0.3,
         "N": _up(_log(rng, 16, 320), 8 if dtype != "tf32" else 4)}
    if rng.random() < 0.5:
        c.update(matrix="irregular", m=_log(rng, 4000, 400000 if op == "wcsr" else 200000), alpha=round(rng.uniform(1.7, 2.3), 2))
    else:
        c.update(matrix="rmat", scale=rng.randint(13, 20 if op == "wcsr" else 17), degree=rng.choice([4, 8, 16, 24]))
    return c


# ----------------------------------------------------------------------------- inputs


class _Handle:
    """A handle as a program keeps it; freed with the object."""

    def __init__(self, h):
        self.h = h

    def __del__(self):
        spmm.spmm_destroy(self.h)


def _gen(seed, salt):
    return torch.Generator(device="cuda").manual_seed(int(seed) * 1000003 + salt)


def _to(x, dtype):
    return x.to(_TORCH[dtype])


def _normal(g, shape, std, dtype):
    out = torch.empty(shape, dtype=_TORCH[dtype], device="cuda")
    step = max(1, (1 << 26) // max(1, shape[1]))
    for r in range(0, shape[0], step):
        part = out[r:r + step]
        part.copy_(torch.randn(part.shape, generator=g, device="cuda").mul_(std))
    return out


def _row_ptr(lens):
    rp = torch.zeros(lens.numel() + 1, dtype=torch.int64, device="cuda")
    torch.cumsum(lens, 0, out=rp[1:])
    return rp


def _blocks_csr(g, m, k, b, density, skewed):
    """CSR of a matrix whose kept b x b blocks are dense: floor(density * #blocks) blocks at random
    places (pruned weights), or, skewed, 10 % of the block-rows full, 20 % empty and the blocks of
    the rest kept with probability density."""
    nbr, nbc = -(-m // b), -(-k // b)
    if not skewed:
        keep = max(1, int(density * nbr * nbc))
        mask = torch.zeros(nbr * nbc, dtype=torch.bool, device="cuda")
        mask[torch.randperm(nbr * nbc, generator=g, device="cuda")[:keep]] = True
        mask = mask.view(nbr, nbc)
    else:
        perm = torch.randperm(nbr, generator=g, device="cuda")
        mask = torch.rand((nbr, nbc), generator=g, device="cuda") < density
        nfull, nempty = round(0.1 * nbr), round(0.2 * nbr)
        mask[perm[:nfull]] = True
        mask[perm[nfull:nfull + nempty]] = False
    width = torch.full((nbc,), b, dtype=torch.int64, device="cuda")
    width[-1] = k - (nbc - 1) * b
    blk_len = (mask * width).sum(1)                       # columns kept in a row of block-row I
    rp = _row_ptr(blk_len.repeat_interleave(b)[:m])
    I, J = mask.nonzero(as_tuple=True)
    cols = (J[:, None] * b + torch.arange(b, device="cuda")).to(torch.int32)
    cols = cols[cols < k]                                 # block-row after block-row, ascending
    start = _row_ptr(blk_len)[:-1]
    row = torch.arange(m, device="cuda")
    base = (start[row // b] - rp[:-1])                    # entry p of row i is column cols[base + p]
    ci = torch.empty(int(rp[-1]), dtype=torch.int32, device="cuda")
    step = 1024
    for r in range(0, m, step):
        r1 = min(m, r + step)
        p0, p1 = int(rp[r]), int(rp[r1])
        off = base[r:r1].repeat_interleave((rp[r + 1:r1 + 1] - rp[r:r1]), output_size=p1 - p0)
        ci[p0:p1] = cols[off + torch.arange(p0, p1, device="cuda")]
    return rp, ci


def _csr_from_keys(keys, m, k):
    keys = torch.unique(keys)                             # sorted
    rows = keys // k
    return _row_ptr(torch.bincount(rows, minlength=m)), (keys - rows * k).to(torch.int32)


def _zipf_lengths(alpha):
    """P(length >= x), x = 1 .. 5000, of min(Zipf(alpha), 5000)."""
    x = torch.arange(1, 200001, dtype=torch.float64)
    w = x ** -alpha
    total = float(w.sum()) + 200000.5 ** (1 - alpha) / (alpha - 1)
    below = torch.cat([torch.zeros(1, dtype=torch.float64), torch.cumsum(w[:4999], 0)]) / total
    return 1.0 - below


def _irregular_csr(g, m, alpha):
    k, band = m, 256
    tail = _zipf_lengths(alpha).cuda()
    u = torch.rand(m, generator=g, device="cuda", dtype=torch.float64)
    length = (5000 - torch.searchsorted(tail.flip(0).contiguous(), u)).clamp_(1, 5000)
    rows = torch.arange(m, device="cuda").repeat_interleave(length)
    n = rows.numel()
    ucol = torch.randint(0, k, (n,), generator=g, device="cuda")
    bcol = (rows + torch.randint(-band, band + 1, (n,), generator=g, device="cuda")).clamp_(0, k - 1)
    col = torch.where(torch.rand(n, generator=g, device="cuda") < 0.5, ucol, bcol)
    return _csr_from_keys(rows * k + col, m, k)


def _rmat_csr(g, scale, degree):
    n = 1 << scale
    parts = []
    for e0 in range(0, degree * n, 1 << 23):
        ne = min(1 << 23, degree * n - e0)
        key = torch.zeros(ne, dtype=torch.int64, device="cuda")
        for _ in range(scale):
            u = torch.rand(ne, generator=g, device="cuda")
            rbit = u >= 0.76
            cbit = ((u >= 0.57) & (u < 0.76)) | (u >= 0.95)
            # row bits from bit `scale` up, column bits below it: both move up together
            key = (key << 1) | (rbit.to(torch.int64) << scale) | cbit.to(torch.int64)
        parts.append(key)
    return _csr_from_keys(torch.cat(parts), n, n)


def _matrix(case, seed):
    """-> m, k, row_ptr, col_idx, values."""
    g = _gen(seed, 1)
    if case["matrix"] == "irregular":
        m = k = case["m"]
        rp, ci = _irregular_csr(g, m, case["alpha"])
        vals = torch.randn(ci.numel(), generator=g, device="cuda")
    else:
        m = k = 1 << case["scale"]
        rp, ci = _rmat_csr(g, case["scale"], case["degree"])
        vals = 1.0 - torch.rand(ci.numel(), generator=g, device="cuda")
    return m, k, rp, ci, _to(vals, case["dtype"])


def _c_dtype(case):
    return _TORCH[case["dtype"]] if case["c16"] else torch.float32


def _opts(case):
    return {"c_type": spmm.C_SAME_AS_INPUT} if case["c16"] else {}


def prepare(case, seed):
    dtype, N = case["dtype"], case["N"]
    stream = torch.cuda.current_stream().cuda_stream
    st = {"op": case["op"], "stream": stream, "N": N}
    if case["op"] == "ffn":
        st["layers"] = []
        for i, (m, k) in enumerate(((case["f"], case["d"]), (case["d"], case["f"]))):
            g = _gen(seed, 10 + i)
            rp, ci = _blocks_csr(g, m, k, case["b"], case["density"], False)
            vals = _to(torch.randn(ci.numel(), generator=g, device="cuda").mul_(0.02 if dtype != "fp8" else 1.0), dtype)
            h = spmm.spmm_bcsr_create_csr_device(m, k, rp.data_ptr(), ci.data_ptr(), vals.data_ptr(), dtype, case["b"], stream,
                                                 layout=spmm.COLMAJOR, **_opts(case))
            spmm.spmm_prepare(h, N)
            st["layers"].append((_Handle(h), _normal(g, (N, k), 1.0, dtype), torch.empty((N, m), dtype=_c_dtype(case), device="cuda")))
        return st
    if case["op"] == "bcsr":
        m, k = case["m"], case["k"]
        g = _gen(seed, 1)
        rp, ci = _blocks_csr(g, m, k, case["b"], case["density"], case["skewed"])
        vals = _to(torch.rand(ci.numel(), generator=g, device="cuda").mul_(2.0).sub_(1.0), dtype)
        h = spmm.spmm_bcsr_create_csr_device(m, k, rp.data_ptr(), ci.data_ptr(), vals.data_ptr(), dtype, case["b"], stream, **_opts(case))
        spmm.spmm_prepare(h, N)
        st["h"] = _Handle(h)
    elif case["op"] == "wcsr":
        m, k, rp, ci, vals = _matrix(case, seed)
        h = spmm.spmm_wcsr_create_csr_device(m, k, rp.data_ptr(), ci.data_ptr(), vals.data_ptr(), dtype, 16, stream, **_opts(case))
        spmm.spmm_prepare(h, N)
        st["h"] = _Handle(h)
    else:
        m, k, rp, ci, vals = _matrix(case, seed)
        st["csr"] = (m, k, rp, ci, vals, dtype)
        st["opts"] = _opts(case)
    st["B"] = _normal(_gen(seed, 2), (k, N), 1.0, dtype)
    st["C"] = torch.empty((m, N), dtype=_c_dtype(case), device="cuda")
    return st


def run(st):
    N, stream = st["N"], st["stream"]
    if st["op"] == "ffn":
        for h, X, Y in st["layers"]:
            spmm.spmm_run(h.h, X.data_ptr(), Y.data_ptr(), N, stream)
        return [Y for _, _, Y in st["layers"]]
    B, C = st["B"], st["C"]
    if st["op"] == "create":
        m, k, rp, ci, vals, dtype = st["csr"]
        h = spmm.spmm_wcsr_create_csr_device(m, k, rp.data_ptr(), ci.data_ptr(), vals.data_ptr(), dtype, 16, stream, **st["opts"])
        spmm.spmm_run(h, B.data_ptr(), C.data_ptr(), N, stream)
        spmm.spmm_destroy(h)
        return C
    spmm.spmm_run(st["h"].h, B.data_ptr(), C.data_ptr(), N, stream)
    return C


# ----------------------------------------------------------------------------- what a pass cannot do without


def _blocks_counts(m, k, b, density, skewed):
    """Expected stored blocks, distinct block columns."""
    nbr, nbc = -(-m // b), -(-k // b)
    if not skewed:
        return nbr * nbc * density, nbc * (1.0 - (1.0 - density) ** nbr)
    full, empty = round(0.1 * nbr), round(0.2 * nbr)
    return full * nbc + (nbr - full - empty) * nbc * density, nbc if full else nbc * (1.0 - (1.0 - density) ** (nbr - empty))


def _blocks_work(m, k, b, density, skewed, es, cs, N):
    nb, cols = _blocks_counts(m, k, b, density, skewed)
    nbr = -(-m // b)
    rows = min(float(k), cols * b)
    return nb * b * b * es + (nbr + 1 + nb) * 4 + rows * N * es + float(m) * N * cs, 2.0 * nb * b * b * N


def _irregular_counts(m, alpha):
    """Expected entries (duplicates ignored), distinct columns (half uniform, half near the diagonal)."""
    n = m * float(_zipf_lengths(alpha).sum())
    return n, m * (1.0 - math.exp(-n / m))


def _rmat_counts(scale, degree):
    n, edges = 1 << scale, degree << scale
    cells = 0.0                                           # occupied cells, by the number of edges' bits of each kind
    for i in range(scale + 1):                            # (0,0) levels
        for j in range(scale + 1 - i):                    # (0,1) and (1,0) levels (equal probability)
            l = scale - i - j
            logw = math.lgamma(scale + 1) - math.lgamma(i + 1) - math.lgamma(j + 1) - math.lgamma(l + 1) + j * math.log(2.0)
            p = math.exp(i * math.log(0.57) + j * math.log(0.19) + l * math.log(0.05))
            cells += math.exp(logw) * -math.expm1(-edges * p)
    cols = sum(math.comb(scale, j) * -math.expm1(-edges * 0.76 ** (scale - j) * 0.24 ** j) for j in range(scale + 1))
    return cells, min(cols, float(n))


def work(case):
    es = _ES[case["dtype"]]
    cs = 2 if case["c16"] else 4
    N = case["N"]
    if case["op"] == "ffn":
        parts = [_blocks_work(m, k, case["b"], case["density"], False, es, cs, N)
                 for m, k in ((case["f"], case["d"]), (case["d"], case["f"]))]
        return {"bytes": sum(p[0] for p in parts), "flops": sum(p[1] for p in parts)}
    if case["op"] == "bcsr":
        by, fl = _blocks_work(case["m"], case["k"], case["b"], case["density"], case["skewed"], es, cs, N)
        return {"bytes": by, "flops": fl}
    # entries with their column index, row pointers, each touched row of B, C
    if case["matrix"] == "irregular":
        m = case["m"]
        nnz, cols = _irregular_counts(m, case["alpha"])
    else:
        m = 1 << case["scale"]
        nnz, cols = _rmat_counts(case["scale"], case["degree"])
    return {"bytes": nnz * (es + 4) + (m + 1) * 4 + cols * N * es + float(m) * N * cs, "flops": 2.0 * nnz * N}


def tolerance(case):
    """About four times the distance to the same products summed in 64 bits, measured on the listed
    and some drawn cases: 1.7e-3 rounding to bf16, 2.1e-4 to fp16, 7.7e-4 for TF32 operands (two
    13-bit truncations per product), 1.7e-5 for fp32 sums of up to 1e5 products in the tensor core."""
    if case["dtype"] == "tf32":
        return {"rel": 3e-3, "max": 0.08}
    if case["c16"]:
        return {"rel": 6.6e-3 if case["dtype"] == "bf16" else 8.5e-4, "max": 0.016}
    return {"rel": 7e-5, "max": 0.013}
