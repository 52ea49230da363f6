"""The work whose speed is measured: calls of the library's public entry points.

A program that uses this library holds a sparse matrix (CSR) or 3-tensor (CSF)
and dense fp32 operands on the GPU and calls one of the seven fused
expressions, again and again with new values: a layer of a graph network
(<SpMM,GEMM>, <SDDMM,SpMM>, <SDDMM,SpMM,GEMM>, <SpMMH,GEMM>) or a sweep of a
tensor factorisation (MTTKRP, <MTTKRP,GEMM>, <SpTTM,SpTTM>).  Sizes are those
of the repository's workloads and tests; structures are the same kinds (R-MAT
graphs, uniform rows, Zipf slices, power-law fibers), drawn here on the GPU.
"""
import functools
import math

import torch

import paper_2205_11622_gb300 as slnr

CSR_OPS = ("spmm_gemm", "sddmm_spmm", "sddmm_spmm_gemm", "spmmh_gemm")
CSF_OPS = ("mttkrp", "mttkrp_gemm", "spttm_ttm")

# Inner widths: the powers of two of the inner-dimension sweep, and widths
# that are multiples of 4 only (feature counts of graph data sets).
POW2 = (16, 32, 64, 128)
OTHER = (12, 20, 48, 96, 100, 200, 256)


def listed():
    return [
        # The smallest call: a 1024 x 1024 matrix of 10 nonzeros a row.  Latency and launches count.
        dict(name="spmm_gemm_1k_32", op="spmm_gemm", n=1024, nnz=10240, graph="uniform", K=32, L=32, tf32=True),
        # A graph-network layer over a large power-law graph: the largest output and gathered matrix.
        dict(name="spmm_gemm_rmat1m_128", op="spmm_gemm", n=1 << 20, nnz=1 << 24, graph="rmat", K=128, L=128, tf32=True),
        # A mid-size layer with tensor cores not allowed: fp32 throughout, K and L different.
        dict(name="spmm_gemm_rmat150k_64_32_fp32", op="spmm_gemm", n=150001, nnz=2400016, graph="rmat", K=64, L=32,
             tf32=False),
        # Graph attention on a 100k-vertex graph, the paper's 64/64.
        dict(name="sddmm_spmm_rmat100k_64", op="sddmm_spmm", n=100000, nnz=2000000, graph="rmat", K=64, L=64, tf32=True),
        # The same on a graph of a few thousand vertices (one mini-batch): a few launches long.
        dict(name="sddmm_spmm_rmat3k_64", op="sddmm_spmm", n=3001, nnz=60020, graph="rmat", K=64, L=64, tf32=True),
        # Widths that are not powers of two (feature counts such as 100): the run-time-width kernels.
        dict(name="sddmm_spmm_rmat30k_100_48", op="sddmm_spmm", n=30011, nnz=600220, graph="rmat", K=48, L=100, tf32=True),
        # Attention, aggregation and the weight matrix in one call.
        dict(name="sddmm_spmm_gemm_rmat100k_64", op="sddmm_spmm_gemm", n=100000, nnz=2000000, graph="rmat", K=64, L=64,
             M=64, tf32=True),
        # Hadamard-product gathers over the large graph: two gathered matrices of 512 MB.
        dict(name="spmmh_gemm_rmat1m_128", op="spmmh_gemm", n=1 << 20, nnz=1 << 24, graph="rmat", K=128, L=128, tf32=True),
        # One mode of a CP decomposition, Zipf slice sizes, rank 32.
        dict(name="mttkrp_10k_32", op="mttkrp", d0=10000, d1=10000, d2=10000, nnz=10000000, L=32, tf32=True),
        # A small tensor of odd sizes, rank 16.
        dict(name="mttkrp_300_16", op="mttkrp", d0=301, d1=203, d2=407, nnz=60001, L=16, tf32=True),
        # MTTKRP times a factor matrix on a mid-size tensor, 32/64.
        dict(name="mttkrp_gemm_4k_32_64", op="mttkrp_gemm", d0=4001, d1=3001, d2=5003, nnz=2000003, L=32, M=64, tf32=True),
        # A chain of two tensor-times-matrix products, power-law fibers of mean length 8.
        dict(name="spttm_ttm_5k_64", op="spttm_ttm", d0=5000, d1=5000, d2=5000, nnz=20000000, L=64, M=64, tf32=True),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _width(rng):
    return rng.choice(POW2) if rng.random() < 0.75 else rng.choice(OTHER)


def draw(rng):
    most = work(listed()[7])
    while True:
        op = rng.choice(CSR_OPS + CSF_OPS)
        tf32 = rng.random() < 0.75
        if op in CSR_OPS:
            n = _log_int(rng, 1000, 1 << 20)
            nnz = int(n * min(n / 8, math.exp(rng.uniform(math.log(3), math.log(40)))))
            case = dict(op=op, n=n, nnz=nnz, graph="rmat" if rng.random() < 0.75 else "uniform", K=_width(rng),
                        L=_width(rng), tf32=tf32)
            if op == "sddmm_spmm_gemm":
                case["M"] = _width(rng)
                if rng.random() < 0.6:  # the usual layer: one feature count for both products
                    case["L"] = case["K"]
        else:
            d0, d1, d2 = (_log_int(rng, 150, 10000) for _ in range(3))
            nnz = min(_log_int(rng, 20000, 20000000), d0 * d1 * d2 // 16)
            case = dict(op=op, d0=d0, d1=d1, d2=d2, nnz=nnz, L=_width(rng), tf32=tf32)
            if op != "mttkrp":
                case["M"] = _width(rng)
        if case.get("nnz", 0) < case.get("d0", 0):
            continue
        w = work(case)
        gathered = case["nnz"] * sum(case.get(k, 0) for k in ("K", "L"))
        if w["bytes"] <= most["bytes"] and w["flops"] <= most["flops"] and gathered <= (1 << 24) * 256:
            return case


# ---- inputs ------------------------------------------------------------------------------

def _rand(g, *shape):
    return torch.rand(shape, generator=g, device="cuda")


def _uniform(g, *shape):  # U[-1, 1]
    return torch.rand(shape, generator=g, device="cuda").mul_(2).sub_(1)


def _normal(g, *shape):
    return torch.randn(shape, generator=g, device="cuda")


def _distinct(g, draw_keys, count):
    """`count` distinct sorted int64 keys out of repeated calls of draw_keys(m)."""
    keys = torch.empty(0, dtype=torch.int64, device="cuda")
    while keys.numel() < count:
        keys = torch.unique(torch.cat([keys, draw_keys(int(1.3 * (count - keys.numel())) + 1024)]))
    extra = keys.numel() - count
    if extra:
        keep = torch.randperm(keys.numel(), generator=g, device="cuda")[:count]
        keys = keys[torch.sort(keep).values]
    return keys


def _rmat_keys(g, n, m):
    """Up to m edges (row n + column) of an R-MAT(0.57, 0.19, 0.19, 0.05) graph; endpoints past n are dropped."""
    row = torch.zeros(m, dtype=torch.int64, device="cuda")
    col = torch.zeros(m, dtype=torch.int64, device="cuda")
    for _ in range(max(1, (n - 1).bit_length())):
        u = _rand(g, m)
        down = u >= 0.76
        row = row * 2 + down
        col = col * 2 + (((u >= 0.57) & ~down) | (u >= 0.95))
    ok = (row < n) & (col < n)
    return (row * n + col)[ok]


@functools.lru_cache(maxsize=16)
def _coprimes(n):
    """Numbers below n without a common divisor with it, as a host tensor."""
    x = torch.arange(1, max(n, 2), dtype=torch.int64)
    return x[torch.gcd(x, torch.tensor(n)) == 1]


def _distinct_in(g, lens, dim):
    """For each length, that many distinct sorted values below dim: (parent of each value, value)."""
    lens = lens.to(torch.int64)
    parent = torch.repeat_interleave(torch.arange(lens.numel(), device="cuda"), lens)
    first = torch.cumsum(lens, 0) - lens
    step = torch.arange(parent.numel(), device="cuda") - first[parent]
    strides = _coprimes(dim).cuda()
    a = (_rand(g, lens.numel()).double() * dim).to(torch.int64).clamp_(max=dim - 1)
    b = strides[(_rand(g, lens.numel()).double() * strides.numel()).to(torch.int64).clamp_(max=strides.numel() - 1)]
    keys = torch.sort(parent * dim + (a[parent] + step * b[parent]) % dim).values
    return keys // dim, keys % dim


def _positions(counts):
    pos = torch.zeros(counts.numel() + 1, dtype=torch.int64, device="cuda")
    pos[1:] = torch.cumsum(counts, 0)
    return pos.to(torch.int32)


def _csr(g, case):
    n, nnz = case["n"], case["nnz"]
    if case["graph"] == "rmat":
        keys = _distinct(g, lambda m: _rmat_keys(g, n, m), nnz)
        row, col = keys // n, keys % n
    else:
        lens = torch.full((n,), nnz // n, dtype=torch.int64, device="cuda")
        lens[: nnz % n] += 1
        row, col = _distinct_in(g, lens, n)
    pos = _positions(torch.bincount(row, minlength=n))
    return pos, col.to(torch.int32)


@functools.lru_cache(maxsize=16)
def _zipf_exponent(max_len, mean):
    """Exponent s of the Zipf law on [1, max_len] whose mean is `mean`."""
    x = torch.arange(1, max_len + 1, dtype=torch.float64)
    lo, hi = 0.0, 6.0
    for _ in range(60):
        s = (lo + hi) / 2
        w = x ** -s
        lo, hi = (s, hi) if float((w * x).sum() / w.sum()) > mean else (lo, s)
    return s


def _levels(i, j, fiber_lens):
    """CSF levels of sorted (i, j) pairs and the lengths of their fibers."""
    slices, counts = torch.unique_consecutive(i, return_counts=True)
    pos1 = torch.tensor([0, slices.numel()], dtype=torch.int32, device="cuda")
    return pos1, slices.to(torch.int32), _positions(counts), j.to(torch.int32), _positions(fiber_lens)


def _fibers(case):
    """Stored (i, j) pairs of an <SpTTM,SpTTM> tensor, and their mean length."""
    mean = min(8.0, case["d2"] / 4)
    return min(case["d0"] * case["d1"] // 2, max(1, round(case["nnz"] / mean))), mean


def _csf(g, case):
    d0, d1, d2, nnz = case["d0"], case["d1"], case["d2"], case["nnz"]
    if case["op"] == "spttm_ttm":  # power-law fiber lengths of mean 8 (nnz is their expected sum), distinct uniform j in a slice
        nf, mean = _fibers(case)
        w = torch.arange(1, d2 + 1, dtype=torch.float64, device="cuda") ** -_zipf_exponent(d2, mean)
        cdf = torch.cumsum(w / w.sum(), 0)
        lens = (torch.searchsorted(cdf, _rand(g, nf).double()) + 1).clamp_(max=d2)
        per_slice = torch.full((d0,), nf // d0, dtype=torch.int64, device="cuda")
        per_slice[torch.randperm(d0, generator=g, device="cuda")[: nf % d0]] += 1
        i, j = _distinct_in(g, per_slice, d1)
        _, k = _distinct_in(g, lens, d2)
        return _levels(i, j, lens) + (k.to(torch.int32),)
    # Zipf(1.2) slice sizes in a shuffled order, at least one nonzero each; (j, k) distinct and uniform in a slice
    most = d1 * d2 // 2
    share = torch.arange(1, d0 + 1, dtype=torch.float64, device="cuda") ** -1.2
    sizes = (share / share.sum() * nnz).to(torch.int64).clamp_(1, most)
    spare = nnz - int(sizes.sum())
    if spare > 0:  # what rounding and the bound leave goes to the smaller slices
        room = most - sizes
        add = torch.minimum(room, torch.full_like(room, spare // d0 + 1))
        before = torch.cumsum(add, 0) - add
        sizes += torch.minimum(add, (spare - before).clamp_(min=0))
    sizes = sizes[torch.randperm(d0, generator=g, device="cuda")]
    slice_of = torch.repeat_interleave(torch.arange(d0, device="cuda"), sizes)
    jk = (_rand(g, slice_of.numel()).double() * d1).to(torch.int64).clamp_(max=d1 - 1) * d2
    jk += (_rand(g, slice_of.numel()).double() * d2).to(torch.int64).clamp_(max=d2 - 1)
    keys = torch.unique(slice_of * (d1 * d2) + jk)
    fibers, lens = torch.unique_consecutive(keys // d2, return_counts=True)
    return _levels(fibers // d1, fibers % d1, lens) + ((keys % d2).to(torch.int32),)


def _inputs(case, seed):
    """(index arrays, values, dense operands) of a case, all made on the GPU from the seed."""
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    op, L, M = case["op"], case["L"], case.get("M")
    if op in CSR_OPS:
        index, n, K = _csr(g, case), case["n"], case["K"]
        nnz = index[1].numel()
        if op == "spmm_gemm":
            uni = case["graph"] == "uniform"
            fill = _uniform if uni else _normal
            return index, _uniform(g, nnz), (fill(g, n, K), fill(g, K, L))
        if op == "spmmh_gemm":
            return index, _uniform(g, nnz), (_normal(g, n, K), _normal(g, n, K), _normal(g, K, L))
        ones = torch.ones(nnz, device="cuda")
        if op == "sddmm_spmm":
            return index, ones, (_normal(g, n, L), _normal(g, n, L), _normal(g, n, K))
        return index, ones, (_normal(g, n, K), _normal(g, n, K), _normal(g, n, L), _normal(g, L, M))
    index = _csf(g, case)
    nnz = index[-1].numel()
    d1, d2 = case["d1"], case["d2"]
    if op == "spttm_ttm":
        return index, _uniform(g, nnz), (_normal(g, d2, L), _normal(g, L, M))
    dense = (_uniform(g, d1, L), _uniform(g, d2, L)) + ((_uniform(g, L, M),) if op == "mttkrp_gemm" else ())
    return index, _rand(g, nnz), dense


def prepare(case, seed):
    index, vals, dense = _inputs(case, seed)
    if case["op"] in CSR_OPS:
        B = slnr.DeviceCSR(case["n"], case["n"], index[0], index[1], vals)
    else:
        B = slnr.DeviceCSF3((case["d0"], case["d1"], case["d2"]), *index, vals)
    return getattr(slnr, case["op"]), B, dense, bool(case["tf32"])


def run(state):
    call, B, dense, tf32 = state
    return call(B, *dense, allow_tf32=tf32)


# ---- what a pass cannot do without ---------------------------------------------------------

def work(case):
    op, nnz, L, M = case["op"], case["nnz"], case["L"], case.get("M", 0)
    if op in CSR_OPS:
        n, K = case["n"], case["K"]
        rows = min(n, nnz)
        sparse = 4 * (n + 1) + 8 * nnz
        if op == "spmm_gemm":
            return {"bytes": sparse + 4 * (n * K + K * L + n * L), "flops": 2 * nnz * K + 2 * rows * K * L}
        if op == "spmmh_gemm":
            return {"bytes": sparse + 4 * (2 * n * K + K * L + n * L), "flops": 3 * nnz * K + 2 * rows * K * L}
        if op == "sddmm_spmm":
            return {"bytes": sparse + 4 * (2 * n * L + 2 * n * K), "flops": nnz * (2 * L + 1 + 2 * K)}
        return {"bytes": sparse + 4 * (2 * n * K + n * L + L * M + n * M),
                "flops": nnz * (2 * K + 1 + 2 * L) + 2 * rows * L * M}
    d0, d1, d2 = case["d0"], case["d1"], case["d2"]
    if op == "spttm_ttm":
        fibers = _fibers(case)[0]
        sparse = 8 * nnz + 2 * 8 * fibers + 2 * 8 * d0  # B's levels, and A's copies of the first two
        return {"bytes": sparse + 4 * (d2 * L + L * M + fibers * M), "flops": 2 * nnz * L + 2 * fibers * L * M}
    norm = sum(r ** -1.2 for r in range(1, d0 + 1))
    fibers = int(sum(d1 * -math.expm1(-nnz * r ** -1.2 / norm / d1) for r in range(1, d0 + 1)))  # expected
    sparse = 8 * nnz + 8 * fibers + 8 * d0
    if op == "mttkrp":
        return {"bytes": sparse + 4 * (d1 + d2 + d0) * L, "flops": 2 * (nnz + fibers) * L}
    return {"bytes": sparse + 4 * ((d1 + d2) * L + L * M + d0 * M), "flops": 2 * (nnz + fibers) * L + 2 * d0 * L * M}


def tolerance(case):
    # Measured against 64 bits over the listed and drawn cases: 8e-8 .. 3.3e-7 of the result's norm in fp32 (up to 1e-6
    # is what sums of these lengths show in another order), and 2.9e-4 .. 3.0e-4 where TF32 is allowed and the dense
    # contraction rounds its operands to 11 bits.
    if case["tf32"] and case["op"] in ("spmm_gemm", "spmmh_gemm", "spttm_ttm", "sddmm_spmm_gemm"):
        return {"rel": 1.2e-3, "max": 2e-2}
    return {"rel": 4e-6, "max": 2e-4}


# ---- the same results in 64 bits, plain torch ------------------------------------------------

def _gather_sum(parent, count, width, term):
    """out[parent[p], :] += term(p0, p1)[p - p0, :] in fp64, a block of entries at a time."""
    out = torch.zeros(count, width, dtype=torch.float64, device="cuda")
    block = max(1, (1 << 27) // width)
    for p0 in range(0, parent.numel(), block):
        p1 = min(parent.numel(), p0 + block)
        out.index_add_(0, parent[p0:p1], term(p0, p1))
    return out


def _parents(pos):
    pos = pos.to(torch.int64)
    return torch.repeat_interleave(torch.arange(pos.numel() - 1, device="cuda"), pos[1:] - pos[:-1])


def exact(case, seed):
    op = case["op"]
    index, vals, dense = _inputs(case, seed)
    v = vals.double()[:, None]
    x = [d.double() for d in dense]
    if op in CSR_OPS:
        n, row, col = case["n"], _parents(index[0]), index[1].to(torch.int64)
        if op == "spmm_gemm":
            return _gather_sum(row, n, x[0].shape[1], lambda a, b: v[a:b] * x[0][col[a:b]]) @ x[1]
        if op == "spmmh_gemm":
            return _gather_sum(row, n, x[0].shape[1], lambda a, b: v[a:b] * x[0][col[a:b]] * x[1][col[a:b]]) @ x[2]
        sampled = lambda a, b: v[a:b] * (x[0][row[a:b]] * x[1][col[a:b]]).sum(1, keepdim=True) * x[2][col[a:b]]  # noqa: E731
        t = _gather_sum(row, n, x[2].shape[1], sampled)
        return t if op == "sddmm_spmm" else t @ x[3]
    pos1, crd1, pos2, crd2, pos3, crd3 = index
    fiber, k = _parents(pos3), crd3.to(torch.int64)
    rows = x[0] if op == "spttm_ttm" else x[1]
    t = _gather_sum(fiber, crd2.numel(), rows.shape[1], lambda a, b: v[a:b] * rows[k[a:b]])
    if op == "spttm_ttm":
        return pos1, crd1, pos2, crd2, t @ x[1]
    i, j = crd1.to(torch.int64)[_parents(pos2)], crd2.to(torch.int64)
    u = _gather_sum(i, case["d0"], t.shape[1], lambda a, b: t[a:b] * x[0][j[a:b]])
    return u if op == "mttkrp" else u @ x[2]
