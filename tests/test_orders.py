"""Which contraction of A = B.X.D comes first, and that neither order costs a
caller anything: values, precision, time-saving routes and workspace.

D first (X.D once per row of X, then sums of its rows) and row first (T = B.X
row by row on chip, times D) give the same sums in another order.  With TF32
the row kernel rounds T once per segment of at most 128 nonzeros, which D first
does not, so the calls that ran row first keep that order wherever a value could
differ by more than 2e-2 of the result's root mean square.
"""
import ctypes

import numpy as np
import pytest

import _parity as P
import oracle
import workloads as wl

import paper_2205_11622_gb300 as slnr

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def gpu():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    slnr.build()
    slnr.lib()


def csr_of(lens, ncols, seed):
    """Rows of the given lengths: distinct columns a + b t mod ncols, sorted."""
    rng = np.random.default_rng(seed)
    coprime = [b for b in range(1, 200) if np.gcd(b, ncols) == 1]
    crd = [np.sort((int(rng.integers(ncols)) + coprime[int(rng.integers(len(coprime)))] *
                    np.arange(n, dtype=np.int64)) % ncols) for n in lens if n]
    pos = np.concatenate([[0], np.cumsum(lens)]).astype(np.int32)
    crd = np.concatenate(crd or [[]]).astype(np.int32)
    return wl.CSR(len(lens), ncols, pos, crd, wl.uniform(wl.Rng(seed), len(crd), -1, 1))


def csf_of(lens, d2, seed, d1=40):
    """Fibers of the given lengths, d1 of them to a slice."""
    f = csr_of(lens, d2, seed)
    nf = len(lens)
    ns = -(-nf // d1)
    pos2 = np.minimum(np.arange(ns + 1) * d1, nf).astype(np.int32)
    return wl.CSF3((ns, d1, d2), np.array([0, ns], np.int32), np.arange(ns, dtype=np.int32), pos2,
                   (np.arange(nf) % d1).astype(np.int32), f.pos, f.crd, f.vals)


def workload(op, lens, ncols, K, L, seed):
    """The call on rows (or fibers) of the given lengths: gathered width K, output width L."""
    r = wl.Rng(seed + 1)
    n = len(lens)
    if op == "spttm_ttm":
        return wl.Workload("order", op, csf_of(lens, ncols, seed),
                           {"C": wl.normal(r, (ncols, K)), "D": wl.normal(r, (K, L))}, {"L": K, "M": L})
    B = csr_of(lens, ncols, seed)
    if op == "spmm_gemm":
        return wl.Workload("order", op, B, {"C": wl.normal(r, (ncols, K)), "D": wl.normal(r, (K, L))}, {"K": K, "L": L})
    if op == "spmmh_gemm":
        return wl.Workload("order", op, B, {"C": wl.normal(r, (ncols, K)), "D": wl.normal(r, (ncols, K)),
                                            "E": wl.normal(r, (K, L))}, {"J": K, "L": L})
    return wl.Workload("order", op, B, {"C": wl.normal(r, (n, K)), "D": wl.normal(r, (ncols, K)),
                                        "F": wl.normal(r, (ncols, K)), "W": wl.normal(r, (K, L))},
                       {"K": K, "L": K, "M": L})


def tf32(x):
    """x rounded to 10 mantissa bits, halves away from zero."""
    u = np.ascontiguousarray(x, np.float32).view(np.uint32)
    return ((u + np.uint32(0x1000)) & np.uint32(0xFFFFE000)).view(np.float32).astype(np.float64)


def row_first(w):
    """The result with T rounded to tf32 once per segment of 128 nonzeros and D once, sums in fp64."""
    d = w.dense
    pos, crd = (w.B.pos3, w.B.crd3) if w.op == "spttm_ttm" else (w.B.pos, w.B.crd)
    X = d["F"] if w.op == "sddmm_spmm_gemm" else d["C"]
    consumer = {"spmm_gemm": "D", "spttm_ttm": "D", "spmmh_gemm": "E", "sddmm_spmm_gemm": "W"}[w.op]
    v = w.B.vals.astype(np.float64)
    rows = np.repeat(np.arange(len(pos) - 1), np.diff(pos))
    if w.op == "sddmm_spmm_gemm":
        v = v * np.einsum("pk,pk->p", d["C"][rows].astype(np.float64), d["D"][crd].astype(np.float64))
    g = X[crd].astype(np.float64)
    if w.op == "spmmh_gemm":
        g *= d["D"][crd]
    starts = np.concatenate([np.arange(a, b, 128) for a, b in zip(pos[:-1], pos[1:]) if a < b])
    seg = np.add.reduceat(v[:, None] * g, starts, axis=0)
    out = np.zeros((len(pos) - 1, d[consumer].shape[1]))
    np.add.at(out, rows[starts], tf32(seg) @ tf32(d[consumer]))
    return out


# A row (fiber) of 50000 nonzeros among short ones: 200 times the root mean square length, so that D first
# differs by 0.1 and more; the row kernel's own order of fp32 sums moves single roundings, 1e-3 at most.
@pytest.mark.gpu
@pytest.mark.parametrize("op,K,L", [("spmm_gemm", 64, 64), ("spmm_gemm", 128, 128), ("spmmh_gemm", 64, 32),
                                    ("sddmm_spmm_gemm", 64, 64), ("spttm_ttm", 64, 64)])
def test_tf32_values_stay_where_rows_are_long(gpu, op, K, L):
    n, ncols = (3000, 50000) if op == "spttm_ttm" else (132000, 132000)
    lens = np.full(n, 1)
    lens[5] = 50000
    w = workload(op, lens.tolist(), ncols, K, L, 0x51A4 + K)
    got, _ = P.phases(w, allow_tf32=True)
    ref = row_first(w)
    rms = np.sqrt(np.mean(ref ** 2))
    assert np.max(np.abs(got.cpu().numpy() - ref) / np.maximum(rms, np.abs(ref))) <= 5e-3


def csr_bytes(op, nrows, ncols, nnz, sizes, tf32=1):
    """Workspace of the fused call; fibers for spttm_ttm (50 to a slice)."""
    n = ctypes.c_size_t(0)
    if op == "spttm_ttm":
        B = slnr.slnr_csf3()
        B.dim[0], B.dim[1], B.dim[2] = -(-nrows // 50), 50, ncols
        B.nnz, B.nslices, B.nfibers = nnz, B.dim[0], nrows
    else:
        B = slnr.slnr_csr(nrows, ncols, nnz, 0x1000, 0x2000, 0x3000)
    o = slnr.slnr_opts(0, tf32, 0, 0, None, None, 0)
    assert getattr(slnr.lib(), f"slnr_{op}_workspace")(ctypes.byref(B), *sizes, ctypes.byref(o), ctypes.byref(n)) == 0
    return n.value


@pytest.mark.parametrize("op,sizes", [("spmm_gemm", (64, 64)), ("spmm_gemm", (128, 128)), ("spmm_gemm", (256, 64)),
                                      ("sddmm_spmm_gemm", (64, 64, 64))])
def test_tf32_graphs_of_many_rows_go_row_first(op, sizes):
    # the workspace tells the order: D first holds X.D, ncols x L floats
    slnr.build()
    narrow = sizes[0] < 256  # the product rounds to tf32 as well
    for n, first in ((16000, True), (1 << 15, narrow), (1 << 16, narrow), (1 << 17, False), (1 << 20, False)):
        assert (csr_bytes(op, n, n, 16 * n, sizes) >= 4 * n * sizes[-1]) == first, n


@pytest.mark.gpu
@pytest.mark.parametrize("n,K,L", [(131077, 64, 64), (131073, 128, 16), (65539, 256, 32)])
def test_hadamard_product_first_gives_the_same_bits(gpu, n, K, L):
    # 9 nonzeros a row and one long row; the product formed here by torch and gathered by the same kernel
    lens = np.full(n, 9)
    lens[7] = 40000
    w = workload("spmmh_gemm", lens.tolist(), n, K, L, 0x51A4 + n)
    B, d = P.to_device(w)
    got, names = P.phases(w, allow_tf32=True)
    assert names == ["seg_count", "seg_write", "hadamard", "tc_spmm_gemm", "combine"]
    assert torch.equal(got, slnr.spmm_gemm(B, d["C"] * d["D"], d["E"], allow_tf32=True))
    # three nonzeros a column: the products in the kernel's gathers
    few = workload("spmmh_gemm", [3] * n, n, 64, L, 0x51A4 + n)
    B, d = P.to_device(few)
    got, names = P.phases(few, allow_tf32=True)
    if n > 1 << 17:
        assert "tc_spmmh_gemm" in names
        assert torch.equal(got, slnr.spmm_gemm(B, d["C"] * d["D"], d["E"], allow_tf32=True))


@pytest.mark.gpu
@pytest.mark.parametrize("K,L,M", [(32, 64, 64), (16, 16, 16), (64, 64, 16), (128, 64, 128), (100, 64, 64)])
def test_sampled_gemm_stays_fp32_at_widths_without_a_tensor_core_kernel(gpu, K, L, M):
    # TF32 allowed or not: the same bits.  36000 nonzeros: past the size from which the tensor cores are taken
    n = 3000
    B = csr_of([12] * n, n, 0x51A4 + K)
    r = wl.Rng(K + L + M)
    w = wl.Workload("sampled", "sddmm_spmm_gemm", B, {"C": wl.normal(r, (n, K)), "D": wl.normal(r, (n, K)),
                                                      "F": wl.normal(r, (n, L)), "W": wl.normal(r, (L, M))},
                    {"K": K, "L": L, "M": M})
    assert torch.equal(P.phases(w, allow_tf32=True)[0], P.phases(w, allow_tf32=False)[0])


@pytest.mark.parametrize("op,nrows,ncols,nnz,sizes,tf32,first", [
    ("spmm_gemm", 4096, 1 << 20, 1 << 20, (256, 256), 0, False),      # 137 GFLOP for 4096 rows
    ("spmm_gemm", 4096, 1 << 20, 1 << 20, (128, 128), 1, False),
    ("spmm_gemm", 1000, 1000000, 1000000, (64, 64), 0, False),
    ("spmmh_gemm", 4096, 1 << 20, 1 << 20, (128, 128), 1, False),
    ("sddmm_spmm_gemm", 1000, 1000000, 1000000, (1024, 1024, 1024), 0, False),
    ("spttm_ttm", 4096, 1 << 20, 1 << 20, (128, 128), 0, False),      # a long third mode
    ("spmm_gemm", 4096, 16384, 16384 * 8, (64, 64), 0, True),         # few columns more: the sums pay for them
    ("spmm_gemm", 150001, 150001, 2400016, (64, 32), 0, True),
    ("spmm_gemm", 264179, 264179, 4830566, (64, 200), 0, False),      # wider rows, beyond what L2 holds of them
    ("spmm_gemm", 726054, 726054, 11070539, (64, 128), 0, False),
    ("spmmh_gemm", 257990, 257990, 5857089, (128, 200), 0, True),     # one row of 200 for two of 128
    ("sddmm_spmm_gemm", 71509, 71509, 1451041, (32, 32, 64), 1, False),
    ("spttm_ttm", 2500000, 5000, 20000000, (64, 64), 0, True),
])
def test_many_columns_and_wider_rows_go_row_first(op, nrows, ncols, nnz, sizes, tf32, first):
    slnr.build()
    assert (csr_bytes(op, nrows, ncols, nnz, sizes, tf32) >= 4 * ncols * sizes[-1]) == first


class Scarce(slnr.Workspace):
    """A device with room for `most` bytes of workspace."""

    def __init__(self, most):
        super().__init__()
        self.most = most

    def get(self, nbytes):
        if nbytes > self.most:
            raise torch.OutOfMemoryError("no room")
        return super().get(nbytes)


@pytest.mark.gpu
@pytest.mark.parametrize("op,K,L,row_kernel", [("spmm_gemm", 64, 64, "tc_spmm_gemm"), ("spmm_gemm", 100, 48, "w_spmm_gemm_tiles"),
                                               ("spmmh_gemm", 64, 64, "tc_spmmh_gemm"),
                                               ("sddmm_spmm_gemm", 64, 64, "tc_sddmm_spmm_gemm"),
                                               ("spttm_ttm", 64, 64, "tc_spmm_gemm")])
def test_a_workspace_that_holds_row_first_is_enough(gpu, op, K, L, row_kernel):
    n = 20000
    w = workload(op, [5] * n, n if op != "spttm_ttm" else 1000, K, L, 0x51A4 + K)
    B, d = P.to_device(w)
    ref, ref_abs = oracle.get().run(w)
    own = slnr.Workspace()
    small = workload(op, [5] * 100, n if op != "spttm_ttm" else 1000, K, L, 1)
    P.phases(small, workspace=own)
    full, names = P.phases(w, workspace=own)  # a small call's workspace before it: the order is the same
    assert names[-1].startswith("flat_"), names
    rows, names = P.phases(w, workspace=Scarce(own.buf.numel() // 2))
    assert row_kernel in names, names
    for got in (full, rows):
        assert P.rel_err(got.cpu().numpy(), ref, ref_abs) <= P.TOL_TF32
    with pytest.raises(torch.OutOfMemoryError):  # not enough for either
        slnr.run(op, B, d, workspace=Scarce(4096))
    class Fixed:  # a workspace of the caller's own: get() is all that the calls need
        def get(self, nbytes, few=torch.empty(4096, dtype=torch.uint8, device="cuda")):
            return few

    with pytest.raises(slnr.SlnrError) as e:
        slnr.run(op, B, d, workspace=Fixed())
    assert e.value.status == 4


# Rows at the row kernels' edges: 127/128/129 straddle the tensor-core segment length, 255/256/257 the light/heavy
# boundary, 5000 is a long heavy row; runs of short rows fill waves and tiles, the number of rows is ragged.
EDGES = ([127, 128, 129, 255, 256, 257, 5000, 1, 0, 3] + [1, 2, 3, 4, 5, 7, 8, 9, 16, 17] * 130 + [0] * 60 + [64, 65, 33] * 11)


@pytest.mark.gpu
@pytest.mark.parametrize("op,K,L", [
    *(("spmm_gemm", *w) for w in [(16, 16), (16, 256), (32, 32), (32, 128), (64, 16), (64, 64), (128, 64), (128, 128),
                                  (128, 256), (256, 16), (256, 64)]),
    *(("spmmh_gemm", *w) for w in [(16, 64), (32, 16), (64, 64), (128, 128), (128, 256), (256, 32)]),
    *(("sddmm_spmm_gemm", *w) for w in [(32, 32), (32, 128), (64, 64), (128, 32), (128, 128)]),
    *(("spttm_ttm", *w) for w in [(16, 16), (64, 64), (128, 128), (256, 64)])])
def test_tensor_core_row_kernel_edges(gpu, op, K, L):
    w = workload(op, EDGES, 6000, K, L, 0x51A4 + K + L)
    assert w.B.nnz >= 1 << 14
    ref, ref_abs = oracle.get().run(w)
    names = P.check_row_first(w, True, ref, ref_abs, P.TOL_TF32)
    assert ("tc_spmm_gemm" if op == "spttm_ttm" else f"tc_{op}") in names, names


@pytest.mark.gpu
@pytest.mark.parametrize("op,K,L,kernel", [
    ("spmm_gemm", 64, 64, "spmm_gemm_tiles"), ("spmm_gemm", 4, 8, "spmm_gemm_tiles"), ("spmm_gemm", 128, 256, "spmm_gemm_tiles"),
    ("spmm_gemm", 100, 36, "w_spmm_gemm_tiles"), ("spmm_gemm", 512, 64, "w_spmm_gemm_tiles"),
    ("spmmh_gemm", 64, 64, "spmm_gemm_tiles"), ("spmmh_gemm", 36, 100, "w_spmm_gemm_tiles"),
    ("sddmm_spmm_gemm", 64, 64, "sddmm_spmm_gemm_tiles"), ("sddmm_spmm_gemm", 8, 32, "sddmm_spmm_gemm_tiles"),
    ("sddmm_spmm_gemm", 256, 16, "sddmm_spmm_gemm_tiles"), ("sddmm_spmm_gemm", 100, 36, "w_sddmm_spmm_gemm_tiles"),
    ("spttm_ttm", 64, 32, "spmm_gemm_tiles"), ("spttm_ttm", 20, 48, "w_spmm_gemm_tiles")])
def test_fp32_row_kernel_edges(gpu, op, K, L, kernel):
    w = workload(op, EDGES, 6000, K, L, 0x51A4 + K + L)
    ref, ref_abs = oracle.get().run(w)
    names = P.check_row_first(w, False, ref, ref_abs, P.TOL_FP32)
    assert kernel in names, names


@pytest.mark.gpu
@pytest.mark.parametrize("L,K", [(4, 4), (4, 64), (32, 4), (8, 32), (16, 16), (64, 16), (16, 64), (64, 64)])
def test_sddmm_spmm_row_kernel(gpu, L, K):
    # fewer than four nonzeros a row: claims of short rows, of long ones and mixed, chunks of heavy rows
    lens = [5000, 257, 256, 255, 9, 8, 7, 0] + [1, 0, 2, 8, 0, 3, 9, 1] * 600 + [0] * 1001
    rng = np.random.default_rng(L + K)
    lens = np.concatenate([lens[:8], rng.permutation(lens[8:])]).tolist()
    r = wl.Rng(0x51A4 + L + K)
    B = csr_of(lens, 6000, 0x51A4 + L)
    assert B.nnz < 4 * B.nrows
    w = wl.Workload("rows", "sddmm_spmm", B, {"C": wl.uniform(r, (B.nrows, L), -1, 1), "D": wl.uniform(r, (6000, L), -1, 1),
                                              "E": wl.uniform(r, (6000, K), -1, 1)}, {"K": K, "L": L})
    ref, ref_abs = oracle.get().run(w)
    got, names = P.phases(w)
    assert names == ["classify", "sddmm_spmm_rows", "combine"]
    assert P.rel_err(got.cpu().numpy(), ref, ref_abs) <= P.TOL_FP32
