"""The nonzero-window kernels (csrc/flat.cu) at the sizes where they can go
wrong, against the oracle (GPU).

Windows hold a fixed number of consecutive nonzeros, so the edges are: rows
that end or start exactly at a window's end, rows over one, a few and hundreds
of windows, fewer nonzeros than one window, runs of empty rows shorter and
longer than the rows a lane group looks at together, and operands that lie on
16-byte but not 32-byte boundaries.  Errors are in units of the magnitude
companion: a chain of n fp32 operations is off by at most n 2^-24 of it, and no
row here has more than about 10000 of them (6e-4); sums of random signs stay far
below the 1e-4 asked for.
"""
import numpy as np
import pytest

import _parity as P
import oracle
import workloads as wl

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def slnr():
    import paper_2205_11622_gb300 as m
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    m.build()
    m.lib()
    return m


def structure(kind, rng):
    """Row lengths."""
    if kind == "one":                # fewer nonzeros than a window
        return [0, 0, 3, 0]
    if kind == "window_ends":        # rows of 1 .. 128 nonzeros, many ending where a window does
        return [16, 16, 32, 1, 15, 64, 48, 128, 8, 8, 4, 2, 2] * 7 + [5]
    if kind == "long":               # one row over hundreds of windows between short ones
        return [3] * 40 + [9000] + [1] * 50 + [700, 0, 0, 33]
    if kind == "empty_runs":         # runs of empty rows around 1 .. 40 times a lane group's rows
        lens = []
        for n in (1, 7, 8, 9, 31, 33, 70, 130, 300, 1300):
            lens += [int(rng.integers(1, 40))] + [0] * n
        return lens + [2] + [0] * 600
    raise ValueError(kind)


def csr(lens, ncols, rng, seed):
    pos = np.concatenate([[0], np.cumsum(lens)]).astype(np.int32)
    crd = np.concatenate([np.sort(rng.choice(ncols, n, replace=False)) for n in lens if n] or [[]]).astype(np.int32)
    vals = wl.uniform(wl.Rng(seed), len(crd), -1.0, 1.0)
    return wl.CSR(len(lens), ncols, pos, crd, vals)


@pytest.mark.parametrize("L,K", [(64, 64), (4, 8), (8, 12), (16, 16), (20, 48), (32, 32), (100, 48), (128, 96), (256, 200),
                                 (512, 260), (1024, 1024)])
@pytest.mark.parametrize("kind", ["one", "window_ends", "long", "empty_runs"])
def test_sddmm_spmm_windows(slnr, L, K, kind):
    rng = np.random.default_rng(L + K)
    B = csr(structure(kind, rng), 9100, rng, 0x51A4 + L)
    r = wl.Rng(0x51A4 + K)
    dense = {"C": wl.uniform(r, (B.nrows, L), -1, 1), "D": wl.uniform(r, (9100, L), -1, 1),
             "E": wl.uniform(r, (9100, K), -1, 1)}
    w = wl.Workload(kind, "sddmm_spmm", B, dense, {"K": K, "L": L})
    ref, ref_abs = oracle.get().run(w)
    dB, dd = P.to_device(w)
    out = torch.full((B.nrows, K), float("nan"), device="cuda")
    slnr.run(w.op, dB, dd, out=out)
    assert slnr.device_flags() == 0
    assert P.rel_err(out.cpu().numpy(), ref, ref_abs) <= P.TOL_FP32
    # again with every operand 16 bytes past a 32-byte boundary: the 16-byte accesses
    off = {k: shifted(v) for k, v in dd.items()}
    dB.crd, dB.vals = shifted(dB.crd, 1), shifted(dB.vals, 1)
    out2 = shifted(torch.full_like(out, float("nan")))
    slnr.run(w.op, dB, off, out=out2)
    assert P.rel_err(out2.cpu().numpy(), ref, ref_abs) <= P.TOL_FP32


def shifted(t, n=4):
    """A contiguous copy of t that starts n elements into its storage."""
    return torch.cat([t.new_zeros(n), t.reshape(-1)])[n:].view(t.shape)


@pytest.mark.parametrize("J,L", [(8, 8), (16, 4), (32, 16), (24, 20), (64, 64), (128, 96), (256, 256), (512, 300), (36, 36)])
@pytest.mark.parametrize("kind", ["window_ends", "long", "empty_runs"])
@pytest.mark.parametrize("op", ["spmm_gemm", "spmmh_gemm"])
def test_premultiplied_sums(slnr, op, J, L, kind):
    # A = B . (X . D): the contraction once per column of B (both in fp32 and,
    # where the widths allow, with X in two tf32 parts), then sums over windows
    rng = np.random.default_rng(J + L)
    lens = structure(kind, rng)
    ncols = {"empty_runs": 45, "window_ends": 2000, "long": 9100}[kind]
    lens = [min(n, ncols) for n in lens]
    lens += [0] * (ncols - len(lens))  # as many rows as columns: the calls that take the product first
    B = csr(lens, ncols, rng, 0x51A4 + J)
    r = wl.Rng(0x51A4 + 7 * L)
    names = ("C", "D") if op == "spmm_gemm" else ("C", "D", "E")
    dense = {k: wl.uniform(r, (ncols, J), -1, 1) for k in names[:-1]}
    dense[names[-1]] = wl.uniform(r, (J, L), -1, 1)
    w = wl.Workload(kind, op, B, dense, {"K": J, "J": J, "L": L})
    ref, ref_abs = oracle.get().run(w)
    dB, dd = P.to_device(w)
    for tf32 in (False, True):
        out = torch.full((B.nrows, L), float("nan"), device="cuda")
        slnr.timing_enable(True)
        try:
            slnr.run(op, dB, dd, out=out, allow_tf32=tf32)
            names = [n for n, _ in slnr.timing_read()]
        finally:
            slnr.timing_enable(False)
        assert "flat_sum" in names, names
        assert slnr.device_flags() == 0
        assert P.rel_err(out.cpu().numpy(), ref, ref_abs) <= P.tolerance(op, tf32)


@pytest.mark.parametrize("K,L", [(16, 16), (32, 128), (64, 64), (128, 128), (128, 16)])
@pytest.mark.parametrize("two", [False, True])
def test_split_product_error(slnr, K, L, two):
    # X enters the tensor cores as two tf32 parts, so only D's rounding is left:
    # with D exactly representable in tf32 the result is as good as fp32's
    # (2^-22 from the parts and K 2^-24 from the sums, well below 1e-5)
    n = 700
    r = wl.Rng(0x51A4 + K + L)
    B = wl.CSR(n, n, np.arange(n + 1, dtype=np.int32) * 30, np.concatenate(
        [np.sort(np.random.default_rng(i).choice(n, 30, replace=False)) for i in range(n)]).astype(np.int32),
        wl.uniform(r, 30 * n, -1, 1))
    D = np.round(wl.uniform(r, (K, L), -1, 1) * 512).astype(np.float32) / 512
    if two:
        w = wl.Workload("split", "spmmh_gemm", B, {"C": wl.uniform(r, (n, K), -1, 1), "D": wl.uniform(r, (n, K), -1, 1),
                                                   "E": D}, {"J": K, "L": L})
    else:
        w = wl.Workload("split", "spmm_gemm", B, {"C": wl.uniform(r, (n, K), -1, 1), "D": D}, {"K": K, "L": L})
    ref, ref_abs = oracle.get().run(w)
    dB, dd = P.to_device(w)
    out = slnr.run(w.op, dB, dd, allow_tf32=True)
    assert P.rel_err(out.cpu().numpy(), ref, ref_abs) <= 1e-5


@pytest.mark.gpu
@pytest.mark.parametrize("K,L", [(16, 16), (64, 32), (128, 128), (48, 12)])
@pytest.mark.parametrize("runs", [[0], [1, 2], [3, 4, 5, 9], [63, 64, 65, 700], [5000, 0, 0, 70000]])
def test_premultiplied_empty_rows(slnr, K, L, runs):
    # runs of empty rows shorter and longer than the window kernel's steps, also after the last nonzero;
    # fp32 sums of 3 products of K terms: below 1e-5 of the absolute sum
    lens, ncols = [], 120
    for i in range(0, 400 if max(runs) < 1000 else 12):
        lens += [1 + i % 3] + [0] * runs[i % len(runs)]
    lens += [40, 0, 0]
    pos = np.concatenate([[0], np.cumsum(lens)]).astype(np.int32)
    r = wl.Rng(0x51A4 + K + L + len(lens))
    crd = np.concatenate([np.sort(np.random.default_rng(i).choice(ncols, n, replace=False))
                          for i, n in enumerate(lens) if n]).astype(np.int32)
    B = wl.CSR(len(lens), ncols, pos, crd, wl.uniform(r, int(pos[-1]), -1, 1))
    w = wl.Workload("empty", "spmm_gemm", B, {"C": wl.uniform(r, (ncols, K), -1, 1), "D": wl.uniform(r, (K, L), -1, 1)},
                    {"K": K, "L": L})
    ref, ref_abs = oracle.get().run(w)
    dB, dd = P.to_device(w)
    out = slnr.run(w.op, dB, dd, allow_tf32=False).cpu().numpy()
    assert P.rel_err(out, ref, ref_abs) <= 1e-5
    assert not out[np.diff(pos) == 0].any()


def columns_workload(ncols, K, L, two, positive=False):
    """A graph over `ncols` columns with enough nonzeros for the tensor cores (2^14) and for each column."""
    per = min(ncols, 30)
    n = max(20000, ncols + 2000) // per + 1
    r = wl.Rng(0x51A4 + ncols + K + L)
    crd = np.concatenate([np.sort(np.random.default_rng(i).choice(ncols, per, replace=False)) for i in range(n)])
    lo = 0.5 if positive else -1
    # as many rows as columns (the others empty): the calls that take the product first
    pos = np.minimum(np.arange(max(n, ncols) + 1), n).astype(np.int32) * per
    B = wl.CSR(len(pos) - 1, ncols, pos, crd.astype(np.int32), wl.uniform(r, per * n, lo, 1))
    X, X2 = wl.uniform(r, (ncols, K), lo, 1), wl.uniform(r, (ncols, K), lo, 1)
    D = np.round(wl.uniform(r, (K, L), lo, 1) * 512).astype(np.float32) / 512
    if two:
        return wl.Workload("columns", "spmmh_gemm", B, {"C": X, "D": X2, "E": D}, {"J": K, "L": L})
    return wl.Workload("columns", "spmm_gemm", B, {"C": X, "D": D}, {"K": K, "L": L})


@pytest.mark.gpu
@pytest.mark.parametrize("two", [False, True])
@pytest.mark.parametrize("ncols,K,L", [(1, 16, 16), (127, 128, 128), (128, 32, 64), (129, 128, 16), (8 * 30 + 1, 16, 32),
                                       (65000, 128, 128), (40000, 64, 64), (19457, 32, 16)])
def test_split_product_rows(slnr, ncols, K, L, two):
    # one tile, its edges, one tile more than a CTA each, several tiles per CTA; the bound is the one above
    w = columns_workload(ncols, K, L, two)
    ref, ref_abs = oracle.get().run(w)
    dB, dd = P.to_device(w)
    slnr.timing_enable(True)
    try:
        out = slnr.run(w.op, dB, dd, allow_tf32=True)
        names = [n for n, _ in slnr.timing_read()]
    finally:
        slnr.timing_enable(False)
    assert names[0] == "tc_premul", names
    assert P.rel_err(out.cpu().numpy(), ref, ref_abs) <= 1e-5


@pytest.mark.gpu
@pytest.mark.parametrize("where", ["C", "D"])
def test_split_product_infinities(slnr, where):
    # positive values, some exact in tf32 (their second part is zero): an
    # infinity stays one, and reaches the entries that it contributes to
    w = columns_workload(500, 64, 64, False, positive=True)
    w.dense["C"][::2] = 0.5
    w.dense[where][3, 5] = np.inf
    dB, dd = P.to_device(w)
    out = slnr.run(w.op, dB, dd, allow_tf32=True).cpu().numpy()
    if where == "D":
        hit = np.zeros_like(out, dtype=bool)
        hit[:, 5] = True
    else:
        rows = np.array([3 in w.B.crd[w.B.pos[i]:w.B.pos[i + 1]] for i in range(w.B.nrows)])
        hit = np.repeat(rows[:, None], 64, axis=1)
    assert np.array_equal(np.isposinf(out), hit) and np.isfinite(out[~hit]).all()


@pytest.mark.gpu
@pytest.mark.parametrize("two", [False, True])
def test_split_product_largest_values(slnr, two):
    # the largest finite values of X (masks), whose upper part must not round to infinity: D of 2^-12 and zeros keeps
    # every sum finite, and 0 times them is 0
    w = columns_workload(500, 64, 64, two)
    most = np.finfo(np.float32).max
    w.dense["C"][3] = np.where(np.arange(64) % 2, most, -most)
    w.dense["C"][4, 5] = most
    if two:
        w.dense["D"][3:5] = 1
    D = w.dense["E" if two else "D"]
    D[:] = 2.0 ** -12
    D[:, ::3] = 0
    w.B.vals[:] *= 0.5
    ref, ref_abs = oracle.get().run(w)
    dB, dd = P.to_device(w)
    out = slnr.run(w.op, dB, dd, allow_tf32=True).cpu().numpy()
    assert np.isfinite(ref).all() and not out[:, ::3].any()
    assert P.rel_err(out, ref, ref_abs) <= 1e-5


def csf(kind, rng, d1, d2, seed):
    """CSF tensors whose slices and fibers end at window edges, span many windows, or are empty in runs."""
    if kind == "few":            # fewer nonzeros than a window
        shape = [[1, 2], [], [3]]
    elif kind == "long":         # one slice over hundreds of windows, single-nonzero slices around it
        shape = [[1]] * 20 + [list(rng.integers(1, 90, 700))] + [[1, 1]] * 9 + [[64] * 16] + [[32], [32], [64]]
    elif kind == "empty_runs":   # runs of empty slices and of empty fibers, shorter and longer than a step
        shape = []
        for n in (1, 7, 9, 40):
            shape += [[5, 1] + [0] * n + [2]] + [[]] * n
        shape += [[0] * 70 + [3] + [0] * 33, [40]] + [[0, 0]] * 12
    pos2, pos3, crd2, crd3 = [0], [0], [], []
    for s in shape:
        crd2 += sorted(rng.choice(d1, len(s), replace=False).tolist())
        for n in s:
            crd3 += sorted(rng.choice(d2, int(n), replace=False).tolist())
            pos3.append(len(crd3))
        pos2.append(len(crd2))
    d0 = 2 * len(shape) + 5
    crd1 = np.sort(rng.choice(d0, len(shape), replace=False))
    a = lambda x: np.asarray(x, np.int32)  # noqa: E731
    return wl.CSF3((d0, d1, d2), a([0, len(shape)]), a(crd1), a(pos2), a(crd2), a(pos3), a(crd3),
                   wl.uniform(wl.Rng(seed), len(crd3), -1, 1))


@pytest.mark.parametrize("L,M", [(4, 8), (8, 4), (12, 36), (16, 16), (32, 64), (48, 100), (64, 32), (128, 260), (256, 16),
                                 (260, 20), (512, 64), (1024, 12)])
@pytest.mark.parametrize("kind", ["few", "long", "empty_runs"])
def test_mttkrp_windows(slnr, L, M, kind):
    rng = np.random.default_rng(L + M)
    d1, d2 = 900, 120
    B = csf(kind, rng, d1, d2, 0x51A4 + L)
    r = wl.Rng(0x51A4 + M)
    C, D, E = wl.uniform(r, (d1, L), -1, 1), wl.uniform(r, (d2, L), -1, 1), wl.uniform(r, (L, M), -1, 1)
    for op, dense, dims in (("mttkrp", {"C": C, "D": D}, {"L": L}), ("mttkrp_gemm", {"C": C, "D": D, "E": E}, {"L": L, "M": M})):
        w = wl.Workload(kind, op, B, dense, dims)
        ref, ref_abs = oracle.get().run(w)
        dB, dd = P.to_device(w)
        for aligned in (True, False):
            out = torch.full((B.dims[0], M if op == "mttkrp_gemm" else L), float("nan"), device="cuda")
            if not aligned:
                out, dd = shifted(out), {k: shifted(v) for k, v in dd.items()}
            slnr.run(op, dB, dd, out=out)
            assert slnr.device_flags() == 0
            assert P.rel_err(out.cpu().numpy(), ref, ref_abs) <= P.TOL_FP32
