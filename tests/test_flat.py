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
