"""Projection of rows that no 16-byte path takes, a thread per short row and a
thread per word of longer ones, at every width, odd strides and alignments;
and the cell table of flat 4-bit rows."""
import numpy as np
import pytest
import torch

import oracle as o
from paper_2109_03513_gb300 import esb, synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    import __graft_entry__
    __graft_entry__.build()


@pytest.mark.parametrize("b,k,signed", [(2, 0, True), (3, 1, False), (4, 2, True), (4, 0, False), (5, 2, True), (6, 5, True),
                                        (7, 3, False), (8, 4, True)])
@pytest.mark.parametrize("rows,cols,ldc_extra,shift", [(1000, 3, 0, 0), (333, 1, 3, 0), (70, 0, 0, 1), (200, 9, 1, 1), (129, 63, 0, 0),
                                                       (5, 1000, 0, 1), (3, 1025, 2, 0), (40, 17, 9, 0),
                                                       (320001, 3, 0, 0),             # several rows a thread: the cell table
                                                       (70, 3, 40, 0), (6001, 3, 40, 0),   # long padding: a thread per word, per row
                                                       (65537, -1, 0, 0), (65535, -1, 1, 0), (300, -1, 1, 1), (300, -2, 1, 0)])
def test_project_any_rows(b, k, signed, rows, cols, ldc_extra, shift):
    cpw = 32 // b
    # the longest short row, the first long one; a word and one code (by rows from 65536 rows on, or at once)
    cols = {0: 2 * cpw, 9: 2 * cpw + 1, -1: cpw + 1, -2: cpw + 5}.get(cols, cols)
    x = synth.normal((rows, cols), seed=rows + cols, std=1.5)
    x[0, 0], x[-1, -1] = float("nan"), -float("inf")
    buf = torch.zeros(rows * cols + 8, dtype=torch.float32, device="cuda")
    xd = buf[shift:shift + rows * cols].view(rows, cols)          # 4-byte aligned only
    xd.copy_(x)
    ldc = esb.esb_row_words(cols, b) + ldc_extra
    out = torch.full((rows, ldc), -1, dtype=torch.int32, device="cuda")
    for alpha in (0.7, 1e-44):                                    # ordinary; thresholds no cell table holds
        esb.esb_project(xd, esb.Fmt(b, k, signed), alpha=alpha, rounding=rows & 1, codes=out, ldc=ldc)
        exp = o.project_packed(x.numpy(), np.float32(alpha), b, k, signed=signed, rounding=rows & 1, ld_words=ldc)
        assert np.array_equal(out.cpu().numpy().view(np.uint32), exp)


@pytest.mark.parametrize("k", [0, 1, 2, 3])
@pytest.mark.parametrize("signed", [True, False])
@pytest.mark.parametrize("alpha", [0.37, 1.0, 3e31, 1e-31, 1e-40])
def test_project_flat_4bit_cell_table(k, signed, alpha):
    """Flat 4-bit projection: every threshold, its neighbours one ulp away,
    zeros, infinities and NaN; alphas whose thresholds leave the table's range
    keep the register search."""
    a = np.float32(alpha)
    q = o.set_nonneg(4, k).astype(np.float64)
    t = (0.5 * (q[1:] + q[:-1]) * float(a)).astype(np.float32)
    bits = t.view(np.uint32).astype(np.int64)
    near = np.concatenate([bits + d for d in range(-3, 4)]).clip(0, 0x7F7FFFFF).astype(np.uint32).view(np.float32)
    x = np.concatenate([near, -near, np.array([0.0, -0.0, np.inf, -np.inf, np.nan, 1e-45, 3e38], np.float32),
                        (synth.normal((3000,), seed=k).numpy() * 4 * a).astype(np.float32)])
    x = np.concatenate([x, np.zeros(-x.size % 128 + 64, np.float32)])[: (x.size + 63) // 8 * 8]
    for rounding in (0, 1):
        codes = esb.esb_project(torch.from_numpy(x).cuda(), esb.Fmt(4, k, signed), alpha=float(a), rounding=rounding, ldc=x.size // 8)
        exp = o.project_packed(x, a, 4, k, signed=signed, rounding=rounding, ld_words=x.size // 8)
        assert np.array_equal(codes.cpu().numpy().view(np.uint32), exp)
