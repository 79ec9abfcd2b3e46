"""GPU parity of the 3-, 5- and 6-bit paths against the CPU oracle at the
sizes where they can go wrong: the cell-table epilogue (passes of 20 or 24
columns, ragged N, residuals, per-channel scales, thresholds no table can
hold) and the tiled GEMM's packed operand runs (48 or 80 codes)."""
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


def u32(t):
    return t.cpu().numpy().view(np.uint32)


def dev_i32(a):
    return torch.from_numpy(np.ascontiguousarray(a).view(np.int32)).cuda()


def random_codes(rows, cols, b, seed, signed=True):
    codes = synth.uniform_ints((rows, cols), 0, 2 ** b, seed)
    return codes if signed else codes & np.uint32((1 << (b - 1)) - 1)


def packed(rows, cols, f, seed, signed=True):
    return o.pack(random_codes(rows, cols, f[0], seed, signed), f[0], f[1], ld_words=esb.esb_row_words(cols, f[0]))


@pytest.mark.parametrize("N,fo,act,per_channel,residual,alpha_out", [
    (5, (6, 3, False), esb.ESB_ACT_RELU, False, False, 0.31),       # one word
    (20, (6, 2, True), esb.ESB_ACT_NONE, True, False, 0.4),         # one whole pass
    (23, (5, 2, False), esb.ESB_ACT_RELU6, True, True, 0.3),        # one column short of a pass
    (25, (5, 2, True), esb.ESB_ACT_NONE, False, True, 0.5),         # one column past a pass
    (96, (5, 1, True), esb.ESB_ACT_RELU, False, True, 0.2),
    (144, (3, 1, False), esb.ESB_ACT_RELU, True, True, 0.9),
    (250, (3, 0, True), esb.ESB_ACT_NONE, False, True, 1.1),
    (333, (6, 3, False), esb.ESB_ACT_RELU, False, True, 0.3),       # several N-tiles
    (70, (6, 4, True), esb.ESB_ACT_NONE, False, False, 0.6),        # more cells than the table holds: bisection
    (48, (5, 2, False), esb.ESB_ACT_RELU, False, False, 1e-44),     # subnormal thresholds: bisection
])
@pytest.mark.parametrize("ldo_extra", [0, 3])
def test_cell_table_epilogue(N, fo, act, per_channel, residual, alpha_out, ldo_extra):
    M, K = 200, 96
    A, B = packed(M, K, (4, 2), 1, signed=False), packed(N, K, (4, 2), 2)
    rng = np.random.default_rng(N)
    sc = (0.01 + 0.01 * rng.random(N)).astype(np.float32) if per_channel else np.full(N, 0.0123, np.float32)
    bi = (rng.standard_normal(N) * 0.3).astype(np.float32) if per_channel else np.full(N, -0.02, np.float32)
    ep = dict(scale0=0.0123, bias0=-0.02, act=act, alpha_out=alpha_out, fmt_out=esb.Fmt(*fo))
    if per_channel:
        ep.update(scale=torch.from_numpy(sc).cuda(), bias=torch.from_numpy(bi).cuda())
    img, kw = None, {}
    if residual:
        res = packed(M, N, fo[:2], 9)
        ep.update(residual=dev_i32(res), res_fmt=esb.Fmt(fo[0], fo[1]), res_scale=0.0625)
        img = np.vectorize(lambda c: o.image(int(c), fo[0], fo[1]))(o.unpack(res, N, fo[0]))
        kw = dict(res_images=img, res_scale=0.0625)
    ldo = esb.esb_row_words(N, fo[0]) + ldo_extra
    out = torch.full((M, ldo), -1, dtype=torch.int32, device="cuda")
    esb.esb_gemm(dev_i32(A), esb.Fmt(4, 2, False), dev_i32(B), esb.Fmt(4, 2), K, ep=esb.Epilogue(**ep), want_acc=False,
                 out_codes=out)
    acc = o.gemm_i64(A, (4, 2), B, (4, 2), M, N, K)
    _, co = o.epilogue(acc, sc, bi, act, alpha_out, fo, **kw)
    assert np.array_equal(u32(out), o.pack(co, fo[0], fo[1], ld_words=ldo))


@pytest.mark.parametrize("M,N,K,f", [
    # few row tiles: N-tiles of 80 columns (96 for 5-bit codes); the full width is in test_gpu_many_tiles.py
    (130, 256, 80, (6, 3)),         # one run, no tail; four N-tiles, the last of 16 columns
    (1, 300, 81, (6, 2)),           # one code past a run
    (200, 481, 47, (5, 2)),         # tail only; six N-tiles, the last of one column
    (129, 260, 1000, (5, 2)),
    (64, 512, 560, (3, 1)),         # whole runs
    (150, 270, 159, (3, 0)),
])
def test_tiled_gemm_packed_widths(M, N, K, f, monkeypatch):
    monkeypatch.setenv("ESB_GEMM_TILED_MIN_MACS", "0")
    A, B = packed(M, K, f, 3, signed=False), packed(N, K, f, 4)
    ws = torch.full((esb.esb_gemm_tiled_workspace_bytes(M, N, K) + 64,), 0x7F, dtype=torch.uint8, device="cuda")
    fo = (f[0], f[1], False)
    acc_o = o.gemm_i64(A, f, B, f, M, N, K)
    s = float(1.0 / max(1.0, np.abs(acc_o).std()))
    want = o.epilogue(acc_o, np.full(N, s, np.float32), np.full(N, 0.05, np.float32), esb.ESB_ACT_RELU, 0.4, fo)
    ep = esb.Epilogue(scale0=s, bias0=0.05, act=esb.ESB_ACT_RELU, alpha_out=0.4, fmt_out=esb.Fmt(*fo))
    Ad, Bd = dev_i32(A), dev_i32(B)
    for full in (False, True):                        # codes only, then every output
        acc, y, codes = esb.esb_gemm(Ad, esb.Fmt(f[0], f[1], False), Bd, esb.Fmt(*f), K, ep=ep, want_acc=full, want_y=full,
                                     want_codes=True, workspace=ws[:-64])
        assert np.array_equal(u32(codes), o.pack(want[1], fo[0], fo[1], ld_words=codes.shape[1]))
        if full:
            assert np.array_equal(acc.cpu().numpy().astype(np.int64), acc_o)
            assert np.array_equal(y.cpu().numpy(), want[0])
    assert bool((ws[-64:] == 0x7F).all())             # nothing written past the stated size
    # too little workspace: served by esb_gemm's kernels, as before
    _, _, codes = esb.esb_gemm(Ad, esb.Fmt(f[0], f[1], False), Bd, esb.Fmt(*f), K, ep=ep, want_acc=False, want_codes=True,
                               workspace=ws[:16])
    assert np.array_equal(u32(codes), o.pack(want[1], fo[0], fo[1], ld_words=codes.shape[1]))


@pytest.mark.parametrize("n,h,w,c,cout", [(1, 7, 9, 64, 40), (3, 17, 5, 24, 16), (2, 16, 8, 160, 96), (1, 1, 1, 32, 8)])
@pytest.mark.parametrize("f", [(4, 2), (5, 2), (3, 1)])
def test_pointwise_convolution_tiles_cross_rows_and_images(n, h, w, c, cout, f):
    """1x1 filters on tiles of 128 consecutive pixels: ragged last tile, one
    and several channel blocks, residual added."""
    X, W = packed(n * h * w, c, f, 5, signed=False), packed(cout, c, f, 6)
    res = packed(n * h * w, cout, f, 7)
    fo = (f[0], f[1], True)
    ep = esb.Epilogue(scale0=0.003, bias0=0.1, residual=dev_i32(res), res_fmt=esb.Fmt(*f), res_scale=0.05, alpha_out=0.5,
                      fmt_out=esb.Fmt(*fo))
    _, _, codes = esb.esb_conv2d_nhwc(dev_i32(X), esb.Fmt(f[0], f[1], False), dev_i32(W), esb.Fmt(*f), n, h, w, c, cout, 1, 1,
                                      1, 0, ep=ep, want_acc=False, want_codes=True)
    acc = o.gemm_i64(X, f, W, f, n * h * w, cout, c)
    img = np.vectorize(lambda v: o.image(int(v), *f))(o.unpack(res, cout, f[0]))
    _, co = o.epilogue(acc, np.full(cout, 0.003, np.float32), np.full(cout, 0.1, np.float32), esb.ESB_ACT_NONE, 0.5, fo,
                       res_images=img, res_scale=0.05)
    assert np.array_equal(u32(codes), o.pack(co, fo[0], fo[1], ld_words=codes.shape[1]))
