"""GPU parity of the persistent kernels with ten tiles a block, against the CPU
oracle on sampled rows: every accumulator buffer is reused (its barriers' phases
flip), both groups of epilogue warps drain an odd and an even number of tiles,
alternately on narrow N-tiles and by columns on wide ones; and the tiled GEMM at
its full N-tile width, several row tiles a block, with a partial last N-tile."""
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


def packed(rows, cols, f, seed, signed=True, ld=None):
    codes = synth.uniform_ints((rows, cols), 0, 2 ** (f[0] if signed else f[0] - 1), seed)
    return o.pack(codes, f[0], f[1], ld_words=ld or esb.esb_row_words(cols, f[0]))


def epilogue_of(fo, act, scale, residual, rows, cols, seed):
    """The Epilogue of a call and the oracle's keywords for the sampled rows."""
    ep = dict(scale0=scale, bias0=0.05, act=act, alpha_out=0.4, fmt_out=esb.Fmt(*fo))
    if not residual:
        return esb.Epilogue(**ep), lambda idx: {}
    res = packed(rows, cols, fo[:2], seed)
    ep.update(residual=dev_i32(res), res_fmt=esb.Fmt(fo[0], fo[1]), res_scale=0.0625)
    table = np.array([o.image(c, fo[0], fo[1]) for c in range(1 << fo[0])])
    return esb.Epilogue(**ep), lambda idx: dict(res_images=table[o.unpack(res[idx], cols, fo[0])], res_scale=0.0625)


OUTPUTS = [((4, 2, False), esb.ESB_ACT_RELU, False), ((4, 2, True), esb.ESB_ACT_NONE, False), ((4, 2, False), esb.ESB_ACT_RELU, True),
           ((6, 3, False), esb.ESB_ACT_RELU, False), ((5, 2, True), esb.ESB_ACT_NONE, True), ((3, 1, False), esb.ESB_ACT_RELU6, True),
           ((8, 4, False), esb.ESB_ACT_RELU, False)]


def compare(codes, y, idx, acc_o, cols, fo, act, scale, kw):
    yo, co = o.epilogue(acc_o, np.full(cols, scale, np.float32), np.full(cols, 0.05, np.float32), act, 0.4, fo, **kw)
    assert np.array_equal(u32(codes[idx]), o.pack(co, fo[0], fo[1], ld_words=codes.shape[1]))
    if y is not None:
        assert np.array_equal(y[idx].cpu().numpy(), yo)
    assert esb.esb_get_status() == 0


@pytest.mark.parametrize("N", [16, 64, 80, 100])
@pytest.mark.parametrize("fo,act,residual", OUTPUTS)
@pytest.mark.parametrize("want_y", [False, True])
def test_gemm_many_row_tiles(N, fo, act, residual, want_y):
    M, K, f = 128 * (152 * 9 + 77) + 5, 40, (4, 2)
    A, B = packed(M, K, f, 1, signed=False), packed(N, K, f, 2)
    s = 0.004
    ep, kw = epilogue_of(fo, act, s, residual, M, N, 3)
    _, y, codes = esb.esb_gemm(dev_i32(A), esb.Fmt(4, 2, False), dev_i32(B), esb.Fmt(*f), K, ep=ep, want_acc=False, want_y=want_y,
                               want_codes=True)
    # rows of every tile of a few blocks, of the ragged end, and others
    rng = np.random.default_rng(N)
    tiles = np.concatenate([b + 152 * np.arange(9) for b in (0, 76, 77, 151)] + [np.array([1443, 1444])])
    idx = np.unique(np.concatenate([tiles * 128 + rng.integers(0, 128, tiles.size), tiles * 128 + 127, [M - 1, M - 5],
                                    rng.integers(0, M, 2000)]))
    compare(codes, y, idx, o.gemm_i64(A[idx], f, B, f, idx.size, N, K), N, fo, act, s, kw(idx))


def conv_images(n, h, w, c, cout, r, stride, pad, f, fo, act, residual, images, kernel):
    geo = (n, h, w, c, cout, r, r, stride, pad)
    assert esb.esb_conv2d_kernel(*geo, esb.Fmt(*f, False), esb.Fmt(*f), out_b=fo[0]) == kernel
    P, Q = esb.conv_out_hw(h, w, r, r, stride, pad)
    ld = esb.esb_row_words(c, f[0])
    X, W = packed(n * h * w, c, f, 5, signed=False), packed(cout * r * r, c, f, 6)
    s = 0.002
    ep, kw = epilogue_of(fo, act, s, residual, n * P * Q, cout, 7)
    _, _, codes = esb.esb_conv2d_nhwc(dev_i32(X), esb.Fmt(*f, False), dev_i32(W), esb.Fmt(*f), *geo, ep=ep, want_acc=False,
                                      want_codes=True)
    Xi = X.reshape(n, h, w, ld)[images]
    acc = o.conv2d_i64(Xi, f, W.reshape(cout, r, r, ld), f, len(images), *geo[1:]).reshape(-1, cout)
    idx = (np.array(images)[:, None] * P * Q + np.arange(P * Q)).ravel()
    compare(codes, None, idx, acc, cout, fo, act, s, kw(idx))


@pytest.mark.parametrize("cout", [16, 64])
@pytest.mark.parametrize("fo,act,residual", OUTPUTS)
def test_halo_many_tiles(cout, fo, act, residual):
    f = fo[:2] if fo[0] < 7 else (4, 2)
    conv_images(55, 56, 56, 16, cout, 3, 1, 1, f, fo, act, residual, [0, 13, 27, 41, 54], esb.ESB_CONV_KERNEL_HALO)


@pytest.mark.parametrize("cout", [16, 64])
@pytest.mark.parametrize("fo,act,residual", OUTPUTS[:6])
def test_stem_many_tiles(cout, fo, act, residual):
    conv_images(48, 64, 252, 3, cout, 3, 2, 1, fo[:2], fo, act, residual, [0, 23, 24, 47], esb.ESB_CONV_KERNEL_STEM)


@pytest.mark.parametrize("N,f", [(2000, (6, 3)), (2000, (5, 2)), (2000, (3, 1)), (2304, (4, 2)), (2100, (4, 1))])
@pytest.mark.parametrize("residual", [False, True])
def test_tiled_gemm_full_width_tiles(N, f, residual, monkeypatch):
    """19 row tiles by 9 N-tiles of 240 (256) columns: more than the SMs, so the
    width stays, and some blocks take two row tiles."""
    monkeypatch.setenv("ESB_GEMM_TILED_MIN_MACS", "0")
    M, K = 2400, 203
    A, B = packed(M, K, f, 3, signed=False), packed(N, K, f, 4)
    fo, s = (f[0], f[1], False), 0.002 if f[0] < 6 else 0.0002
    ep, kw = epilogue_of(fo, esb.ESB_ACT_RELU, s, residual, M, N, 8)
    ws = torch.empty(esb.esb_gemm_tiled_workspace_bytes(M, N, K), dtype=torch.uint8, device="cuda")
    _, _, codes = esb.esb_gemm(dev_i32(A), esb.Fmt(f[0], f[1], False), dev_i32(B), esb.Fmt(*f), K, ep=ep, want_acc=False,
                               want_codes=True, workspace=ws)
    idx = np.unique(np.concatenate([np.arange(0, M, 41), np.arange(127, M, 128), [M - 1]]))
    compare(codes, None, idx, o.gemm_i64(A[idx], f, B, f, idx.size, N, K), N, fo, esb.ESB_ACT_RELU, s, kw(idx))
