"""GPU parity of convolutions whose pixel rows, filter rows and code widths do
not line up, against the CPU oracle: input rows padded beyond the filter's, and
four-word rows at stride 1 off the halo kernel (whole rows or single words in
the im2col K)."""
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


def packed(rows, cols, f, seed, ld, signed=True):
    codes = synth.uniform_ints((rows, cols), 0, 2 ** (f[0] if signed else f[0] - 1), seed)
    return o.pack(codes, f[0], f[1], ld_words=ld)


def check(X, fx, Wd, W, fw, geo):
    n, h, w, c, cout, r, s, stride, pad = geo
    acc_o = o.conv2d_i64(X.reshape(n, h, w, -1), fx, W.reshape(cout, r, s, -1), fw, *geo).reshape(-1, cout)
    s0 = float(1.0 / max(1.0, np.abs(acc_o).std()))
    fo = (4, 2, False)
    yo, co = o.epilogue(acc_o, np.full(cout, s0, np.float32), np.full(cout, 0.05, np.float32), esb.ESB_ACT_RELU, 0.4, fo)
    ep = esb.Epilogue(scale0=s0, bias0=0.05, act=esb.ESB_ACT_RELU, alpha_out=0.4, fmt_out=esb.Fmt(*fo))
    acc, y, codes = esb.esb_conv2d_nhwc(dev_i32(X), esb.Fmt(*fx, False), Wd, esb.Fmt(*fw), *geo, ep=ep, want_acc=True, want_y=True,
                                        want_codes=True)
    assert np.array_equal(acc.cpu().numpy().astype(np.int64), acc_o)
    assert np.array_equal(y.cpu().numpy(), yo)
    assert np.array_equal(u32(codes), o.pack(co, fo[0], fo[1], ld_words=codes.shape[1]))
    assert esb.esb_get_status() == 0


@pytest.mark.parametrize("f,c,ldx", [((4, 2), 64, 12), ((4, 2), 33, 12), ((5, 2), 54, 16), ((6, 3), 30, 12), ((3, 1), 70, 12),
                                     ((6, 4), 30, 12), ((4, 2), 20, 8)])
@pytest.mark.parametrize("r,stride", [(3, 1), (3, 2), (1, 1)])
def test_input_rows_longer_than_filter_rows(f, c, ldx, r, stride):
    """The words of a pixel past its channels take no part, whatever they hold,
    and no filter word past the last is read: the filters end where other
    codes begin."""
    n, h, w, cout, pad = 2, 9, 11, 24, r // 2
    ldw = esb.esb_row_words(c, f[0])
    X = packed(n * h * w, c, f, 3, ldx, signed=False)
    X[:, (c + 32 // f[0] - 1) // (32 // f[0]):] = 0x5A5A5A5A        # beyond the channels' words
    W = packed(cout * r * r, c, f, 4, ldw)
    guarded = torch.full((cout * r * r + 2, ldw), 0x15151515, dtype=torch.int32, device="cuda")
    guarded[:-2] = dev_i32(W)
    check(X, f, guarded[:-2], W, f, (n, h, w, c, cout, r, r, stride, pad))


@pytest.mark.parametrize("n,h,w,c,cout,r,fx,fw", [
    (1, 6, 140, 3, 24, 3, (4, 2), (4, 2)),           # wider than the halo kernel's tile, few tiles: whole rows
    (3, 200, 210, 3, 16, 3, (4, 2), (4, 2)),         # many tiles: single words
    (3, 200, 210, 3, 16, 3, (6, 3), (6, 3)),
    (3, 200, 210, 10, 16, 3, (4, 2), (4, 2)),        # two words of channels
    (2, 20, 20, 16, 40, 3, (4, 1), (4, 1)),          # too little of the halo tile used
    (2, 20, 20, 3, 40, 5, (5, 2), (5, 2)),
    (2, 7, 7, 6, 16, 5, (3, 1), (3, 1)),
    (1, 24, 200, 3, 96, 11, (4, 2), (4, 2)),         # whole rows would not stay resident
    (1, 24, 200, 9, 96, 11, (4, 2), (4, 2)),
    (2, 19, 21, 3, 24, 3, (8, 5), (8, 5)),           # significand planes
    (2, 19, 21, 5, 24, 3, (6, 4), (5, 2)),
    (2, 19, 21, 3, 24, 3, (4, 2), (6, 3)),           # filters of another width
    (2, 56, 56, 16, 24, 3, (4, 2), (3, 1)),
])
def test_four_word_rows_off_the_halo_kernel(n, h, w, c, cout, r, fx, fw):
    geo = (n, h, w, c, cout, r, r, 1, r // 2)
    assert esb.esb_conv2d_kernel(*geo, esb.Fmt(*fx, False), esb.Fmt(*fw)) in (esb.ESB_CONV_KERNEL_IM2COL, esb.ESB_CONV_KERNEL_STREAMED)
    X = packed(n * h * w, c, fx, 5, esb.esb_row_words(c, fx[0]), signed=False)
    W = packed(cout * r * r, c, fw, 6, esb.esb_row_words(c, fw[0]))
    check(X, fx, dev_i32(W), W, fw, geo)
