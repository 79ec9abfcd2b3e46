"""GPU parity of the strided few-channel convolution (first layers) against
the CPU oracle: every channel count, strides 2 and 4, filters that span one
or two chunk pairs, odd sizes, several column segments, tiles that cross
images, every code width and mixed widths, each epilogue."""
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


CASES = [
    # n, h, w, c, cout, r, s, stride, pad, fx, fw
    (2, 23, 64, 3, 64, 7, 7, 2, 3, (4, 2), (4, 2)),
    (64, 13, 66, 3, 32, 3, 3, 2, 1, (4, 2), (4, 2)),          # about three tiles per block, across images
    (1, 40, 227, 3, 96, 11, 11, 4, 2, (4, 1), (4, 1)),        # two chunk pairs per filter row, stride 4
    (1, 9, 601, 1, 24, 5, 5, 2, 2, (5, 2), (5, 2)),           # three column segments, one channel
    (2, 11, 75, 2, 40, 3, 9, 2, 0, (6, 3), (6, 3)),           # nine taps a row, no padding
    (3, 17, 90, 4, 70, 3, 3, 2, 2, (3, 1), (3, 1)),           # four channels, ragged N
    (1, 30, 130, 3, 300, 7, 7, 2, 3, (2, 0), (2, 0)),         # two N-tiles
    (1, 12, 70, 3, 16, 2, 2, 2, 0, (7, 3), (4, 2)),           # mixed widths, even filter
    (2, 15, 257, 3, 48, 4, 1, 4, 0, (4, 3), (5, 1)),
    (1, 8, 52, 3, 8, 8, 8, 2, 7, (4, 0), (6, 2)),             # padding of seven
    (40, 9, 252, 3, 64, 7, 7, 2, 3, (4, 2), (4, 2)),          # full tile rows, two tiles a block
]


@pytest.mark.parametrize("n,h,w,c,cout,r,s,stride,pad,fx,fw", CASES)
def test_stem_convolution_matches_oracle(n, h, w, c, cout, r, s, stride, pad, fx, fw):
    check(n, h, w, c, cout, r, s, stride, pad, fx, fw, esb.ESB_CONV_KERNEL_STEM)


@pytest.mark.parametrize("n,h,w,c,cout,r,s,stride,pad,fx,fw", [
    (40, 51, 51, 3, 287, 2, 2, 2, 1, (3, 0), (3, 0)),         # a fifth of the tile rows used, a costly epilogue
    (60, 40, 40, 3, 64, 3, 3, 2, 1, (2, 1), (2, 1)),
    (60, 31, 31, 2, 40, 3, 3, 2, 1, (6, 3), (6, 3)),
    (200, 40, 20, 4, 64, 3, 3, 4, 1, (4, 2), (4, 2)),
])
def test_strided_layers_left_to_im2col_match_oracle(n, h, w, c, cout, r, s, stride, pad, fx, fw):
    check(n, h, w, c, cout, r, s, stride, pad, fx, fw, esb.ESB_CONV_KERNEL_IM2COL)


def check(n, h, w, c, cout, r, s, stride, pad, fx, fw, kernel):
    signed_x = (n + h) % 2 == 0
    assert esb.esb_conv2d_kernel(n, h, w, c, cout, r, s, stride, pad, esb.Fmt(*fx, signed_x), esb.Fmt(*fw), out_b=fx[0]) == kernel
    x = (synth.normal if signed_x else synth.half_normal)((n * h * w, c), seed=h + c).numpy()
    wt = synth.he_normal((cout * r * s, c), fan_in=r * s * c, seed=cout + r).numpy()
    ax, _ = o.calibrate(x, *fx, signed_x)
    aw, _ = o.calibrate(wt, *fw, True)
    ldx, ldw = esb.esb_row_words(c, fx[0]), esb.esb_row_words(c, fw[0])
    X = o.project_packed(x, ax, *fx, signed_x, ld_words=ldx)
    W = o.project_packed(wt, aw, *fw, True, ld_words=ldw)
    acc_o = o.conv2d_i64(X.reshape(n, h, w, ldx), fx, W.reshape(cout, r, s, ldw), fw, n, h, w, c, cout, r, s, stride,
                         pad).reshape(-1, cout)
    s0 = esb.esb_dequant_scale(ax, esb.Fmt(*fx), aw, esb.Fmt(*fw))
    Xd, Wd = dev_i32(X), dev_i32(W)
    fx_, fw_ = esb.Fmt(*fx, signed_x), esb.Fmt(*fw)
    geo = (n, h, w, c, cout, r, s, stride, pad)
    for act, fo in ((esb.ESB_ACT_RELU, (fx[0], fx[1], False)), (esb.ESB_ACT_NONE, (4, 2, True)), (esb.ESB_ACT_RELU6, (4, 2, False))):
        yo, co = o.epilogue(acc_o, np.full(cout, s0, np.float32), np.full(cout, 0.05, np.float32), act, 0.6, fo)
        ep = esb.Epilogue(scale0=s0, bias0=0.05, act=act, alpha_out=0.6, fmt_out=esb.Fmt(*fo))
        _, _, codes = esb.esb_conv2d_nhwc(Xd, fx_, Wd, fw_, *geo, ep=ep, want_acc=False, want_codes=True)
        assert np.array_equal(u32(codes), o.pack(co, fo[0], fo[1], ld_words=codes.shape[1]))
    acc, y, _ = esb.esb_conv2d_nhwc(Xd, fx_, Wd, fw_, *geo, ep=ep, want_acc=True, want_y=True)
    assert np.array_equal(acc.cpu().numpy().astype(np.int64), acc_o)
    assert np.array_equal(y.cpu().numpy(), yo)
    assert esb.esb_get_status() == 0
