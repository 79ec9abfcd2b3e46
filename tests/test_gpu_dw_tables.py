"""Depthwise 3x3 of 4-bit codes with per-channel scale and bias: the integer
threshold tables (large layers), their refusal by a channel whose scale is
not positive, and the per-element path (small layers), against the oracle."""
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


def dev_i32(a):
    return torch.from_numpy(np.ascontiguousarray(a).view(np.int32)).cuda()


@pytest.mark.parametrize("n,h,w,c,stride", [(8, 57, 55, 20, 1), (20, 41, 43, 36, 2), (1, 9, 9, 200, 1)])
@pytest.mark.parametrize("fo,act", [((4, 2, False), esb.ESB_ACT_RELU6), ((4, 1, False), esb.ESB_ACT_NONE),
                                    ((4, 2, True), esb.ESB_ACT_RELU), ((4, 0, True), esb.ESB_ACT_NONE)])
@pytest.mark.parametrize("odd", ["", "zero", "negative", "nan", "extreme"])
def test_depthwise_per_channel(n, h, w, c, stride, fo, act, odd):
    ldx = esb.esb_row_words(c, 4)
    # every code pattern, so sums reach their bound of 1296
    X = o.pack(synth.uniform_ints((n * h * w, c), 0, 16, 3), 4, 2, ld_words=ldx)
    W = o.pack(synth.uniform_ints((9, c), 0, 16, 4), 4, 2, ld_words=ldx)
    rng = np.random.default_rng(c)
    sc = (0.002 + 0.02 * rng.random(c)).astype(np.float32)
    bi = rng.standard_normal(c).astype(np.float32)
    if odd == "zero":
        sc[c // 2] = 0.0
    elif odd == "negative":
        sc[c // 3] = -0.01
    elif odd == "nan":
        bi[c // 4] = np.nan
    elif odd == "extreme":                            # thresholds out of reach, cancellation, overflow to infinity
        sc[0], bi[0] = 1e-30, 0.3
        sc[1], bi[1] = 3e38, -1e38
        sc[2], bi[2] = 1e-6, 1e6
        sc[3], bi[3] = 1e-6, -1e6
    ep = esb.Epilogue(scale=torch.from_numpy(sc).cuda(), bias=torch.from_numpy(bi).cuda(), act=act, alpha_out=0.61, fmt_out=esb.Fmt(*fo))
    _, _, codes = esb.esb_conv2d_nhwc(dev_i32(X), esb.Fmt(4, 2), dev_i32(W), esb.Fmt(4, 2), n, h, w, c, c, 3, 3, stride, 1,
                                      groups=c, ep=ep, want_acc=False, want_codes=True)
    acc = o.dwconv_i64(X.reshape(n, h, w, ldx), (4, 2), W.reshape(3, 3, -1), (4, 2), n, h, w, c, 3, 3, stride, 1).reshape(-1, c)
    with np.errstate(all="ignore"):
        _, co = o.epilogue(acc, sc, bi, act, 0.61, fo)
    assert np.array_equal(codes.cpu().numpy().view(np.uint32), o.pack(co, 4, fo[1], ld_words=codes.shape[1]))
