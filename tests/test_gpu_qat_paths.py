"""The training kernels at the edges of their paths: every width of
dn_project (flat 4-bit granules, a thread per word by thresholds on |x - mu| or
by division, a sigma no threshold can stand for), and dn_backward where fp32 pairs cannot carry
the values (infinities, underflow, constant inputs) or pointers are not
16-byte aligned."""
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


# the last: more words than the wide formats divide for
@pytest.mark.parametrize("rows,cols", [(1, 8), (37, 24), (5, 136), (3, 1), (2, 331), (80001, 16)])
@pytest.mark.parametrize("fmt", [(2, 0, True), (3, 1, True), (4, 2, True), (4, 1, False), (5, 2, True), (6, 5, True),
                                 (7, 3, True), (8, 4, False)])
@pytest.mark.parametrize("sigma", [1.7, 0.0, float("inf"), float("nan")])
def test_dn_project_widths(rows, cols, fmt, sigma):
    x = synth.normal((rows, cols), seed=rows + cols, mean=0.3, std=2.0)
    x[0, 0] = float("inf")
    if cols > 2:
        x[-1, 1], x[-1, 2] = float("nan"), -float("inf")
    st = torch.tensor([0.3, sigma], dtype=torch.float64, device="cuda")
    codes, xq = esb.esb_dn_project(x.cuda(), st, esb.Fmt(*fmt), rounding=rows & 1)
    a = float(np.float32(esb.esb_alpha_star(fmt[0], fmt[1])[0]))
    with np.errstate(all="ignore"):
        co, xqo = o.dn_project(x.numpy(), 0.3, sigma, a, *fmt, rounding=rows & 1)
    assert np.array_equal(codes.cpu().numpy().view(np.uint32), o.pack(co.reshape(rows, cols), fmt[0], fmt[1], ld_words=codes.shape[1]))
    assert np.array_equal(xq.cpu().numpy().ravel(), xqo)


@pytest.mark.parametrize("n,shift", [(1, 0), (3, 0), (4097, 0), (70001, 1)])
@pytest.mark.parametrize("kind", ["ordinary", "small", "tiny", "huge", "inf", "zero", "mean"])
def test_dn_backward_ranges(n, shift, kind):
    """Against fp64: one rounding to fp32 (2^-24 relative), plus 2^-40 of the two
    terms that are subtracted and of the mean's term.  The pairs carry some 46
    bits (their low parts are plain fp32 sums), fewer than fp64's 53, and x - mu
    loses those of mu / sigma (13 at a mean of 1e4, where c is small against g)."""
    x = synth.normal((n + shift,), seed=n, mean=0.4, std=1.3)
    g = synth.normal((n + shift,), seed=n + 1)
    if kind == "small":
        g = g * 1e-22
    elif kind == "tiny":
        g = g * 1e-36
    elif kind == "huge":
        g, x = g * 1e30, x * 1e25
    elif kind == "inf":
        g[n // 2 + shift] = float("inf")
    elif kind == "zero":
        g.zero_()
    elif kind == "mean":
        x = x + 1e4
    xd, gd = x.cuda()[shift:], g.cuda()[shift:]
    xc, gc = x[shift:].double(), g[shift:].double()
    mu, sg = float(xc.mean()), float((xc - xc.mean()).square().mean().sqrt())
    st = torch.tensor([mu, sg], dtype=torch.float64, device="cuda")
    got = esb.esb_dn_backward(gd, xd, st).cpu().double()
    s = sg + 1e-7
    t1, c = (gc - gc.mean()) / s, xc - mu
    t2 = c * ((gc * c).sum() / (n * sg * s * s)) if sg > 0 else torch.zeros_like(c)
    exp = t1 - t2
    if kind == "inf":
        assert torch.equal(torch.isfinite(got), torch.isfinite(exp)) and torch.equal(torch.isnan(got), torch.isnan(exp))
        return
    mean_err = 2.0 ** -40 * float(gc.abs().mean()) / s
    tol = 2.0 ** -24 * exp.abs() + 2.0 ** -40 * (t1.abs() + t2.abs()) + mean_err + 2.0 ** -149
    assert bool(((got - exp).abs() <= tol).all())


@pytest.mark.parametrize("n", [5, 4097, 70001])
@pytest.mark.parametrize("kind", ["g", "gx"])
def test_dn_backward_sums_that_overflow_between_lanes(n, kind):
    """Every lane's own sum is finite in fp32 but a warp's is not: the sum of
    g (constant 2e37), or only that of g (x - mu) (g = 1e37 (x - mu) alternating
    in sign, so that g itself sums to about zero)."""
    x = synth.normal((n,), seed=n, mean=0.4, std=1.3)
    if kind == "g":
        g = torch.full((n,), 2e37)
    else:
        x = 0.4 + 1.3 * (1.0 - 2.0 * (torch.arange(n) % 2)).float()
        g = 1e37 * (x - 0.4)
    xc, gc = x.double(), g.double()
    mu, sg = float(xc.mean()), float((xc - xc.mean()).square().mean().sqrt())
    got = esb.esb_dn_backward(g.cuda(), x.cuda(), torch.tensor([mu, sg], dtype=torch.float64, device="cuda")).cpu().double()
    s, c = sg + 1e-7, xc - mu
    t1, t2 = (gc - gc.mean()) / s, c * ((gc * c).sum() / (n * sg * s * s))
    # recomputed in fp64: the sums are trees of some 30 levels (2^-48 of the magnitudes summed), and
    # |x - mu| is at most about 4 sigma
    tol = 2.0 ** -24 * (t1 - t2).abs() + 2.0 ** -44 * (t1.abs() + t2.abs() + float(gc.abs().mean()) / s)
    assert bool(((got - (t1 - t2)).abs() <= tol).all())


@pytest.mark.parametrize("mu,sigma", [(0.0, float("nan")), (float("nan"), 1.0), (float("nan"), 0.0), (0.5, float("inf")), (0.5, 0.0)])
def test_dn_backward_of_no_gradient(mu, sigma):
    """A gradient of zeros is zero, but NaN where the statistics or x make the fp64 expression so."""
    x = torch.tensor([0.5, -1.0, float("inf"), float("nan"), 3.0])
    g = torch.zeros(5)
    st = torch.tensor([mu, sigma], dtype=torch.float64)
    got = esb.esb_dn_backward(g.cuda(), x.cuda(), st.cuda()).cpu().double()
    c, s = x.double() - mu, sigma + 1e-7
    k2 = float((g.double() * c).sum()) / (5 * sigma * s * s) if sigma > 0 else 0.0
    assert torch.equal(got.isnan(), ((g.double() - 0.0) / s - c * k2).isnan()) and bool((got[~got.isnan()] == 0).all())
