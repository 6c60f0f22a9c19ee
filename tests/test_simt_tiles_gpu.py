"""CUDA-core kernels at the sizes where their token tiles and runs can go wrong: one token, a tile less and more than one
token (16 / 32 tokens in the small form, 64 / 128 and 128 / 256 in the large one), runs of tiles that cross from one (b,h)
pair into another, and the change from the small to the large form.  fp32 storage, so that nothing hides behind rounding.

Tolerance: the kernels and the oracle differ by fp32 rounding only.  A logit is a sum of d <= 128 products, S a sum over n
tokens kept in up to 25 partial sums, o a sum of d products: with random signs each contributes about
sqrt(128) * 2^-25 = 3e-7 of its terms' size, and the outputs are smaller than their terms by up to a factor 3 (zero-mean V).
"""
import pytest
import torch

from oracle import ref as oracle
from paper_2510_08318_b200 import linattn, synth
from util import errors, row_errors

pytestmark = pytest.mark.gpu
TOL = 3e-6


def check(got, want, what):
    rel, _ = errors(got, want)
    worst, idx = row_errors(got, want)
    assert rel <= TOL and worst <= 10 * TOL, f"{what}: rel-L2 {rel:.2e}, worst row {idx} {worst:.2e}"


# (B, H, n): small form, edges of 16 and 32 tokens; then the large form (296 tiles of 64 or 128 tokens on the key side,
# 148 of 128 or 256 on the query side) with runs that cross pairs and ragged last tiles
SHAPES = [(1, 2, 1), (1, 3, 15), (2, 1, 17), (1, 2, 33), (1, 1, 255), (1, 5, 1003), (1, 13, 2945), (2, 3, 6401), (1, 2, 19009)]


@pytest.mark.parametrize("d", [64, 128])
@pytest.mark.parametrize("B,H,n", SHAPES, ids=[f"B{b}H{h}n{n}" for b, h, n in SHAPES])
def test_forward_tiles_and_runs(B, H, n, d):
    x = synth.make_inputs(1, B=B, H=H, n=n, d=d)
    ctx = linattn.LinAttn(H, d, max_B=B, max_n=n)
    ctx.set_feature_map(x["Wq"].cuda(), x["Wk"].cuda())
    out = torch.full((B, H, n, d), float("nan"), device="cuda")
    ctx.forward(x["q"].cuda(), x["k"].cuda(), x["v"].cuda(), out=out)
    ctx.check()
    S, z = ctx.read_state(B)
    want, Sr, zr = oracle.ref_linear(x["q"], x["k"], x["v"], x["Wq"], x["Wk"], return_state=True)
    check(out.cpu().numpy(), want, "out")
    check(S.numpy(), Sr, "S")
    check(z.numpy(), zr, "z")
    ctx.destroy()


@pytest.mark.parametrize("splits", [1, 7, 64])
def test_forced_splits(splits):
    """LINATTN_OPT_SPLITS: the same number of partial sums for every pair, small and large tiles."""
    for n, d in [(777, 128), (5000, 64)]:
        x = synth.make_inputs(1, B=1, H=3, n=n, d=d)
        ctx = linattn.LinAttn(3, d, max_B=1, max_n=n)
        ctx.set_option(linattn.OPT_SPLITS, splits)
        ctx.set_feature_map(x["Wq"].cuda(), x["Wk"].cuda())
        out = ctx.forward(x["q"].cuda(), x["k"].cuda(), x["v"].cuda())
        ctx.check()
        check(out.cpu().numpy(), oracle.ref_linear(x["q"], x["k"], x["v"], x["Wq"], x["Wk"]), f"splits={splits} n={n}")
        ctx.destroy()


# gradients: tiles of 16 / 32 tokens while the large ones (64 / 128) number fewer than 148, then the large form; ragged last
# tiles, runs that cross pairs
BWD_SHAPES = [(1, 2, 2), (1, 3, 15), (2, 1, 17), (1, 2, 33), (2, 3, 777), (1, 3, 3201), (2, 2, 5003)]


@pytest.mark.parametrize("d", [64, 128])
@pytest.mark.parametrize("B,H,n", BWD_SHAPES, ids=[f"B{b}H{h}n{n}" for b, h, n in BWD_SHAPES])
def test_backward_tiles_and_runs(B, H, n, d):
    """A gradient passes through two more products than the output (dphi, then dx or dW): twice the bound."""
    x = synth.make_inputs(1, B=B, H=H, n=n, d=d)
    dout = torch.randn(B, H, n, d, generator=torch.Generator().manual_seed(n))
    want = oracle.ref_backward(x["q"], x["k"], x["v"], x["Wq"], x["Wk"], dout)
    ctx = linattn.LinAttn(H, d, max_B=B, max_n=n)
    ctx.set_feature_map(x["Wq"].cuda(), x["Wk"].cuda())
    args = [x[t].cuda() for t in ("q", "k", "v")] + [dout.cuda()]
    got = ctx.backward(*args)
    ctx.check()
    for name, g, w in zip(("dq", "dk", "dv", "dWq", "dWk"), got, want):
        rel, _ = errors(g.cpu().numpy(), w)
        assert rel <= 2 * TOL, f"{name}: rel-L2 {rel:.2e}"
    again = ctx.backward(*args)
    assert all(torch.equal(a, b) for a, b in zip(got, again))
    ctx.destroy()


@pytest.mark.parametrize("d,n", [(128, 3201), (64, 100)])
def test_shared_weight_gradients_and_other_kernel_function(d, n):
    """One matrix for eleven heads (every slice of the weight-gradient sum takes whole pairs), and the ReLU kernel function's
    gradients, token-major, against the oracle."""
    H = 11
    x = synth.make_inputs(1, B=1, H=H, n=n, d=d)
    dout = torch.randn(1, H, n, d, generator=torch.Generator().manual_seed(n))
    ctx = linattn.LinAttn(H, d, max_B=1, max_n=n)
    ctx.set_feature_map(x["Wq"][0].contiguous().cuda(), x["Wk"][0].contiguous().cuda())
    args = [x[t].cuda() for t in ("q", "k", "v")] + [dout.cuda()]
    got = ctx.backward(*args, per_head=False)
    ctx.check()
    want = oracle.ref_backward(x["q"], x["k"], x["v"], x["Wq"][0], x["Wk"][0], dout)
    for name, g, w in zip(("dq", "dk", "dv", "dWq", "dWk"), got, want):
        assert errors(g.cpu().numpy(), w)[0] <= 2 * TOL, name
    ctx.set_option(linattn.OPT_KERNEL_FUNCTION, linattn.PHI_RELU)
    ctx.set_option(linattn.OPT_LAYOUT, linattn.LAYOUT_BNHD)
    tm = [a.transpose(1, 2).contiguous().view(1, H, n, d) for a in args]
    got = ctx.backward(*tm)
    ctx.check()
    want = oracle.ref_relu_backward(x["q"], x["k"], x["v"], dout)
    for name, g, w in zip(("dq", "dk", "dv"), got, want):
        # a query whose phi meets few keys' divides by a small denominator: the bound on a row grows with 1 / den
        g = g.view(1, n, H, d).transpose(1, 2)
        assert errors(g.cpu().numpy(), w)[0] <= 4 * TOL, name
    ctx.destroy()
