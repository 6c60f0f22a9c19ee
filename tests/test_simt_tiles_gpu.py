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
