"""Tensor-core gradients at fp32 accuracy (bf16 activations; head dimension 64, or fp32 feature-map weights): ragged last tiles,
runs of tiles that cross units, odd numbers of heads (a last pair without a second head), both layouts, shared weights, Eq. 8,
the rule that hands small problems to the CUDA-core kernels, and the time-out path.

Bounds: dq, dk, dv are rounded to bf16 once, at most 2^-9 of each element (1.953e-3), so that is the bound on their relative
L2 error but for the 2^-17 of their last product.  dW: four products follow one another (logits, dO S^T, dS, x^T du), each of
8 truncated additions of its leading parts (2^-24 each at the accumulator's size then, half of the final one on average):
4 * 8 * 2^-25 = 9.5e-7.
"""
import pytest
import torch

from oracle import ref as oracle
from paper_2510_08318_b200 import linattn, synth
from util import errors

pytestmark = pytest.mark.gpu
TOL_BF16 = 1.98e-3
TOL_DW = 9.5e-7


def inputs(B, H, n, d, weights):
    x = synth.make_inputs(2, B=B, H=H, n=n, d=d)
    g = torch.Generator().manual_seed(n + d)
    if weights == torch.float32:
        x["Wq"], x["Wk"] = (torch.randn(x["Wq"].shape, generator=g) for _ in range(2))
    x["dout"] = torch.randn(B, H, n, d, generator=g).bfloat16()
    x["a"] = (0.02 * torch.randn(B, H, n, d, generator=g)).bfloat16()
    return x


def context(x, per_head=True, layout=0):
    B, H, n, d = x["q"].shape
    ctx = linattn.LinAttn(H, d, max_B=B, max_n=n)
    ctx.set_option(linattn.OPT_LAYOUT, layout)
    W = [x[k] if per_head else x[k][0].contiguous() for k in ("Wq", "Wk")]
    ctx.set_feature_map(W[0].cuda(), W[1].cuda())
    return ctx, W


def on_gpu(t, layout):
    t = t.cuda()
    return t.transpose(1, 2).contiguous().view(t.shape) if layout else t


def back(t, layout):
    B, H, n, d = t.shape
    return (t.view(B, n, H, d).transpose(1, 2) if layout else t).float().cpu().numpy()


def kernels(ctx, fn):
    ctx.set_option(linattn.OPT_PROFILE, 1)
    fn()
    names = [k["name"] for k in ctx.kernel_times()]
    ctx.set_option(linattn.OPT_PROFILE, 0)
    return names


# tiles of 128 tokens over 148 CTAs: fewer tiles than CTAs, a few per CTA with runs that cross units, one row in the last tile
SHAPES = [(1, 3, 1003, 128, torch.float32, 0, True), (2, 2, 769, 128, torch.float32, 1, True), (1, 5, 8193, 128, torch.float32, 0, False),
          (1, 33, 1100, 64, torch.bfloat16, 0, True), (3, 11, 1153, 64, torch.bfloat16, 1, False), (1, 5, 9001, 64, torch.float32, 1, True)]


@pytest.mark.parametrize("B,H,n,d,weights,layout,per_head", SHAPES)
def test_gradients(B, H, n, d, weights, layout, per_head):
    x = inputs(B, H, n, d, weights)
    ctx, W = context(x, per_head, layout)
    args = [on_gpu(x[k], layout) for k in ("q", "k", "v", "dout")]
    assert "qside_bwd_split_tc" in kernels(ctx, lambda: ctx.backward(*args, per_head=per_head))
    got = ctx.backward(*args, per_head=per_head)
    ctx.check()
    assert ctx.last_launch_count() == 7
    S, z = ctx.read_state(B)
    want = oracle.ref_backward(x["q"], x["k"], x["v"], W[0], W[1], x["dout"])
    for name, g, w in zip(("dq", "dk", "dv"), got, want):
        assert errors(back(g, layout), w)[0] <= TOL_BF16, name
    for name, g, w in zip(("dWq", "dWk"), got[3:], want[3:]):
        assert errors(g.cpu().numpy(), w)[0] <= TOL_DW, name
    _, Sr, zr = oracle.ref_linear(x["q"], x["k"], x["v"], W[0], W[1], rows=[0], return_state=True)
    assert errors(S.numpy(), Sr)[0] <= TOL_DW and errors(z.numpy(), zr)[0] <= TOL_DW
    again = ctx.backward(*args, per_head=per_head)
    assert all(torch.equal(a, b) for a, b in zip(got, again))
    ctx.destroy()


@pytest.mark.parametrize("H,n,d,weights", [(3, 1003, 128, torch.float32), (33, 1100, 64, torch.bfloat16)])
def test_gradients_through_mixed_attention(H, n, d, weights):
    x, r = inputs(1, H, n, d, weights), 0.3
    ctx, W = context(x)
    got = ctx.backward_mixed(*[x[k].cuda() for k in ("q", "k", "v", "a")], r, x["dout"].cuda())
    ctx.check()
    want = oracle.ref_backward_mixed(x["q"], x["k"], x["v"], W[0], W[1], x["a"], r, x["dout"])
    for i, (g, w) in enumerate(zip(got, want)):
        # dr is one sum of n H d products with random signs, of which the fp32 sums keep 2^-24 each
        tol = TOL_BF16 if i in (0, 1, 2, 5) else TOL_DW if i < 5 else 1e-5
        assert errors(g.float().cpu().numpy(), w)[0] <= tol, i
    ctx.destroy()


def test_values_with_a_large_mean():
    """dphi(q) = S dnum + dden z cancels where the rows of S / z resemble o: the parts of S must survive that."""
    x = inputs(1, 3, 1003, 128, torch.float32)
    x["v"] = (x["v"].float() + 0.5).bfloat16()
    ctx, W = context(x)
    args = [x[k].cuda() for k in ("q", "k", "v", "dout")]
    got = ctx.backward(*args)
    ctx.set_option(linattn.OPT_PATH, linattn.PATH_SIMT)
    simt = ctx.backward(*args)
    want = oracle.ref_backward(x["q"], x["k"], x["v"], W[0], W[1], x["dout"])
    for g, s, w in zip(got, simt, want):
        assert errors(g.float().cpu().numpy(), w)[0] <= 2 * errors(s.float().cpu().numpy(), w)[0]
    ctx.destroy()


@pytest.mark.parametrize("H,n,d,weights,split", [(1, 2945, 128, torch.float32, True), (1, 2944, 128, torch.float32, False),
                                                 (33, 1023, 64, torch.bfloat16, False), (37, 1024, 64, torch.bfloat16, True)])
def test_rule(H, n, d, weights, split):
    """24 tiles of 128-feature heads; one tile per SM (148) and 1024 tokens for 64-feature heads."""
    x = inputs(1, H, n, d, weights)
    ctx, _ = context(x)
    args = [x[k].cuda() for k in ("q", "k", "v", "dout")]
    assert ("qside_bwd_split_tc" in kernels(ctx, lambda: ctx.backward(*args))) == split
    ctx.set_option(linattn.OPT_PATH, linattn.PATH_TENSOR)
    with pytest.raises(linattn.LinAttnError):   # what needs fp32 accuracy is not what this option asks for
        ctx.backward(*args)
    ctx.destroy()


@pytest.mark.parametrize("side", [2, 3])
def test_a_wait_that_runs_out_is_reported(side):
    """The first tile's logits are never announced: the waits run out, every role unwinds, and the context stays usable."""
    x = inputs(1, 5, 8193, 128, torch.float32)
    ctx, _ = context(x)
    args = [x[k].cuda() for k in ("q", "k", "v", "dout")]
    before = ctx.backward(*args)
    ctx.check()
    ctx.set_option(linattn.OPT_WAIT_LIMIT_US, 1000)
    ctx.set_option(linattn.OPT_TEST_UNMET_ARRIVAL, side)
    ctx.backward(*args)
    with pytest.raises(linattn.LinAttnError) as err:
        ctx.check()
    assert err.value.status == linattn.ERR_TIMEOUT
    ctx.set_option(linattn.OPT_TEST_UNMET_ARRIVAL, 0)
    ctx.set_option(linattn.OPT_WAIT_LIMIT_US, 2000000)
    after = ctx.backward(*args)
    ctx.check()
    assert all(torch.equal(a, b) for a, b in zip(before, after))
    ctx.destroy()
