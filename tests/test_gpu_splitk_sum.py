"""Few output tiles of a long reduction: K ranges on every CTA pair, their fp32 partials added by a second kernel.

Against the fp64 product of the same operands.  Bound: a bf16 result is off by half an ulp (at most 2^-8 relative).  Each of the
fp32 additions is off by at most 2^-23 of a partial sum (the adder truncates), itself about sqrt(K) of a term where signs are
random; the sum of |terms| is about K of a term, so the errors add up to about 2^-23 of it: four times that.  (A dropped stage of
64 terms at K = 8192 is some sqrt(64) / 8192 = 2^-10 of it.)
"""
import gc

import pytest
import torch

from paper_2409_09099_b200 import binding as B
from paper_2409_09099_b200.layer import SsteLinear

pytestmark = pytest.mark.gpu


@pytest.fixture(autouse=True)
def give_memory_back():
    yield
    gc.collect()


def _close(got, a, b):
    ref, mag = a.double() @ b.double(), a.double().abs() @ b.double().abs()
    bound = ref.abs() * 2.0 ** -8 + mag * 2.0 ** -21 + 1e-30
    assert bool(((got.double() - ref).abs() <= bound).all())


# (O, I, T): which product has the long reduction, with a ragged 256-row tile, a ragged last column tile, several tiles,
# and an odd number of stages; the last one has all three products split
SHAPES = [(128, 8192, 128), (384, 6400, 128), (128, 5248, 640), (8192, 128, 128), (4992, 384, 384), (128, 128, 8192),
          (384, 640, 4992), (2048, 2048, 128)]


@pytest.mark.parametrize("shape", SHAPES)
@pytest.mark.parametrize("fp8", [False, True])
def test_products_and_layer(shape, fp8):
    O, I, T = shape
    dt = B.E4M3 if fp8 else B.BF16
    ctx = B.Context(0)
    gen = torch.Generator(device="cuda").manual_seed(O + I + T)
    mk = lambda r, c, s: torch.empty((r, c), dtype=torch.bfloat16, device="cuda").normal_(0.0, s, generator=gen)
    W, X, dY = mk(O, I, 0.02), mk(T, I, 1.0), mk(T, O, 1e-2)
    lin = SsteLinear(ctx, W, T, tensor_id=1, seed=3, fp8=fp8)
    lin.init_beta()
    lin.prune()
    Y = lin.forward(X).clone()
    dX, dW = (t.clone() for t in lin.backward(dY))
    # the same operands through the single calls: same ranges or others, so equal up to the order of the fp32 sums
    amax = lin._amax
    y_amax = torch.zeros(1, dtype=torch.float32, device="cuda")
    Y1, dW1, dX1 = torch.empty_like(Y), torch.empty_like(dW), torch.empty_like(dX)
    Xop, Gop = (lin.Xq, lin.dYq) if fp8 else (X, dY)
    ctx.linear_fwd(Xop, lin.vals, lin.meta, Y1, x_amax_dev=amax(0), w_amax_dev=amax(1), y_amax_out_dev=y_amax)
    ctx.linear_bwd_weight(lin.gvals, lin.gmeta, Xop, dW1, g_amax_dev=amax(2), x_amax_dev=amax(0))
    ctx.linear_bwd_input(Gop, lin.w_dense, dX1, g_amax_dev=amax(2), w_amax_dev=amax(1))
    torch.cuda.synchronize()
    assert torch.equal(Y, Y1) and float(y_amax) == float(Y1.abs().max())
    inv = [1.0, 1.0, 1.0]
    if fp8:
        inv = [float(a) / m for a, m in zip(lin.amax, (448.0, 448.0, 57344.0))]
    wd = lin.w_dense.double() * inv[1]
    xd, gd = Xop.double() * inv[0], Gop.double() * inv[2]
    G = torch.empty((O, T), dtype=lin.gvals.dtype, device="cuda")
    ctx.decompress(lin.gvals, lin.gmeta, G)
    Gd = G.double() * inv[2]
    for y in (Y, Y1):
        _close(y, xd, wd.T)
    for w in (dW, dW1):
        _close(w, Gd, xd)
    for x in (dX, dX1):
        _close(x, gd, wd)


def test_shapes_take_the_path():
    plans = [B.plan(p, B.BF16, *s) for s, p in zip(SHAPES, (0, 0, 0, 2, 2, 1, 1, 2))]
    assert all(p[1] > 2 and p[2] == 0 for p in plans), plans
    assert B.joint_plan(B.BF16, 128, 128, 8192)[11] == 1 and B.joint_plan(B.BF16, 8192, 128, 128)[10] > 1


def test_same_bits_every_time_and_without_workspace():
    """The ranges are added in order: repeated calls agree bit for bit; a context without a workspace takes whole tiles."""
    gen = torch.Generator(device="cuda").manual_seed(5)
    mk = lambda r, c, s: torch.empty((r, c), dtype=torch.bfloat16, device="cuda").normal_(0.0, s, generator=gen)
    W, X = mk(128, 8192, 0.02), mk(256, 8192, 1.0)
    ctx, small = B.Context(0), B.Context(0, minimal_workspace=True)
    lin = SsteLinear(ctx, W, 256, tensor_id=1, seed=3)
    lin.init_beta()
    lin.prune()
    Y = lin.forward(X).clone()
    for _ in range(20):
        assert torch.equal(lin.forward(X), Y)
    Z = torch.empty_like(Y)
    small.linear_fwd(X, lin.vals, lin.meta, Z)
    wd = lin.w_dense.double()
    _close(Y, X.double(), wd.T)
    _close(Z, X.double(), wd.T)
