"""Products whose pairs work through several tiles: both accumulators of every width in turn, two of which share columns at 256.

Against the fp64 product of the same operands.  Bound as in test_gpu_splitk_sum.py: half a unit in the last place of a bf16 result
(2^-8 relative), and fp32 additions that are off by about 2^-23 of the sum of magnitudes: four times that.
"""
import pytest
import torch

from paper_2409_09099_b200 import binding as B
from paper_2409_09099_b200.layer import SsteLinear

pytestmark = pytest.mark.gpu


def _mk(gen, r, c, s):
    return torch.empty((r, c), dtype=torch.bfloat16, device="cuda").normal_(0.0, s, generator=gen)


def _close(got, a, b):
    ref, mag = a.double() @ b.double(), a.double().abs() @ b.double().abs()
    bound = ref.abs() * (2.0 ** -8 if got.dtype == torch.bfloat16 else 0.0) + mag * 2.0 ** -21 + 1e-30
    assert bool(((got.double() - ref).abs() <= bound).all())


# 10 x 20 tiles of 256 (200 on 74 pairs), both edges ragged; one stage, an odd number of them, more than the pipeline holds
@pytest.mark.parametrize("K", [128, 384, 2176])
@pytest.mark.parametrize("width,fp8,out_dtype", [(w, f, torch.bfloat16) for w in (256, 224, 192, 128) for f in (False, True)]
                         + [(256, f, torch.float32) for f in (False, True)])
def test_forward_and_weight_gradient(width, fp8, out_dtype, K):
    M, N = 2432, 4992
    ctx = B.Context(0)
    try:
        gen = torch.Generator(device="cuda").manual_seed(K)
        ctx.debug_force_tile_width(width)
        ctx.debug_force_splits(1)
        # forward [M, N] over K features; weight gradient [M, N] over K tokens
        fwd = SsteLinear(ctx, _mk(gen, M, K, 0.02), N, fp8=fp8, out_dtype=out_dtype)
        bwd = SsteLinear(ctx, _mk(gen, M, N, 0.02), K, fp8=fp8, out_dtype=out_dtype)
        fwd.init_beta(); fwd.prune()
        X = _mk(gen, N, K, 1.0)
        Y = fwd.forward(X)
        inv = lambda lin, i: float(lin.amax[i]) / (448.0, 448.0, 57344.0)[i] if fp8 else 1.0
        _close(Y, (fwd.Xq if fp8 else X).double() * inv(fwd, 0), fwd.w_dense.double().T * inv(fwd, 1))
        bwd.init_beta(); bwd.prune()
        X = _mk(gen, K, N, 1.0)
        bwd.forward(X)
        bwd.sparsify_grad(_mk(gen, K, M, 1e-2))
        G = torch.empty((M, K), dtype=bwd.gvals.dtype, device="cuda")
        ctx.decompress(bwd.gvals, bwd.gmeta, G)
        _close(bwd.grad_weight(), G.double() * inv(bwd, 2), (bwd.Xq if fp8 else X).double() * inv(bwd, 0))
        assert ctx.poll_device_status() == 0
    finally:
        ctx.debug_force_tile_width(0)
        ctx.debug_force_splits(0)
        ctx.close()


@pytest.mark.parametrize("fp8", [False, True])
def test_products_that_read_the_previous_one(fp8):
    """Each kernel's roles wait for the previous kernel by themselves: a chain of products through two buffers, and the gradients
    of each link, queued without a pause, against the same calls one at a time."""
    D, T, links = 1280, 1152, 24
    ctx = B.Context(0)
    try:
        gen = torch.Generator(device="cuda").manual_seed(7)
        layers = []
        for i in range(4):
            lin = SsteLinear(ctx, _mk(gen, D, D, 0.05), T, tensor_id=i, seed=3, fp8=fp8, dense_copy=i % 2 == 0)
            lin.init_beta()
            layers.append(lin)
        X0, ping, pong = _mk(gen, T, D, 1.0), *(torch.empty((T, D), dtype=torch.bfloat16, device="cuda") for _ in range(2))

        def run(between):
            x = X0
            for k in range(links):
                lin = layers[k % 4]
                lin.Y = pong if x is ping else ping
                lin.prune(); between()
                y = lin.forward(x); between()
                dX, dW = lin.backward(y, step=k); between()
                x = y
            return [x.clone()] + [t.clone() for lin in layers for t in (lin.dX, lin.dW, lin.vals, lin.meta, lin.gvals, lin.gmeta)]

        want = run(torch.cuda.synchronize)
        assert float(want[0].float().abs().max()) > 0 and bool(torch.isfinite(want[0].float()).all())
        for _ in range(10):
            got = run(lambda: None)
            assert all(torch.equal(a.view(torch.uint8), b.view(torch.uint8)) for a, b in zip(got, want))
        assert ctx.poll_device_status() == 0
    finally:
        ctx.close()
