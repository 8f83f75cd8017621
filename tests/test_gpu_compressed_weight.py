"""grad_X from the compressed weight where the workspace has no room for a dense copy: the kernel that expands the operand itself.

The contexts here have a workspace for partial sums but not for a copy beside them (a copy needs 80 MB more), so that these calls
do not end in the dense kernel.  The reference is the dense kernel with the same tile width and the same K ranges: the same bits.
"""
import pytest
import torch

from paper_2409_09099_b200 import binding as B
from tests.gpu_util import DEV, context_with_workspace

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    c = context_with_workspace(40 << 20)
    yield c
    assert c.poll_device_status() == 0
    c.close()


@pytest.fixture(autouse=True)
def hooks_off(ctx):
    yield
    ctx.debug_force_splits(0)
    ctx.debug_force_tile_order(0)
    ctx.debug_force_tile_width(0)


def _operands(ctx, O, I, T, fp8):
    gen = torch.Generator(device=DEV).manual_seed(O + I + T)
    mk = lambda r, c, s: torch.empty((r, c), dtype=torch.bfloat16, device=DEV).normal_(0.0, s, generator=gen)
    wdt = B.E4M3 if fp8 else B.BF16
    one = lambda v: torch.full((1,), v, dtype=torch.float32, device=DEV)
    amax = dict(w_amax_dev=one(0.3), g_amax_dev=one(0.05)) if fp8 else {}
    vals, meta = ctx.alloc_compressed(O, I, wdt)
    dense = torch.empty((O, I), dtype=B._TORCH_DT[wdt], device=DEV)
    ctx.project_compress(mk(O, I, 0.02), one(1.25), vals, meta, dense, w_amax_dev=amax.get("w_amax_dev"))
    dY = mk(T, O, 1e-2)
    if fp8:
        q = torch.empty((T, O), dtype=torch.float8_e5m2, device=DEV)
        ctx.quantize_fp8(dY, amax["g_amax_dev"], q)
        dY = q
    return dY, dense, vals, meta, amax


def _both(ctx, ops, out_dtype=torch.bfloat16):
    """(launches, grad_X) from the compressed operand, after comparing it with the dense one's; a guard row behind the result."""
    dY, dense, vals, meta, amax = ops
    out = []
    ctx.debug_force_tile_width(256)
    for kw in (dict(vals=vals, meta=meta), {}):
        whole = torch.full((dY.shape[0] + 1, dense.shape[1]), 7.0, dtype=out_dtype, device=DEV)
        xa = torch.full((1,), 1e9, device=DEV)
        before = B.launch_count()
        ctx.linear_bwd_input(dY, None if kw else dense, whole[:-1], dx_amax_out_dev=xa, **amax, **kw)
        out.append((B.launch_count() - before, whole[:-1], xa))
        assert bool((whole[-1] == 7.0).all())
    (n, got, ga), (m, want, wa) = out
    assert torch.equal(got.view(torch.uint8), want.view(torch.uint8))
    assert ga.item() == wa.item() == want.float().abs().max().item()
    assert n == m                                         # no pass that expands the weight
    return n, got


@pytest.mark.parametrize("out_dtype", [torch.bfloat16, torch.float32])
@pytest.mark.parametrize("O,I,T", [(128, 128, 128), (384, 640, 1152), (256, 256, 512), (640, 384, 19200)])
@pytest.mark.parametrize("fp8", [False, True])
def test_whole_tiles(ctx, O, I, T, out_dtype, fp8):
    """One tile, ragged tiles and K stages, several waves."""
    ctx.debug_force_splits(1)
    _both(ctx, _operands(ctx, O, I, T, fp8), out_dtype)


@pytest.mark.parametrize("splits", [2, 3, 4])
@pytest.mark.parametrize("O,I,T", [(4096, 256, 512), (4224, 640, 384), (2048, 1280, 5120)])
@pytest.mark.parametrize("fp8", [False, True])
def test_ranges_that_exchange(ctx, O, I, T, splits, fp8):
    """Few tiles; a ragged tile and an odd number of stages; 100 tiles, of which the last 26 are split (2 and 4 ranges)."""
    ctx.debug_force_splits(splits)
    ops = _operands(ctx, O, I, T, fp8)
    first = _both(ctx, ops)[1].clone()
    for _ in range(3):                                    # counters left at zero, the same order of sums
        assert torch.equal(_both(ctx, ops)[1].view(torch.uint8), first.view(torch.uint8))


@pytest.mark.parametrize("O,I,T", [(8192, 128, 128), (4992, 384, 384)])
@pytest.mark.parametrize("fp8", [False, True])
def test_ranges_added_afterwards(ctx, O, I, T, fp8):
    n, _ = _both(ctx, _operands(ctx, O, I, T, fp8))
    assert n == 2                                         # the product and the sum


@pytest.mark.parametrize("group_m", [1, 3, 1000])
@pytest.mark.parametrize("splits", [1, 2])
def test_tile_order(ctx, group_m, splits):
    ops = _operands(ctx, 1280, 768, 1792, False)
    ctx.debug_force_splits(splits)
    want = _both(ctx, ops)[1].clone()
    ctx.debug_force_tile_order(group_m)
    assert torch.equal(_both(ctx, ops)[1].view(torch.uint8), want.view(torch.uint8))
