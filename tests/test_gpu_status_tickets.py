"""The arrival counters of split products are zero after every poll that reports an error, whichever error it is.

A product that gave up on a wait leaves counters half counted.  The status word holds one error, so a degenerate beta recorded
before it must not hide that.  The state such a product leaves is written into the workspace here.
"""
import ctypes

import pytest
import torch

from paper_2409_09099_b200 import binding as B

pytestmark = pytest.mark.gpu

STATUS_OFF = 0                                        # offsets in the workspace: csrc/common.cuh
TICKETS_OFF = (256 + 2 * 8 * 1024 + 1023) // 1024 * 1024
TICKETS = 8192


def _words(ctx, offset, n):
    return ctx.workspace[offset: offset + 4 * n].view(torch.int32)


@pytest.mark.parametrize("status", [B.ERR_DEGENERATE, B.ERR_TIMEOUT])
def test_poll_clears_half_counted_tickets(status):
    ctx = B.Context(0)
    gen = torch.Generator(device="cuda").manual_seed(3)
    O, I, T = 256, 256, 4096
    dY = torch.empty((T, O), dtype=torch.bfloat16, device="cuda").normal_(0.0, 1.0, generator=gen)
    X = torch.empty((T, I), dtype=torch.bfloat16, device="cuda").normal_(0.0, 1.0, generator=gen)
    gvals, gmeta = ctx.alloc_compressed(O, T)
    ctx.mvue_sparsify(dY, 1, 0, 0, gvals, gmeta)
    want, got = (torch.empty((O, I), dtype=torch.bfloat16, device="cuda") for _ in range(2))
    ctx.debug_force_splits(2)
    try:
        ctx.linear_bwd_weight(gvals, gmeta, X, want)
        assert ctx.poll_device_status() == B.OK
        assert not _words(ctx, TICKETS_OFF, TICKETS).any()
        _words(ctx, TICKETS_OFF, TICKETS).fill_(0x10001)            # one of two units claimed and finished
        _words(ctx, STATUS_OFF, 1).fill_(status)
        assert ctx.poll_device_status() == status
        assert not _words(ctx, TICKETS_OFF, TICKETS).any()
        ctx.linear_bwd_weight(gvals, gmeta, X, got)
        assert torch.equal(got.view(torch.int16), want.view(torch.int16))
        assert ctx.poll_device_status() == B.OK
    finally:
        ctx.debug_force_splits(0)
    ctx.close()


@pytest.mark.parametrize("recorded", [0, B.ERR_DEGENERATE])
def test_a_timeout_is_reported_over_a_degenerate_beta(recorded):
    """The stall hook of the one-tile product: its wait runs out after a millisecond and the kernel returns."""
    ctx = B.Context(0)
    dY = torch.ones((128, 256), dtype=torch.bfloat16, device="cuda")
    w = torch.ones((256, 128), dtype=torch.bfloat16, device="cuda")
    dX = torch.empty((128, 128), dtype=torch.bfloat16, device="cuda")
    _words(ctx, STATUS_OFF, 1).fill_(recorded)
    ctx.debug_inject_stall(True)
    try:
        ctx.linear_bwd_input(dY, w, dX)
        torch.cuda.synchronize()
    finally:
        ctx.debug_inject_stall(False)
    assert ctx.poll_device_status() == B.ERR_TIMEOUT
    ctx.linear_bwd_input(dY, w, dX)
    assert bool((dX == 256).all()) and ctx.poll_device_status() == B.OK
    ctx.close()


def test_layout_of_the_workspace():
    lib = B.load()
    lib.sste_workspace_bytes.restype = ctypes.c_size_t
    assert (lib.sste_workspace_bytes() + 1023) // 1024 * 1024 == TICKETS_OFF
