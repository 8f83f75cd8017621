"""A context's workspace at its two ends: ready when the constructor returns, untouched by others while a product still uses it."""
import pytest
import torch

from paper_2409_09099_b200 import binding as B

pytestmark = pytest.mark.gpu

O, I, T = 256, 256, 4096                                     # few tiles, a long reduction: grad_W goes through the workspace
BUSY = 100_000_000                                           # clocks that a stream is kept busy with, about 50 ms


def _operands():
    gen = torch.Generator(device="cuda").manual_seed(4)
    mk = lambda r, c: torch.empty((r, c), dtype=torch.bfloat16, device="cuda").normal_(0.0, 1.0, generator=gen)
    ctx = B.Context(0)
    gvals, gmeta = ctx.alloc_compressed(O, T)
    dY, X = mk(T, O), mk(T, I)
    ctx.mvue_sparsify(dY, 1, 0, 0, gvals, gmeta)
    want = torch.empty((O, I), dtype=torch.bfloat16, device="cuda")
    ctx.linear_bwd_weight(gvals, gmeta, X, want)
    torch.cuda.synchronize()
    return gvals, gmeta, X, want


@pytest.mark.parametrize("own_stream", [False, True])
def test_first_product_on_another_stream(own_stream):
    gvals, gmeta, X, want = _operands()
    got = torch.empty_like(want)
    made_on, used_on = torch.cuda.Stream() if own_stream else torch.cuda.current_stream(), torch.cuda.Stream()
    n = B.load().sste_workspace_bytes_recommended()
    with torch.cuda.stream(made_on):
        dirty = torch.full((n // 4,), 0x10001, dtype=torch.int32, device="cuda")      # the memory the workspace comes from
        del dirty
        torch.cuda._sleep(BUSY)
        ctx = B.Context(0)
    with torch.cuda.stream(used_on):
        ctx.linear_bwd_weight(gvals, gmeta, X, got)
    torch.cuda.synchronize()
    assert torch.equal(got.view(torch.int16), want.view(torch.int16)) and ctx.poll_device_status() == B.OK
    ctx.close()


def test_close_leaves_the_workspace_to_work_in_flight():
    """Closing frees nothing: memory allocated right afterwards is not the workspace of a product that has yet to run."""
    gvals, gmeta, X, want = _operands()
    got, side = torch.empty_like(want), torch.cuda.Stream()
    ctx = B.Context(0)
    with torch.cuda.stream(side):
        torch.cuda._sleep(BUSY)
        ctx.linear_bwd_weight(gvals, gmeta, X, got)
    ctx.close()
    other = torch.full_like(ctx.workspace, 0x5a)             # on this stream, beside the side stream's work
    torch.cuda.synchronize()
    assert torch.equal(got.view(torch.int16), want.view(torch.int16)) and bool((other == 0x5a).all())
