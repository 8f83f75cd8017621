"""Forward products whose pairs store whole tiles, two output boxes at a time, and split ones, box by box, from the same buffers.

Another split of an fp32 sum changes it by about 1e-6 of the sum of magnitudes, which moves the bf16 result by at most one unit in
the last place (2^-7 of the value at the start of a binade) wherever it is not much smaller than those.
"""
import pytest
import torch

from paper_2409_09099_b200 import binding as B
from paper_2409_09099_b200.layer import SsteLinear

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("O,I,T,fp8", [(640, 5120, 8192, False), (5248, 5120, 1024, False), (8064, 8448, 640, False),
                                       (1664, 8192, 8192, True), (768, 10240, 8192, True)])
def test_whole_tiles_and_then_split_ones(O, I, T, fp8):
    ctx = B.Context(0)
    try:
        gen = torch.Generator(device="cuda").manual_seed(O + I + T)
        mk = lambda r, c, s: torch.empty((r, c), dtype=torch.bfloat16, device="cuda").normal_(0.0, s, generator=gen)
        lin = SsteLinear(ctx, mk(O, I, 0.02), T, fp8=fp8)
        lin.init_beta(); lin.prune()
        X = mk(T, I, 1.0)
        Y = lin.forward(X).clone()
        for _ in range(30):
            lin.Y.fill_(7.0)
            assert torch.equal(lin.forward(X).view(torch.int16), Y.view(torch.int16))
        ctx.debug_force_splits(1)
        try:
            ref = lin.forward(X).float()
        finally:
            ctx.debug_force_splits(0)
        assert bool(((Y.float() - ref).abs() <= 2.0 ** -7 * ref.abs() + 1e-5 * ref.abs().max()).all())
        assert ctx.poll_device_status() == 0
    finally:
        ctx.close()
