"""Padding and cropping at sizes where a 16-byte vector is cut by a row end or an array end, and at odd addresses.

dst is compared whole, with elements in front of and behind it that must stay as they were.
"""
import gc

import pytest
import torch

from tests.gpu_util import DEV

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    from paper_2409_09099_b200 import binding
    c = binding.Context(0)
    yield c
    assert c.poll_device_status() == 0
    c.close()
    gc.collect()      # models of earlier tests hold GPU memory through reference cycles: not left to chance


def _at(offset, rows, cols, fill=None):
    """A contiguous [rows, cols] view `offset` elements into a buffer with 16 guard elements on either side."""
    buf = torch.randint(1, 1 << 14, (16 + offset + rows * cols + 16,), dtype=torch.int16, device=DEV)
    if fill is not None:
        buf.fill_(fill)
    return buf, buf[16 + offset: 16 + offset + rows * cols].view(rows, cols).view(torch.bfloat16)


@pytest.mark.parametrize("offset", [0, 1, 3])
@pytest.mark.parametrize("rows,cols", [(1, 1), (1, 9), (3, 7), (7, 8), (5, 128), (129, 77), (40, 1001)])
def test_pad_and_crop(ctx, rows, cols, offset):
    rows_p, cols_p = (rows + 127) // 128 * 128, (cols + 127) // 128 * 128
    _, src = _at(offset, rows, cols)
    buf, dst = _at(0, rows_p, cols_p, fill=7)
    ctx.pad_2d(src, dst)
    want = torch.zeros((rows_p, cols_p), dtype=torch.int16, device=DEV)
    want[:rows, :cols] = src.view(torch.int16)
    assert torch.equal(dst.view(torch.int16), want)
    assert bool((buf[:16] == 7).all()) and bool((buf[-16:] == 7).all())
    buf, back = _at(offset, rows, cols, fill=9)
    ctx.crop_2d(dst, back)
    assert torch.equal(back.view(torch.int16), src.view(torch.int16))
    assert bool((buf[: 16 + offset] == 9).all()) and bool((buf[-16:] == 9).all())


@pytest.mark.parametrize("fp8", [False, True])
def test_compressed_weight_route_with_and_without_workspace(fp8):
    """grad_X from the compressed weight: expanded into the workspace, or tile by tile where there is no room for it."""
    from paper_2409_09099_b200 import binding as B, synth
    from paper_2409_09099_b200.layer import SsteLinear
    from tests.gpu_util import dbf16
    O, I, T = 384, 256, 640
    W, X, dY = (dbf16(synth.gaussian_bf16(s, sh, sig)) for s, sh, sig in ((51, (O, I), 0.02), (52, (T, I), 1.0), (53, (T, O), 1e-2)))
    out = []
    for minimal in (False, True):
        c = B.Context(0, minimal_workspace=minimal)
        lin = SsteLinear(c, W, T, seed=3, fp8=fp8, dense_copy=False)
        lin.init_beta(); lin.prune(); lin.forward(X); lin.backward(dY)
        out.append(lin.dX.clone())
        assert c.poll_device_status() == 0
        c.close()
    assert torch.equal(out[0].view(torch.int16), out[1].view(torch.int16))
