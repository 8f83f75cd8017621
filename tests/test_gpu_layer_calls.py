"""The one-call-per-phase path of a layer (sste_layer_prune / _forward / _backward) against the single calls.

The layer takes the single calls when a `mark` callback wants to see them, so both paths run on the same buffers' shapes
and must leave the same bits.  The FP8 maxima come without a memset there (a scratch word that every call leaves zero):
checked over repeated iterations with maxima that shrink, and for a tensor of zeros.
"""
import pytest
import torch

from paper_2409_09099_b200 import synth
from tests.gpu_util import DEV, dbf16

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    from paper_2409_09099_b200 import binding
    c = binding.Context(0)
    yield c
    assert c.poll_device_status() == 0
    c.close()


def _bits(t):
    return t.contiguous().view(torch.uint8)


@pytest.mark.parametrize("fp8,dense_copy", [(False, True), (False, False), (True, True), (True, False)])
@pytest.mark.parametrize("O,I,T", [(128, 128, 128), (384, 640, 256)])
def test_layer_calls_equal_single_calls(ctx, O, I, T, fp8, dense_copy):
    from paper_2409_09099_b200.layer import SsteLinear
    W = dbf16(synth.gaussian_bf16(O + 11, (O, I), 0.02))
    layers = [SsteLinear(ctx, W, T, tensor_id=4, seed=17, fp8=fp8, dense_copy=dense_copy) for _ in range(2)]
    layers[1].mark = lambda label: None                     # the single calls
    for step, scale in enumerate((1.0, 0.25, 0.0)):
        X = dbf16(synth.gaussian_bf16(O + 12 + step, (T, I), 1.0)) * scale
        dY = dbf16(synth.gaussian_bf16(O + 22 + step, (T, O), 1e-2)) * scale
        for lin in layers:
            if step == 0:
                lin.init_beta()
            lin.prune()
            lin.forward(X)
            lin.backward(dY, step=step, token_offset=4 * step)
        a, b = layers
        for name in ("vals", "meta", "gvals", "gmeta", "Y", "dX", "dW"):
            assert torch.equal(_bits(getattr(a, name)), _bits(getattr(b, name))), (step, name)
        if fp8:
            assert torch.equal(a.amax, b.amax) and not a._scratch.any()
        assert a.launches == b.launches


def test_described_buffers_follow_the_attributes(ctx):
    """A replaced buffer, exchanged weight storage or a shorter batch takes effect in the next call."""
    from paper_2409_09099_b200.layer import SsteLinear
    O, I, T = 256, 128, 256
    W1, W2 = (dbf16(synth.gaussian_bf16(s, (O, I), 0.02)) for s in (31, 32))
    X = dbf16(synth.gaussian_bf16(33, (T, I), 1.0))
    lin = SsteLinear(ctx, W1.clone(), T)
    lin.init_beta(); lin.prune()
    Y1 = lin.forward(X).clone()
    lin.W.data = W2                                          # same tensor object, other storage
    lin.prune()
    Y2 = lin.forward(X).clone()
    ref = SsteLinear(ctx, W2, T)
    ref.beta.copy_(lin.beta); ref.beta_ready = True
    ref.prune()
    assert torch.equal(Y2, ref.forward(X)) and not torch.equal(Y1, Y2)
    lin.Y = torch.empty_like(lin.Y)
    assert lin.forward(X) is lin.Y and torch.equal(lin.Y, Y2)
    lin.Y.fill_(7.0)
    lin.forward(X[:128])                                     # a shorter batch fills the first rows only
    assert torch.equal(lin.Y[:128], Y2[:128]) and bool((lin.Y[128:] == 7.0).all())


@pytest.mark.parametrize("fp8", [False, True])
@pytest.mark.parametrize("O,I,T", [(128, 128, 128), (128, 256, 4096), (768, 768, 2048), (3072, 768, 1024), (1280, 1280, 2176),
                                   (2432, 2560, 512), (384, 5120, 640)])
def test_one_launch_gradients_equal_two_launches(ctx, O, I, T, fp8):
    """sste_layer_grads against the two single calls: the same sums, of which only the split may differ.

    Another split of an fp32 sum changes it by about 1e-6 of the sum of magnitudes, which moves the bf16 result by at most
    one unit in the last place (2^-7 of the value at the start of a binade) wherever it is not much smaller than those."""
    from paper_2409_09099_b200.layer import SsteLinear
    W = dbf16(synth.gaussian_bf16(O + 61, (O, I), 0.02))
    X = dbf16(synth.gaussian_bf16(O + 62, (T, I), 1.0))
    dY = dbf16(synth.gaussian_bf16(O + 63, (T, O), 1e-2))
    lin = SsteLinear(ctx, W, T, tensor_id=4, seed=17, fp8=fp8)
    lin.init_beta(); lin.prune(); lin.forward(X)
    for rep in range(2):                                     # the tickets of split tiles must be left at zero
        lin.dX.fill_(7.0); lin.dW.fill_(7.0)
        dX, dW = (t.clone() for t in lin.backward(dY, step=3))
        ref_w, ref_x = lin.grad_weight().float(), lin.grad_input(dY).float()
        for got, ref in ((dW.float(), ref_w), (dX.float(), ref_x)):
            assert bool(((got - ref).abs() <= 2.0 ** -7 * ref.abs() + 1e-5 * ref.abs().max()).all())


@pytest.mark.parametrize("fp8", [False, True])
@pytest.mark.parametrize("O,I,T", [(203, 80, 72), (128, 80, 128), (200, 128, 1000), (1, 3, 5)])
def test_padded_calls_equal_single_calls(ctx, O, I, T, fp8):
    """sste_padded_forward / _backward against the single calls; columns that need a crop, rows only, neither."""
    from paper_2409_09099_b200.layer import SsteLinearPadded
    W = dbf16(synth.gaussian_bf16(O + 81, (O, I), 0.02))
    layers = [SsteLinearPadded(ctx, O, I, T, tensor_id=4, seed=17, fp8=fp8) for _ in range(2)]
    layers[1].inner.mark = lambda label: None               # the single calls
    for step in range(2):
        X = dbf16(synth.gaussian_bf16(O + 82 + step, (T, I), 1.0))
        dY = dbf16(synth.gaussian_bf16(O + 92 + step, (T, O), 1e-2))
        for lin in layers:
            lin.set_weight(W)
            if step == 0:
                lin.init_beta()
            lin.prune()
            assert lin.forward(X) is lin.Y
            lin.backward(dY, step=step)
        a, b = layers
        for name in ("Y", "dX", "dW"):
            assert torch.equal(_bits(getattr(a, name)), _bits(getattr(b, name))), (step, name)
        assert tuple(a.Y.shape) == (T, O) and tuple(a.dX.shape) == (T, I) and tuple(a.dW.shape) == (O, I)
