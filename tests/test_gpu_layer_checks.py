"""What the one-call phases of a layer must not take: tensors and states that the single calls refuse or follow."""
import pytest
import torch

from paper_2409_09099_b200 import binding as B, synth
from paper_2409_09099_b200.layer import SsteLinear, SsteLinearPadded
from tests.gpu_util import dbf16

pytestmark = pytest.mark.gpu

O, I, T = 256, 128, 128                                  # T = I: a transposed X has the right shape


@pytest.fixture(scope="module")
def ctx():
    c = B.Context(0)
    yield c
    assert c.poll_device_status() == 0
    c.close()


def _same(a, b):
    return torch.equal(a.contiguous().view(torch.uint8), b.contiguous().view(torch.uint8))


def _layer(ctx, seed=41, cls=SsteLinear, **kw):
    lin = cls(ctx, dbf16(synth.gaussian_bf16(seed, (O, I), 0.02)), T, tensor_id=2, **kw)
    lin.init_beta(); lin.prune()
    return lin


X1 = lambda: dbf16(synth.gaussian_bf16(42, (T, I), 1.0))
DY = lambda: dbf16(synth.gaussian_bf16(43, (T, O), 1e-2))


@pytest.mark.parametrize("call", ["backward", "overlap"])
@pytest.mark.parametrize("what", ["transposed", "fp32", "host"])
def test_a_saved_input_that_the_products_cannot_read_is_refused(ctx, call, what):
    """X of the backward comes from the forward or from whoever keeps activations; only bf16, contiguous, on the device."""
    lin, X, dY = _layer(ctx), X1(), DY()
    lin.forward(X)
    lin.X = {"transposed": X.t(), "fp32": X.float(), "host": X.cpu()}[what]
    lin.sparsify_grad(dY)
    with pytest.raises((AssertionError, B.SsteError)):
        if call == "backward":
            lin.backward(dY)
        else:
            lin.grad_weight_and_input(dY, ctx, torch.cuda.Stream())
    lin.X = X.t().contiguous()                           # the same values where they can be read
    lin.backward(dY)
    ref = _layer(ctx)
    ref.forward(X.t().contiguous())
    ref.backward(dY)
    assert _same(lin.dW, ref.dW)
