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


@pytest.mark.parametrize("fp8", [False, True])
def test_buffers_given_other_storage(ctx, fp8):
    """`t.data = ...` on any buffer between two phases: the next phase works on the new storage and leaves the old alone."""
    lin, ref, X, dY = _layer(ctx, fp8=fp8), _layer(ctx, fp8=fp8), X1(), DY()
    names = ["W", "beta", "vals", "meta", "w_dense", "gvals", "gmeta", "Y", "dX", "dW"] + (["amax", "Xq", "dYq"] if fp8 else [])
    for l in (ref, lin):
        l.prune(); l.forward(X); l.backward(dY, step=1)
    old = {}
    for phase in ("prune", "forward", "backward"):
        for n in names:
            t = getattr(lin, n)
            old[n] = t.data
            t.data = t.data.clone()
            old[n].view(torch.uint8).fill_(0x55)
        for l in (ref, lin):
            {"prune": l.prune, "forward": lambda: l.forward(X), "backward": lambda: l.backward(dY, step=2)}[phase]()
        for n in names:
            assert bool((old[n].view(torch.uint8) == 0x55).all()), (phase, n)
            assert _same(getattr(lin, n), getattr(ref, n)), (phase, n)
    assert lin._desc.fits and lin._desc.buffers.W == lin.W.data_ptr()      # described again, not left to the single calls


def test_padded_buffers_given_other_storage(ctx):
    lin = SsteLinearPadded(ctx, 200, 100, 72, seed=5)
    W, X, dY = (dbf16(synth.gaussian_bf16(s, sh, sg)) for s, sh, sg in ((51, (200, 100), 0.02), (52, (72, 100), 1.0), (53, (72, 200), 1e-2)))
    lin.set_weight(W); lin.init_beta(); lin.prune()
    want = [lin.forward(X).clone()] + [t.clone() for t in lin.backward(dY, step=1)]
    old = []
    for t in (lin.Xp, lin.dYp, lin.Y, lin.dX, lin.dW):
        old.append(t.data)
        t.data = torch.zeros_like(t.data)
        old[-1].view(torch.int16).fill_(0x5555)
    got = [lin.forward(X), *lin.backward(dY, step=1)]
    assert all(_same(a, b) for a, b in zip(got, want)) and all(bool((t.view(torch.int16) == 0x5555).all()) for t in old)


def test_a_weight_turned_into_a_view_that_is_not_contiguous_is_refused(ctx):
    W = dbf16(synth.gaussian_bf16(61, (256, 256), 0.02))
    lin = SsteLinear(ctx, W, T)
    lin.init_beta(); lin.prune()
    lin.W.data = lin.W.data.t()                          # same address, same sizes
    with pytest.raises(AssertionError):
        lin.prune()


@pytest.mark.parametrize("how", ["subclass", "attribute", "context"])
@pytest.mark.parametrize("call", ["backward", "overlap"])
def test_single_calls_that_someone_overrides_are_still_made(ctx, how, call):
    """A layer whose grad_weight does something more (an all-reduce, a count), or a context that watches its calls."""
    seen = []

    class Watching(SsteLinear):
        def grad_weight(self):
            seen.append("W")
            return super().grad_weight()

    class WatchingContext(B.Context):
        def linear_bwd_weight(self, *a, **kw):
            seen.append("W")
            return super().linear_bwd_weight(*a, **kw)

    ctx_ = WatchingContext(0) if how == "context" else ctx
    side_ctx, side = (WatchingContext if how == "context" else B.Context)(0), torch.cuda.Stream()
    lin, X, dY = _layer(ctx_, cls=Watching if how == "subclass" else SsteLinear), X1(), DY()
    lin.forward(X)
    if how == "attribute":
        plain = lin.grad_weight
        lin.grad_weight = lambda: (seen.append("W"), plain())[1]
    if call == "backward":
        lin.backward(dY)
    else:
        lin.sparsify_grad(dY)
        lin.grad_weight_and_input(dY, side_ctx, side)
    assert seen == ["W"]
    ref = _layer(ctx)
    ref.forward(X); ref.backward(dY)
    torch.testing.assert_close(lin.dW.float(), ref.dW.float(), rtol=2.0 ** -7, atol=1e-5 * float(ref.dW.float().abs().max()))
    assert lin.ctx is ctx_


def test_padded_backward_uses_the_inner_layers_input(ctx):
    """No forward, no input: refused.  An input that somebody gave the inner layer (recomputed activations) is the one used."""
    W, X, dY = (dbf16(synth.gaussian_bf16(s, sh, sg)) for s, sh, sg in ((71, (200, 100), 0.02), (72, (72, 100), 1.0), (73, (72, 200), 1e-2)))
    lin, ref = (SsteLinearPadded(ctx, 200, 100, 72, seed=5) for _ in range(2))
    for l in (lin, ref):
        l.set_weight(W); l.init_beta(); l.prune()
    with pytest.raises(AttributeError):
        lin.backward(dY)
    lin.forward(torch.zeros_like(X))
    ref.forward(X)
    lin.inner.X = ref.Xp
    for a, b in zip(lin.backward(dY), ref.backward(dY)):
        assert _same(a, b)


@pytest.mark.parametrize("kind", ["int64", "uint64", "int32"])
def test_seeds_and_ids_from_numpy(ctx, kind):
    import numpy as np
    n = getattr(np, kind)
    lin, ref, X, dY = _layer(ctx), _layer(ctx), X1(), DY()
    lin.seed, lin.tensor_id, lin.T, lin.counter_cols = n(77), n(3), n(T), n(0)
    ref.seed, ref.tensor_id = 77, 3
    for l in (lin, ref):
        l.prune(); l.forward(X); l.backward(dY, step=n(4), token_offset=n(8))
    assert _same(lin.dW, ref.dW) and _same(lin.gmeta, ref.gmeta)
