"""The one-call phases of a layer refuse what their kernels cannot take before the first of them is launched (no GPU needed).

The context and the buffers are addresses that nothing looks at: a call that gets as far as the device returns ERR_CUDA here.
"""
import ctypes

import pytest

from paper_2409_09099_b200 import binding as B, build

CTX = ctypes.create_string_buffer(4096)              # device 0, null pointers: only ever asked for the device
BUFFERS = ("W", "vals", "meta", "w_dense", "gvals", "gmeta", "Xq", "dYq", "Y", "dX", "dW")


@pytest.fixture(scope="module")
def lib():
    import torch
    if torch.cuda.is_available():
        pytest.skip("addresses without memory behind them: not where a device could be asked")
    build.build()
    return B.load()


def _layer(fp8, **changes):
    d = B.LayerBuffers(O=256, I=128, T=128, op_dtype=B.E4M3 if fp8 else B.BF16, out_dtype=B.BF16)
    for i, name in enumerate(BUFFERS + ("beta",) + (("amax", "scratch") if fp8 else ())):
        setattr(d, name, 0x100000 * (i + 1))
    if not fp8:
        d.Xq = d.dYq = None
    for k, v in changes.items():
        setattr(d, k, v)
    return d


def _calls(lib, d, X=0x10000000, dY=0x20000000, token_offset=0):
    at = ctypes.byref(d)
    return {"prune": lambda: lib.sste_layer_prune(CTX, at, None),
            "forward": lambda: lib.sste_layer_forward(CTX, at, X, None, None),
            "backward": lambda: lib.sste_layer_backward(CTX, at, X, dY, 0, token_offset, None),
            "grads": lambda: lib.sste_layer_grads(CTX, at, X, dY, None)}


@pytest.mark.parametrize("fp8", [False, True])
@pytest.mark.parametrize("phase", ["prune", "forward", "backward", "grads"])
def test_sizes(lib, phase, fp8):
    for name in ("O", "I", "T"):
        for bad in (0, -128, 100, 192, -2 ** 31):
            want = B.ERR_CUDA if (phase, name) == ("prune", "T") else B.ERR_SHAPE      # a prune does not look at T
            assert _calls(lib, _layer(fp8, **{name: bad}))[phase]() == want, (name, bad)
    assert _calls(lib, _layer(fp8))[phase]() == B.ERR_CUDA                      # nothing wrong: as far as the device


@pytest.mark.parametrize("fp8", [False, True])
@pytest.mark.parametrize("phase,reads", [("prune", ("W", "vals", "meta", "w_dense")), ("forward", ("vals", "meta", "Y")),
                                         ("backward", ("gvals", "gmeta", "w_dense", "dX", "dW")),
                                         ("grads", ("gvals", "gmeta", "w_dense", "dX", "dW"))])
def test_alignment_and_missing_buffers(lib, phase, reads, fp8):
    extra = {"prune": (), "forward": ("Xq",)}.get(phase, ("Xq", "dYq")) if fp8 else ()
    for name in reads + extra:
        assert _calls(lib, _layer(fp8, **{name: 0x900040}))[phase]() == B.ERR_ALIGN, name
        if name != "w_dense":
            assert _calls(lib, _layer(fp8, **{name: None}))[phase]() == B.ERR_INVALID_ARG, name
    other = set(BUFFERS) - set(reads) - set(extra) - {"Xq", "dYq"}
    for name in other:                                                          # what a phase does not touch does not matter
        assert _calls(lib, _layer(fp8, **{name: 0x900040}))[phase]() == B.ERR_CUDA, name
    if fp8:
        assert _calls(lib, _layer(True, scratch=0x900004))[phase]() == B.ERR_ALIGN
    if phase in ("backward", "grads"):                                          # grad_X from the compressed operand
        assert _calls(lib, _layer(fp8, w_dense=None))[phase]() == B.ERR_CUDA
        assert _calls(lib, _layer(fp8, w_dense=None, vals=0x900040))[phase]() == B.ERR_ALIGN
        assert _calls(lib, _layer(fp8, w_dense=None, meta=None))[phase]() == B.ERR_INVALID_ARG


@pytest.mark.parametrize("fp8", [False, True])
def test_other_arguments(lib, fp8):
    assert _calls(lib, _layer(fp8), token_offset=2)["backward"]() == B.ERR_SHAPE
    for cols in (-1, 257):
        assert _calls(lib, _layer(fp8, counter_cols=cols))["backward"]() == B.ERR_INVALID_ARG
    for phase in ("forward", "backward", "grads"):
        assert _calls(lib, _layer(fp8, out_dtype=B.E4M3))[phase]() == B.ERR_DTYPE
        assert _calls(lib, _layer(fp8), X=0x10000002, dY=0x20000002)[phase]() == (B.ERR_CUDA if fp8 and phase == "grads" else B.ERR_ALIGN)
    assert _calls(lib, _layer(fp8), X=0x10000010)["forward"]() == (B.ERR_CUDA if fp8 else B.ERR_ALIGN)


@pytest.mark.parametrize("fp8", [False, True])
def test_padded(lib, fp8):
    def status(call, inner=None, ptr=0x30000000, **changes):
        p = B.PaddedLayerBuffers(inner or _layer(fp8), 200, 100, 72, 0, 0x40000000, 0x50000000, 0x60000000, 0x70000000, 0x71000000)
        for k, v in changes.items():
            setattr(p, k, v)
        if call == "forward":
            return lib.sste_padded_forward(CTX, ctypes.byref(p), ptr, None)
        return lib.sste_padded_backward(CTX, ctypes.byref(p), ptr, 0, 0, None)

    for call, own in (("forward", ("Y",)), ("backward", ("dX", "dW"))):
        assert status(call) == B.ERR_CUDA
        assert status(call, ptr=0x30000001) == B.ERR_ALIGN
        for name in own:
            assert status(call, **{name: 0x60000001}) == B.ERR_ALIGN            # 2-byte elements at an odd address
            assert status(call, **{name: 0x60000002}) == status(call, **{name: None}) == B.ERR_CUDA
        assert status(call, inner=_layer(fp8, **{own[0]: 0x900040})) == B.ERR_ALIGN
        assert status(call, Xp=0x40000010) == (B.ERR_CUDA if fp8 else B.ERR_ALIGN)
    assert status("backward", dYp=0x50000010) == B.ERR_ALIGN
