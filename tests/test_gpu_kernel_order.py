"""A kernel is scheduled while the one in front of it in the stream still runs, and reads nothing before that one is done.

Every input of every call is written by a kernel of the library right in front of the call, with the queue backed up so that the two
meet; the results are those of the same calls one at a time.
"""
import pytest
import torch

from paper_2409_09099_b200 import binding as B
from paper_2409_09099_b200.layer import SsteLinear

pytestmark = pytest.mark.gpu

O, I, T = 1024, 2048, 1024
BF, E4, E5, U8 = torch.bfloat16, torch.float8_e4m3fn, torch.float8_e5m2, torch.uint8


@pytest.fixture(scope="module")
def ctx():
    c = B.Context(0)
    yield c
    assert c.poll_device_status() == 0
    c.close()


class _Tail:
    """a tensor at the end of a buffer that a kernel takes a while to write"""

    def __init__(self, t):
        self.whole = torch.zeros(1 << 25, dtype=U8, device="cuda")
        self.t = self.whole[-max(128, t.nbytes):].view(t.dtype)[:t.numel()].view(t.shape)
        self.t.copy_(t)


class _Scalar(_Tail):
    def __init__(self, value):
        super().__init__(torch.tensor([value], dtype=torch.float32, device="cuda"))


def _empty(shape, dtype):
    return torch.empty(shape, dtype=dtype, device="cuda")


def _calls(ctx):
    """name -> (inputs by name, call(inputs) -> outputs); nothing but the call's own kernels is launched by it before it is done"""
    gen = torch.Generator(device="cuda").manual_seed(3)
    rnd = lambda r, c, s: _empty((r, c), BF).normal_(0.0, s, generator=gen)
    W, X, dY = rnd(O, I, 0.02), rnd(T, I, 1.0), rnd(T, O, 1e-2)
    calls = {}
    for fp8 in (False, True):
        k, tag = B.E4M3 if fp8 else B.BF16, "fp8 " if fp8 else ""
        lin = SsteLinear(ctx, W, T, seed=5, fp8=fp8)
        lin.init_beta(); lin.prune(); lin.forward(X); lin.backward(dY)
        # operands of the single calls, as the layer left them
        xa, wa, ga = (_Scalar(float(lin.amax[i])) if fp8 else None for i in range(3))
        beta = _Scalar(float(lin.beta))
        val = lambda s: None if s is None else s.t
        x, g = (lin.Xq, lin.dYq) if fp8 else (X, dY)

        def project(d, k=k, fp8=fp8):
            vals, meta = ctx.alloc_compressed(O, I, k)
            dense = _empty((O, I), E4 if fp8 else BF)
            ctx.project_compress(d["W"], val(d["beta"]), vals, meta, dense, w_amax_dev=val(d.get("w_amax")))
            return vals, meta, dense

        def forward(d):
            Y = _empty((T, O), BF)
            ctx.linear_fwd(d["X"], d["vals"], d["meta"], Y, x_amax_dev=val(d.get("x_amax")), w_amax_dev=val(d.get("w_amax")))
            return (Y,)

        def sparsify(d, fp8=fp8):
            vals, meta = ctx.alloc_compressed(O, T, B.E5M2 if fp8 else B.BF16)
            q = _empty((T, O), E5) if fp8 else None
            ctx.mvue_sparsify(d["dY"], 7, 1, 0, vals, meta, dense_q_out=q, g_amax_dev=val(d.get("g_amax")))
            return (vals, meta) + ((q,) if fp8 else ())

        def grad_w(d):
            dW = _empty((O, I), BF)
            ctx.linear_bwd_weight(d["vals"], d["meta"], d["X"], dW, g_amax_dev=val(d.get("g_amax")), x_amax_dev=val(d.get("x_amax")))
            return (dW,)

        def grad_x(d):
            dX = _empty((T, I), BF)
            ctx.linear_bwd_input(d["dY"], d.get("w"), dX, g_amax_dev=val(d.get("g_amax")), w_amax_dev=val(d.get("w_amax")),
                                 vals=d.get("vals"), meta=d.get("meta"))
            return (dX,)

        def decompress(d, fp8=fp8):
            out = _empty((O, I), E4 if fp8 else BF)
            ctx.decompress(d["vals"], d["meta"], out)
            return (out,)

        def canonical(d, k=k):
            out = _empty((O, I // 16), torch.int16)
            ctx.meta_to_canonical(d["meta"], O, I, k, out)
            return (out,)

        def prune(d, lin=lin):
            lin.W = d["W"]
            lin.beta = val(d["beta"])
            lin.prune()
            return tuple(t.clone() for t in (lin.vals, lin.meta, lin.w_dense))

        def layer_forward(d, lin=lin):
            return (lin.forward(d["X"]).clone(),)

        def layer_backward(d, lin=lin):
            return tuple(t.clone() for t in lin.backward(d["dY"]))

        amaxes = lambda **kw: {n: s for n, s in kw.items() if s is not None}
        vals, meta, gvals, gmeta = (t.clone() for t in (lin.vals, lin.meta, lin.gvals, lin.gmeta))
        calls[tag + "project"] = dict(W=W, beta=beta, **amaxes(w_amax=wa)), project
        calls[tag + "forward"] = dict(X=x.clone(), vals=vals, meta=meta, **amaxes(x_amax=xa, w_amax=wa)), forward
        calls[tag + "sparsify"] = dict(dY=dY, **amaxes(g_amax=ga)), sparsify
        calls[tag + "grad_w"] = dict(vals=gvals, meta=gmeta, X=x.clone(), **amaxes(g_amax=ga, x_amax=xa)), grad_w
        calls[tag + "grad_x"] = dict(dY=g.clone(), w=lin.w_dense.clone(), **amaxes(g_amax=ga, w_amax=wa)), grad_x
        calls[tag + "grad_x compressed"] = dict(dY=g.clone(), vals=vals, meta=meta, **amaxes(g_amax=ga, w_amax=wa)), grad_x
        calls[tag + "decompress"] = dict(vals=vals, meta=meta), decompress
        calls[tag + "canonical"] = dict(meta=meta), canonical
        calls[tag + "layer prune"] = dict(W=W, beta=beta), prune
        calls[tag + "layer forward"] = dict(X=X), layer_forward
        calls[tag + "layer backward"] = dict(dY=dY), layer_backward

    def scalar_of(f):
        out = _empty(1, torch.float32)

        def call(d):
            f(d, out)
            return (out.clone(),)
        return call

    def quantize(d):
        q = _empty((T, I), E4)
        ctx.quantize_fp8(d["X"], val(d["amax"]), q)
        return (q,)

    def flips(d):
        n = _empty(1, torch.int64)
        ctx.flip_count(d["a"], d["b"], O, I, n)
        return (n,)

    decayed = W.clone()

    def decay(d):
        ctx.srste_decay(d["W"], d["meta"], B.BF16, 0.5, decayed)
        out = decayed.clone()
        decayed.copy_(W)
        return (out,)

    def crop(d):
        out = _empty((T - 3, I - 5), BF)
        ctx.crop_2d(d["X"], out)
        return (out,)

    def pad(d):
        out = _empty((T + 128, I + 128), BF)
        ctx.pad_2d(d["X"], out)
        return (out,)

    bmeta = calls["project"][1](dict(W=rnd(O, I, 0.02), beta=_Scalar(1.0)))[1]
    meta = calls["canonical"][0]["meta"]
    calls["beta"] = dict(W=W), scalar_of(lambda d, out: ctx.beta_init(d["W"], out))
    calls["amax"] = dict(X=X), scalar_of(lambda d, out: ctx.amax(d["X"], out))
    calls["project_amax"] = dict(W=W, beta=_Scalar(1.3)), scalar_of(lambda d, out: ctx.project_amax(d["W"], val(d["beta"]), out))
    calls["quantize"] = dict(X=X, amax=_Scalar(5.0)), quantize
    calls["flip_count"] = dict(a=meta, b=bmeta), flips
    calls["srste_decay"] = dict(W=W, meta=meta), decay
    calls["crop"] = dict(X=X), crop
    calls["pad"] = dict(X=X), pad
    return calls


def test_inputs_that_the_kernel_in_front_writes(ctx):
    bad = set()
    for name, (new, call) in _calls(ctx).items():
        new = {n: s if isinstance(s, _Tail) else _Tail(s) for n, s in new.items()}
        mine = {n: _Tail(s.t) for n, s in new.items()}        # the call's own copies
        given = {n: s if isinstance(new[n], _Scalar) else s.t for n, s in mine.items()}
        torch.cuda.synchronize()
        want = [t.clone() for t in call(given)]
        for last in new:
            t = new[last].t
            for rep in range(8):
                # something else, until the kernel in front of the call writes it (metadata: any of the six codes)
                mine[last].t.copy_(torch.full_like(t, 0x44) if t.dtype is U8 else torch.zeros_like(t) if rep % 2 else t.flip(0) * 0.5
                                   if t.dtype in (BF, torch.float32) else t.flip(0))
                torch.cuda.synchronize()
                torch.cuda._sleep(400000)
                ctx.pad_2d(new[last].whole.view(BF).view(-1, 128), mine[last].whole.view(BF).view(-1, 128))
                got = call(given)
                torch.cuda.synchronize()
                if not all(torch.equal(a.view(U8), b.view(U8)) for a, b in zip(got, want)):
                    bad.add((name, last))
    assert not bad, sorted(bad)
