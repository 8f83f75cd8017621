"""One S-STE linear layer as a user of the library sees it: buffers + the call sequence.

This is bookkeeping only (which buffer goes to which C-ABI call, in the order the
paper's training iteration prescribes); every computation runs in libsste.
Straight-through estimator (Eq. 3): ``dW`` is the gradient with respect to the
sparse weight and is meant to be applied to the dense weight unchanged.
"""
from __future__ import annotations

import ctypes
from operator import index

import torch

from . import binding as B

# attributes the sste_layer descriptor is made of: setting one makes the next call build it anew
_DESCRIBED = frozenset(("ctx", "W", "T", "tensor_id", "seed", "fp8", "counter_cols", "beta", "vals", "meta", "w_dense",
                        "gvals", "gmeta", "Y", "dX", "dW", "amax", "Xq", "dYq", "_scratch", "sparsify_grad", "grad_weight",
                        "grad_input"))
# what a one-call phase stands for; a layer or context that brings its own version of one of these gets the single calls
_LAYER_CALLS = ("sparsify_grad", "grad_weight", "grad_input")
_CONTEXT_CALLS = ("project_amax", "project_compress", "amax", "quantize_fp8", "linear_fwd", "mvue_sparsify", "linear_bwd_weight",
                  "linear_bwd_input", "pad_2d", "crop_2d")
_bf16, _raw_stream, _device = torch.bfloat16, torch._C._cuda_getCurrentRawStream, torch._C._cuda_getDevice


def _as_defined(obj, cls, names):
    """Whether `obj` is a `cls` whose methods `names` are those of `cls` (no subclass, no attribute, overrides them)."""
    t = type(obj)
    return (isinstance(obj, cls) and vars(obj).keys().isdisjoint(names)
            and (t is cls or all(getattr(t, n) is getattr(cls, n) for n in names)))


def _takes(t, shape):
    """Whether a one-call phase can read `t` as it is; anything else goes to the single calls, which check it."""
    return t.dtype is _bf16 and t.shape == shape and t.is_cuda and t.is_contiguous()


def _same_places(tensors):
    """A check that the storage of `tensors` is where it is now.

    Unrolled for the bf16 phases of a layer with a dense copy, where the host sets the pace (0.3 us for five tensors, 0.5 in a
    loop)."""
    calls, at = [t.data_ptr for t in tensors], [t.data_ptr() for t in tensors]
    if len(calls) == 3:
        (a, b, c), (p, q, r) = calls, at
        return lambda: a() == p and b() == q and c() == r
    if len(calls) == 5:
        (a, b, c, d, e), (p, q, r, s, t) = calls, at
        return lambda: a() == p and b() == q and c() == r and d() == s and e() == t
    return lambda: [call() for call in calls] == at


class _Described:
    """sste_layer of a layer's buffers; per phase the C call and the check that the buffers it works on are where they were.

    A tensor may be given other storage without being replaced (`t.data = ...`, a storage resized to 0 and back)."""
    __slots__ = ("fits", "buffers", "at", "x_shape", "g_shape", "w_shape", "prune", "prune_there", "forward", "forward_there",
                 "backward", "backward_there", "grads")


class SsteLinear:
    """W[O, I] dense master weight (bf16); forward Y = X S(W)^T, backward (dX, dW).

    ``fp8=True`` selects the whole-process FP8 variant (Sec. 5.2): E4M3 forward
    operands, E5M2 output gradient, per-tensor scale = fp8_max / amax; the state of a
    quantised tensor is its amax (one device float), from which every consumer forms the
    scale itself.  ``dense_copy=True`` (the default, the faster route on B200) also keeps w~ as a
    dense [O, I] tensor and feeds grad_X from it; with ``dense_copy=False`` the layer keeps none and
    grad_X expands the compressed operand for the length of the call (less memory, slower).
    ``track_flips=True`` keeps the previous iteration's metadata and counts the mask entries
    that changed at every prune (flip rate, Sec. 3.1).
    """

    def __init__(self, ctx: B.Context, W: torch.Tensor, T: int, tensor_id: int = 0, seed: int = 0,
                 fp8: bool = False, out_dtype: torch.dtype = torch.bfloat16, track_flips: bool = False,
                 dense_copy: bool = True, counter_cols: int = 0):
        assert W.dtype == torch.bfloat16 and W.is_cuda
        O, I = W.shape
        dev, empty = W.device, torch.empty
        wdt, gdt = (B._TORCH_DT[B.E4M3], B._TORCH_DT[B.E5M2]) if fp8 else (_bf16, _bf16)
        # scalars in one zeroed tensor: beta; FP8: max|X|, max|w~| (bf16 projection), max|dY| and the amax passes' scratch
        scalars = torch.zeros(4 + B.LAYER_SCRATCH_BYTES // 4 if fp8 else 1, dtype=torch.float32, device=dev)
        buffers = dict(
            ctx=ctx, W=W, T=T, tensor_id=tensor_id, seed=seed, fp8=fp8, O=O, I=I, counter_cols=counter_cols,
            beta=scalars[0:1] if fp8 else scalars, beta_ready=False,
            vals=empty((O, I // 2), dtype=wdt, device=dev), meta=empty(O * I // 8, dtype=torch.uint8, device=dev),
            w_dense=empty((O, I), dtype=wdt, device=dev) if dense_copy else None,
            gvals=empty((O, T // 2), dtype=gdt, device=dev), gmeta=empty(O * T // 8, dtype=torch.uint8, device=dev),
            Y=empty((T, O), dtype=out_dtype, device=dev), dX=empty((T, I), dtype=out_dtype, device=dev),
            dW=empty((O, I), dtype=out_dtype, device=dev),
            launches=0,        # library calls, also those that a phase call stands for
            mark=None,         # optional callback(label), called before every C-ABI call (a benchmark records events)
            track_flips=track_flips,
            amax=scalars[1:4] if fp8 else None,
            Xq=empty((T, I), dtype=wdt, device=dev) if fp8 else None,
            dYq=empty((T, O), dtype=gdt, device=dev) if fp8 else None,
            _scratch=scalars[4:] if fp8 else None,
            _desc=None, _as_made=W.is_contiguous())
        self.__dict__.update(buffers)
        if track_flips:
            self.meta_prev = torch.empty_like(self.meta)
            self.flips = torch.zeros(1, dtype=torch.int64, device=dev)   # mask entries changed by the last prune
            self._have_prev = False

    def __setattr__(self, name, value):
        d = self.__dict__
        if name in _DESCRIBED:
            d["_desc"] = None
            d["_as_made"] = False
        d[name] = value

    # One C call per phase (prune, forward, backward) on buffers described once: what a small layer costs is host time.
    # The per-call path below it runs when something wants to see the single calls or the tensors are of other sizes.
    def _describe(self):
        tensors = (self.W, self.beta, self.amax, self.vals, self.meta, self.w_dense, self.gvals, self.gmeta, self.Xq,
                   self.dYq, self.Y, self.dX, self.dW, self._scratch)
        x_shape, g_shape = torch.Size((self.T, self.I)), torch.Size((self.T, self.O))
        self.__dict__["_desc"] = desc = _Described()
        # a layer whose buffers were replaced by ones of other sizes or types is not described: the single calls check it
        desc.fits = (_as_defined(self, SsteLinear, _LAYER_CALLS) and _as_defined(self.ctx, B.Context, _CONTEXT_CALLS)
                     and (self._as_made or self._replaced_fit(x_shape, g_shape, tensors)))
        if not desc.fits:
            desc.prune_there = desc.forward_there = desc.backward_there = lambda: True
            return desc
        scratch_bytes = B.LAYER_SCRATCH_BYTES if self.fp8 and self._scratch.nbytes >= B.LAYER_SCRATCH_BYTES else 0
        d = B.LayerBuffers(self.O, self.I, self.T, B.E4M3 if self.fp8 else B.BF16, B._CODE_OF[self.Y.dtype],
                           self.counter_cols, index(self.tensor_id) & 0xffffffff, scratch_bytes, index(self.seed) & 0xffffffffffffffff,
                           *[None if t is None else t.data_ptr() for t in tensors])
        lib = self.ctx.lib
        desc.buffers, desc.at, desc.x_shape, desc.g_shape = d, ctypes.addressof(d), x_shape, g_shape
        desc.w_shape = torch.Size((self.O, self.I))
        w = (self.vals, self.meta) if self.w_dense is None else (self.w_dense,)
        there = lambda *tensors: _same_places([t for t in tensors if t is not None])
        desc.prune, desc.forward, desc.backward, desc.grads = (lib.sste_layer_prune, lib.sste_layer_forward,
                                                               lib.sste_layer_backward, lib.sste_layer_grads)
        fp8 = (self.amax, self._scratch)
        desc.prune_there = there(self.W, self.beta, self.vals, self.meta, self.w_dense, *fp8)
        desc.forward_there = there(self.vals, self.meta, self.Y, self.Xq, *fp8)
        desc.backward_there = there(self.gvals, self.gmeta, self.dW, self.dX, *w, self.Xq, self.dYq, *fp8)
        return desc

    def _moved(self):
        self.__dict__["_as_made"] = False
        return self._describe()

    def _replaced_fit(self, x_shape, g_shape, tensors):
        wdt, gdt = (B._TORCH_DT[B.E4M3], B._TORCH_DT[B.E5M2]) if self.fp8 else (_bf16, _bf16)
        w_shape = (self.O, self.I)
        return (all(t is None or (t.is_cuda and t.is_contiguous()) for t in tensors)
                and self.W.dtype is _bf16 and tuple(self.W.shape) == w_shape and self.beta.dtype is torch.float32
                and self.beta.numel() >= 1 and self.meta.nbytes == self.O * self.I // 8
                and self.gmeta.nbytes == self.O * self.T // 8
                and self.vals.dtype is wdt and tuple(self.vals.shape) == (self.O, self.I // 2)
                and self.gvals.dtype is gdt and tuple(self.gvals.shape) == (self.O, self.T // 2)
                and (self.w_dense is None or (self.w_dense.dtype is wdt and tuple(self.w_dense.shape) == w_shape))
                and self.Y.shape == g_shape and self.dX.shape == x_shape and tuple(self.dW.shape) == w_shape
                and self.dX.dtype is self.Y.dtype and self.dW.dtype is self.Y.dtype
                and (not self.fp8 or (self.amax.dtype is torch.float32 and self.amax.numel() == 3
                                      and self._scratch.nbytes >= 8 and self.Xq.dtype is wdt and self.Xq.shape == x_shape
                                      and self.dYq.dtype is gdt and self.dYq.shape == g_shape)))

    def _amax(self, k):
        return self.amax[k:k + 1] if self.fp8 else None

    def _m(self, label):
        if self.mark is not None:
            self.mark(label)

    # (0) first iteration only: beta is computed once and then frozen (Sec. 4.2)
    def init_beta(self):
        self.ctx.beta_init(self.W, self.beta)
        self.beta_ready = True
        self.launches += 1

    # (1) prune: w~ = beta * S_soft(W), compressed for the sparse products (and for grad_X)
    def prune(self):
        assert self.beta_ready, "call init_beta() in the first iteration"
        if self.mark is None and not self.track_flips:
            desc = self._desc or self._describe()
            if not desc.prune_there():
                desc = self._moved()
            W = self.W                                            # the caller's: it may be another view by now
            if desc.fits and W.dtype is _bf16 and W.shape == desc.w_shape and W.is_contiguous():
                st = desc.prune(self.ctx.handle, desc.at, _raw_stream(_device()))
                if st:
                    self.ctx._check(st)
                self.__dict__["launches"] += 2 if self.fp8 else 1
                return
        c = self.ctx
        if self.track_flips:
            self.meta, self.meta_prev = self.meta_prev, self.meta     # last iteration's image becomes "previous"
        if self.fp8:
            # the scale of w~ needs amax(w~) first: one read-only pass over W, then the cast to E4M3
            self._m("project_amax")
            c.project_amax(self.W, self.beta, self.amax[1:2])
            self.launches += 1
        self._m("project_compress")
        c.project_compress(self.W, self.beta, self.vals, self.meta, self.w_dense, w_amax_dev=self._amax(1))
        self.launches += 1
        if self.track_flips:
            if self._have_prev:
                self._m("flip_count")
                c.flip_count(self.meta_prev, self.meta, self.O, self.I, self.flips)
                self.launches += 1
            self._have_prev = True

    def flip_rate(self) -> float:
        """r_k of the last prune (synchronises); 0 before the second prune."""
        return float(self.flips.item()) / (self.O * self.I)

    # (2a) forward with the sparse weight
    def forward(self, X, y_amax_out=None):
        if self.mark is None:
            desc = self._desc or self._describe()
            if not desc.forward_there():
                desc = self._moved()
            if desc.fits and _takes(X, desc.x_shape):
                st = desc.forward(self.ctx.handle, desc.at, X.data_ptr(), None if y_amax_out is None else B._ptr(y_amax_out),
                                  _raw_stream(_device()))
                if st:
                    self.ctx._check(st)
                d = self.__dict__
                if self.fp8:
                    d["launches"] += 3
                else:
                    d["X"] = X
                    d["launches"] += 1
                return self.Y
        c = self.ctx
        if not self.fp8:
            self.X = X
            self._m("linear_fwd")
            c.linear_fwd(X, self.vals, self.meta, self.Y, y_amax_out_dev=y_amax_out)
            self.launches += 1
            return self.Y
        self._m("amax_x")
        c.amax(X, self.amax[0:1])
        self._m("quantize_x")
        c.quantize_fp8(X, self.amax[0:1], self.Xq)
        self._m("linear_fwd")
        c.linear_fwd(self.Xq, self.vals, self.meta, self.Y, x_amax_dev=self.amax[0:1], w_amax_dev=self.amax[1:2],
                     y_amax_out_dev=y_amax_out)
        self.launches += 3
        return self.Y

    # (2b) backward: MVUE on the output gradient for grad_W, dense product for grad_X
    def backward(self, dY, step: int = 0, token_offset: int = 0):
        if self.mark is None:
            desc = self._desc or self._describe()
            if not desc.backward_there():
                desc = self._moved()
            X = None if self.fp8 else self.X
            if desc.fits and _takes(dY, desc.g_shape) and (X is None or _takes(X, desc.x_shape)):
                st = desc.backward(self.ctx.handle, desc.at, None if X is None else X.data_ptr(), dY.data_ptr(), step,
                                      token_offset, _raw_stream(_device()))
                if st:
                    self.ctx._check(st)
                self.__dict__["launches"] += 4 if self.fp8 else 3
                return self.dX, self.dW
        self.sparsify_grad(dY, step, token_offset)
        self.grad_weight()
        self.grad_input(dY)
        return self.dX, self.dW

    def grad_input_mvue_weight(self, dY, step: int = 0, tensor_id_w: int | None = None):
        """Ablation (Sec. 5.1, the variant the paper rejects): grad_X = dY MVUE(S(W)^T)^T on sparse tensor cores.

        The sparsified operand must be 2:4 along the contraction dim O, so MVUE runs on w~ viewed as [O, I]
        (groups of four consecutive rows), giving the compressed [I, O] operand; the product is then the
        forward-type call with dY as the K-major operand.  bf16 only.  Composed of existing calls.
        """
        assert not self.fp8
        c = self.ctx
        if not hasattr(self, "wt_vals"):
            self.wt_vals, self.wt_meta = c.alloc_compressed(self.I, self.O, B.BF16)
            self.wt_dense = torch.empty((self.O, self.I), dtype=torch.bfloat16, device=self.W.device)
        tid = self.tensor_id + (1 << 16) if tensor_id_w is None else tensor_id_w     # a stream of its own
        c.decompress(self.vals, self.meta, self.wt_dense)
        c.mvue_sparsify(self.wt_dense, self.seed, tid, step, self.wt_vals, self.wt_meta)
        c.linear_fwd(dY, self.wt_vals, self.wt_meta, self.dX)
        self.launches += 3
        return self.dX

    def grad_weight_and_input(self, dY, side_ctx: B.Context, side_stream: torch.cuda.Stream):
        """grad_W and grad_X at the same time: they are independent once MVUE has run.  Where one launch for both is the
        clearly faster way (bf16 results, see sste_layer_grads_beside), it runs on the current stream and shares the SMs between them;
        otherwise grad_W runs on `side_stream` (through `side_ctx`: its own split-K workspace) beside grad_X, which takes about
        as long as one after the other (10496 x 768, 4096 tokens, FP8: 54.0 against 56.7 us; 8064 x 384, 4352 tokens: 53.3 against
        51.0).  `backward` alone is often faster by now: it takes one launch more often.
        Both are complete in current-stream order on return."""
        if self.mark is None:
            desc = self._desc or self._describe()
            if not desc.backward_there():
                desc = self._moved()
            X = None if self.fp8 else self.X
            if (desc.fits and _takes(dY, desc.g_shape) and (X is None or _takes(X, desc.x_shape))
                    and not self.ctx.lib.sste_layer_grads_beside(self.ctx.handle, desc.at)):
                st = desc.grads(self.ctx.handle, desc.at, None if X is None else X.data_ptr(), dY.data_ptr(),
                                   _raw_stream(_device()))
                if st:
                    self.ctx._check(st)
                self.__dict__["launches"] += 2
                return self.dX, self.dW
        main = torch.cuda.current_stream()
        side_stream.wait_stream(main)
        with torch.cuda.stream(side_stream):
            saved, self.__dict__["ctx"] = self.ctx, side_ctx       # (not a new context of the layer: nothing to describe)
            try:
                self.grad_weight()
            finally:
                self.__dict__["ctx"] = saved
        self.grad_input(dY)
        main.wait_stream(side_stream)
        return self.dX, self.dW

    # (2b.1) MVUE(dY^T): 2:4 along tokens, compressed and transposed for the grad_W product
    def sparsify_grad(self, dY, step: int = 0, token_offset: int = 0):
        c = self.ctx
        if self.fp8:
            self._m("amax_g")
            c.amax(dY, self.amax[2:3])
            self.launches += 1
        self._m("mvue_sparsify")
        c.mvue_sparsify(dY, self.seed, self.tensor_id, step, self.gvals, self.gmeta,
                        dense_q_out=self.dYq if self.fp8 else None, g_amax_dev=self._amax(2),
                        token_offset=token_offset, counter_cols=self.counter_cols)
        self.launches += 1

    # (2b.2) grad_W = MVUE(dY^T) X, sparse
    def grad_weight(self, ctx: B.Context | None = None):
        self._m("linear_bwd_weight")
        (ctx or self.ctx).linear_bwd_weight(self.gvals, self.gmeta, self.Xq if self.fp8 else self.X, self.dW,
                                            g_amax_dev=self._amax(2), x_amax_dev=self._amax(0))
        self.launches += 1
        return self.dW

    # (2b.3) grad_X = dY w~, dense; w~ from the compressed operand unless a dense copy is kept
    def grad_input(self, dY, dx_amax_out=None):
        g = self.dYq if self.fp8 else dY
        self._m("linear_bwd_input")
        if self.w_dense is not None:
            self.ctx.linear_bwd_input(g, self.w_dense, self.dX, g_amax_dev=self._amax(2), w_amax_dev=self._amax(1),
                                      dx_amax_out_dev=dx_amax_out)
        else:
            self.ctx.linear_bwd_input(g, None, self.dX, g_amax_dev=self._amax(2), w_amax_dev=self._amax(1),
                                      vals=self.vals, meta=self.meta, dx_amax_out_dev=dx_amax_out)
        self.launches += 1
        return self.dX


class SsteLinearPadded:
    """An S-STE linear of ANY shape (W[O, I], T tokens), run on zero-padded copies.

    The library's kernels want multiples of 128.  Zero groups are fixed points of the projection (Eq. 4) and of
    the MVUE rule and add nothing to beta, to an amax or to a product, so padding W, X and dY with zeros and
    cropping Y, dX and dW gives the unpadded results; the MVUE counter runs over the unpadded column count.
    The pad and crop passes are library kernels too (sste_pad_2d / sste_crop_2d); a result whose columns need no
    cropping is the first rows of the inner layer's buffer.
    """

    def __init__(self, ctx: B.Context, O: int, I: int, T: int, **kw):
        self.ctx, self.O, self.I, self.T = ctx, O, I, T
        self.Op, self.Ip, self.Tp = B.padded_dim(O), B.padded_dim(I), B.padded_dim(T)
        dev = f"cuda:{ctx.device}"
        bf = dict(dtype=torch.bfloat16, device=dev)
        self.Wp = torch.empty((self.Op, self.Ip), **bf)
        self.Xp = torch.empty((self.Tp, self.Ip), **bf)
        self.dYp = torch.empty((self.Tp, self.Op), **bf)
        self.inner = SsteLinear(ctx, self.Wp, self.Tp, counter_cols=O, **kw)
        rows = lambda t, r, c: t[:r] if t.dtype is _bf16 and t.shape[1] == c else torch.empty((r, c), **bf)
        self.Y, self.dX, self.dW = rows(self.inner.Y, T, O), rows(self.inner.dX, T, I), rows(self.inner.dW, O, I)
        self._desc = None

    @property
    def beta(self):
        return self.inner.beta

    def set_weight(self, W):
        self.ctx.pad_2d(W, self.Wp)

    def init_beta(self):
        self.inner.init_beta()

    def prune(self):
        self.inner.prune()

    # Descriptor of the one-call path for the inner layer's `of`, made anew when that is or when a buffer of this layer is
    # replaced or given other storage; None: the single calls take it.
    def _described(self, of):
        d = self._desc
        if d is not None and d[0] is of and d[2]():
            xp, dyp, y, dx, dw = d[1]
            if self.Xp is xp and self.dYp is dyp and self.Y is y and self.dX is dx and self.dW is dw:
                return d[4] if d[3] else None
        bufs, inner = (self.Xp, self.dYp, self.Y, self.dX, self.dW), self.inner
        crop = lambda t, whole: None if t.data_ptr() == whole.data_ptr() else B._ptr(t)
        p = B.PaddedLayerBuffers(of.buffers, self.O, self.I, self.T, 0, B._ptr(self.Xp), B._ptr(self.dYp),
                                 crop(self.Y, inner.Y), crop(self.dX, inner.dX), crop(self.dW, inner.dW))
        fits = (inner.Y.dtype is _bf16 and tuple(self.Xp.shape) == (self.Tp, self.Ip)
                and tuple(self.dYp.shape) == (self.Tp, self.Op) and tuple(self.Y.shape) == (self.T, self.O)
                and tuple(self.dX.shape) == (self.T, self.I) and tuple(self.dW.shape) == (self.O, self.I)
                and all(t.dtype is _bf16 and t.is_cuda and t.is_contiguous() for t in bufs))
        self._desc = of, bufs, _same_places(bufs), fits, ctypes.addressof(p), p
        return ctypes.addressof(p) if fits else None

    def _crop(self, src, dst):
        if src.data_ptr() != dst.data_ptr():
            self.ctx.crop_2d(src, dst)

    def forward(self, X):
        inner = self.inner
        at = None
        if inner.mark is None and _takes(X, (self.T, self.I)):
            of = inner._desc or inner._describe()
            if not of.forward_there():
                of = inner._moved()
            at = self._described(of) if of.fits else None
        if at is not None:
            st = self.ctx.lib.sste_padded_forward(self.ctx.handle, at, X.data_ptr(), _raw_stream(_device()))
            if st:
                self.ctx._check(st)
            inner = inner.__dict__
            if not self.inner.fp8:
                inner["X"] = self.Xp
            inner["launches"] += 3 if self.inner.fp8 else 1
            return self.Y
        self.ctx.pad_2d(X, self.Xp)
        self.inner.forward(self.Xp)
        self._crop(self.inner.Y, self.Y)
        return self.Y

    def backward(self, dY, step: int = 0):
        # (the inner layer's input is Xp after a forward; without one, or after somebody gave it another, the single calls tell)
        inner = self.inner
        at = None
        if inner.mark is None and (inner.fp8 or inner.__dict__.get("X") is self.Xp) and _takes(dY, (self.T, self.O)):
            of = inner._desc or inner._describe()
            if not of.backward_there():
                of = inner._moved()
            at = self._described(of) if of.fits else None
        if at is not None:
            st = self.ctx.lib.sste_padded_backward(self.ctx.handle, at, dY.data_ptr(), step, 0, _raw_stream(_device()))
            if st:
                self.ctx._check(st)
            self.inner.__dict__["launches"] += 4 if self.inner.fp8 else 3
            return self.dX, self.dW
        self.ctx.pad_2d(dY, self.dYp)
        self.inner.backward(self.dYp, step=step)
        self._crop(self.inner.dX, self.dX)
        self._crop(self.inner.dW, self.dW)
        return self.dX, self.dW
