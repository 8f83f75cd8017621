"""The elementwise rules on values whose sums overflow, on infinities and on NaNs, against the rules restated in fp32 here.

Finite values are enough to need this: three gradients of 1e38 and one of 3e38 in a group have a sum beyond fp32.  A comparison
with a NaN is false and a NaN is never a maximum; results are compared bit for bit, NaNs as NaNs.
"""
import numpy as np
import pytest
import torch

from oracle import sste_oracle as orc
from paper_2409_09099_b200 import binding as B, synth
from tests.gpu_util import DEV, bits16, bits8, canonical_meta, dbf16

pytestmark = pytest.mark.gpu

INF, NAN = np.float32(np.inf), np.float32(np.nan)
# bf16 values; no two in a group of four are far enough apart to hide a third
ALPHABET = np.array([0.0, -0.0, 1.0, -2.0, 2.0 ** 125, -1.5 * 2.0 ** 126, 1.75 * 2.0 ** 127, -1.5 * 2.0 ** 127, INF, -INF, NAN,
                     2.0 ** -133], np.float32)


@pytest.fixture(scope="module")
def ctx():
    c = B.Context(0)
    yield c
    assert c.poll_device_status() == 0
    c.close()


def _groups():
    n = len(ALPHABET)
    return ALPHABET[np.stack(np.meshgrid(*[np.arange(n)] * 4, indexing="ij"), -1).reshape(-1, 4)]


def _f32(bits):
    return np.asarray(bits, np.uint32).view(np.float32)


def mvue_rule(a, u):
    """q0, q1, v0, v1 of groups a [n, 4] with uniforms u [n]: the rule of Sec. 5.1 by selections, every step one fp32 operation."""
    with np.errstate(all="ignore"):
        m = np.abs(a)
        mx = np.fmax.reduce(m, axis=1)
        hit = m[:, :3] == mx[:, None]
        x = np.where(hit.any(1), hit.argmax(1), 3)
        without = np.where(np.arange(4)[None] == x[:, None], np.float32(0), m)
        z = np.add.accumulate(without, axis=1, dtype=np.float32)
        s = np.add.accumulate(m, axis=1, dtype=np.float32)
        rest = z[:, 3]
        clipped = mx >= rest
        h = np.where(clipped, rest, np.float32(0.5) * s[:, 3])
        c = np.where(clipped[:, None], z[:, :3], s[:, :3])
        r1 = u * h
        r2 = r1 + h
        below = _f32(rest.view(np.uint32) - np.uint32(1))
        r1 = np.where(clipped, np.fmin(r1, below), r1)
        j1 = (c <= r1[:, None]).sum(1)
        n2 = (c <= r2[:, None]).sum(1)
        ia = np.where(clipped, np.where(rest == 0, np.where(x == 0, 1, 0), j1), np.minimum(j1, 2))
        ib = np.where(clipped, x, np.minimum(np.maximum(j1 + 1, n2), 3))
        rows = np.arange(len(a))
        sign = lambda i: np.where(h == 0, np.uint32(0), a[rows, i].view(np.uint32) & np.uint32(0x80000000))
        va = _f32(sign(ia) | h.view(np.uint32))
        vb = np.where(clipped, a[rows, ib], _f32(sign(ib) | h.view(np.uint32)))
    swap = ia > ib
    return np.minimum(ia, ib), np.maximum(ia, ib), np.where(swap, vb, va), np.where(swap, va, vb)


def _equal(got, want, is_nan):
    """Equal codes, or both NaN (whose payload and sign are the conversion's)."""
    return bool(((got == want) | (is_nan(got) & is_nan(want))).all())


_nan16 = lambda b: (b & 0x7fff) > 0x7f80
_nan_e5m2 = lambda b: (b & 0x7f) > 0x7c
_nan_e4m3 = lambda b: (b & 0x7f) == 0x7f


def _as_tokens(groups):
    """[T, O] with T = 768, O = 128: group i in column i % 128, token group i // 128."""
    g = np.zeros((192 * 128, 4), np.float32)
    g[: len(groups)] = groups
    return synth.to_bf16_bits(np.ascontiguousarray(g.reshape(192, 128, 4).transpose(0, 2, 1).reshape(768, 128)))


def _columns(bits):
    return synth.bf16_bits_to_f32(bits).reshape(192, 4, 128).transpose(2, 0, 1).reshape(-1, 4)        # [column, token group]


def test_mvue_groups(ctx):
    a = synth.bf16_bits_to_f32(synth.to_bf16_bits(_groups()))
    n = len(a)
    for k24 in (np.zeros(n, np.int64), np.full(n, (1 << 24) - 1), np.random.default_rng(3).integers(0, 1 << 24, n)):
        pos = torch.zeros(n, dtype=torch.int32, device=DEV)
        val = torch.zeros((n, 2), dtype=torch.float32, device=DEV)
        ctx.debug_mvue_groups(dbf16(synth.to_bf16_bits(a)), torch.from_numpy(k24.astype(np.int32)).to(DEV), pos, val)
        q0, q1, v0, v1 = mvue_rule(a, k24.astype(np.float32) * np.float32(2.0 ** -24))
        assert np.array_equal(pos.cpu().numpy(), q0 | (q1 << 2))
        nan = lambda b: (b & 0x7fffffff) > 0x7f800000
        assert _equal(val.cpu().numpy().view(np.uint32), np.stack([v0, v1], 1).view(np.uint32), nan)


@pytest.mark.parametrize("counter_cols", [0, 101])
@pytest.mark.parametrize("fp8", [False, True])
def test_mvue_sparsify(ctx, fp8, counter_cols):
    dY = _as_tokens(_groups())
    T, O = dY.shape
    seed, tid, step = 11, 3, 5
    cols = counter_cols or O
    # the uniforms: one Philox word per group (the oracle's stream, itself checked against known answers)
    g = (np.arange(T // 4, dtype=np.uint64)[None, :] * np.uint64(cols) + np.arange(O, dtype=np.uint64)[:, None]).reshape(-1)
    u = (_uniforms(seed, tid, step, g) * np.float32(2.0 ** -24)).astype(np.float32)
    q0, q1, v0, v1 = mvue_rule(_columns(dY), u)
    for amax in ((2.0 ** 127, np.inf, np.nan, 2.0 ** -140, 0.0) if fp8 else (None,)):
        dt = B.E5M2 if fp8 else B.BF16
        gvals, gmeta = ctx.alloc_compressed(O, T, dt)
        q = torch.zeros((T, O), dtype=torch.float8_e5m2, device=DEV) if fp8 else None
        ctx.mvue_sparsify(dbf16(dY), seed, tid, step, gvals, gmeta, dense_q_out=q, counter_cols=counter_cols,
                          g_amax_dev=torch.tensor([amax], dtype=torch.float32, device=DEV) if fp8 else None)
        v = np.stack([v0, v1], 1).reshape(O, T // 2)
        with np.errstate(all="ignore"):
            if fp8:
                s = np.float32(1) if amax == 0 else np.float32(57344) / np.float32(amax)
                assert _equal(bits8(gvals), orc.f32_to_fp8(v * s, orc.E5M2), _nan_e5m2)
                assert _equal(bits8(q), orc.f32_to_fp8(synth.bf16_bits_to_f32(dY) * s, orc.E5M2), _nan_e5m2)
            else:
                assert _equal(bits16(gvals), orc.f32_to_bf16(v), _nan16)
        code = (q0 | (q1 << 2)).reshape(O, T // 16, 4).astype(np.uint16)
        want = code[..., 0] | (code[..., 1] << 4) | (code[..., 2] << 8) | (code[..., 3] << 12)
        assert np.array_equal(canonical_meta(ctx, gmeta, O, T, dt), want)


def test_mvue_of_a_padded_gradient(ctx):
    """The pass that pads and sparsifies: the same results as padding first."""
    from paper_2409_09099_b200.layer import SsteLinearPadded
    rows, cols = 766, 101
    dY = dbf16(_as_tokens(_groups()))[:rows, :cols].contiguous()
    layers = [SsteLinearPadded(ctx, cols, 40, rows, seed=3) for _ in range(2)]
    layers[1].inner.mark = lambda label: None                          # the single calls
    W, X = dbf16(synth.gaussian_bf16(1, (cols, 40), 0.02)), dbf16(synth.gaussian_bf16(2, (rows, 40), 1.0))
    for l in layers:
        l.set_weight(W); l.init_beta(); l.prune(); l.forward(X); l.backward(dY, step=2)
    a, b = (l.inner for l in layers)
    assert torch.equal(a.gvals.view(torch.int16), b.gvals.view(torch.int16)) and torch.equal(a.gmeta, b.gmeta)


def _uniforms(seed, tid, step, g):
    """24-bit uniforms of group indices g."""
    block = g >> np.uint64(2)
    first, last = int(block.min()), int(block.max())
    words = np.empty((last - first + 1, 4), np.uint32)
    for i in range(first, last + 1):
        words[i - first] = orc.philox4x32_10((i & 0xffffffff, i >> 32, tid, step), (seed & 0xffffffff, seed >> 32))
    return (words[(block - np.uint64(first)).astype(np.int64), (g & np.uint64(3)).astype(np.int64)] >> 8).astype(np.float32)


def projection_rule(a, beta, s):
    """Kept positions and the four values of groups a [n, 4] (bf16 values): rank by magnitude bits, t the second-smallest."""
    key = (a.view(np.uint32) & np.uint32(0x7fffffff)).astype(np.int64) * 4 + (3 - np.arange(4))
    order = np.argsort(-key, axis=1)
    p = np.sort(order[:, :2], axis=1)
    with np.errstate(all="ignore"):
        t = np.abs(a[np.arange(len(a)), order[:, 2]])[:, None]
        v = (a - np.copysign(t, a)) * np.float32(beta) * np.float32(s)
        v = np.where(np.abs(a) > t, v, np.float32(0))
    return p, v.astype(np.float32)


@pytest.mark.parametrize("beta", [1.5, 0.0, np.inf, np.nan])
@pytest.mark.parametrize("fp8", [False, True])
def test_projection(ctx, fp8, beta):
    a = np.zeros((128 * 768 // 4, 4), np.float32)
    a[: len(_groups())] = _groups()
    W = synth.to_bf16_bits(a.reshape(128, 768))
    a = synth.bf16_bits_to_f32(W).reshape(-1, 4)
    dt = B.E4M3 if fp8 else B.BF16
    for amax in ((1.0, 2.0 ** 127, 2.0 ** -140, np.inf, np.nan) if fp8 else (None,)):
        vals, meta = ctx.alloc_compressed(128, 768, dt)
        dense = torch.empty((128, 768), dtype=B._TORCH_DT[dt], device=DEV)
        f32 = lambda x: torch.tensor([x], dtype=torch.float32, device=DEV)
        ctx.project_compress(dbf16(W), f32(beta), vals, meta, dense, w_amax_dev=f32(amax) if fp8 else None)
        with np.errstate(all="ignore"):
            p, v = projection_rule(a, beta, np.float32(448) / np.float32(amax) if fp8 else 1.0)
        code, nan, bits = ((lambda x: orc.f32_to_fp8(x, orc.E4M3), _nan_e4m3, bits8) if fp8 else (orc.f32_to_bf16, _nan16, bits16))
        assert _equal(bits(dense), code(v).reshape(128, 768), nan)
        assert _equal(bits(vals), code(np.take_along_axis(v, p, 1)).reshape(128, 384), nan)
        nib = (p[:, 0] | (p[:, 1] << 2)).reshape(128, 48, 4).astype(np.uint16)
        want = nib[..., 0] | (nib[..., 1] << 4) | (nib[..., 2] << 8) | (nib[..., 3] << 12)
        assert np.array_equal(canonical_meta(ctx, meta, 128, 768, dt), want)
