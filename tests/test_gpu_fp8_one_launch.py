"""FP8 layers: maximum and quantisation of X, maximum and projection of W in one launch each, against the two single calls.

Bit for bit, at the sizes where the work per block changes, at the largest that one launch takes and beyond it; also with most SMs
busy, so that blocks which run work out the chunks of those that do not.
"""
import pytest
import torch

from paper_2409_09099_b200 import binding as B
from paper_2409_09099_b200.layer import SsteLinear

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    c = B.Context(0)
    yield c
    assert c.poll_device_status() == 0
    c.close()


def _randn(rows, cols, seed):
    return torch.empty((rows, cols), dtype=torch.bfloat16, device="cuda").normal_(
        generator=torch.Generator(device="cuda").manual_seed(seed))


def _bits(t):
    return t.contiguous().view(torch.uint8)


def _slots_empty(ctx, *layers):
    """the context's counters, in front of the partial tiles, and the layers' scratch are zero again"""
    torch.cuda.synchronize()
    return not ctx.workspace[17408:17408 + 4 * 8192].any() and not any(lin._scratch.view(torch.int32).any() for lin in layers)


def _check_x(ctx, X, Xq, amax):
    ref_amax, ref_q = torch.empty_like(amax), torch.empty_like(Xq)
    ctx.amax(X, ref_amax)
    ctx.quantize_fp8(X, ref_amax, ref_q)
    assert torch.equal(amax, ref_amax) and torch.equal(_bits(Xq), _bits(ref_q))


# T x I: the largest of two launches, the smallest of one; 296 blocks of one vector per thread, then two; four; the largest of one
# launch, the next of two
@pytest.mark.parametrize("T,I", [(1024, 896), (1024, 1024), (128, 9472), (128, 9600), (512, 9472), (1024, 9344), (1024, 9472), (1024, 9600)])
def test_quantised_input(ctx, T, I):
    W = _randn(128, I, 1) * 0.02
    lin = SsteLinear(ctx, W, T, fp8=True)
    lin.init_beta()
    lin.prune()
    X = _randn(T, I, T + I)
    X[-1, -1] = 77.0                                  # the maximum in the last chunk, then everywhere zero, then small again
    for scale in (1.0, 0.0, 0.25):
        lin.forward(X * scale)
        _check_x(ctx, X * scale, lin.Xq, lin.amax[0:1])
        assert _slots_empty(ctx, lin)


# O x I: one tile of 32 x 128 per block up to 592 of them, two up to 1184, four up to 1776, then two launches
@pytest.mark.parametrize("O,I", [(128, 128), (4736, 512), (2432, 1024), (4736, 1024), (4864, 1024), (7040, 1024), (7168, 1024)])
@pytest.mark.parametrize("dense_copy", [True, False])
def test_projected_weight(ctx, O, I, dense_copy):
    W = _randn(O, I, O + I) * 0.02
    W[-1, -4:] = torch.tensor([3.0, -2.0, 0.5, 0.25], dtype=torch.bfloat16)
    layers = [SsteLinear(ctx, W, 128, fp8=True, dense_copy=dense_copy) for _ in range(2)]
    layers[1].mark = lambda label: None               # the single calls
    for factor in (1.0, 0.5):
        for lin in layers:
            lin.init_beta()
            lin.prune()
        a, b = layers
        assert torch.equal(a.amax[1:2], b.amax[1:2])
        for name in ("vals", "meta") + (("w_dense",) if dense_copy else ()):
            assert torch.equal(_bits(getattr(a, name)), _bits(getattr(b, name))), name
        assert _slots_empty(ctx, *layers)
        W.mul_(factor * 0.5)


def test_blocks_that_cannot_run_are_not_waited_for(ctx):
    """A product on 80 SMs of another stream (its context cannot split it) leaves room for half of the blocks: the results are the same.
    (Whether blocks are overtaken here is a matter of time; test_chunks_that_others_work_out makes it so.)"""
    other, side = B.Context(0, minimal_workspace=True), torch.cuda.Stream()
    M, K = 10240, 16384
    busy = SsteLinear(other, _randn(M, 256, 3) * 0.02, K)          # grad_W: 40 tiles of the whole reduction
    busy.init_beta()
    busy.prune()
    busy.forward(_randn(K, 256, 4))
    busy.sparsify_grad(_randn(K, M, 5))
    T, I = 1024, 9472
    lin = SsteLinear(ctx, _randn(3712, I // 74, 6) * 0.02, 128, fp8=True)
    wide = SsteLinear(ctx, _randn(128, I, 7) * 0.02, T, fp8=True)
    for l in (lin, wide):
        l.init_beta()
        l.prune()
    X = _randn(T, I, 8)
    wide.forward(X)
    torch.cuda.synchronize()
    vals, codes = lin.vals.clone(), wide.Xq.clone()
    for _ in range(3):
        lin.vals.zero_()
        wide.Xq.zero_()
        torch.cuda.synchronize()
        with torch.cuda.stream(side):
            for _ in range(3):
                busy.grad_weight()
        wide.forward(X)
        lin.prune()
        torch.cuda.synchronize()
        assert torch.equal(_bits(wide.Xq), _bits(codes)) and torch.equal(_bits(lin.vals), _bits(vals))
        assert _slots_empty(ctx, lin, wide)
    assert other.poll_device_status() == 0


# one tile of W per block, two, four; one vector of X per thread, two, four, eight
@pytest.mark.parametrize("O,I,T", [(4736, 512, 2176), (4736, 1024, 2304), (6912, 1024, 4608), (128, 1024, 9216)])
def test_chunks_that_others_work_out(ctx, O, I, T):
    """Every other block keeps its maximum to itself: the others take its chunk over, and the words are empty afterwards all the same."""
    lin = SsteLinear(ctx, _randn(O, I, 1) * 0.02, T, fp8=True)
    lin.init_beta()
    lin.prune()
    X = _randn(T, I, 2)
    lin.forward(X)
    want = [t.clone() for t in (lin.amax, lin.vals, lin.meta, lin.w_dense, lin.Xq, lin.Y)]
    taken = torch.zeros(1, dtype=torch.int32, device="cuda")
    tiles = O // 32 * (I // 128)
    chunks = -(-tiles // (1 if tiles <= 592 else 2 if tiles <= 1184 else 4))
    vectors = T * I // 8
    chunks_x = -(-vectors // (512 * next(v for v in (1, 2, 4, 8) if vectors <= 296 * 512 * v)))
    ctx.debug_withhold_maxima(taken)
    try:
        for _ in range(20):
            lin.amax.zero_(), lin.vals.zero_(), lin.meta.zero_(), lin.w_dense.zero_(), lin.Xq.zero_(), taken.zero_()
            lin.prune()
            pruned = taken.clone()
            lin.forward(X)
            assert int(pruned) >= chunks // 2 and int(taken) - int(pruned) >= chunks_x // 2
            assert _slots_empty(ctx, lin)
            for a, b in zip((lin.amax, lin.vals, lin.meta, lin.w_dense, lin.Xq, lin.Y), want):
                assert torch.equal(_bits(a), _bits(b))
    finally:
        ctx.debug_withhold_maxima(None)


_UNUSUAL = [float("inf"), -float("inf"), float("nan"), 3.3e38, -3.3e38, 2.0 ** 127, 2.0 ** -133, -0.0]


def _with_unusual(t, at):
    """`t` with two unusual values in each of the groups of four `at`, every pair of them in turn"""
    flat, pick, k = t.clone().view(-1, 4), torch.tensor(_UNUSUAL, dtype=t.dtype, device=t.device), torch.arange(len(at), device=t.device)
    flat[list(at), 0], flat[list(at), 1] = pick[k % 8], pick[k // 8 % 8]
    return flat.view_as(t)


# one tile of W per block, two, four (of which the last block has fewer than four)
@pytest.mark.parametrize("O,I", [(4736, 512), (2432, 1024), (4864, 1024), (6912, 1024)])
@pytest.mark.parametrize("where", ["first", "last", "everywhere"])
def test_projection_of_any_values(ctx, O, I, where):
    groups = O * I // 4
    at = {"first": range(64), "last": range(groups - 64, groups), "everywhere": range(5, groups, groups // 300)}[where]
    W = _with_unusual(_randn(O, I, O) * 0.02, at)
    layers = [SsteLinear(ctx, W, 128, fp8=True) for _ in range(2)]
    layers[1].mark = lambda label: None               # the single calls
    for beta in (1.5, 0.0, float("inf"), float("nan")):
        for lin in layers:
            lin.beta.fill_(beta)
            lin.beta_ready = True
            lin.prune()
        a, b = layers
        assert torch.equal(_bits(a.amax[1:2]), _bits(b.amax[1:2])), beta
        for name in ("vals", "meta", "w_dense"):
            assert torch.equal(_bits(getattr(a, name)), _bits(getattr(b, name))), (beta, name)
        assert _slots_empty(ctx, *layers)


# one vector of X per thread, two, four, eight
@pytest.mark.parametrize("T,I", [(1024, 1024), (2176, 1024), (4608, 1024), (9216, 1024)])
def test_quantisation_of_any_values(ctx, T, I):
    lin = SsteLinear(ctx, _randn(128, I, 1) * 0.02, T, fp8=True)
    lin.init_beta()
    lin.prune()
    X = _randn(T, I, T)
    last = T * I // 4 - 1
    for at in (range(0), range(64), range(last - 63, last + 1), range(3, last, last // 500)):
        for values in ((0, 1, 2, 3, 4, 5, 6, 7), (3, 4, 5), (0, 3), (2, 6)):
            Z = X.clone().view(-1, 4)
            k = torch.arange(len(at), device="cuda")
            Z[list(at), k % 4] = torch.tensor([_UNUSUAL[v] for v in values], dtype=X.dtype, device="cuda")[k % len(values)]
            Z = Z.view_as(X)
            lin.forward(Z)
            ref_amax, ref_q = torch.empty_like(lin.amax[0:1]), torch.empty_like(lin.Xq)
            ctx.amax(Z, ref_amax)
            ctx.quantize_fp8(Z, ref_amax, ref_q)
            assert torch.equal(_bits(lin.amax[0:1]), _bits(ref_amax)) and torch.equal(_bits(lin.Xq), _bits(ref_q))
            assert _slots_empty(ctx, lin)


def test_layers_of_one_context_side_by_side(ctx):
    """Prunes need no context of their own (a product does): two at once leave what one after the other leaves."""
    own = B.Context(0)
    a, b, c = (SsteLinear(k, _randn(O, I, O) * s, 2048, seed=1, fp8=True)
               for k, O, I, s in ((ctx, 3072, 768, 0.02), (ctx, 768, 3072, 0.7), (own, 1280, 1280, 3.0)))
    X = _randn(2048, 1280, 5)
    for lin in (a, b, c):
        lin.init_beta()
        lin.prune()
    Y = c.forward(X).clone()
    watched = [t for lin in (a, b) for t in (lin.amax[1:2], lin.vals, lin.meta, lin.w_dense)]
    want = [t.clone() for t in watched]
    side = torch.cuda.Stream()
    for _ in range(50):
        for t in watched:
            t.zero_()
        c.Y.zero_()
        torch.cuda.synchronize()
        a.prune()
        with torch.cuda.stream(side):
            b.prune()
        c.forward(X)
        with torch.cuda.stream(side):
            b.prune()
        assert _slots_empty(ctx, a, b, c)
        assert all(torch.equal(_bits(t), _bits(w)) for t, w in zip(watched, want)) and torch.equal(_bits(c.Y), _bits(Y))
    assert own.poll_device_status() == 0
    own.close()


@pytest.mark.parametrize("minimal", [False, True])
def test_launches(minimal):
    """One launch in front of the product where the scratch has room, whatever the workspace; two with the former 8 bytes."""
    ctx = B.Context(0, minimal_workspace=minimal)
    try:
        lin = SsteLinear(ctx, _randn(256, 1024, 1) * 0.02, 1024, fp8=True)
        X = _randn(1024, 1024, 2)
        got = []
        for scratch in (lin._scratch, torch.zeros(2, dtype=torch.float32, device="cuda")):
            lin._scratch = scratch
            lin.init_beta()
            before = B.launch_count()
            lin.prune()
            pruned = B.launch_count()
            lin.forward(X)
            got.append((pruned - before, B.launch_count() - pruned, lin.Y.clone(), lin.vals.clone(), lin.amax.clone()))
            assert _slots_empty(ctx, lin)
        assert got[0][:2] == (1, 2) and got[1][:2] == (2, 3)
        assert all(torch.equal(_bits(p), _bits(q)) for p, q in zip(got[0][2:], got[1][2:]))
    finally:
        ctx.close()
