"""Performance cases of the S-STE linear layer, through the layer classes a training or serving program uses.

A case is one layer shape and one thing done with it:

  op = "train"    one training iteration of the layer: prune the dense weight, forward, backward (grad_X, grad_W)
  op = "forward"  the forward alone with a weight that was pruned before (evaluation, serving)

with O, I, T = out features, in features, tokens, and the options of the layer: `fp8` (the whole-process FP8 variant),
`dense_copy` (False: no dense copy of the pruned weight is kept), `overlap` (grad_W on a side stream beside grad_X) and
`padded` (a shape that is not a multiple of 128, run through SsteLinearPadded).

Sizes are those of `synth.CONFIGS` (GPT-2-small, GPT-2-large and 7B-shaped linears) and of the padded-shape tests.
"""
from __future__ import annotations

import torch

from paper_2409_09099_b200 import binding as B
from paper_2409_09099_b200.layer import SsteLinear, SsteLinearPadded

# widest layer and longest batch of the shipped configurations
MAX_FEATURES, MAX_TOKENS, MIN_DIM = 11008, 16384, 128
# the largest listed case in multiply-adds of one dense product, a bf16 one counted twice (half the FP8 rate)
LARGEST = 11008 * 4096 * 16384


def _case(op, O, I, T, fp8=False, dense_copy=True, overlap=False, padded=False):
    return dict(op=op, O=O, I=I, T=T, fp8=fp8, dense_copy=dense_copy, overlap=overlap, padded=padded)


def listed():
    return [
        # the smallest layer of the repository's configurations: launches and host work are what it costs
        dict(name="layer_256", **_case("train", 256, 256, 512)),
        # GPT-2-small block, 8 x 1024 tokens: attention output, both MLP layers; the second with the backward's two
        # products on two streams, as the benchmark runs them
        dict(name="small_proj", **_case("train", 768, 768, 8192)),
        dict(name="small_fc1", **_case("train", 3072, 768, 8192)),
        dict(name="small_fc2_overlap", **_case("train", 768, 3072, 8192, overlap=True)),
        # the same MLP layer in FP8
        dict(name="small_fc1_fp8", **_case("train", 3072, 768, 8192, fp8=True)),
        # GPT-2-large block, 16 x 1024 tokens; the second MLP layer without the dense weight copy, to save memory
        dict(name="large_qkv", **_case("train", 3840, 1280, 16384)),
        dict(name="large_fc2_lean", **_case("train", 1280, 5120, 16384, dense_copy=False)),
        # 7B-shaped FFN in FP8: the largest workload
        dict(name="ffn_up_fp8", **_case("train", 11008, 4096, 16384, fp8=True)),
        # vocabulary projection on a batch of 1000 tokens, and a small odd shape: padded and cropped on the way
        dict(name="vocab_padded", **_case("train", 50257, 768, 1000, padded=True)),
        dict(name="odd_padded", **_case("train", 203, 80, 72, padded=True)),
        # serving: a short batch through one layer, bf16 and FP8
        dict(name="serve_small", **_case("forward", 3072, 768, 128)),
        dict(name="serve_ffn_fp8", **_case("forward", 4096, 11008, 256, fp8=True)),
    ]


def draw(rng):
    while True:
        def size(hi):
            return int(round(MIN_DIM * (hi / MIN_DIM) ** rng.random()))

        op = "forward" if rng.random() < 0.25 else "train"
        fp8 = rng.random() < 0.35
        O, I, T = size(MAX_FEATURES), size(MAX_FEATURES), size(MAX_TOKENS)
        padded = rng.random() < 0.2
        if not padded:
            O, I, T = (max(MIN_DIM, (v + 64) // 128 * 128) for v in (O, I, T))
        train = op == "train" and not padded
        dense_copy = not (train and rng.random() < 0.15)
        overlap = train and rng.random() < 0.2
        # the compressed-weight route and the padding passes cost more than the plain layer
        cost = O * I * T * (1 if fp8 else 2) * (1 if dense_copy else 2) * (2 if padded else 1)
        if cost <= LARGEST:
            return _case(op, O, I, T, fp8, dense_copy, overlap, padded)


_contexts = None


def _ctx():
    """One context for the main stream and one for the side stream, kept for the life of the program."""
    global _contexts
    if _contexts is None:
        _contexts = (B.Context(0), B.Context(0), torch.cuda.Stream())
    return _contexts


def prepare(case, seed):
    ctx, side_ctx, side_stream = _ctx()
    O, I, T = case["O"], case["I"], case["T"]
    gen = torch.Generator(device="cuda").manual_seed(seed)

    def gaussian(rows, cols, sigma):
        return torch.empty((rows, cols), dtype=torch.bfloat16, device="cuda").normal_(0.0, sigma, generator=gen)

    W, X = gaussian(O, I, 0.02), gaussian(T, I, 1.0)
    s = dict(case=case, X=X, W=W, step=seed % 1000, side_ctx=side_ctx, side_stream=side_stream)
    if case["op"] == "train":
        s["dY"] = gaussian(T, O, 1e-2)
    if case["padded"]:
        lin = SsteLinearPadded(ctx, O, I, T, tensor_id=3, seed=seed, fp8=case["fp8"])
        lin.set_weight(W)
    else:
        lin = SsteLinear(ctx, W, T, tensor_id=3, seed=seed, fp8=case["fp8"], dense_copy=case["dense_copy"])
    lin.init_beta()       # first iteration only: beta is frozen afterwards
    lin.prune()
    s["lin"] = lin
    return s


def run(state):
    case, lin = state["case"], state["lin"]
    if case["op"] == "forward":
        return {"Y": lin.forward(state["X"])}
    if case["padded"]:
        lin.set_weight(state["W"])       # the optimiser has updated the dense weight
        inner = lin.inner
    else:
        inner = lin
    lin.prune()
    Y = lin.forward(state["X"])
    if case["overlap"]:
        lin.sparsify_grad(state["dY"], step=state["step"])
        dX, dW = lin.grad_weight_and_input(state["dY"], state["side_ctx"], state["side_stream"])
    else:
        dX, dW = lin.backward(state["dY"], step=state["step"])
    return {"Y": Y, "dX": dX, "dW": dW, "vals": inner.vals, "meta": inner.meta}


def work(case):
    O, I, T = case["O"], case["I"], case["T"]
    elt = 1 if case["fp8"] else 2
    compressed = O * I * (0.5 * elt + 0.125)
    if case["op"] == "forward":
        # X and the compressed weight in, Y out; half of the multiply-adds of the dense product
        return {"bytes": 2 * T * I + compressed + 2 * T * O, "flops": 1 * T * O * I}
    # W, X, dY in; Y, dX, dW and the compressed weight out; forward and grad_W at half the multiply-adds, grad_X dense
    return {"bytes": 2 * (2 * O * I + 2 * T * I + 2 * T * O) + compressed, "flops": 4 * T * O * I}


def tolerance(case):
    # bf16 results of fp32 sums: half a unit in the last place is 2^-9 of a value; metadata bytes are exact
    return {"rel": 1e-2}
