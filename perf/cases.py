"""The work a user of the 2:4-sparse linear layer has the library do, as cases that can be timed and compared.

Five kinds of pass, each through the calls of ``paper_2608_24070_b200.binding`` in the order a program makes them:

* ``train``  one layer's training step: forward (with the lazy adapters fused in when there are any), adapter
             gradients, input gradient from the doubly pruned weight, compressed weight gradient;
* ``infer``  the four linears of a decoder block at inference: q, k, v stacked, o, gate and up stacked, down;
* ``setup``  both pruning passes of a weight matrix in one launch, compressed copies, metadata and masks;
* ``tail``   what the optimizer step leaves to the library: weight decay on the compressed gradient, refresh of the
             transposed copy from the new weights;
* ``nm``     one training step of a layer whose N:M pattern is re-selected every step and emulated on dense products.

Weights, masks, adapter factors and output buffers are what a program keeps between steps; every pass reads all its
inputs and writes all its outputs anew.
"""
import math

import torch

from paper_2608_24070_b200 import binding as B


def listed():
    return [
        # one small layer at a small batch: three short launches, bound by latency and by the cost of a call
        {"name": "train_512", "kind": "train", "tokens": 256, "d_in": 512, "d_out": 512, "r": 0},
        # an attention input projection of a small model with a ragged batch and the narrowest adapters
        {"name": "train_qkv_ragged", "kind": "train", "tokens": 1000, "d_in": 768, "d_out": 2304, "r": 16},
        # the MLP of a small model at its pretraining batch: short reductions, many tokens
        {"name": "train_gpt2_fc", "kind": "train", "tokens": 8192, "d_in": 768, "d_out": 3072, "r": 0},
        # a square attention projection of a 7B model in the adapter phase, at its pretraining batch
        {"name": "train_7b_q", "kind": "train", "tokens": 16384, "d_in": 4096, "d_out": 4096, "r": 64},
        # the down projection of the same model before the adapters come in (most of the training run)
        {"name": "train_7b_down", "kind": "train", "tokens": 16384, "d_in": 11008, "d_out": 4096, "r": 0},
        # the gate / up projection of a 13B model with wide adapters, half the batch
        {"name": "train_13b_up", "kind": "train", "tokens": 8192, "d_in": 5120, "d_out": 13824, "r": 128},
        # decoding one sequence: a block's weights are read for a single token
        {"name": "decode_7b_1", "kind": "infer", "tokens": 1, "d": 4096, "ffn": 11008, "r": 0},
        # decoding a small batch with adapters
        {"name": "decode_7b_8_r64", "kind": "infer", "tokens": 8, "d": 4096, "ffn": 11008, "r": 64},
        # a prompt of odd length with adapters
        {"name": "prefill_7b_500_r64", "kind": "infer", "tokens": 500, "d": 4096, "ffn": 11008, "r": 64},
        # pruning a 7B gate / up matrix when the masks are made
        {"name": "setup_7b_up", "kind": "setup", "d_in": 4096, "d_out": 11008},
        # every step's refresh of a 13B gate / up matrix
        {"name": "tail_13b_up", "kind": "tail", "d_in": 5120, "d_out": 13824},
        # an accuracy experiment with 2:8 sparsity on a 7B attention projection
        {"name": "nm_2of8_7b_q", "kind": "nm", "tokens": 2048, "d_in": 4096, "d_out": 4096, "n": 2, "m": 8},
    ]


def _log_uniform(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def _dim(rng, lo, hi):
    """A layer width: a multiple of 128, as the library takes them."""
    return 128 * max(1, round(_log_uniform(rng, lo, hi) / 128))


def _cap_tokens(tokens, n_weights, most):
    return max(1, min(tokens, int(most // n_weights)))


def draw(rng):
    kind = rng.choices(["train", "infer", "setup", "tail", "nm"], [8, 6, 2, 2, 2])[0]
    rank = lambda: rng.choice([0, 0, 16, 32, 64, 64, 128, 256])
    if kind == "train":
        d_in, d_out = _dim(rng, 512, 13824), _dim(rng, 512, 13824)
        tokens = _cap_tokens(round(_log_uniform(rng, 256, 16384)), d_in * d_out, 16384 * 4096 * 8192)
        return {"kind": kind, "tokens": tokens, "d_in": d_in, "d_out": d_out, "r": rank()}
    if kind == "infer":
        d = _dim(rng, 768, 5120)
        ffn = 128 * round(d * rng.uniform(2.5, 4.0) / 128)
        return {"kind": kind, "tokens": round(_log_uniform(rng, 1, 2048)), "d": d, "ffn": ffn, "r": rank()}
    if kind in ("setup", "tail"):
        return {"kind": kind, "d_in": _dim(rng, 768, 13824), "d_out": _dim(rng, 768, 13824)}
    d_in, d_out = _dim(rng, 512, 5120), _dim(rng, 512, 13824)
    n, m = rng.choice([(1, 2), (2, 4), (1, 4), (2, 8), (4, 8), (4, 16), (8, 16)])
    return {"kind": kind, "tokens": round(_log_uniform(rng, 256, 8192)), "d_in": d_in, "d_out": d_out, "n": n, "m": m}


def _block(case):
    """(d_in, d_out) of the four linears of a decoder block, in the order it runs them."""
    d, ffn = case["d"], case["ffn"]
    return [(d, 3 * d), (d, d), (d, 2 * ffn), (ffn, d)]


class _Layer:
    """The compressed weight of one layer, its masks and adapter factors, as a program keeps them."""

    def __init__(self, new, d_in, d_out, r, backward):
        W = new(d_out, d_in, sigma=0.02)
        self.d_in, self.d_out, self.r = d_in, d_out, r
        self.vals, self.meta, self.mask1 = B.alloc_compressed(d_out, d_in)
        if backward:
            self.vals_t, self.meta_t, _ = B.alloc_compressed(d_in, d_out)
            B.slope_prune_24_double(W, self.vals, self.meta, self.mask1, self.vals_t, self.meta_t, None)
        else:
            B.slope_prune_24(W, self.vals, self.meta, None)
        if r:
            self.L, self.R = new(d_in, r, sigma=0.01), new(r, d_out, sigma=0.01)


def prepare(case, seed):
    gen = torch.Generator(device="cuda").manual_seed(seed)
    new = lambda *shape, sigma=1.0: torch.randn(shape, device="cuda", generator=gen, dtype=torch.bfloat16).mul_(sigma)
    empty = lambda *shape: torch.empty(shape, device="cuda", dtype=torch.bfloat16)
    kind, s = case["kind"], dict(case)
    if kind == "infer":
        b, r = case["tokens"], case["r"]
        s["layers"] = [_Layer(new, d_in, d_out, r, False) for d_in, d_out in _block(case)]
        s["X"] = [new(b, layer.d_in) for layer in s["layers"]]
        s["Y"] = [empty(b, layer.d_out) for layer in s["layers"]]
        s["T"] = [empty(b, r) for _ in s["layers"]] if r else None
        return s
    d_in, d_out = case["d_in"], case["d_out"]
    if kind == "setup":
        s["W"] = new(d_out, d_in, sigma=0.02)
        s["copy"], s["copy_t"] = B.alloc_compressed(d_out, d_in), B.alloc_compressed(d_in, d_out)
        s["mask2"] = torch.empty_like(s["copy"][2])
    elif kind == "tail":
        s["layer"] = _Layer(new, d_in, d_out, 0, True)
        s["dWc"] = new(d_out, d_in // 2)
        s["decayed"] = torch.empty_like(s["dWc"])
        # the optimizer has just written new weights into the forward copy
        s["layer"].vals.add_(new(d_out, d_in // 2, sigma=0.002))
    elif kind == "train":
        b, r = case["tokens"], case["r"]
        s["layer"] = _Layer(new, d_in, d_out, r, True)
        s["X"], s["dY"] = new(b, d_in), new(b, d_out)
        s["Y"], s["dX"], s["dWc"] = empty(b, d_out), empty(b, d_in), empty(d_out, d_in // 2)
        if r:
            s["T"], s["dT"], s["dL"], s["dR"] = empty(b, r), empty(b, r), empty(d_in, r), empty(r, d_out)
            s["workspace"] = torch.empty(max(16, B.slope_adapter_workspace_bytes(b, d_out, d_in, r)), dtype=torch.uint8,
                                         device="cuda")
    else:
        b = case["tokens"]
        s["W"], s["X"], s["dY"] = new(d_out, d_in, sigma=0.02), new(b, d_in), new(b, d_out)
        s["WR"], s["WRC"], s["dW"], s["Y"], s["dX"] = (empty(d_out, d_in), empty(d_out, d_in), empty(d_out, d_in),
                                                       empty(b, d_out), empty(b, d_in))
        s["mask1"], s["mask2"] = (torch.empty((d_out, d_in // 8), dtype=torch.uint8, device="cuda") for _ in range(2))
    return s


def run(s):
    kind = s["kind"]
    if kind == "train":
        layer, X, dY = s["layer"], s["X"], s["dY"]
        if layer.r:
            B.slope_linear_fwd_adapter(X, layer.vals, layer.meta, layer.d_out, layer.L, layer.R, s["T"], s["Y"])
            B.slope_adapter_fwd_bwd(1, X, dY, layer.L, layer.R, X.shape[0], layer.d_out, layer.d_in, layer.r, T=s["T"],
                                    dT=s["dT"], dL=s["dL"], dR=s["dR"], workspace=s["workspace"])
            B.slope_linear_bwd_dx(dY, layer.vals_t, layer.meta_t, layer.d_in, s["dX"], s["dT"], layer.L)
            B.slope_linear_bwd_dw_masked(dY, X, layer.mask1, s["dWc"])
            return s["Y"], s["dX"], s["dWc"], s["dL"], s["dR"]
        B.slope_linear_fwd(X, layer.vals, layer.meta, layer.d_out, s["Y"])
        B.slope_linear_bwd_dx(dY, layer.vals_t, layer.meta_t, layer.d_in, s["dX"])
        B.slope_linear_bwd_dw_masked(dY, X, layer.mask1, s["dWc"])
        return s["Y"], s["dX"], s["dWc"]
    if kind == "infer":
        for i, layer in enumerate(s["layers"]):
            if layer.r:
                B.slope_linear_fwd_adapter(s["X"][i], layer.vals, layer.meta, layer.d_out, layer.L, layer.R, s["T"][i],
                                           s["Y"][i])
            else:
                B.slope_linear_fwd(s["X"][i], layer.vals, layer.meta, layer.d_out, s["Y"][i])
        return s["Y"]
    if kind == "setup":
        (vals, meta, mask1), (vals_t, meta_t, _) = s["copy"], s["copy_t"]
        B.slope_prune_24_double(s["W"], vals, meta, mask1, vals_t, meta_t, s["mask2"])
        return vals, meta, mask1, vals_t, meta_t, s["mask2"]
    if kind == "tail":
        layer = s["layer"]
        B.slope_sparse_add(s["dWc"], layer.vals, 1.0 / 128.0, 0.1, s["decayed"])
        B.slope_update_sparse_matrix(layer.vals, layer.mask1, layer.meta_t, layer.vals_t)
        return s["decayed"], layer.vals_t
    n, m = s["n"], s["m"]
    B.slope_prune_nm(s["W"], n, m, s["WR"], s["mask1"])
    B.slope_double_prune_nm(s["WR"], s["mask1"], n, m, s["WRC"], s["mask2"])
    B.slope_dense_linear_fwd(s["X"], s["WR"], s["Y"])
    B.slope_dense_linear_bwd_dx(s["dY"], s["WRC"], s["dX"])
    B.slope_dense_linear_bwd_dw(s["dY"], s["X"], s["dW"])
    B.slope_apply_mask(s["dW"], s["mask1"], s["dW"])
    return s["WR"], s["WRC"], s["mask1"], s["mask2"], s["Y"], s["dX"], s["dW"]


def work(case):
    """Bytes: every input read once, every output written once.  A compressed copy is 1.125 bytes per weight element (half
    of the values, 4 metadata bits per group of four), a mask 0.125.  Flops: products with the entries that are kept."""
    kind = case["kind"]
    if kind == "infer":
        b, r, total = case["tokens"], case["r"], {"bytes": 0, "flops": 0}
        for d_in, d_out in _block(case):
            total["bytes"] += 1.125 * d_in * d_out + 2 * (b + r) * (d_in + d_out)
            total["flops"] += b * d_in * d_out + 2 * b * r * (d_in + d_out)
        return total
    d_in, d_out = case["d_in"], case["d_out"]
    n_weights = d_in * d_out
    if kind == "setup":
        return {"bytes": (2 + 2 * 1.125 + 2 * 0.125) * n_weights, "flops": 0}
    if kind == "tail":
        # the forward copy's values serve both calls
        return {"bytes": (1 + 1 + 1 + 0.125 + 0.125 + 1) * n_weights, "flops": 1.5 * n_weights}
    b = case["tokens"]
    activations = 2 * 2 * b * (d_in + d_out)                      # X, dY in; Y, dX out
    if kind == "train":
        r = case["r"]
        return {"bytes": activations + (2 * 1.125 + 0.125 + 1) * n_weights + 2 * 2 * r * (d_in + d_out),
                "flops": 3 * b * n_weights + 3 * 2 * b * r * (d_in + d_out)}
    kept = case["n"] / case["m"]
    # the two pruned matrices and masks, and the masked gradient, are outputs
    return {"bytes": activations + (2 + 2 * 2 + 2 * 0.125 + 2) * n_weights, "flops": 3 * 2 * b * n_weights * kept}


def tolerance(case):
    """Relative to the same pass in 64 bits, outputs rounded once to bf16 are off by 1.7e-3 (norm) and half a unit in the
    last place (2^-8 of a value at most); adapter gradients, products with an operand that was itself rounded, by 2.4e-3 and
    about 1e-2 of the root mean square.  Four times that.  Selection is exact."""
    if case["kind"] == "setup":
        return "exact"
    if case.get("r"):
        return {"rel": 1e-2, "max": 4e-2}
    return {"rel": 7e-3, "max": 1.6e-2}
