"""Performance cases of the token-tree verification library.

Each case is one call that a program built on this library makes over and over: verify a draft tree
(from device or from host buffers, bf16 or INT4 weights, one token up to 128 nodes), grow a draft tree on
the generating side, fill the cache from a prompt, roll the cache back, or run the tree attention on its
own. Sizes come from `inputs.MODELS` / `inputs.WORKLOADS`; models that would not fit the card three times
over keep their widths and lose layers.

    listed()            the cases
    draw(rng)           one more case from the same ranges
    prepare(case, seed) the state a program holds before the call (weights packed, prefix in the cache)
    run(state)          the call, and its outputs
    work(case)          bytes and operations that one call cannot do without
    tolerance(case)     how far two correct implementations may be apart
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2309_04255_b200 import binding as B
from paper_2309_04255_b200 import inputs as gen

DEV = "cuda:0"
# a small decoder of the generating side: the widths of the repository's small bf16 model
SMALL = gen.ModelConfig("small-bf16", 2, 512, 4, 128, 1408, 2048, "bf16")


def _cfg(case) -> gen.ModelConfig:
    base = SMALL if case["model"] == "small" else gen.MODELS[case["model"]]
    return gen.shrink(base, case["layers"])


def listed():
    return [
        # The smallest whole pass: fp32, a few dozen short kernels. Launches and latency.
        {"name": "tiny_f32_verify", "op": "verify", "model": "tiny", "layers": 2, "prefix": 32, "nodes": 15, "levels": 4,
         "branching": "binary", "int4": False},
        # The generating side: a small draft model adds 12 nodes to a tree of 8 and wants the four best successors of each.
        {"name": "small_extend", "op": "extend", "model": "small", "layers": 2, "prefix": 300, "old": 8, "nodes": 20, "levels": 8,
         "branching": "uniform4", "top_k": 4},
        # Acceptance and rollback alone, on a 7B-shaped cache: a scheduler that has its own argmax.
        {"name": "rollback_7b", "op": "rollback", "model": "7b", "layers": 32, "prefix": 512, "nodes": 32, "levels": 8,
         "branching": "uniform4"},
        # Tree attention on its own, shortest and longest prefix of the attention sweep.
        {"name": "attention_p256_n8", "op": "attention", "heads": 32, "prefix": 256, "nodes": 8, "levels": 6, "branching": "uniform4"},
        {"name": "attention_p8192_n128", "op": "attention", "heads": 32, "prefix": 8192, "nodes": 128, "levels": 12,
         "branching": "uniform4"},
        # Plain decoding step of the target: a tree of the root alone.
        {"name": "decode_7b", "op": "verify", "model": "7b", "layers": 32, "prefix": 512, "nodes": 1, "levels": 1, "branching": "chain",
         "int4": False},
        # The ordinary verification pass (workload C2).
        {"name": "verify_7b_n32", "op": "verify", "model": "7b", "layers": 32, "prefix": 512, "nodes": 32, "levels": 8,
         "branching": "uniform4", "int4": False},
        # The same pass with INT4 weights, which is how the method's own target model is held.
        {"name": "verify_7b_int4_n32", "op": "verify", "model": "7b", "layers": 32, "prefix": 512, "nodes": 32, "levels": 8,
         "branching": "uniform4", "int4": True},
        # The same model driven from host buffers, logits copied back, ragged sizes.
        {"name": "verify_host_7b_n45", "op": "verify_host", "model": "7b", "layers": 32, "prefix": 701, "nodes": 45, "levels": 9,
         "branching": "geometric4", "int4": False},
        # Workload C3 at half its depth.
        {"name": "verify_13b_n64", "op": "verify", "model": "13b", "layers": 20, "prefix": 1024, "nodes": 64, "levels": 10,
         "branching": "geometric4", "int4": False},
        # Workload C5 at a fifth of its depth: the largest tree, the longest prefix, the widest model.
        {"name": "verify_30b_n128", "op": "verify", "model": "30b", "layers": 12, "prefix": 2048, "nodes": 128, "levels": 12,
         "branching": "uniform4", "int4": False},
        # A prompt into the cache, with the logits of its last token.
        {"name": "prefill_7b_512", "op": "prefill", "model": "7b", "layers": 32, "prefix": 0, "nodes": 512, "int4": False},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _tree(rng, n):
    # deep enough for n nodes at four children each, and shaped like the listed trees
    levels = rng.randint(8, 14) if n > 1 else 1
    return {"nodes": n, "levels": levels, "branching": rng.choice(["uniform4", "geometric4"]) if n > 1 else "chain"}


def draw(rng):
    op = rng.choice(["verify", "verify", "verify", "int4", "verify_host", "prefill", "extend", "attention", "rollback", "tiny"])
    model = rng.choice(["7b", "7b", "13b", "30b"])
    layers = rng.randint(4, {"7b": 32, "13b": 20, "30b": 12}[model])
    prefix = _log_int(rng, 16, 2048)
    nodes = _log_int(rng, 1, 128)
    if op == "verify":
        return {"op": "verify", "model": model, "layers": layers, "prefix": prefix, "int4": False, **_tree(rng, nodes)}
    if op == "int4":
        return {"op": "verify", "model": model, "layers": layers, "prefix": prefix, "int4": True, **_tree(rng, nodes)}
    if op == "verify_host":
        return {"op": "verify_host", "model": model, "layers": layers, "prefix": prefix, "int4": False, **_tree(rng, nodes)}
    if op == "prefill":
        return {"op": "prefill", "model": "7b", "layers": rng.randint(3, 12), "prefix": rng.choice([0, _log_int(rng, 16, 1024)]),
                "nodes": _log_int(rng, 8, 1024), "int4": rng.random() < 0.25}
    if op == "extend":
        n = max(2, nodes)
        small = rng.random() < 0.5
        return {"op": "extend", "model": "small" if small else "7b", "layers": rng.randint(2, 8), "prefix": prefix,
                "old": rng.randint(0, n - 1), "top_k": rng.randint(1, 8), **_tree(rng, n)}
    if op == "attention":
        return {"op": "attention", "heads": rng.choice([4, 12, 32, 40]), "prefix": _log_int(rng, 16, 6400), **_tree(rng, nodes)}
    if op == "rollback":
        return {"op": "rollback", "model": model, "layers": layers, "prefix": prefix, **_tree(rng, max(2, nodes))}
    return {"op": "verify", "model": "tiny", "layers": rng.randint(1, 4), "prefix": _log_int(rng, 1, 512), "int4": False,
            **_tree(rng, nodes)}


def _parents(case, seed):
    return gen.gen_tree(gen.Workload("case", "", case["prefix"], case["nodes"], case["levels"], case["branching"]), seed)


def _dev(a):
    return torch.as_tensor(np.ascontiguousarray(a, dtype=np.int32), device=DEV)


def _verifier(cfg, max_seq, seed, int4=False):
    """The weights of a model, packed, and a cache whose prefix holds N(0, 1) rows."""
    v = B.Verifier(cfg, max_seq, flags=B.FLAG_INT4_WEIGHTS if int4 else 0, device=DEV)
    v.pack_globals({k: gen.gen_tensor_device(cfg, k, -1, DEV, seed) for k in ("tok_embed", "final_norm", "lm_head")})
    for layer in range(cfg.n_layers):
        v.pack_layer(layer, {k: gen.gen_tensor_device(cfg, k, layer, DEV, seed) for k in gen.LAYER_TENSORS})
    _fill_cache(v, seed)
    return v


def _fill_cache(v, seed):
    v.kv_view().normal_(generator=torch.Generator(device=DEV).manual_seed(seed + 1))


def prepare(case, seed):
    op = case["op"]
    if op == "attention":
        H, P, n = case["heads"], case["prefix"], case["nodes"]
        cfg = gen.ModelConfig("attention", 0, H * 128, H, 128, 256, 512, "bf16")
        g = torch.Generator(device=DEV).manual_seed(seed + 1)
        q, k, v = (torch.randn(s, generator=g, device=DEV, dtype=torch.bfloat16) for s in ((n, H, 128), (H, P + n, 128), (H, P + n, 128)))
        return {"op": op, "v": B.Verifier(cfg, 16, device=DEV), "q": q, "k": k, "v_": v, "P": P, "parent": _dev(_parents(case, seed))}
    cfg = _cfg(case)
    P, n = case["prefix"], case["nodes"]
    if op == "prefill":
        return {"op": op, "v": _verifier(cfg, P + n + 8, seed, case["int4"]), "P": P, "tokens": _dev(gen.gen_prefix_tokens(cfg, n, seed))}
    parent, tokens = _parents(case, seed), gen.gen_tokens(cfg, n, seed)
    if op == "rollback":
        # the cache and the target's choices, some of which agree with the draft
        v = B.Verifier(cfg, P + 128 + 8, device=DEV)
        _fill_cache(v, seed)
        argmax = gen.gen_tokens(cfg, n, seed + 1)
        planted = gen.plant_tokens(parent, tokens, argmax, seed, prob=0.9)
        return {"op": op, "v": v, "P": P, "tokens": _dev(planted), "parent": _dev(parent), "argmax": _dev(argmax)}
    v = _verifier(cfg, P + 128 + 8, seed, case.get("int4", False))
    s = {"op": op, "v": v, "P": P}
    if op == "verify_host":
        s["tokens"], s["parent"] = (torch.from_numpy(np.ascontiguousarray(a, dtype=np.int32)).pin_memory() for a in (tokens, parent))
        s["out"] = {"logits": torch.empty((n, cfg.vocab), dtype=torch.float32).pin_memory(), "argmax": torch.empty(n, dtype=torch.int32).pin_memory(),
                    "accepted_path": torch.full((n,), -1, dtype=torch.int32).pin_memory(), "scalars": torch.zeros(8, dtype=torch.int32).pin_memory()}
        return s
    s["tokens"], s["parent"] = _dev(tokens), _dev(parent)
    if op == "extend":
        s["old"], s["top_k"] = case["old"], case["top_k"]
        if s["old"]:        # the tree's first nodes are in the cache already
            v.extend_tree(P, s["tokens"][:s["old"]], s["parent"][:s["old"]], 0, top_k=1, want_logits=False)
    return s


def run(s):
    v, P = s["v"], s["P"]
    if s["op"] == "attention":
        return v.tree_attention(s["q"], s["k"], s["v_"], P, s["parent"])
    if s["op"] == "rollback":
        path, scalars = v.accept_compact(P, s["tokens"], s["parent"], s["argmax"])
        return {"path": path, "scalars": scalars, "cache": v.kv_view()}
    if s["op"] == "prefill":
        logits = v.prefill(P, s["tokens"], want_logits=True)
        return {"logits": logits, "cache": v.kv_view()[:, :, :, :P + s["tokens"].numel()]}
    if s["op"] == "extend":
        out = v.extend_tree(P, s["tokens"], s["parent"], s["old"], top_k=s["top_k"])
        return {**out, "cache": v.kv_view()[:, :, :, :P + s["tokens"].numel()]}
    if s["op"] == "verify_host":
        out = v.verify_tree_host(P, s["tokens"], s["parent"], s["out"])
    else:
        out = v.verify_tree(P, s["tokens"], s["parent"])
    # of the cache, the prefix and the root's row are defined whatever was accepted
    return {**out, "cache": v.kv_view()[:, :, :, :P + 1]}


def work(case):
    n, P = case["nodes"], case["prefix"]
    if case["op"] == "attention":
        d = case["heads"] * 128
        return {"bytes": 2 * (2 * (P + n) * d + 2 * n * d), "flops": 4 * n * (P + n) * d}
    cfg = _cfg(case)
    L, d, f, V, e = cfg.n_layers, cfg.d_model, cfg.d_ffn, cfg.vocab, cfg.elem_bytes
    if case["op"] == "rollback":
        # every row of an accepted path of typical length, read and written once in K and V of every layer
        return {"bytes": 2 * min(3, n) * 2 * L * d * e, "flops": 0}
    new = n - case.get("old", 0)
    layer_elems = cfg.layer_weight_elems()
    weights = L * layer_elems * e
    if case.get("int4"):
        weights = int(L * layer_elems * (0.5 + 1.0 / 64))
    rows = 1 if case["op"] == "prefill" else new          # nodes whose logits are wanted
    cache = 2 * L * d * e * (P + case.get("old", 0) + new)  # prefix read, new rows written
    pairs = new * P + new * (new + 1) // 2 if case["op"] == "prefill" else new * (P + n)
    return {"bytes": weights + V * d * e + cache + new * d * e + rows * V * 4,
            "flops": 2 * new * L * layer_elems + 4 * L * pairs * d + 2 * rows * V * d}


def tolerance(case):
    if case["op"] == "rollback":
        return "exact"
    if case["op"] == "attention":
        # bf16 outputs and bf16 softmax weights: 2^-9 each, rounded independently
        return {"rel": 6e-3, "max": 6e-2}
    if case["model"] == "tiny":
        return {"rel": 1e-5, "max": 2e-4, "differ": 0.01}
    # Activations carry 16 significant bits through the layers, rows enter the cache as bf16 (2^-9): logits of two
    # correct implementations agree to a few 1e-4, single cache entries to a bf16 step.
    return {"rel": 2e-3, "max": 3e-2, "differ": 0.01}
