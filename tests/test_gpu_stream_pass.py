"""The one-kernel bf16 pass over few nodes (pass_stream.cu) against the oracle, at the edges of how it cuts its work: models
with fewer pairs of rows than CTAs, K that ends inside a k-block, an odd vocabulary, rows of a CTA on both sides of a weight
tile, prefixes around a tile of 32 keys, trees whose first nodes are in the cache already, prompts of a few tokens."""
import time

import numpy as np
import pytest
import torch

from paper_2309_04255_b200 import binding as B
from paper_2309_04255_b200 import inputs as gen

from gpu_util import BF16_TOL, Twin, argmax_agrees_where_decided, check_acceptance_against_oracle, kernels_of, logits_close

pytestmark = pytest.mark.gpu
DEV = "cuda:0"

MODELS = {"one-head": gen.ModelConfig("one-head", 1, 128, 1, 128, 352, 512, "bf16"),
          "odd": gen.ModelConfig("odd", 3, 640, 5, 128, 1376, 2051, "bf16"),
          "small": gen.ModelConfig("small", 2, 512, 4, 128, 1408, 2048, "bf16"),
          "two-heads": gen.ModelConfig("two-heads", 4, 256, 2, 128, 704, 2048, "bf16"),
          "7b": gen.shrink(gen.MODELS["7b"], 1), "13b": gen.shrink(gen.MODELS["13b"], 1), "30b": gen.shrink(gen.MODELS["30b"], 1)}
# Activations carry 16 bits (hi + lo planes, 2^-17 each) into at most 4 x 3 layers of products and the sums are fp32: some 1e-5 of
# the largest logit. K and V of a pass's own nodes are rounded to bf16 (2^-9 each) only in the cache, where earlier nodes of
# a tree are read back.
TOL = 1e-4


def tree(n, seed):
    return gen.tree_random(n, 4, "uniform4", seed) if n > 1 else np.array([-1], np.int32)


def rising_keys(tw, P):
    """Makes the keys of the prefix grow towards its end, on both sides, so that every tile raises the running maximum."""
    for l, (k, v) in list(tw._prefix.items()):
        k = (k.float() * torch.linspace(0.1, 2.0, P)[None, :, None]).to(k.dtype)
        tw._prefix[l] = (k, v)
        tw.v.kv_view()[l, 0, :, :P] = k.to(DEV)


@pytest.mark.parametrize("model,P,n", [("one-head", 0, 1), ("one-head", 31, 4), ("odd", 33, 3), ("odd", 1, 2), ("odd", 300, 4), ("small", 0, 4),
                                       ("small", 32, 1), ("small", 100, 3), ("7b", 33, 1), ("7b", 128, 4), ("30b", 40, 2)])
def test_pass_over_few_nodes(model, P, n):
    cfg = MODELS[model]
    tw = Twin(cfg, P + n + 40, scale=3.0 if cfg.d_model < 1024 else 1.0, seed=n)
    tw.fill_prefix_synthetic(P)
    parent, tokens = tree(n, P), gen.gen_tokens(cfg, n, P)
    ref = tw.oracle_pass(P, tokens, parent)
    before, launches = tw.v.kv_view().clone(), tw.v.launch_count()
    out = tw.gpu_pass(P, tokens, parent)
    assert tw.v.launch_count() - launches == 3        # the pass, argmax, search: this kernel, not the one per step
    logits_close(out["logits"], ref.logits, TOL)
    argmax_agrees_where_decided(out["argmax"], ref.logits, BF16_TOL)
    acc = check_acceptance_against_oracle(out, tokens, parent)
    after = tw.v.kv_view()
    assert torch.equal(after[:, :, :, :P], before[:, :, :, :P]) and torch.equal(after[:, :, :, P + n:], before[:, :, :, P + n:])
    for layer in range(cfg.n_layers):
        for which, rows in ((0, ref.tree_k[layer]), (1, ref.tree_v[layer])):
            want = rows[acc.path].reshape(acc.accepted_len, cfg.n_heads, cfg.head_dim).transpose(1, 0, 2)
            have = after[layer, which, :, P:P + acc.accepted_len].double().cpu().numpy()
            assert np.abs(have - want).max() <= 2 ** -8 * np.abs(want).max()
    again = tw.gpu_pass(P, tokens, parent)
    assert np.array_equal(again["logits"], out["logits"]) and np.array_equal(again["scalars"], out["scalars"])


# tiles of 32 keys per CTA (148 SMs): 12, 12, 17 to 18, 10 to 11, 5 to 6, 5 to 6, 4 to 5
@pytest.mark.parametrize("model,P,n,rising", [("7b", 1500, 1, True), ("7b", 1500, 4, False), ("30b", 1100, 3, True), ("13b", 1024, 2, True),
                                              ("odd", 5000, 3, True), ("odd", 5000, 4, False), ("one-head", 20000, 2, True)])
def test_pass_over_few_nodes_behind_many_key_tiles(model, P, n, rising):
    """More tiles than a CTA has pairs of warps: a pair takes several and rescales what it has, rows are merged within a CTA
    and between the CTAs of a head, and attention items wrap around the ring."""
    cfg = MODELS[model]
    tw = Twin(cfg, P + n + 8, scale=3.0 if cfg.d_model < 1024 else 1.0, seed=n)
    tw.fill_prefix_synthetic(P)
    if rising:
        rising_keys(tw, P)
    parent, tokens = tree(n, P), gen.gen_tokens(cfg, n, P)
    ref = tw.oracle_pass(P, tokens, parent)
    out = tw.gpu_pass(P, tokens, parent)
    logits_close(out["logits"], ref.logits, TOL)
    check_acceptance_against_oracle(out, tokens, parent)
    again = tw.gpu_pass(P, tokens, parent)
    assert np.array_equal(again["logits"], out["logits"])


def us_per_pass(v, P, tokens, parent, reps=50):
    t, p = (torch.as_tensor(np.asarray(a, np.int32), device=DEV) for a in (tokens, parent))
    out, best = v.new_outputs(len(tokens)), float("inf")
    for _ in range(8):
        a, b = (torch.cuda.Event(enable_timing=True) for _ in range(2))
        torch.cuda._sleep(2_000_000)        # the host gets ahead
        a.record()
        for _ in range(reps):
            v.verify_tree(P, t, p, out=out)
        b.record()
        b.synchronize()
        best = min(best, a.elapsed_time(b) * 1e3 / reps)
    return best


@pytest.mark.parametrize("model,P", [("two-heads", 1900), ("two-heads", 2048), ("one-head", 4096)])
def test_few_heads_with_a_long_prefix_are_not_slower_than_one_kernel_per_step(model, P):
    """One or two heads have a key range for every tile of the prefix to spare, and a merge that takes them one by one: with a
    tile per range these passes take 1.1 to 1.4 of what a context with pinned kernels takes, with four 0.9 and less."""
    cfg = MODELS[model]
    times = []
    for flags in (0, B.FLAG_MMA_ATTN):
        tw = Twin(cfg, P + 8, flags=flags, scale=3.0, keep_host=False)
        tw.fill_prefix_synthetic(P)
        times.append(us_per_pass(tw.v, P, gen.gen_tokens(cfg, 4), tree(4, P)))
    assert times[0] < times[1]


@pytest.mark.parametrize("model,P,cuts", [("odd", 30, [3, 4, 8, 9]), ("small", 300, [30, 33, 70, 74]), ("7b", 40, [1, 5, 8]), ("7b", 1500, [34, 37, 41])])
def test_extension_by_few_nodes(model, P, cuts):
    """A tree grown by one to four nodes per call behind calls of any size: earlier nodes are keys with a mask."""
    cfg = MODELS[model]
    n = cuts[-1]
    tw = Twin(cfg, P + n + 8, scale=3.0 if cfg.d_model < 1024 else 1.0)
    tw.fill_prefix_synthetic(P)
    parent, tokens = gen.tree_random(n, 12, "uniform4", n), gen.gen_tokens(cfg, n)
    ref = tw.oracle_pass(P, tokens, parent)
    old = 0
    for m in cuts:
        out = tw.v.extend_tree(P, torch.as_tensor(tokens[:m], device=DEV), torch.as_tensor(parent[:m], device=DEV), old, top_k=2)
        assert out["status"].item() == 0
        logits_close(out["logits"].cpu().numpy(), ref.logits[old:m], BF16_TOL)
        old = m


def one_kernel_passes(names):
    return sum("stream_pass_kernel" in k for k in names)


@pytest.mark.parametrize("P,n", [(0, 1), (0, 4), (257, 2), (30, 257), (0, 260)])
def test_prompts_that_are_or_end_in_few_tokens(P, n):
    """The last row's logits and the cache of a prompt of a few tokens, or whose last chunk is (chunks are of 256), as one pass over
    the same chain gives them."""
    cfg = MODELS["small"]
    tw = Twin(cfg, P + n + 8, scale=3.0, keep_host=False)
    tw.fill_prefix_synthetic(P)
    tokens = torch.as_tensor(gen.gen_tokens(cfg, n), device=DEV)
    last = tw.v.prefill(P, tokens, want_logits=True)
    assert tw.v.last_status() == 0
    assert one_kernel_passes(kernels_of(lambda: tw.v.prefill(P, tokens, want_logits=True))) == 1
    cache = tw.v.kv_view()[:, :, :, :P + n].clone()
    # the same prompt in two calls, cut elsewhere
    if n > 1:
        tw.v.prefill(P, tokens[:n - 1])
        again = tw.v.prefill(P + n - 1, tokens[n - 1:], want_logits=True)
        logits_close(again.cpu().numpy()[None], last.double().cpu().numpy()[None], BF16_TOL)
        d = (tw.v.kv_view()[:, :, :, :P + n].double() - cache.double()).abs().max().item()
        assert d <= BF16_TOL * cache.double().abs().max().item()
    bad = tokens.clone()
    bad[-1] = cfg.vocab
    tw.v.prefill(P, bad)
    assert tw.v.last_status() == B.ERR_BAD_TOKEN


@pytest.mark.parametrize("bad_at", [0, 200, 256, 258])
def test_bad_tokens_of_prompts_that_end_in_few_tokens(bad_at):
    """259 tokens: a chunk of 256 and three through the one-kernel pass, which keeps the error of the chunk before it (its weights,
    already asked for, land and nothing is written) or finds its own. Then the good prompt is what it was."""
    cfg, n = MODELS["small"], 259
    tw = Twin(cfg, n + 8, scale=3.0, keep_host=False)
    tokens = torch.as_tensor(gen.gen_tokens(cfg, n), device=DEV)
    last = tw.v.prefill(0, tokens, want_logits=True)
    cache = tw.v.kv_view().clone()
    bad = tokens.clone()
    bad[bad_at] = cfg.vocab + 7
    assert one_kernel_passes(kernels_of(lambda: tw.v.prefill(0, bad))) == 1
    for _ in range(2):
        tw.v.kv_view().fill_(7.0)
        tw.v.prefill(0, bad, want_logits=True)
        assert tw.v.last_status() == B.ERR_BAD_TOKEN
        assert (tw.v.kv_view()[:, :, :, 256:] == 7.0).all()
        if bad_at >= 256:
            assert torch.equal(tw.v.kv_view()[:, :, :, :256], cache[:, :, :, :256])
    again = tw.v.prefill(0, tokens, want_logits=True)
    assert tw.v.last_status() == 0
    assert torch.equal(again, last) and torch.equal(tw.v.kv_view()[:, :, :, :n], cache[:, :, :, :n])


@pytest.mark.parametrize("model,P,flags", [("small", 40, 0), ("odd", 700, 0), ("7b", 200, 0), ("small", 40, B.FLAG_INT4_WEIGHTS)])
def test_bounded_waits_run_out_and_the_context_survives(model, P, flags):
    """With the limit at 1 ms and the inputs withheld behind the first grid barrier, the waits of consumers, producers and the
    loader of every CTA run out: TIMEOUT, promptly, with nothing written, and again. The barrier words are back at zero
    afterwards: passes of one and four nodes (P = 700: several key ranges per head and their counters) are bit for bit what
    they were."""
    cfg = MODELS[model]
    tw = Twin(cfg, P + 16, flags=flags, scale=3.0 if cfg.d_model < 1024 else 1.0, keep_host=False)
    tw.fill_prefix_synthetic(P)
    passes = [(tree(n, P), gen.gen_tokens(cfg, n, P)) for n in (1, 4)]
    before = [tw.gpu_pass(P, tokens, parent) for parent, tokens in passes]
    cache = tw.v.kv_view().clone()
    with pytest.raises(B.LlmcadError) as e:          # refuses to run with the default limit of 2 s
        tw.v.selftest_pass_timeout()
    assert e.value.code == B.ERR_INVALID_ARG
    tw.v.set_wait_limit_ns(1_000_000)
    for _ in range(2):
        t0 = time.perf_counter()
        assert tw.v.selftest_pass_timeout() == B.ERR_TIMEOUT
        assert time.perf_counter() - t0 < 1.0
    assert torch.equal(tw.v.kv_view(), cache)
    tw.v.set_wait_limit_ns(0)
    for (parent, tokens), was in zip(passes, before):
        now = tw.gpu_pass(P, tokens, parent)
        assert now["scalars"][B.S_STATUS] == 0
        for key in ("logits", "argmax", "scalars", "accepted_path"):
            assert np.array_equal(now[key], was[key]), key


def test_timeout_self_test_is_refused_where_the_kernel_is_not_taken():
    cfg = MODELS["small"]
    for flags in (B.FLAG_MMA_ATTN, B.FLAG_SIMT_GEMM):
        tw = Twin(cfg, 64, flags=flags, keep_host=False)
        tw.v.set_wait_limit_ns(1_000_000)
        with pytest.raises(B.LlmcadError) as e:
            tw.v.selftest_pass_timeout()
        assert e.value.code == B.ERR_UNSUPPORTED


@pytest.mark.parametrize("other_nodes", [20, 2])
def test_two_contexts_on_two_streams(other_nodes):
    """The one-kernel pass of one context beside another context's passes, of many kernels or of one, on a stream of its own:
    neither waits for ever, and both give what they give alone."""
    cfg = MODELS["small"]
    P, passes = 300, []
    for n, seed in ((3, 1), (other_nodes, 2)):
        tw = Twin(cfg, P + n + 8, scale=3.0, seed=seed, keep_host=False)
        tw.fill_prefix_synthetic(P)
        t, p = (torch.as_tensor(np.asarray(a, np.int32), device=DEV) for a in (gen.gen_tokens(cfg, n, seed), gen.tree_random(n, 6, "uniform4", n)))
        passes.append((tw.v, t, p, tw.v.verify_tree(P, t, p)["logits"].clone(), torch.cuda.Stream()))
    torch.cuda.synchronize()
    outs = []
    for _ in range(40):
        for v, t, p, alone, st in passes:
            with torch.cuda.stream(st):
                outs.append((v.verify_tree(P, t, p), alone))
    torch.cuda.synchronize()
    for out, alone in outs:
        assert out["scalars"][B.S_STATUS].item() == 0 and torch.equal(out["logits"], alone)
