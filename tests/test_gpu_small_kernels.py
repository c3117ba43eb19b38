"""GPU parity of the short kernels around the decoder forward, at the sizes where their splits change: the
verified-path search by pointer doubling, the rollback that rides in the same kernel, and the top-k that
keeps a row of logits in registers as long as it fits."""
import numpy as np
import pytest
import torch

from oracle import oracle as orc
from paper_2309_04255_b200 import binding as B
from paper_2309_04255_b200 import inputs as gen

from gpu_util import BF16_TOL, F32_TOL, Twin, argmax_agrees_where_decided, check_acceptance_against_oracle, logits_close

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


def dev_i32(a):
    return torch.as_tensor(np.asarray(a, np.int32), device=DEV)


@pytest.mark.parametrize("n", [1, 2, 3, 5, 31, 32, 33, 64, 65, 127, 128])
@pytest.mark.parametrize("broken", [False, True])
def test_search_and_rollback_along_chains(n, broken):
    """A chain is the deepest tree of its size: every doubling round is needed. Accepted whole, or up to a
    wrong link in its middle; the entries behind the path are -1."""
    cfg = gen.ModelConfig("chain", 2, 256, 2, 128, 256, 512, "bf16")
    parent = gen.tree_chain(n)
    tokens, amax = np.arange(n, dtype=np.int32), np.arange(1, n + 1, dtype=np.int32)
    if broken and n > 1:
        tokens[n // 2] = 400
    v = B.Verifier(cfg, 7 + n + 1)
    v.kv_view().normal_()
    before = v.kv_view().clone()
    path, sc = v.accept_compact(7, dev_i32(tokens), dev_i32(parent), dev_i32(amax))
    acc = orc.accept(parent, tokens, amax)
    assert sc.cpu().numpy()[:7].tolist() == [acc.accepted_len, acc.next_token, 7 + acc.accepted_len, acc.n_correct, acc.n_all, acc.rectified, 0]
    assert path.cpu().numpy().tolist() == acc.path.tolist() + [-1] * (128 - acc.accepted_len)
    assert torch.equal(v.kv_view(), before)      # a chain's path is already in place


@pytest.mark.parametrize("vocab", [8, 31, 1023, 1024, 1025, 32767, 32768, 32769, 40000])
def test_topk_of_short_and_long_rows(vocab):
    """Rows that fill part of the block, all of its registers, and more than those. The oracle works on the
    kernel's own logits, so the ids are exact (ties included: half the rows of the lm_head repeat); a
    probability is one rounded exponential over a sum of up to 40000 of them, added in blocks: 1e-5."""
    cfg = gen.ModelConfig("topk", 1, 64, 1, 64, 64, vocab, "f32")
    v = B.Verifier(cfg, 16)
    g = gen.gen_globals(cfg)
    g["lm_head"] = g["lm_head"] * 20
    g["lm_head"][vocab // 2: 2 * (vocab // 2)] = g["lm_head"][: vocab // 2]
    v.pack_globals(g)
    v.pack_layer(0, gen.gen_layer(cfg, 0))
    out = v.extend_tree(3, dev_i32([1, 2, 5]), dev_i32([-1, 0, 0]), 0, top_k=8)
    assert out["status"].item() == 0
    ids, probs = orc.topk_softmax(out["logits"].cpu().numpy(), 8)
    assert out["topk_ids"].cpu().numpy().tolist() == ids.tolist()
    np.testing.assert_allclose(out["topk_probs"].cpu().numpy(), probs, rtol=1e-5)


@pytest.mark.parametrize("P,n,H,hd,f,V", [(0, 1, 2, 64, 136, 129), (5, 8, 4, 64, 688, 1024), (63, 9, 2, 128, 264, 1001), (700, 3, 1, 128, 512, 300),
                                          (2000, 40, 4, 64, 688, 512), (130, 65, 5, 64, 1200, 640), (31, 128, 4, 64, 688, 1024)])
def test_one_kernel_fp32_pass(P, n, H, hd, f, V):
    """The fp32 pass in one kernel where its cuts change: node blocks of eight and their remainders, several
    staged chunks (128 nodes of 688 columns), one and two nodes per attention task, one and several key
    ranges, both head widths, odd vocabularies; the verified path against the oracle's search."""
    cfg = gen.ModelConfig("f32", 2, H * hd, H, hd, f, V, "f32")
    tw = Twin(cfg, P + n + 8, scale=3.0)
    tw.fill_prefix_synthetic(P)
    parent = gen.tree_random(n, 12, "uniform4", n) if n > 1 else np.array([-1], np.int32)
    tokens = gen.gen_tokens(cfg, n)
    l0 = tw.v.launch_count()
    ref = tw.oracle_pass(P, tokens, parent)
    planted = gen.plant_tokens(parent, tokens, ref.logits.argmax(1).astype(np.int32), 1, prob=0.9)
    for t in (tokens, planted):
        ref = tw.oracle_pass(P, t, parent)
        out = tw.gpu_pass(P, t, parent)
        logits_close(out["logits"], ref.logits, F32_TOL)
        argmax_agrees_where_decided(out["argmax"], ref.logits, F32_TOL)
        check_acceptance_against_oracle(out, t, parent)
        assert out["accepted_path"][out["scalars"][B.S_ACCEPTED_LEN]:].tolist() == [-1] * (128 - out["scalars"][B.S_ACCEPTED_LEN])
    assert tw.v.launch_count() - l0 == 2


def ctas_of_next_gemm(v, run):
    """CTAs of the streaming kernel in the one GEMM that run() launches, by their time stamps."""
    trace = torch.zeros(1, 256, 16, dtype=torch.int64, device=DEV)
    v.set_gemm_trace(trace)
    y = run()
    torch.cuda.synchronize()
    v.set_gemm_trace(None)
    assert v.last_status() == 0
    return y, int((trace[0, :, 0] != 0).sum())


def pair_plan(n_out, n_in):
    """CTAs when pairs of them share items of (two weight tiles, two k-blocks)."""
    items = -(-n_out // 256) * -(-n_in // 128)
    groups = min(torch.cuda.get_device_properties(0).multi_processor_count // 2, items)
    return 2 * -(-items // -(-items // groups))


@pytest.mark.parametrize("n_out,n_in,n", [(128, 64, 96), (100, 136, 128), (300, 520, 128), (640, 128, 96), (257, 72, 128), (4096, 1000, 120), (9600, 4096, 128)])
def test_gemm_on_cta_pairs(n_out, n_in, n):
    """Weight tiles paired over two CTAs: one tile only (its pair is empty), an odd number of them, a ragged last
    k-block, an odd number of k-blocks, half of the activation rows per CTA. bf16 inputs, fp32 sums: the error of
    a sum of n_in products is at most n_in * 2^-24 of the sum of their magnitudes; 2e-6 * sqrt(n_in) of the largest
    result is far inside what the random signs leave of that and far below a single wrong element."""
    cfg = gen.ModelConfig("g", 0, 256, 2, 128, 256, 512, "bf16")
    v = B.Verifier(cfg, 16)
    g = torch.Generator(device=DEV).manual_seed(n_out + n_in + n)
    w = torch.randn(n_out, n_in, generator=g, device=DEV).to(torch.bfloat16)
    x = torch.randn(n, n_in, generator=g, device=DEV).to(torch.bfloat16)
    tiled = v.tile_weight(w)
    y, ctas = ctas_of_next_gemm(v, lambda: v.skinny_gemm_tiled(tiled, n_out, x))
    assert ctas == pair_plan(n_out, n_in)
    ref = x.double() @ w.double().t()
    assert (y.double() - ref).abs().max() <= 2e-6 * n_in ** 0.5 * ref.abs().max()


@pytest.mark.parametrize("n_out,n_in,n", [(128, 64, 96), (100, 192, 128), (300, 576, 128), (640, 128, 96), (4096, 1088, 120)])
def test_int4_gemm_cut_for_cta_pairs(n_out, n_in, n):
    """The INT4 GEMM deals its tiles out as the bf16 GEMM does on CTA pairs, at the same edges: bit for bit the bf16 GEMM
    over the dequantised weights, and that within the bound above."""
    cfg = gen.ModelConfig("g", 0, 256, 2, 128, 256, 512, "bf16")
    v = B.Verifier(cfg, 16)
    g = torch.Generator(device=DEV).manual_seed(n_out + n_in + n)
    w = torch.randn(n_out, n_in, generator=g, device=DEV).to(torch.bfloat16)
    x = torch.randn(n, n_in, generator=g, device=DEV).to(torch.bfloat16)
    q, e = B.quantize_int4(w)
    wq = (q.view(n_out, -1, 64).double() * torch.exp2(e.double())[:, :, None]).view(n_out, n_in).to(torch.bfloat16)
    packed, tiled = v.tile_weight_int4(w), v.tile_weight(wq)
    y, ctas = ctas_of_next_gemm(v, lambda: v.skinny_gemm_tiled_int4(packed, n_out, x))
    assert ctas == pair_plan(n_out, n_in)
    assert torch.equal(y, v.skinny_gemm_tiled(tiled, n_out, x))
    ref = x.double() @ wq.double().t()
    assert (y.double() - ref).abs().max() <= 2e-6 * n_in ** 0.5 * ref.abs().max()


PROMPT_CFG = gen.ModelConfig("prompt", 2, 512, 4, 128, 1408, 1000, "bf16")


@pytest.mark.parametrize("cuts", [[129], [200], [255], [256], [257], [300, 140], [64, 191], [400]])
def test_prompt_chunks_of_up_to_256_tokens(cuts):
    """Prompts whose chunks are wider than a tree (129..256 tokens on CTA pairs, two row blocks in the attention kernel),
    in one or two calls that start at odd cache positions, against sequential decoding: the logits of the last token
    within the bf16 bound of the repository (2e-2 of the largest; rows of earlier chunks are read back rounded), cache
    rows within a bf16 rounding step plus that bound, a second run bit for bit."""
    total = sum(cuts)
    twin = Twin(PROMPT_CFG, total + 8, scale=3.0)
    tokens = gen.gen_prefix_tokens(PROMPT_CFG, total, seed=total)
    dec = orc.SequentialDecoder(PROMPT_CFG, twin.glob, [twin.layer(l) for l in range(2)], total + 1)
    for t in tokens:
        ref = dec.step(int(t))
    runs = []
    for _ in range(2):
        twin.v.kv_view().zero_()
        done = 0
        for m in cuts:
            lg = twin.v.prefill(done, dev_i32(tokens[done:done + m]), want_logits=True)
            assert twin.v.last_status() == 0
            done += m
        runs.append((lg.clone(), twin.v.kv_view().clone()))
    assert torch.equal(runs[0][0], runs[1][0]) and torch.equal(runs[0][1], runs[1][1])
    logits_close(runs[0][0].cpu().numpy(), ref, BF16_TOL)
    rows = runs[0][1][:, :, :, :total].double().cpu().numpy()
    for l in range(2):
        for got, want in zip(rows[l], dec.cache_heads(l, total)):
            assert np.abs(got - want).max() <= (2.0 ** -8 + BF16_TOL) * np.abs(want).max()


def test_prompts_with_cta_pairs_at_every_size():
    """The threshold of the CTA pairs is a tuning aid (read once per process, hence the child): from 16 nodes on, where the
    last row's lm_head, which has 16 padded nodes whatever the prompt, would take them too."""
    import os, subprocess, sys
    here = os.path.dirname(os.path.abspath(__file__))
    script = ("import sys; sys.path[:0] = [sys.argv[1], sys.argv[1] + '/..']; import test_gpu_small_kernels as T\n"
              "for cuts in ([5], [64, 191], [300, 140]): T.test_prompt_chunks_of_up_to_256_tokens(cuts)\nprint('ok')")
    r = subprocess.run([sys.executable, "-c", script, here], env=dict(os.environ, LLMCAD_CTA_PAIR_MIN="16"), capture_output=True,
                       text=True, timeout=300)
    assert r.returncode == 0 and r.stdout.strip().endswith("ok"), r.stdout[-2000:] + r.stderr[-4000:]


def test_wide_prompt_chunks_are_as_exact_as_narrow_ones():
    """The last token's logits of a model without attention (wo = 0: no rounded cache entry reaches them) against 64 bits,
    256 tokens in one chunk and the same token at the end of a chunk of 128. Both carry 16-bit activations (2^-17 each) and
    lose up to 5.8e-8 per k-block of 64 products to the accumulators, over at most 64 (gate, up) or 86 (down) of them:
    below 2e-5 of the norm, where a lost lo plane costs 2e-3; and they agree to 10 % (the cuts of the k ranges differ),
    where accumulating both planes in one sum costs 30 %."""
    cfg = gen.ModelConfig("ffn", 2, 4096, 32, 128, 11008, 2048, "bf16")
    errs = {128: [], 256: []}
    for seed in range(3):
        v = B.Verifier(cfg, 264)
        glob = {k: gen.gen_tensor_device(cfg, k, -1, DEV, seed) for k in ("tok_embed", "final_norm", "lm_head")}
        v.pack_globals(glob)
        tokens = dev_i32(gen.gen_prefix_tokens(cfg, 256, seed))
        norm = lambda x, g: x * torch.rsqrt((x * x).mean() + cfg.rms_eps) * g.double()
        x = glob["tok_embed"][int(tokens[-1])].double()
        for l in range(cfg.n_layers):
            w = {k: gen.gen_tensor_device(cfg, k, l, DEV, seed) for k in gen.LAYER_TENSORS}
            w["wo"].zero_()
            v.pack_layer(l, w)
            h = norm(x, w["ffn_norm"])
            x = x + w["w_down"].double() @ (torch.nn.functional.silu(w["w_gate"].double() @ h) * (w["w_up"].double() @ h))
        ref = glob["lm_head"].double() @ norm(x, glob["final_norm"])
        for n in errs:
            got = v.prefill(0, tokens[256 - n:], want_logits=True).double()
            assert v.last_status() == 0
            errs[n].append(((got - ref).norm() / ref.norm()).item())
    assert max(errs[128] + errs[256]) <= 2e-5
    assert sum(errs[256]) <= 1.1 * sum(errs[128])


def test_prompt_with_a_bad_token_in_a_wide_chunk():
    twin = Twin(PROMPT_CFG, 300)
    tokens = gen.gen_prefix_tokens(PROMPT_CFG, 250, seed=1)
    tokens[200] = PROMPT_CFG.vocab
    twin.v.prefill(0, dev_i32(tokens))
    assert twin.v.last_status() == B.ERR_BAD_TOKEN
