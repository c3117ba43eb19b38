"""How the GEMMs of a pass over 33 to 64 nodes cut their work: ring items of one k-block up to 48 nodes in wide models, cut by
two where K has an even number of them, and CTA pairs from 49 on in wider ones. Whole passes against the oracle, and bit for bit
against an INT4 context, whose kernel is cut the same way and shares no ring with them."""
import numpy as np
import pytest
import torch

from paper_2309_04255_b200 import binding as B
from paper_2309_04255_b200 import inputs as gen

from gpu_util import argmax_agrees_where_decided, check_acceptance_against_oracle, kernels_of, logits_close
from test_gpu_int4 import Int4Twin
from test_gpu_small_kernels import ctas_of_next_gemm, pair_plan

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [33, 48, 49, 64])
@pytest.mark.parametrize("d,heads,f", [(512, 4, 1408), (512, 4, 1344), (128, 1, 320), (640, 5, 64)])      # K of 22, 21, 5, 1 k-blocks
def test_passes_of_33_to_64_nodes(d, heads, f, n):
    cfg = gen.ModelConfig("cut", 2, d, heads, 128, f, 1000, "bf16")
    twin = Int4Twin(cfg, 50 + n + 8, scale=3.0, seed=n)
    twin.fill_prefix_synthetic(50)
    twin.v16.kv_view()[:, :, :, :50] = twin.v.kv_view()[:, :, :, :50]
    parent, tokens = gen.tree_random(n, 10, "uniform4", n), gen.gen_tokens(cfg, n, n)
    out, ref = twin.gpu_pass(50, tokens, parent), twin.oracle_pass(50, tokens, parent)
    logits_close(out["logits"], ref.logits, 1e-3)           # hi + lo activations: some 1e-5
    argmax_agrees_where_decided(out["argmax"], ref.logits, 1e-3)
    check_acceptance_against_oracle(out, tokens, parent)
    t, p = (torch.as_tensor(np.asarray(a, np.int32), device=twin.v16.device) for a in (tokens, parent))
    o16 = twin.v16.verify_tree(50, t, p)
    assert np.array_equal(o16["logits"].cpu().numpy(), out["logits"])
    assert np.array_equal(o16["scalars"].cpu().numpy(), out["scalars"])


def small_model(d, f, max_seq):
    cfg = gen.ModelConfig("width", 1, d, d // 128, 128, f, 1000, "bf16")
    v = B.Verifier(cfg, max_seq)
    v.pack_globals({k: gen.gen_tensor_device(cfg, k, -1, v.device) for k in ("tok_embed", "final_norm", "lm_head")})
    v.pack_layer(0, {k: gen.gen_tensor_device(cfg, k, 0, v.device) for k in gen.LAYER_TENSORS})
    return cfg, v


def tree(v, cfg, n):
    return (torch.as_tensor(np.asarray(a, np.int32), device=v.device) for a in (gen.gen_tokens(cfg, n, n), gen.tree_random(n, 10, "uniform4", n)))


def stream_variants(names):
    """k-blocks per ring item of the streaming GEMM kernels among `names`."""
    return sorted({int(n.split("gemm_stream_kernelILi")[1][0]) for n in names if "gemm_stream_kernelILi" in n})


@pytest.mark.parametrize("d,f,n,k_blocks", [(512, 1408, 33, 2), (512, 1408, 48, 2), (2048, 5632, 48, 2), (3072, 8192, 33, 1), (3072, 8192, 48, 1), (3072, 8192, 32, 2)])
def test_which_passes_take_ring_items_of_one_k_block(d, f, n, k_blocks):
    """Narrow models lose by them at 33 to 48 nodes (the sums are the same either way)."""
    cfg, v = small_model(d, f, n + 16)
    t, p = tree(v, cfg, n)
    out = v.verify_tree(0, t, p)
    assert out["scalars"][B.S_STATUS].item() == 0
    assert stream_variants(kernels_of(lambda: v.verify_tree(0, t, p, out=out))) == [k_blocks]


@pytest.mark.parametrize("n,tiled", [(48, True), (96, False), (128, False), (112, True)])
def test_gemm_on_its_own_keeps_ring_items_of_two_k_blocks(n, tiled):
    """As many columns of the MMA as a pass of 48 nodes and more, and a twentieth to a sixth slower with one."""
    n_out, n_in = 1536, 512
    v = B.Verifier(gen.ModelConfig("g", 0, 256, 2, 128, 256, 512, "bf16"), 16)
    w, x = (torch.randn(s, device=v.device).to(torch.bfloat16) for s in ((n_out, n_in), (n, n_in)))
    wt = v.tile_weight(w)
    call = (lambda: v.skinny_gemm_tiled(wt, n_out, x)) if tiled else (lambda: v.skinny_gemm(w, x))
    call()
    assert stream_variants(kernels_of(call)) == [2]


def single_plan(n_out, n_in):
    """CTAs when each has items of (one weight tile, two k-blocks) of its own."""
    items = -(-n_out // 128) * -(-n_in // 128)
    groups = min(torch.cuda.get_device_properties(0).multi_processor_count, items)
    return -(-items // -(-items // groups))


# widths at which the two plans differ in their number of CTAs (148 SMs)
@pytest.mark.parametrize("d,f,n,pairs", [(640, 1408, 49, False), (640, 1408, 64, False), (1152, 3072, 64, False), (4096, 11008, 49, True), (4096, 11008, 64, True),
                                         (4096, 11008, 48, False)])
def test_which_passes_of_up_to_64_nodes_take_cta_pairs(d, f, n, pairs):
    """Narrow models lose by pairs at 49 to 64 nodes, wide ones gain; by the CTAs of the first QKV GEMM of a pass."""
    cfg, v = small_model(d, f, n + 16)
    t, p = tree(v, cfg, n)
    assert single_plan(3 * d, d) != pair_plan(3 * d, d)
    out, ctas = ctas_of_next_gemm(v, lambda: v.verify_tree(0, t, p))
    assert out["scalars"][B.S_STATUS].item() == 0
    assert ctas == (pair_plan if pairs else single_plan)(3 * d, d)


@pytest.mark.parametrize("n", [49, 64])
def test_gemm_on_its_own_takes_no_cta_pairs_up_to_64_nodes(n):
    n_out, n_in = 640, 640
    v = B.Verifier(gen.ModelConfig("g", 0, 256, 2, 128, 256, 512, "bf16"), 16)
    g = torch.Generator(device=v.device).manual_seed(n)
    w, x = (torch.randn(s, generator=g, device=v.device).to(torch.bfloat16) for s in ((n_out, n_in), (n, n_in)))
    tiled = v.tile_weight(w)
    y, ctas = ctas_of_next_gemm(v, lambda: v.skinny_gemm_tiled(tiled, n_out, x))
    assert ctas == single_plan(n_out, n_in) != pair_plan(n_out, n_in)
    ref = x.double() @ w.double().t()
    assert (y.double() - ref).abs().max() <= 2e-6 * n_in ** 0.5 * ref.abs().max()
