"""How the GEMMs of a pass over 33 to 64 nodes cut their work: ring items of one k-block up to 48 nodes, cut by two where K
has an even number of them, and CTA pairs from 49 on. Whole passes against the oracle, and bit for bit against an INT4
context, whose kernel is cut the same way and shares no ring with them."""
import numpy as np
import pytest
import torch

from paper_2309_04255_b200 import inputs as gen

from gpu_util import argmax_agrees_where_decided, check_acceptance_against_oracle, logits_close
from test_gpu_int4 import Int4Twin

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
