"""What the entry points promise their callers around the pass itself: which outputs are written, how far, and in
which order with other work of the stream."""
import numpy as np
import pytest
import torch

from oracle import oracle as orc
from paper_2309_04255_b200 import binding as B
from paper_2309_04255_b200 import inputs as gen

from gpu_util import Twin, check_acceptance_against_oracle

pytestmark = pytest.mark.gpu
DEV = "cuda:0"

SMALL = {"f32": gen.ModelConfig("f32", 2, 256, 4, 64, 688, 1024, "f32"),
         "bf16": gen.ModelConfig("bf16", 2, 512, 4, 128, 1408, 2048, "bf16")}


def planted(twin, P, parent, tokens, seed, rounds=4):
    """Tokens of which the target accepts several levels: each round plants its choices one level deeper."""
    for _ in range(rounds):
        tokens = gen.plant_tokens(parent, tokens, twin.gpu_pass(P, tokens, parent)["argmax"], seed, prob=1.0)
    return tokens


def host_buffers(n, vocab):
    return {"logits": torch.empty((n, vocab), dtype=torch.float32).pin_memory(), "argmax": torch.empty(n, dtype=torch.int32).pin_memory(),
            "accepted_path": torch.full((n + 3,), 77, dtype=torch.int32).pin_memory(), "scalars": torch.zeros(8, dtype=torch.int32).pin_memory()}


@pytest.mark.parametrize("dtype", ["f32", "bf16"])
def test_host_entry_returns_the_verified_path(dtype):
    """llmcad_verify_tree_host on trees of which several levels are accepted, two different ones in a row on one context:
    all n entries of the path, 0 behind it, and nothing past them; everything else as the device entry gives it. A
    refused tree gives an empty path."""
    cfg, P = SMALL[dtype], 40
    twin = Twin(cfg, P + 40, scale=3.0)
    twin.fill_prefix_synthetic(P)
    lengths = set()
    for seed, n in ((3, 24), (5, 31), (3, 24)):
        parent = gen.tree_random(n, 8, "uniform4", seed)
        tokens = planted(twin, P, parent, gen.gen_tokens(cfg, n, seed), seed)
        dev = twin.gpu_pass(P, tokens, parent)
        acc = check_acceptance_against_oracle(dev, tokens, parent)
        assert acc.accepted_len >= 3 and acc.path.tolist() != list(range(acc.accepted_len))
        lengths.add(tuple(acc.path.tolist()))
        host = host_buffers(n, cfg.vocab)
        twin.v.verify_tree_host(P, torch.as_tensor(tokens).pin_memory(), torch.as_tensor(parent).pin_memory(), host)
        for k in ("logits", "argmax", "scalars"):
            assert np.array_equal(host[k].numpy(), dev[k]), k
        assert host["accepted_path"].tolist() == acc.path.tolist() + [0] * (n - acc.accepted_len) + [77] * 3
    assert len(lengths) == 2
    bad = parent.copy()
    bad[2] = 2
    host = host_buffers(n, cfg.vocab)
    twin.v.verify_tree_host(P, torch.as_tensor(tokens).pin_memory(), torch.as_tensor(bad).pin_memory(), host)
    assert host["scalars"].tolist() == [0, -1, P, 0, 0, 0, B.ERR_BAD_TREE, 0]
    assert host["accepted_path"].tolist() == [0] * n + [77] * 3


def test_paths_stay_inside_the_callers_buffers():
    """llmcad_accept_compact on a path buffer of n entries, and verify_tree on outputs of the caller whose path has n: the
    path, -1 up to n, and nothing behind (the buffers are the front of larger ones, so that a longer write would show). A
    path length below n is refused."""
    cfg, P, n = SMALL["f32"], 9, 20
    twin = Twin(cfg, P + n + 1, scale=3.0)
    twin.fill_prefix_synthetic(P)
    v = twin.v
    parent = gen.tree_random(n, 8, "uniform4", 4)
    tokens = planted(twin, P, parent, gen.gen_tokens(cfg, n, 4), 4)
    ref = twin.gpu_pass(P, tokens, parent)
    acc = check_acceptance_against_oracle(ref, tokens, parent)
    want = acc.path.tolist() + [-1] * (n - acc.accepted_len) + [77] * (256 - n)
    t, p, amax = (torch.as_tensor(np.asarray(a, np.int32), device=DEV) for a in (tokens, parent, ref["argmax"]))
    for q, expect in ((p, want), (torch.full_like(p, 5), [-1] * n + [77] * (256 - n))):     # the second tree is refused
        room = torch.full((256,), 77, dtype=torch.int32, device=DEV)
        sc = torch.zeros(8, dtype=torch.int32, device=DEV)
        args = (v.ctx, None, P, t.data_ptr(), q.data_ptr(), amax.data_ptr(), n, room.data_ptr())
        assert B.lib().llmcad_accept_compact(*args, sc.data_ptr(), B._stream()) == B.OK
        assert room.tolist() == expect
    assert B.lib().llmcad_accept_compact_fill(*args, n - 1, sc.data_ptr(), B._stream()) == B.ERR_INVALID_ARG
    out = v.new_outputs(n)
    room = torch.full((256,), 77, dtype=torch.int32, device=DEV)
    out["accepted_path"] = room[:n]
    assert v.verify_tree(P, t, p, out=out)["accepted_path"] is out["accepted_path"]
    assert room.tolist() == want and out["scalars"].tolist() == ref["scalars"].tolist()


@pytest.mark.parametrize("op", ["verify", "prefill"])
def test_weights_packed_right_before_a_pass_are_the_ones_it_uses(op):
    """Two sets of weights packed in turn, each followed by a pass on the same stream with nothing in between: every pass
    gives bit for bit what it gives after a synchronisation. (The first GEMM requests weights ahead of its dependency; that
    it does so after the packing is an order of launches which no single run proves.)"""
    cfg, P, n = SMALL["bf16"], 30, 16
    m = 150 if op == "prefill" else n             # a wide chunk starts with a kernel of its own
    v = B.Verifier(cfg, P + m + 1)
    v.kv_view().normal_(generator=torch.Generator(device=DEV).manual_seed(1))
    tokens = torch.as_tensor(gen.gen_tokens(cfg, m, 2), device=DEV)
    parent = torch.as_tensor(gen.tree_random(n, 6, "uniform4", 2), device=DEV)
    sets = []
    for seed in (0, 1):
        glob = {k: w.to(DEV) for k, w in gen.gen_globals(cfg, seed).items()}
        layers = [{k: w.to(DEV) for k, w in gen.gen_layer(cfg, l, seed).items()} for l in range(cfg.n_layers)]
        sets.append((glob, layers))

    def pack(s):                                   # as the binding does, without its synchronisation
        glob, layers = sets[s]
        g = B.GlobalWeights(**{k: w.data_ptr() for k, w in glob.items()})
        B._check(B.lib().llmcad_pack_globals(v.ctx, g, v.packed.data_ptr(), B._stream()), "pack")
        for l, w in reversed(list(enumerate(layers))):      # the layer that the pass reads first comes last
            lw = B.LayerWeights(**{k: t.data_ptr() for k, t in w.items()})
            B._check(B.lib().llmcad_pack_layer(v.ctx, l, lw, v.packed.data_ptr(), B._stream()), "pack")

    def run():
        return v.verify_tree(P, tokens, parent)["logits"] if op == "verify" else v.prefill(P, tokens, want_logits=True)

    refs = []
    for s in (0, 1):
        pack(s)
        torch.cuda.synchronize()
        refs.append(run().clone())
    assert not torch.equal(refs[0], refs[1])
    outs = []
    for i in range(40):
        pack(i & 1)
        outs.append(run().clone())
    torch.cuda.synchronize()
    assert all(torch.equal(o, refs[i & 1]) for i, o in enumerate(outs))


def test_a_replaced_cache_is_the_one_in_use_and_the_old_one_is_freed():
    """The binding keeps its view of the cache between calls; neither another tensor in `kv` nor another storage under the
    same tensor leaves it on old memory, and a dropped cache is freed at once."""
    cfg = gen.ModelConfig("cache", 2, 512, 4, 128, 1408, 2048, "bf16")
    v = B.Verifier(cfg, 4096)
    nbytes = v.kv.numel()
    v.kv_view().fill_(1)
    held = torch.cuda.memory_allocated()
    v.kv = None
    assert torch.cuda.memory_allocated() <= held - nbytes
    v.kv = torch.zeros(nbytes, dtype=torch.uint8, device=DEV)
    assert v.kv_view().data_ptr() == v.kv.data_ptr() and not v.kv_view().any()
    v.kv.data = torch.full((nbytes,), 0, dtype=torch.uint8, device=DEV)
    v.kv_view().fill_(2)
    assert v.kv_view().data_ptr() == v.kv.data_ptr() and v.kv.any()


@pytest.mark.parametrize("dtype,flags,mb", [("f32", 0, 24), ("bf16", B.FLAG_INT4_WEIGHTS, 82), ("bf16", B.FLAG_SIMT_GEMM, 24)])
def test_a_context_holds_no_room_for_chunks_it_never_runs(dtype, flags, mb):
    """Only bf16 contexts on the tensor cores run prompts in chunks of 256; the others hold activations of 128 nodes. d 4096,
    f 11008: 128 rows of x, xn, q, att (d) and h (f) are 14 MB in fp32, 8 in bf16; with INT4, where hi and lo plane lie 256
    rows apart, they and the remainders of K and V are 24, the segments of the GEMMs 53."""
    import ctypes
    cfg = gen.ModelConfig("room", 1, 4096, 32, 128, 11008, 512, dtype)
    c = B.make_config(cfg, 64, flags=flags)
    torch.cuda.synchronize()
    free = torch.cuda.mem_get_info()[0]
    h = ctypes.c_void_p()
    assert B.lib().llmcad_create(ctypes.byref(c), ctypes.byref(h)) == B.OK
    used = free - torch.cuda.mem_get_info()[0]
    B.lib().llmcad_destroy(h)
    assert 4e6 < used <= mb * 1e6
