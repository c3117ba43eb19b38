"""Streams that have only some of the device's SMs (green contexts). The one-kernel passes want them all at once; calls on such
streams go through the kernels per step. Nothing is launched there: calls are captured into a graph and its kernels read."""
import numpy as np
import pytest
import torch

from paper_2309_04255_b200 import binding as B
from paper_2309_04255_b200 import inputs as gen

from gpu_util import Twin, kernels_of

pytestmark = pytest.mark.gpu
SMALL = gen.ModelConfig("small", 2, 512, 4, 128, 1408, 2048, "bf16")


@pytest.fixture()
def stream_of_64_sms():
    from cuda.bindings import driver as drv

    def ok(r):
        assert int(r[0]) == 0, r[0]
        return r[1] if len(r) == 2 else r[1:]

    torch.cuda.synchronize()        # the primary context is there
    dev = ok(drv.cuDeviceGet(0))
    sms = ok(drv.cuDeviceGetDevResource(dev, drv.CUdevResourceType.CU_DEV_RESOURCE_TYPE_SM))
    groups, _, _ = ok(drv.cuDevSmResourceSplitByCount(1, sms, 0, 64))
    ctx = ok(drv.cuGreenCtxCreate(ok(drv.cuDevResourceGenerateDesc(groups[:1], 1)), dev, drv.CUgreenCtxCreate_flags.CU_GREEN_CTX_DEFAULT_STREAM))
    raw = ok(drv.cuGreenCtxStreamCreate(ctx, drv.CUstream_flags.CU_STREAM_NON_BLOCKING, 0))
    yield torch.cuda.ExternalStream(int(raw))
    torch.cuda.synchronize()
    ok(drv.cuStreamDestroy(raw) + (None,))
    ok(drv.cuGreenCtxDestroy(ctx) + (None,))


@pytest.mark.parametrize("cfg,one_kernel", [(SMALL, "stream_pass_kernel"), (gen.MODELS["tiny"], "small_pass_kernel")])
def test_one_kernel_passes_only_where_every_sm_is_there(stream_of_64_sms, cfg, one_kernel):
    tw = Twin(cfg, 64, scale=3.0 if cfg is SMALL else 1.0, keep_host=False)
    tw.fill_prefix_synthetic(40)
    n = 3
    t, p = (torch.as_tensor(np.asarray(a, np.int32), device=tw.v.device) for a in (gen.gen_tokens(cfg, n), [-1, 0, 0]))
    out = tw.v.new_outputs(n)
    calls = {"verify": lambda: tw.v.verify_tree(40, t, p, out=out),
             "extend": lambda: tw.v.extend_tree(40, t, p, 1, top_k=2),
             "prefill": lambda: tw.v.prefill(40, t, want_logits=True)}
    for name, call in calls.items():
        call()
        assert sum(one_kernel in k for k in kernels_of(call)) == 1, name
        on_part = kernels_of(call, stream_of_64_sms)
        assert len(on_part) > 8 and not any("stream_pass_kernel" in k or "small_pass_kernel" in k for k in on_part), name
