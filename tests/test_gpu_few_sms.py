"""A context with some of the SMs only (a green context): a cooperative launch of one block per SM of the
device is refused there, and the quantizer takes its two passes."""
import pytest
import torch

from paper_2609_13031_b200 import api

pytestmark = pytest.mark.gpu


@pytest.fixture
def stream_of_16_sms():
    cu = pytest.importorskip("cuda.bindings.driver")
    if not hasattr(cu, "cuGreenCtxCreate"):
        pytest.skip("no green contexts in these bindings")
    torch.zeros(1, device="cuda")

    def ok(r):
        assert int(r[0]) == 0, r[0]
        return r[1:]
    dev, = ok(cu.cuDeviceGet(torch.cuda.current_device()))
    sms, = ok(cu.cuDeviceGetDevResource(dev, cu.CUdevResourceType.CU_DEV_RESOURCE_TYPE_SM))
    groups = ok(cu.cuDevSmResourceSplitByCount(1, sms, 0, 16))[0]
    desc, = ok(cu.cuDevResourceGenerateDesc(groups, 1))
    ctx, = ok(cu.cuGreenCtxCreate(desc, dev, cu.CUgreenCtxCreate_flags.CU_GREEN_CTX_DEFAULT_STREAM))
    stream, = ok(cu.cuGreenCtxStreamCreate(ctx, cu.CUstream_flags.CU_STREAM_NON_BLOCKING, 0))
    yield int(stream)
    torch.cuda.synchronize()
    cu.cuStreamDestroy(stream)
    cu.cuGreenCtxDestroy(ctx)


@pytest.mark.parametrize("H,n,m,stages", [(2, 3000, 100, 1), (8, 20011, 301, 8)])
def test_refused_cooperative_launch_takes_two_passes(stream_of_16_sms, H, n, m, stages):
    assert api.quantize_stages(3, 1, H, n, m, 128) == stages
    x = [torch.randn((1, H, r, 128), device="cuda").to(torch.bfloat16) for r in (n, n, n, m)]
    ws = api.new_workspace(1, H)
    want = api.quantize_qkv(*x, ws, flags=api.QKV_TWO_LAUNCHES)
    out = {name: torch.zeros_like(t) for name, t in want.items()}
    code, scale = torch.zeros_like(out["k8"]), torch.zeros_like(out["sk"])
    torch.cuda.synchronize()
    p = lambda t: t.data_ptr()
    lib = api.load()
    for _ in range(2):
        rc = lib.fp8attn_quantize_qkv(*(p(t) for t in x), 1, H, n, m, 128, *(p(out[k]) for k in ("q8", "k8", "v8", "t8", "sq", "sk", "sv")),
                                      p(ws), ws.numel(), stream_of_16_sms)
        assert rc == api.OK
        rc = lib.fp8attn_quantize(p(x[1]), 1, H, n, 128, None, p(code), p(scale), p(ws), ws.numel(), stream_of_16_sms)
        assert rc == api.OK
        torch.cuda.synchronize()
        assert all(torch.equal(out[k], want[k]) for k in want)
        assert torch.equal(code, want["k8"]) and torch.equal(scale, want["sk"])
    got = api.quantize_qkv(*x, ws)                      # with all SMs again, in one pass
    assert all(torch.equal(got[k], want[k]) for k in want)
    assert api.last_device_status(ws) == (0, 0)
