"""The device-side error path: a bounded wait that runs out is reported through the
workspace status words, the kernel returns normally, the error is sticky until it
has been read, and the context stays usable.  The wait is made to expire on a
barrier that nothing signals (no fault, trap or hang is involved)."""
import pytest
import torch

from paper_2609_13031_b200 import api

pytestmark = pytest.mark.gpu


def test_expired_wait_is_reported_is_sticky_and_clears():
    ws = api.new_workspace(1, 2)
    assert api.last_device_status(ws) == (0, 0)
    api.selftest_wait_timeout(ws, limit_us=500)
    torch.cuda.synchronize()                                   # the kernel came back by itself
    # while the error is pending, an attention launch on this workspace does nothing
    q = torch.randint(0, 100, (1, 2, 256, 64), dtype=torch.uint8, device="cuda")
    s = torch.ones((1, 2), dtype=torch.float32, device="cuda")
    out = torch.full((1, 2, 256, 64), 7.0, dtype=torch.bfloat16, device="cuda")
    api.icl_forward_fp8(q, None, q, q, s, s, s, ws, out_train=out)
    torch.cuda.synchronize()
    assert torch.all(out == 7.0)
    status, detail = api.last_device_status(ws)
    assert status == api.ERR_TIMEOUT
    assert detail >> 24 == 11                                   # the self-test's wait id
    assert "timed out" in api.status_string(status)
    # read once -> cleared; the same workspace and context work again
    assert api.last_device_status(ws) == (0, 0)
    api.icl_forward_fp8(q, None, q, q, s, s, s, ws, out_train=out)
    assert api.last_device_status(ws) == (0, 0)
    assert not torch.all(out == 7.0) and torch.isfinite(out.float()).all()


@pytest.mark.parametrize("n,m,stages", [(512, 128, -1), (3000, 200, 1), (8192, 2048, 2)])
def test_small_fused_quantization_writes_nothing_while_an_error_is_pending(n, m, stages):
    assert api.quantize_stages(3, 1, 8, n, m, 64) == stages
    q, k, v = (torch.randn((1, 8, n, 64), device="cuda").to(torch.bfloat16) for _ in range(3))
    t = torch.randn((1, 8, m, 64), device="cuda").to(torch.bfloat16)
    ws = api.new_workspace(1, 8)
    want = api.quantize_qkv(q, k, v, t, ws, flags=api.QKV_TWO_LAUNCHES)
    out = {name: torch.full_like(x, 7) for name, x in want.items()}
    api.selftest_wait_timeout(ws, limit_us=500)
    api.quantize_qkv(q, k, v, t, ws, out=out)
    assert all((x == 7).all() for x in out.values())
    code, scale = api.quantize(k, ws)                              # tensors by themselves are quantized all the same
    assert torch.equal(code, want["k8"]) and torch.equal(scale, want["sk"])
    status, detail = api.last_device_status(ws)
    assert status == api.ERR_TIMEOUT and detail >> 24 == 11         # the self-test's, not one of the quantizer's
    api.quantize_qkv(q, k, v, t, ws, out=out)
    assert all(torch.equal(out[name], want[name]) for name in want)
    assert api.last_device_status(ws) == (0, 0)


@pytest.mark.parametrize("H,n,d,stages", [(4, 3000, 64, 1), (8, 20011, 128, 3), (3, 40000, 128, 3), (16, 12289, 64, 2)])
@pytest.mark.parametrize("limit", [1, 2000, 6000, 20000])
def test_one_pass_quantizer_gives_up_cleanly(H, n, d, stages, limit):
    """Waits that run out (at once, or in the middle of a stage whose copies are under way): the call
    comes back, says so, leaves its words at zero and writes nowhere else; the next call is right."""
    assert api.quantize_stages(1, 1, H, n, 0, d) == stages
    torch.manual_seed(n + limit)
    x = torch.randn((1, H, n, d), device="cuda").to(torch.bfloat16)
    want, want_scale = torch.empty_like(x, dtype=torch.uint8), torch.empty((1, H), device="cuda")
    api.quantize_noalloc(x, want, want_scale)
    ws = api.new_workspace(1, H)
    guarded = torch.full((x.numel() + 8192,), 0x55, dtype=torch.uint8, device="cuda")
    codes, scale = guarded[4096:-4096].view(x.shape), torch.zeros((1, H), device="cuda")
    for _ in range(3):
        api.selftest_quantize_timeout(x, ws, codes, scale, limit_clocks=limit)
        torch.cuda.synchronize()
        left = ws.clone()
        assert not left[16:].any()                             # counter, words and accumulators
        assert (guarded[:4096] == 0x55).all() and (guarded[-4096:] == 0x55).all()
        status, detail = api.last_device_status(ws)
        assert status in (api.OK, api.ERR_TIMEOUT) and (limit > 1 or status == api.ERR_TIMEOUT)
        assert (detail >> 24) == (32 if status else 0)
        if status == api.OK:
            assert torch.equal(codes, want) and torch.equal(scale, want_scale)
        got, got_scale = api.quantize(x, ws)
        assert torch.equal(got, want) and torch.equal(got_scale, want_scale)
        assert api.last_device_status(ws) == (0, 0)


def test_selftest_argument_checks():
    lib = api.load()
    ws = api.new_workspace(1, 1)
    assert lib.fp8attn_selftest_wait_timeout(ws.data_ptr(), ws.numel(), 0, None) == api.ERR_INVALID_ARG
    assert lib.fp8attn_selftest_wait_timeout(None, ws.numel(), 10, None) == api.ERR_WORKSPACE
    x = torch.zeros((1, 1, 1025, 64), dtype=torch.bfloat16, device="cuda")
    o, s = torch.empty_like(x, dtype=torch.uint8), torch.empty((1, 1), device="cuda")
    call = lambda rows, limit, w=ws.data_ptr(): lib.fp8attn_selftest_quantize_timeout(
        x.data_ptr(), 1, 1, rows, 64, o.data_ptr(), s.data_ptr(), limit, w, ws.numel(), None)
    assert call(1025, 0) == call(0, 10) == call(1025, 200000000) == api.ERR_INVALID_ARG
    assert call(1024, 10) == api.ERR_UNSUPPORTED                # a block per head: no waits
    assert call(1025, 10, None) == api.ERR_WORKSPACE
    torch.cuda.synchronize()
    assert api.last_device_status(ws) == (0, 0)
