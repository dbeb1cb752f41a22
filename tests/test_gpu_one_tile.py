"""CTAs of one 128-row tile, in launches that leave SMs free: the same rows bit for bit as CTAs of two tiles
give in a launch with more test rows, at the edges of tiles and key steps, and within the oracle's bounds."""
import numpy as np
import pytest
import torch

import oracle
from helpers import Guarded, check_bf16_attention, check_fp8_attention, sample_rows
from paper_2609_13031_b200 import api

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("B,H,n,m,d", [
    (1, 1, 1, 1, 64), (1, 2, 127, 129, 128), (1, 3, 128, 0, 64), (1, 2, 129, 31, 64), (2, 2, 257, 256, 128),
    (1, 8, 1000, 333, 128), (1, 8, 1152, 1100, 64), (1, 2, 4100, 700, 128), (1, 1, 9000, 65, 64),
])
@pytest.mark.parametrize("kind", ["fp8", "bf16", "fp16"])
def test_same_rows_as_with_two_tiles(B, H, n, m, d, kind):
    g = torch.Generator(device="cuda")
    g.manual_seed(n + m)
    dt = torch.float16 if kind == "fp16" else torch.bfloat16
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    many = m + (sms // (B * H) + 1) * 128
    assert api.attention_rows_per_cta(B, H, n, m, d) == 128
    assert api.attention_rows_per_cta(B, H, n, many, d) == 256
    q, k, v, t = (torch.randn((B, H, r, d), device="cuda", generator=g).to(dt) for r in (n, n, n, many))
    ws = api.new_workspace(B, H)
    if kind == "fp8":
        o = api.quantize_qkv(q, k, v, t, ws)
        q, k, v, t = (o[c] for c in ("q8", "k8", "v8", "t8"))
        scales = tuple(o[c] for c in ("sq", "sk", "sv"))
        call = lambda test, *outs: api.icl_forward_fp8(q, test, k, v, *scales, ws, 0.0, *outs)
    else:
        call = lambda test, *outs: api.icl_forward_bf16(q, test, k, v, ws, 0.0, *outs)
    want_train, want_test = call(t)
    few = t[:, :, :m].contiguous() if m else None
    train, test = Guarded((B, H, n, d), dt if kind != "fp8" else torch.bfloat16), Guarded((B, H, m, d), want_test.dtype)
    call(few, train.t, test.t if m else None)
    assert api.last_device_status(ws) == (0, 0)
    train.check()
    test.check()
    assert torch.equal(train.t, want_train)
    if m:
        assert torch.equal(test.t, want_test[:, :, :m])
    # the oracle's bounds on some rows of the larger call (equal to the smaller one's where both have them)
    rows = sample_rows(n, 5, 3)
    bits = [x.cpu().numpy() if kind == "fp8" else x.view(torch.int16).cpu().numpy().view(np.uint16) for x in (q, k, v)]
    got = train.t[:, :, torch.from_numpy(rows).cuda()].float().cpu().numpy().astype(np.float64)
    if kind == "fp8":
        A, Abs, Bnd = oracle.icl_attention_rows(*bits, rows, **dict(zip(("sq", "sk", "sv"), (s.cpu().numpy() for s in scales))))
        check_fp8_attention(got, A, Abs, Bnd, diffuse=False, label="one tile", named_config=False)
    else:
        A, Abs, _ = oracle.icl_attention_rows(*bits, rows, dtype16=kind)
        check_bf16_attention(got, A, Abs, label="one tile", rounding=2.0 ** (-12 if kind == "fp16" else -9))


@pytest.mark.parametrize("flags", [api.TEST_ROWS_USE_KV_HEAD0, api.TEST_ROWS_ONLY, api.TEST_ROWS_USE_KV_HEAD0 | api.TEST_ROWS_ONLY])
@pytest.mark.parametrize("B,H,n,m,d", [(1, 3, 500, 129, 64), (2, 4, 385, 31, 128)])
@pytest.mark.parametrize("fp8", [True, False])
def test_flags_give_the_same_rows_as_with_two_tiles(B, H, n, m, d, fp8, flags):
    torch.manual_seed(n + flags)
    many = m + (torch.cuda.get_device_properties(0).multi_processor_count // (B * H) + 1) * 128
    assert [api.attention_rows_per_cta(B, H, n, r, d, flags) for r in (m, many)] == [128, 256]
    q, k, v, t = (torch.randn((B, H, r, d), device="cuda").to(torch.bfloat16) for r in (n, n, n, many))
    ws = api.new_workspace(B, H)
    o = api.quantize_qkv(q, k, v, t, ws)
    if fp8:
        q, k, v, t = (o[c] for c in ("q8", "k8", "v8", "t8"))
    call = (lambda x: api.icl_forward_fp8(None if flags & api.TEST_ROWS_ONLY else q, x, k, v, o["sq"], o["sk"], o["sv"], ws, flags=flags)) \
        if fp8 else (lambda x: api.icl_forward_bf16(None if flags & api.TEST_ROWS_ONLY else q, x, k, v, ws, flags=flags))
    want_train, want = call(t)
    train, test = call(t[:, :, :m].contiguous())
    assert torch.equal(test, want[:, :, :m])
    assert (train is None and want_train is None) if flags & api.TEST_ROWS_ONLY else torch.equal(train, want_train)
    assert api.last_device_status(ws) == (0, 0)


@pytest.mark.parametrize("n,m,d,rows", [(16384, 65, 64, 128), (16385, 65, 64, 256), (16384, 129, 128, 128), (16385, 129, 128, 256)])
def test_both_sides_of_the_limit_of_keys(n, m, d, rows):
    """One head, test rows alone: the same rows as in a launch of enough test rows for two tiles."""
    torch.manual_seed(n)
    flags, many = api.TEST_ROWS_ONLY, m + 148 * 128
    assert [api.attention_rows_per_cta(1, 1, n, r, d, flags) for r in (m, many)] == [rows, 256]
    k, v, t = (torch.randn((1, 1, r, d), device="cuda").to(torch.bfloat16) for r in (n, n, many))
    ws = api.new_workspace(1, 1)
    _, want = api.icl_forward_bf16(None, t, k, v, ws, flags=flags)
    _, got = api.icl_forward_bf16(None, t[:, :, :m].contiguous(), k, v, ws, flags=flags)
    assert torch.equal(got, want[:, :, :m]) and api.last_device_status(ws) == (0, 0)


@pytest.mark.parametrize("H,n,m,d", [(8, 1930, 250, 64), (8, 1930, 250, 128), (8, 2200, 0, 128)])
def test_one_tile_where_the_keys_could_be_split(H, n, m, d):
    """FP8ATTN_SPLIT_TAIL where one tile is over sooner than a split in two: the same call as without the flag."""
    torch.manual_seed(n)
    assert api.attention_rows_per_cta(1, H, n, m, d, api.SPLIT_TAIL) == 128
    q, k, v, t = (torch.randn((1, H, r, d), device="cuda").to(torch.bfloat16) for r in (n, n, n, m))
    ws = api.new_workspace(1, H, n_train=n, n_test=m, d=d)
    before = api.launch_count()
    got = api.icl_forward_bf16(q, t if m else None, k, v, ws, flags=api.SPLIT_TAIL)
    assert api.launch_count() - before == 1
    want = api.icl_forward_bf16(q, t if m else None, k, v, ws)
    assert all(a is b is None or torch.equal(a, b) for a, b in zip(got, want)) and api.last_device_status(ws) == (0, 0)


def test_three_tiles_where_their_split_is_over_sooner():
    """300 test rows of 49 heads against 4,000 keys: 49 blocks of three tiles in three ranges, by the oracle's bounds."""
    H, n, m, d, flags = 49, 4000, 300, 64, api.SPLIT_TAIL | api.TEST_ROWS_ONLY
    assert api.attention_rows_per_cta(1, H, n, m, d, flags) == 384
    torch.manual_seed(n)
    q, k, v, t = (torch.randn((1, H, r, d), device="cuda").to(torch.bfloat16) for r in (n, n, n, m))
    ws = api.new_workspace(1, H, n_train=n, n_test=m, d=d)
    o = api.quantize_qkv(q, k, v, t, ws)
    before = api.launch_count()
    _, got = api.icl_forward_fp8(None, o["t8"], o["k8"], o["v8"], o["sq"], o["sk"], o["sv"], ws, flags=flags)
    assert api.launch_count() - before == 2 and api.last_device_status(ws) == (0, 0)
    rows = sample_rows(m, 8, 3)
    z = {c: o[c].cpu().numpy() for c in ("t8", "k8", "v8", "sq", "sk", "sv")}
    A, Abs, Bnd = oracle.icl_attention_rows(z["t8"], z["k8"], z["v8"], rows, sq=z["sq"], sk=z["sk"], sv=z["sv"])
    check_fp8_attention(got[:, :, torch.from_numpy(rows).cuda()].float().cpu().numpy().astype(np.float64), A, Abs, Bnd,
                        diffuse=False, label="three tiles", named_config=False)
