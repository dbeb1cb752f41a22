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
