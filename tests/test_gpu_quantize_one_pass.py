"""The one-pass forms of the quantizer (heads held on chip between the maximum and the conversion, by
one block each or by all SMs together) against the two-launch form, which the other tests hold
against the oracle: same codes and scales, bit for bit.  Shapes at their edges: one stage and several, a
shorter last stage, heads just below and above what a block and what the chip holds, test rows that
outnumber the train rows, every call twice on one workspace (it has to leave its words clean)."""
import numpy as np
import pytest
import torch

import oracle
from paper_2609_13031_b200 import api

pytestmark = pytest.mark.gpu


def tensors(B, H, rows, d, dtype, seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    return [torch.empty((B, H, r, d), dtype=dtype, device="cuda").normal_(generator=g) if r else None for r in rows]


@pytest.mark.parametrize("B,H,n,m,d,dtype,flags,stages", [
    (1, 1, 1, 0, 64, "bf16", 0, -1),
    (1, 3, 1, 5, 128, "fp16", 0, -1),
    (1, 2, 257, 31, 64, "bf16", 0, -1),
    (2, 5, 1000, 77, 128, "fp16", api.QUERY_SCALE_FROM_ALL_ROWS, 1),
    (4, 16, 63, 9, 64, "bf16", 0, -1),
    (1, 7, 9001, 300, 128, "bf16", 0, 3),               # 21 units, seven at a time
    (1, 11, 12289, 64, 128, "bf16", 0, 7),              # 33 units, five at a time, then three
    (1, 11, 12289, 64, 128, "bf16", api.QUERY_SCALE_FROM_ALL_ROWS, 0),    # too many heads whose rows enter the maximum
    (1, 6, 8000, 1333, 128, "fp16", api.QUERY_SCALE_FROM_ALL_ROWS, 3),    # 18 units, six at a time
    (1, 2, 33203, 77, 128, "bf16", 0, 0),               # 6 units, one at a time, half a stage empty
    (1, 7, 20011, 3001, 128, "bf16", 0, 7),             # 21 units, three at a time
    (1, 4, 30001, 0, 128, "fp16", 0, 6),                # 12 units, two at a time
    (1, 2, 65536, 1, 128, "bf16", 0, 6),                # the largest head that fits
    (1, 1, 65600, 100, 128, "bf16", 0, 0),              # the first that does not
    (1, 3, 300, 40000, 64, "bf16", 0, -1),              # test rows outnumber the train rows
    (3, 100, 16, 4, 64, "bf16", 0, -1),
    (1, 2, 1024, 130, 64, "fp16", 0, -1),               # the longest head that one block holds
    (1, 2, 1025, 130, 64, "fp16", 0, 1),                # the first that it does not
    (1, 1, 1100, 60001, 64, "bf16", 0, 1),              # test rows fill the SMs, shares of a few KB
    (1, 1, 1000, 70001, 64, "bf16", 0, -1),             # test rows in pieces, a shorter last one
    (100, 8, 130, 3, 64, "bf16", 0, -1),                # heads fill the SMs: no pieces
    (16, 16, 40, 41, 64, "fp16", 0, -1),                # more test rows than train rows: pieces again
    (2, 3, 512, 512, 128, "bf16", api.QUERY_SCALE_FROM_ALL_ROWS, -1),     # the longest test head that enters the maximum
    (2, 3, 512, 513, 128, "bf16", api.QUERY_SCALE_FROM_ALL_ROWS, 0),
    (1, 2, 500, 3000, 64, "bf16", api.QUERY_SCALE_FROM_ALL_ROWS, 0),
])
def test_one_pass_matches_two_launches(B, H, n, m, d, dtype, flags, stages):
    assert api.quantize_stages(3, B, H, n, m, d, flags) == stages
    assert api.quantize_stages(3, B, H, n, m, d, flags | api.QKV_TWO_LAUNCHES) == 0
    tdt = torch.bfloat16 if dtype == "bf16" else torch.float16
    ws = api.new_workspace(B, H)
    for seed in (1, 2):
        x = tensors(B, H, (n, n, n, m), d, tdt, seed)
        got = api.quantize_qkv(*x, ws, flags=flags)
        want = api.quantize_qkv(*x, ws, flags=flags | api.QKV_TWO_LAUNCHES)
        again = api.quantize_qkv(*x, ws, flags=flags)
        for name in ("q8", "k8", "v8", "t8", "sq", "sk", "sv"):
            assert torch.equal(got[name], want[name]), name
            assert torch.equal(again[name], want[name]), name
        assert (api.quantize_stages(1, B, H, n, 0, d) != 0) == (n <= 65536)
        for extra in (0, api.QKV_TWO_LAUNCHES):
            before = api.launch_count()
            code, scale = api.quantize(x[1], ws, flags=extra)
            assert not extra or api.launch_count() - before == 2
            assert torch.equal(code, want["k8"]) and torch.equal(scale, want["sk"])
    assert api.last_device_status(ws) == (0, 0)


@pytest.mark.parametrize("H,n,m,stages", [(7, 9001, 300, 3), (2, 65000, 1000, 6)])
def test_several_stages_match_oracle(H, n, m, stages):
    assert api.quantize_stages(3, 1, H, n, m, 128) == stages
    x = tensors(1, H, (n, n, n, m), 128, torch.bfloat16, 5)
    ws = api.new_workspace(1, H)
    o = api.quantize_qkv(*x, ws)
    bits = [t.view(torch.int16).cpu().numpy().view(np.uint16) for t in x]
    for i, (code, scale) in enumerate((("q8", "sq"), ("k8", "sk"), ("v8", "sv"))):
        want, s = oracle.quantize(bits[i])
        assert np.array_equal(o[code].cpu().numpy(), want) and np.array_equal(o[scale].cpu().numpy(), s)
        if i == 0:
            want_t, _ = oracle.quantize(bits[3], scale_in=s)
    assert np.array_equal(o["t8"].cpu().numpy(), want_t)


def test_workspace_shared_with_other_calls():
    """The words of the one-pass kernel are its own: perturbation, ordered quantization and the
    two-launch form in between change nothing."""
    x = tensors(1, 4, (3000, 3000, 3000, 100), 64, torch.bfloat16, 3)
    ws = api.new_workspace(1, 4)
    first = api.quantize_qkv(*x, ws)
    api.perturb(x[1], 0.05, 1, 1, ws)
    api.quantize_qkv(*x, ws, order_keys=True)
    api.quantize_qkv(*x, ws, flags=api.QKV_TWO_LAUNCHES)
    second = api.quantize_qkv(*x, ws)
    for name in ("q8", "k8", "v8", "t8", "sq", "sk", "sv"):
        assert torch.equal(first[name], second[name]), name
    assert api.last_device_status(ws) == (0, 0)
