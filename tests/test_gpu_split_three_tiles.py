"""The key split of three-tile CTAs (d = 64), in more ranges than one combine batch holds, and in as few as
two with many rows, against the oracle; and scratch of the smallest accepted size."""
import dataclasses

import numpy as np
import pytest
import torch

import oracle
from helpers import check_bf16_attention, check_fp8_attention, sample_rows
from paper_2609_13031_b200 import api
from paper_2609_13031_b200 import workloads as W

pytestmark = pytest.mark.gpu


def f64(t):
    return t.float().cpu().numpy().astype(np.float64)


@pytest.mark.parametrize("B,H,n,m,test_only,launches,rows_per_cta,d", [
    (1, 8, 20011, 300, True, 2, 384, 64),      # three tiles, 18 ranges
    (1, 2, 17000, 129, True, 2, 256, 64),      # 33 ranges of four steps
    (4, 16, 4200, 300, False, 3, 384, 64),     # full rounds, then 28 blocks in five ranges
    (1, 8, 4100, 2048, True, 2, 256, 64),      # 64 blocks in two ranges: three tiles would not pay
    (1, 16, 4100, 700, True, 2, 256, 64),      # 48 blocks in three
    (1, 7, 3700, 700, True, 2, 256, 128),      # 21 blocks in seven
])
@pytest.mark.parametrize("kind", ["fp8", "fp16"])
def test_split_against_oracle(B, H, n, m, test_only, launches, rows_per_cta, d, kind):
    w = dataclasses.replace(W.CONFIGS["C4"].scaled(n, m), B=B, H=H, d=d)
    g = W.generate(w)
    flags = api.SPLIT_TAIL | (api.TEST_ROWS_ONLY if test_only else 0)
    assert api.attention_rows_per_cta(B, H, n, m, d, flags) == rows_per_cta
    ws = api.new_workspace(B, H, n_train=n, n_test=m, d=d)
    dev = lambda a: torch.from_numpy(a).cuda()
    rows_tr, rows_te = sample_rows(n, 6, 3), np.unique(np.concatenate([sample_rows(m, 12, 3), np.arange(max(0, m - 50), m, 7)]))
    calls = (("test", rows_te),) if test_only else (("train", rows_tr), ("test", rows_te))
    before = api.launch_count()
    if kind == "fp8":
        q8, sq = oracle.quantize(g["q_train"])
        k8, sk = oracle.quantize(g["k"])
        v8, sv = oracle.quantize(g["v"])
        t8, _ = oracle.quantize(g["q_test"], scale_in=sq)
        out = dict(zip(("train", "test"), api.icl_forward_fp8(dev(q8), dev(t8), dev(k8), dev(v8), dev(sq), dev(sk), dev(sv),
                                                              ws, flags=flags)))
    else:
        half = {k: W.bf16_bits_to_f32(v).astype(np.float16) for k, v in g.items()}
        x = {k: torch.from_numpy(v).cuda() for k, v in half.items()}
        out = dict(zip(("train", "test"), api.icl_forward_bf16(x["q_train"], x["q_test"], x["k"], x["v"], ws, flags=flags)))
    assert api.launch_count() - before == launches
    assert api.last_device_status(ws) == (0, 0)
    for name, rows in calls:
        got = f64(out[name][:, :, torch.from_numpy(rows).cuda()])
        if kind == "fp8":
            A, Abs, Bnd = oracle.icl_attention_rows(q8 if name == "train" else t8, k8, v8, rows, sq=sq, sk=sk, sv=sv)
            check_fp8_attention(got, A, Abs, Bnd, diffuse=False, label=f"split three tiles/{name}", named_config=False)
        else:
            bits = {k: v.view(np.uint16) for k, v in half.items()}
            A, Abs, _ = oracle.icl_attention_rows(bits["q_train" if name == "train" else "q_test"], bits["k"], bits["v"],
                                                  rows, dtype16="fp16")
            check_bf16_attention(got, A, Abs, label=f"split three tiles fp16/{name}", rounding=2.0 ** -12)


def test_many_ranges_cost_no_precision():
    """Every range rounds P against a maximum of its own, which is never above the row's: the error against
    64 bits of a launch in 36 ranges is that of the unsplit one (0.90 .. 1.01 of it over 8,192 .. 524,288 keys,
    16 .. 2,048 rows, both head sizes and all types; 1.06 leaves three times the spread of a sample this size)."""
    torch.manual_seed(5)
    B, H, n, m, d = 1, 2, 18500, 250, 64
    q, k, v = (torch.randn((B, H, n, d), device="cuda").to(torch.bfloat16) for _ in range(3))
    t = torch.randn((B, H, m, d), device="cuda").to(torch.bfloat16)
    ws = api.new_workspace(B, H, n_train=n, n_test=m, d=d)
    o = api.quantize_qkv(q, k, v, t, ws)
    deq = lambda c, s: o[c].view(torch.float8_e4m3fn).double() * o[s].double()[:, :, None, None]
    want = torch.softmax(deq("t8", "sq") @ deq("k8", "sk").transpose(2, 3) * d ** -0.5, dim=3) @ deq("v8", "sv")
    err = {}
    for flags in (0, api.SPLIT_TAIL):
        _, out = api.icl_forward_fp8(None, o["t8"], o["k8"], o["v8"], o["sq"], o["sk"], o["sv"], ws,
                                     flags=flags | api.TEST_ROWS_ONLY)
        err[flags] = ((out.double() - want).norm() / want.norm()).item()
    assert err[api.SPLIT_TAIL] < 1.06 * err[0], err


def test_smallest_scratch_is_accepted():
    """Scratch for 256 rows per SM, the size the flag has always asked for."""
    torch.manual_seed(0)
    B, H, n, m, d = 1, 8, 20000, 300, 64
    mk = lambda r: torch.randint(0, 0x60, (B, H, r, d), dtype=torch.uint8, device="cuda")
    t, k, v = mk(m), mk(n), mk(n)
    s = torch.full((B, H), 0.01, dtype=torch.float32, device="cuda")
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    small = api.workspace_bytes(B, H) + sms * 256 * (d + 4) * 4
    flags = api.TEST_ROWS_ONLY | api.SPLIT_TAIL
    outs = []
    for nbytes in (small, api.workspace_bytes(B, H, n, m, d)):
        ws = torch.zeros(nbytes + 4096, dtype=torch.uint8, device="cuda")
        ws[nbytes:] = 0xA5
        outs.append(api.icl_forward_fp8(None, t, k, v, s, s, s, ws[:nbytes], flags=flags)[1].float())
        assert api.last_device_status(ws) == (0, 0) and bool((ws[nbytes:] == 0xA5).all())
    # P is rounded against other maxima: about sqrt(2) x 2.6 % of a weight, averaged over the row
    assert ((outs[0] - outs[1]).norm() / outs[1].norm()).item() < 0.04
    with pytest.raises(api.Fp8AttnError) as e:
        api.icl_forward_fp8(None, t, k, v, s, s, s, torch.zeros(small - 1, dtype=torch.uint8, device="cuda"), flags=flags)
    assert e.value.status == api.ERR_WORKSPACE
