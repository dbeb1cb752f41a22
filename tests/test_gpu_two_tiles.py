"""The random shapes and flags of test_gpu_fuzz.py once more, in launches of so many tables that a CTA takes two tiles
(they are small enough for one tile otherwise): the first and the last table against the oracle."""
import dataclasses

import numpy as np
import pytest
import torch

import oracle
from helpers import Guarded, bf16_bits_to_f64, check_bf16_attention, check_fp8_attention
from paper_2609_13031_b200 import api
from paper_2609_13031_b200 import workloads as W
from test_gpu_fuzz import cases, head0

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("i,cfg,n,m,fp8,half,gqa,test_only", cases(96, 2609))
def test_random_shapes_and_flags(i, cfg, n, m, fp8, half, gqa, test_only):
    w = W.CONFIGS[cfg].scaled(n, m)
    test_only = test_only and m > 0
    flags = (api.TEST_ROWS_USE_KV_HEAD0 if gqa else 0) | (api.TEST_ROWS_ONLY if test_only else 0)
    tiles = lambda rows: (rows + 127) // 128
    per_table = w.H * (tiles(m) + (0 if test_only else tiles(n)))
    w = dataclasses.replace(w, B=torch.cuda.get_device_properties(0).multi_processor_count // per_table + 1)
    assert api.attention_rows_per_cta(w.B, w.H, n, m, w.d, flags) == 256
    g = W.generate(w)
    if half:
        g = {k: np.ascontiguousarray(bf16_bits_to_f64(v).astype(np.float16)).view(np.uint16) for k, v in g.items()}
    dtype16, tdt = ("fp16", torch.float16) if half else ("bf16", torch.bfloat16)
    ws = api.new_workspace(w.B, w.H)
    x = {k: torch.from_numpy(v.view(np.int16)).cuda().view(tdt) for k, v in g.items()}
    q_test = x["q_test"] if m else None
    out = {"train": None if test_only else Guarded((w.B, w.H, n, w.d), tdt), "test": Guarded((w.B, w.H, m, w.d), tdt) if m else None}
    into = dict(flags=flags, out_train=out["train"] and out["train"].t, out_test=out["test"] and out["test"].t)
    if fp8:
        o = api.quantize_qkv(x["q_train"], x["k"], x["v"], q_test, ws)
        api.icl_forward_fp8(None if test_only else o["q8"], o["t8"] if m else None, o["k8"], o["v8"], o["sq"], o["sk"],
                            o["sv"], ws, **into)
    else:
        api.icl_forward_bf16(None if test_only else x["q_train"], q_test, x["k"], x["v"], ws, **into)
    assert api.last_device_status(ws) == (0, 0)
    tables = sorted({0, w.B - 1})
    some = lambda a: np.ascontiguousarray(a[tables])
    for name, nq in (("train", n), ("test", m)):
        if out[name] is None:
            continue
        label = f"two tiles {i}/{cfg}/{w.B}x{n}+{m}/fp8={fp8}/half={half}/gqa={gqa}/test_only={test_only}/{name}"
        out[name].check(label)
        got = out[name].t[tables].float().cpu().numpy().astype(np.float64)
        kv0 = head0 if gqa and name == "test" else lambda a: a
        k, v, q = (some(g[c]) for c in ("k", "v", "q_train" if name == "train" else "q_test"))
        if fp8:
            q8, sq = oracle.quantize(some(g["q_train"]), dtype16=dtype16)
            if name == "test":
                q8, _ = oracle.quantize(q, scale_in=sq, dtype16=dtype16)
            (k8, sk), (v8, sv) = (oracle.quantize(a, dtype16=dtype16) for a in (k, v))
            A, Abs, Bnd = oracle.icl_attention_rows(q8, kv0(k8), kv0(v8), np.arange(nq), sq=sq, sk=kv0(sk), sv=kv0(sv))
            check_fp8_attention(got, A, Abs, Bnd, diffuse=False, label=label, named_config=False)
        else:
            A, Abs, _ = oracle.icl_attention_rows(q, kv0(k), kv0(v), np.arange(nq), dtype16=dtype16)
            check_bf16_attention(got, A, Abs, label=label, rounding=2.0 ** -12 if half else 2.0 ** -9)


def bits_of(w):
    return {k: torch.from_numpy(v.view(np.int16)).cuda().view(torch.bfloat16) for k, v in W.generate(w).items()}


@pytest.mark.parametrize("d", [64, 128])
def test_test_rows_are_batch_invariant_and_share_kv_with_train_rows(d):
    """The batch-invariance properties of the one-tile launches, with 19 heads of eight tiles: 152 CTAs of one tile."""
    w = dataclasses.replace(W.CONFIGS["C1"].scaled(640, 300), H=19, d=d)
    assert [api.attention_rows_per_cta(1, w.H, 640, m, d) for m in (300, 129)] == [256, 128]
    x, ws = bits_of(w), api.new_workspace(1, w.H)
    x["q_test"][:, :, 7] = x["q_train"][:, :, 500]
    o = api.quantize_qkv(x["q_train"], x["k"], x["v"], x["q_test"], ws)
    call = lambda t: api.icl_forward_fp8(o["q8"], t, o["k8"], o["v8"], o["sq"], o["sk"], o["sv"], ws)
    train, test = call(o["t8"])
    assert torch.equal(test[:, :, 7], train[:, :, 500])
    perm = torch.randperm(300, generator=torch.Generator().manual_seed(1)).cuda()
    again, shuffled = call(o["t8"][:, :, perm].contiguous())
    assert torch.equal(shuffled, test[:, :, perm]) and torch.equal(again, train)
    _, few = call(o["t8"][:, :, 130:259].contiguous())       # 133 CTAs of one tile
    assert torch.equal(few, test[:, :, 130:259])
    assert api.last_device_status(ws) == (0, 0)
