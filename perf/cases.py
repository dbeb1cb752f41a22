"""What the library is asked to do in use, as cases that can be timed and compared.

Every case goes through the public functions of ``paper_2609_13031_b200.api``.  Kinds:

``fp8``       quantize Q, K, V and the test queries of one ICL-attention layer, then both attention
              calls in FP8 (the whole path; one call per layer and table batch)
``gated``     the same layer below the 8,192-row gate, where the final configuration stays in 16 bits
``attn16``    the 16-bit attention calls on their own (callers that do not quantize)
``predict``   new test rows against a long train context whose quantized keys and values are kept:
              quantize the test queries with the train-query scale, run the test call alone
``quant_qkv`` the four quantizations of a layer, for callers that keep the codes
``quant_one`` one tensor quantized on its own
``host``      the host-to-host step: tables in page-locked host memory, results back there
``perturb``   seeded Gaussian noise on one tensor, the noise study's stand-in for quantization

Value distributions follow the workloads of this repository: N(0,1), a few outlier channels,
log-normal row gains, keys with a constant offset.
"""
import math

import torch

from paper_2609_13031_b200 import api

# dtype "bf16" / "fp16"; dist: "normal", "outlier", "rowgain", "kshift"; split: balance the last round
# of a small launch; order: keys of largest norm first
_DEFAULT = dict(kind="fp8", B=1, H=8, d=64, n_train=1024, n_test=256, dtype="bf16", dist="normal",
                split=True, order=False)


def _case(name=None, **kw):
    c = dict(_DEFAULT, **kw)
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # a tiny table, two heads: launches and host time are all there is
        _case("fp8_512", H=2, n_train=512, n_test=128, split=False),
        # a table just at the gate, with outlier channels
        _case("fp8_8k", n_train=8192, n_test=2048, dist="outlier"),
        # a mid-size table of no round size, d = 128
        _case("fp8_20k_ragged", d=128, n_train=20011, n_test=3001, dist="rowgain"),
        # the large single table of the benchmark, d = 128, keys of largest norm first
        _case("fp8_64k", d=128, n_train=65536, n_test=16384, dist="rowgain", order=True),
        # a batch of four very large tables
        _case("fp8_4x256k", B=4, H=4, n_train=262144, n_test=65536, dist="kshift"),
        # a small fp16 table of odd size below the gate
        _case("gated_3k_ragged", kind="gated", d=128, n_train=3001, n_test=777, dtype="fp16", split=False),
        # the 16-bit path on a mid-size table
        _case("attn16_32k", kind="attn16", n_train=32768, n_test=8192, dist="outlier"),
        # a few hundred new rows against a long context
        _case("predict_300_of_256k", kind="predict", n_train=262144, n_test=300),
        # codes of a large layer
        _case("quant_qkv_64k", kind="quant_qkv", d=128, n_train=65536, n_test=16384, dist="rowgain"),
        # one odd-sized fp16 tensor of two tables
        _case("quant_one_12k", kind="quant_one", B=2, n_train=12289, n_test=0, dtype="fp16"),
        # a mid-size table that lives in host memory
        _case("host_16k", kind="host", d=128, n_train=16384, n_test=4096, dist="rowgain"),
        # noise on the keys of a large layer
        _case("perturb_64k", kind="perturb", d=128, n_train=65536, n_test=0),
    ]


def _spread(rng, lo, hi):
    """A whole number spread over the logarithm of [lo, hi]; odd sizes among them, and round ones."""
    n = int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))
    if rng.random() < 0.3:
        n = max(lo, n // 256 * 256)
    return min(max(n, lo), hi)


def draw(rng):
    kind = rng.choice(["fp8"] * 5 + ["gated", "attn16", "attn16", "predict", "quant_qkv", "quant_one", "host", "perturb"])
    d = rng.choice([64, 128])
    B, H = rng.choice([(1, 2), (1, 4), (1, 8), (1, 8), (1, 8), (2, 8), (4, 4), (1, 16)])
    dist = rng.choice(["normal", "outlier", "rowgain", "kshift"])
    dtype = rng.choice(["bf16", "bf16", "bf16", "fp16"])
    order = False
    if kind == "fp8":
        n_train = _spread(rng, 256, 131072)
        n_test = _spread(rng, 32, max(64, n_train // 4))
        order = n_train >= 32768 and rng.random() < 0.5
    elif kind == "gated":
        n_train, n_test = _spread(rng, 256, 8192), _spread(rng, 32, 2048)
    elif kind == "attn16":
        n_train = _spread(rng, 512, 65536)
        n_test = _spread(rng, 32, max(64, n_train // 4))
    elif kind == "predict":
        n_train, n_test = _spread(rng, 8192, 524288), _spread(rng, 16, 2048)
    elif kind == "host":
        n_train = _spread(rng, 512, 32768)
        n_test = _spread(rng, 32, max(64, n_train // 4))
    else:
        n_train, n_test = _spread(rng, 256, 131072), _spread(rng, 32, 32768) if kind == "quant_qkv" else 0
    if kind == "perturb":
        dtype = "bf16"
    return _case(kind=kind, B=B, H=H, d=d, n_train=n_train, n_test=n_test, dtype=dtype, dist=dist,
                 split=rng.random() < 0.8, order=order)


def _inputs(case, seed, names):
    """16-bit tensors on the GPU, made from the seed alone."""
    B, H, d = case["B"], case["H"], case["d"]
    dtype = torch.bfloat16 if case["dtype"] == "bf16" else torch.float16
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    gain = None
    if case["dist"] == "outlier":      # four channels of a head, the same ones in all its tensors
        gain = torch.ones((B, H, 1, d), dtype=dtype, device="cuda")
        gain.scatter_(3, torch.rand((B, H, 1, d), device="cuda", generator=g).topk(4, dim=3).indices, 20.0)
    out = {}
    for name in names:
        rows = case["n_test"] if name == "q_test" else case["n_train"]
        x = torch.empty((B, H, rows, d), dtype=dtype, device="cuda").normal_(generator=g)
        if gain is not None:
            x.mul_(gain)
        elif case["dist"] == "rowgain":
            x.mul_(torch.randn((B, H, rows, 1), device="cuda", generator=g).mul_(0.5).exp_().to(dtype))
        elif case["dist"] == "kshift" and name == "k":
            x.add_(3.0)
        out[name] = x
    return out


def prepare(case, seed):
    B, H, d, n_train, n_test = (case[k] for k in ("B", "H", "d", "n_train", "n_test"))
    kind = case["kind"]
    s = {"kind": kind, "order": case["order"], "flags": api.SPLIT_TAIL if case["split"] else 0}
    if kind in ("quant_one", "perturb"):
        s.update(_inputs(case, seed, ("k",)))
        s["ws"] = api.new_workspace(B, H)
        if kind == "quant_one":
            s["codes"] = torch.empty((B, H, n_train, d), dtype=torch.uint8, device="cuda")
            s["scale"] = torch.empty((B, H), dtype=torch.float32, device="cuda")
        else:
            s["noisy"] = torch.empty_like(s["k"])
            s["seed"] = seed
        return s
    s.update(_inputs(case, seed, ("q_train", "k", "v", "q_test")))
    if kind == "host":
        for name in ("q_train", "k", "v", "q_test"):
            pinned = torch.empty(s[name].shape, dtype=s[name].dtype, pin_memory=True)
            pinned.copy_(s[name])
            s[name] = pinned
        s["out_train"] = torch.empty(s["k"].shape, dtype=s["k"].dtype, pin_memory=True)
        s["out_test"] = torch.empty(s["q_test"].shape, dtype=s["k"].dtype, pin_memory=True)
        s["scratch"] = torch.empty(api.host_step_scratch_bytes(B, H, n_train, n_test, d), dtype=torch.uint8,
                                   device="cuda")
        return s
    s["ws"] = api.new_workspace(B, H, n_train=n_train, n_test=n_test, d=d)
    if kind == "predict":
        # fitted once and kept: quantized keys and values, and the train-query scale
        kept = api.quantize_qkv(s.pop("q_train"), s.pop("k"), s.pop("v"), None, s["ws"])
        s["kept"] = {n: kept[n] for n in ("k8", "v8", "sq", "sk", "sv")}
    elif kind == "quant_qkv" or s["order"]:
        # a caller with buffers of its own
        dev = dict(dtype=torch.uint8, device="cuda")
        s["codes"] = {"q8": torch.empty((B, H, n_train, d), **dev), "k8": torch.empty((B, H, n_train, d), **dev),
                      "v8": torch.empty((B, H, n_train, d), **dev), "t8": torch.empty((B, H, n_test, d), **dev),
                      "sq": torch.empty((B, H), device="cuda"), "sk": torch.empty((B, H), device="cuda"),
                      "sv": torch.empty((B, H), device="cuda")}
        if s["order"]:
            s["codes"]["key_dest"] = torch.empty((B, H, n_train), dtype=torch.int32, device="cuda")
            s["out_train"] = torch.empty_like(s["k"])
            s["out_test"] = torch.empty_like(s["q_test"])
    return s


def run(s):
    kind = s["kind"]
    if kind == "fp8" and not s["order"]:
        return api.icl_attention(s["q_train"], s["q_test"], s["k"], s["v"], s["ws"], flags=s["flags"])
    if kind == "fp8":
        o = api.quantize_qkv(s["q_train"], s["k"], s["v"], s["q_test"], s["ws"], out=s["codes"], order_keys=True)
        return api.icl_forward_fp8(o["q8"], o["t8"], o["k8"], o["v8"], o["sq"], o["sk"], o["sv"], s["ws"],
                                   out_train=s["out_train"], out_test=s["out_test"], flags=s["flags"])
    if kind == "gated":
        return api.icl_attention_gated(s["q_train"], s["q_test"], s["k"], s["v"], s["ws"])
    if kind == "attn16":
        return api.icl_forward_bf16(s["q_train"], s["q_test"], s["k"], s["v"], s["ws"], flags=s["flags"])
    if kind == "predict":
        o = s["kept"]
        t8, _ = api.quantize(s["q_test"], s["ws"], scale_in=o["sq"])
        _, out = api.icl_forward_fp8(None, t8, o["k8"], o["v8"], o["sq"], o["sk"], o["sv"], s["ws"],
                                     flags=s["flags"] | api.TEST_ROWS_ONLY)
        return out
    if kind == "quant_qkv":
        return api.quantize_qkv(s["q_train"], s["k"], s["v"], s["q_test"], s["ws"], out=s["codes"])
    if kind == "quant_one":
        return api.quantize(s["k"], s["ws"], out=s["codes"], scale_out=s["scale"])
    if kind == "host":
        return api.icl_step_host(s["q_train"], s["k"], s["v"], s["q_test"], s["scratch"],
                                 out_train=s["out_train"], out_test=s["out_test"])
    return api.perturb(s["k"], 0.0265, s["seed"], 1, s["ws"], out=s["noisy"])


def work(case):
    B, H, d, n_train, n_test = (case[k] for k in ("B", "H", "d", "n_train", "n_test"))
    kind = case["kind"]
    train, test = B * H * d * n_train, B * H * d * n_test      # elements
    both = 4.0 * B * H * d * n_train * (n_train + n_test)       # Q K^T and P V of both calls
    if kind in ("fp8", "gated", "attn16", "host"):
        # four 16-bit tensors in, two out
        return {"bytes": 2 * (3 * train + test) + 2 * (train + test), "flops": both}
    if kind == "predict":
        return {"bytes": 2 * train + 4 * test, "flops": 4.0 * B * H * d * n_train * n_test}
    if kind == "quant_qkv":
        return {"bytes": 3 * (3 * train + test), "flops": 0}
    return {"bytes": (3 if kind == "quant_one" else 4) * train, "flops": 0}


def tolerance(case):
    """About four times what the path shows against itself with K and V in another key order (which
    moves the online softmax's reference maxima and so the rounding of P).  Peaked softmax (outlier
    channels, row gains): a few weights of a row dominate and keep their rounding, relative error
    2e-3 .. 6e-3 in FP8, 3e-4 .. 1e-3 in bf16.  Diffuse softmax: the outputs are small averages and
    carry the rounding of P in full, 2.4e-2 .. 3.6e-2 in FP8, 2.7e-3 in bf16, 3.4e-4 in fp16.  The
    largest single difference is 0.28 of the rms in FP8, 1.5e-2 in bf16 and 2e-3 in fp16."""
    kind = case["kind"]
    if kind in ("quant_qkv", "quant_one"):
        return "exact"
    if kind == "perturb":
        # noise in fp32, rounded to bf16: under 0.5 % of the elements land one bf16 step away
        return {"rel": 6e-4}
    peaked = case["dist"] in ("outlier", "rowgain")
    if kind in ("fp8", "predict", "host"):
        return {"rel": 0.03 if peaked else 0.14, "max": 0.9}
    if case["dtype"] == "fp16":
        return {"rel": 1.5e-3, "max": 1.5e-2}
    return {"rel": 4e-3 if peaked else 1.1e-2, "max": 0.08}


def _codes64(x, scale=None):
    """The paper's Eq. 2 per head: (e4m3 values of x / scale, times that scale, in 64 bits; the scale)."""
    if scale is None:
        amax = x.abs().amax(dim=(2, 3)).float()
        scale = torch.where(amax == 0, torch.ones_like(amax), amax / torch.full_like(amax, 448.0))  # the IEEE division
    s = scale[:, :, None, None]
    codes = (x.float() / s).clamp(-448.0, 448.0).to(torch.float8_e4m3fn)
    return codes.double() * s.double(), scale


def _attention64(q, k, v):
    out = torch.empty_like(q)
    rows = max(1, (1 << 27) // k.shape[2])      # a block of scores of about 1 GB
    for b in range(q.shape[0]):
        for h in range(q.shape[1]):
            for r in range(0, q.shape[2], rows):
                p = torch.softmax(q[b, h, r:r + rows] @ k[b, h].T * q.shape[3] ** -0.5, dim=1)
                out[b, h, r:r + rows] = p @ v[b, h]
    return out


def _shift_down(x, n):
    """An int64 tensor shifted down by n as an unsigned word."""
    return (x >> n) & ((1 << (64 - n)) - 1)


def _mix64(x):
    """The counter hash that ``perturb`` documents, on int64 tensors."""
    def signed(c):
        return c - (1 << 64) if c >= 1 << 63 else c
    x = x + signed(0x9E3779B97F4A7C15)
    x = (x ^ _shift_down(x, 30)) * signed(0xBF58476D1CE4E5B9)
    x = (x ^ _shift_down(x, 27)) * signed(0x94D049BB133111EB)
    return x ^ _shift_down(x, 31)


def _perturbed64(x, epsilon, seed, stream):
    B, H, rows, d = x.shape
    x = x.reshape(B * H, rows * d // 2, 2).double()
    rho = x.square().mean(dim=(1, 2)).sqrt()
    dev = dict(dtype=torch.int64, device=x.device)
    odd = 0x9E3779B97F4A7C15 - (1 << 64)
    words = torch.arange(rows * d // 2, **dev) * odd
    out = torch.empty_like(x)
    for head in range(B * H):
        key = _mix64(_mix64(torch.tensor(seed, **dev)) ^ (stream * (0xD6E8FEB86659FD93 - (1 << 64))))
        bits = _mix64(words ^ _mix64(key ^ head))
        u1, u2 = ((u.double() + 0.5) * 2.0 ** -32 for u in (_shift_down(bits, 32), bits & 0xffffffff))
        r, angle = (-2.0 * u1.log()).sqrt(), 2.0 * math.pi * u2
        out[head] = x[head] + epsilon * rho[head] * torch.stack((r * angle.cos(), r * angle.sin()), dim=1)
    return out.reshape(B, H, rows, d), rho.reshape(B, H)


def exact(case, seed):
    """Where codes enter the attention, they are the definition's: what remains is what the kernels
    lose in the scores, the weights, the sums and the results."""
    kind = case["kind"]
    if kind == "perturb":
        return _perturbed64(_inputs(case, seed, ("k",))["k"], 0.0265, seed, 1)
    if kind == "quant_one":
        return [None, _inputs(case, seed, ("k",))["k"].abs().amax(dim=(2, 3)).double() / 448.0]
    if kind != "quant_qkv":
        rows = case["n_test"] + (0 if kind == "predict" else case["n_train"])
        if case["B"] * case["H"] * case["n_train"] * rows > 5e11:
            return None     # about 20 seconds of 64-bit matrix products
    x = _inputs(case, seed, ("q_train", "k", "v", "q_test"))
    if kind == "quant_qkv":
        return {"s" + n[0]: x[n].abs().amax(dim=(2, 3)).double() / 448.0 for n in ("q_train", "k", "v")}
    if kind in ("gated", "attn16"):
        q, k, v, t = (x[n].double() for n in ("q_train", "k", "v", "q_test"))
    else:
        q, scale_q = _codes64(x["q_train"])
        k, v, t = _codes64(x["k"])[0], _codes64(x["v"])[0], _codes64(x["q_test"], scale_q)[0]
    out_test = _attention64(t, k, v)
    return out_test if kind == "predict" else (_attention64(q, k, v), out_test)
