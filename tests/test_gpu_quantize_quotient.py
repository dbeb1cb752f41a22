"""The quantizer's division: every mantissa of a head's maximum against every input mantissa, both
signs and both zeros, bit for bit.  The kernels divide by multiplication with one correction, which
has to give the IEEE quotient for all of them."""
import numpy as np
import pytest
import torch

import oracle
from paper_2609_13031_b200 import api

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype,mant_bits", [("bf16", 7), ("fp16", 10)])
@pytest.mark.parametrize("flags", [0, api.QKV_TWO_LAUNCHES])
def test_every_mantissa_pair(dtype, mant_bits, flags):
    n = 1 << mant_bits
    one = 0x3F80 if dtype == "bf16" else 0x3C00                    # bits of 1.0
    amax = (one + np.arange(n) + (n << 2)).astype(np.uint16)       # (1.m) * 2^4, one per head
    # all mantissas at six exponents below the maximum's, then the zeros and the maximum itself
    vals = np.concatenate([one + (e << mant_bits) + np.arange(n) for e in (-7, -4, -1, 1, 2, 3)] + [np.zeros(62, int)])
    rows = -(-(2 * vals.size + 4) // 64)
    x = np.zeros((1, n, rows * 64), dtype=np.uint16)
    x[:, :, :vals.size] = vals
    x[:, :, vals.size:2 * vals.size] = vals | 0x8000
    x[:, :, -1] = amax
    x = x.reshape(1, n, rows, 64)
    t = x.copy()                                                   # test rows: four times the maximum too
    t[:, :, 0, 0] = amax + (2 << mant_bits)
    t[:, :, 0, 1] = (amax + (2 << mant_bits)) | 0x8000
    tdt = torch.bfloat16 if dtype == "bf16" else torch.float16
    dev = lambda a: torch.from_numpy(a.view(np.int16)).cuda().view(tdt)
    ws = api.new_workspace(1, n)
    o = api.quantize_qkv(dev(x), dev(x), dev(x), dev(t), ws, flags=flags)
    one_codes, one_scale = api.quantize(dev(x), ws)
    want, s = oracle.quantize(x, dtype16=dtype)
    want_t, _ = oracle.quantize(t, scale_in=s, dtype16=dtype)
    assert api.last_device_status(ws) == (0, 0)
    for got in (o["q8"], o["k8"], o["v8"], one_codes):
        assert np.array_equal(got.cpu().numpy(), want)
    assert np.array_equal(o["t8"].cpu().numpy(), want_t)
    for got in (o["sq"], o["sk"], o["sv"], one_scale):
        assert np.array_equal(got.cpu().numpy(), s)
