"""The noise at the ends of what its formula meets: uniforms next to 1, whose logarithm is next to 0, and strengths
whose product with the RMS is next to the largest fp32 number."""
import numpy as np
import pytest
import torch

import oracle
from helpers import bf16_bits_to_f64
from paper_2609_13031_b200 import api

pytestmark = pytest.mark.gpu

M = (1 << 64) - 1
GOLDEN, STREAM = 0x9E3779B97F4A7C15, 0xD6E8FEB86659FD93


def mix(z):
    z = (z + GOLDEN) & M
    z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9 & M
    z = (z ^ (z >> 27)) * 0x94D049BB133111EB & M
    return z ^ (z >> 31)


def unmix(z):
    z = z ^ (z >> 31) ^ (z >> 62)
    z = z * pow(0x94D049BB133111EB, -1, 1 << 64) & M
    z = z ^ (z >> 27) ^ (z >> 54)
    z = z * pow(0xBF58476D1CE4E5B9, -1, 1 << 64) & M
    z = z ^ (z >> 30) ^ (z >> 60)
    return (z - GOLDEN) & M


def seed_of(bits, pair, stream_id):
    """The seed that makes `bits` the 64 random bits of that pair of elements of head 0."""
    key = unmix(bits) ^ (pair * GOLDEN & M)
    return unmix(unmix(unmix(key)) ^ (stream_id * STREAM & M))


def test_uniforms_next_to_one():
    """Every u1 that the conversion to fp32 can give in [1 - 2^-12, 1], with an angle whose sine and cosine both count.
    The kernel's log2 may be off by 2^-22 there (the documented bound of lg2.approx), so z^2 by 2 ln 2 times that."""
    assert mix(unmix(0x123456789ABCDEF0)) == 0x123456789ABCDEF0
    pair, stream_id, turn = 13, 3, 0x20000000                   # turn / 2^32 = an eighth
    x = torch.ones((1, 1, 1, 64), dtype=torch.bfloat16, device="cuda")
    x[..., 2 * pair:2 * pair + 2] = 0
    ws = api.new_workspace(1, 1)
    u = [min(k << 8, (1 << 32) - 1) for k in range((1 << 24) - 4096, (1 << 24) + 1)]
    out = torch.empty((len(u), 1, 1, 1, 64), dtype=torch.bfloat16, device="cuda")
    for i, hi in enumerate(u):
        api.perturb(x, 1.0, seed_of(hi << 32 | turn, pair, stream_id), stream_id, ws, out=out[i])
    got = out[..., 2 * pair:2 * pair + 2].reshape(-1, 2).double().cpu().numpy()
    assert torch.isfinite(out.float()).all()
    z = np.sqrt(-2 * np.log((np.array(u) + 0.5) / 2.0 ** 32) / 2)       # (half of z^2 each)
    rho = np.sqrt(62 / 64)
    off = np.log(2) * 2.0 ** -22
    # (got + step)^2 and so on: a bf16 rounding of the result around the bound on its square
    for col in (0, 1):
        lo = rho * np.sqrt(np.maximum(z ** 2 - off, 0)) * (1 - 2.0 ** -8)
        hi = rho * np.sqrt(z ** 2 + off) * (1 + 2.0 ** -8)
        assert np.all(got[:, col] >= lo) and np.all(got[:, col] <= hi), (got[:, col], z)
    assert api.last_device_status(ws) == (0, 0)


def test_strengths_next_to_the_largest_number():
    """epsilon * rho = 1e38: z up to 3 fits bf16, and the same elements are finite as in the oracle."""
    x = torch.full((1, 1, 256, 64), 1e10, dtype=torch.bfloat16, device="cuda")
    bits = x.view(torch.int16).cpu().numpy().view(np.uint16)
    ws = api.new_workspace(1, 1)
    out, rho = api.perturb(x, 1e28, 11, 2, ws)
    ref, _ = oracle.perturb(bits, 1e28, 11, 2)
    want, got = bf16_bits_to_f64(ref), out.double().cpu().numpy()
    fits = np.abs(want) < 3e38
    assert fits.mean() > 0.99 and np.abs(want[fits]).max() > 2.5e38
    assert np.isfinite(got[fits]).all()
    assert np.all(np.abs(got - want)[fits] <= 2.0 ** -7 * np.abs(want)[fits] + 1e-5 * 1e38)
