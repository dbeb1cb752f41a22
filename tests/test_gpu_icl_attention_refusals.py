"""What icl_attention refuses on the host, each with everything else in order and before anything is launched: the
kernels read as many values from every address as k's sizes say."""
import pytest
import torch

from paper_2609_13031_b200 import api

pytestmark = pytest.mark.gpu

B, H, N, M, D = 2, 3, 40, 24, 64
TOGETHER, TYPE, SPACE = "of k's batch", "of one type", "workspace"


def rows(n, B=B, H=H, d=D, dtype=torch.bfloat16, device="cuda"):
    return torch.ones((B, H, n, d), dtype=dtype, device=device)


@pytest.mark.parametrize("which,make,message", [
    ("q_train", lambda: None, "expected tensors"), ("v", lambda: None, "expected tensors"), ("k", lambda: None, "contiguous CUDA"),
    ("k", lambda: rows(N, device="cpu"), "contiguous CUDA"), ("k", lambda: rows(N).transpose(1, 2), "contiguous CUDA"),
    ("k", lambda: rows(N).view(B * H, N, D), "contiguous CUDA"),
    ("q_train", lambda: rows(N, dtype=torch.float16), TYPE), ("v", lambda: rows(N).float(), TYPE),
    ("q_test", lambda: rows(M, dtype=torch.float16), TYPE),
    ("q_train", lambda: rows(N - 1), TOGETHER), ("v", lambda: rows(N + 1), TOGETHER), ("v", lambda: rows(N, H=H - 1), TOGETHER),
    ("v", lambda: rows(N, B=1), TOGETHER), ("v", lambda: rows(N, d=D // 2), TOGETHER),
    ("q_train", lambda: rows(D, d=N), TOGETHER), ("q_train", lambda: torch.ones(B * H * N * D, dtype=torch.bfloat16, device="cuda"), TOGETHER),
    ("v", lambda: rows(N, device="cpu"), TOGETHER), ("v", lambda: rows(N, B=N, H=H, d=D)[:B, :, :1].expand(B, H, N, D), TOGETHER),
    ("q_train", lambda: torch.ones((B, N, H, D), dtype=torch.bfloat16, device="cuda").transpose(1, 2), TOGETHER),
    ("q_test", lambda: rows(M, H=1), TOGETHER), ("q_test", lambda: rows(M, d=2 * D), TOGETHER), ("q_test", lambda: rows(M, device="cpu"), TOGETHER),
    ("q_test", lambda: torch.ones((B, H, D, M), dtype=torch.bfloat16, device="cuda").transpose(2, 3), TOGETHER),
    ("workspace", lambda: api.new_workspace(B, H, device="cpu"), SPACE),
    ("workspace", lambda: torch.zeros(1, dtype=torch.uint8, device="cuda").expand(1 << 20), SPACE),
])
def test_refused_before_any_launch(which, make, message):
    args = dict(q_train=rows(N), q_test=rows(M), k=rows(N), v=rows(N), workspace=api.new_workspace(B, H))
    args[which] = make()
    before = api.launch_count()
    with pytest.raises(AssertionError, match=message):
        api.icl_attention(**args)
    assert api.launch_count() == before


def test_heads_folded_into_one_dimension_stay_accepted():
    torch.manual_seed(1)
    q, t, k, v = (torch.randn((B, H, r, D), device="cuda").to(torch.bfloat16) for r in (N, M, N, N))
    ws = api.new_workspace(B, H)
    want = api.icl_attention(q, t, k, v, ws)
    got = api.icl_attention(q.view(B * H, N, D), t, k, v.view(B * H, N, D), ws.view(16, -1))
    assert torch.equal(got[0], want[0]) and torch.equal(got[1], want[1])
    assert api.last_device_status(ws) == (0, 0)
