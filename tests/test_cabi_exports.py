"""The C-ABI library builds, loads on a machine without a GPU, and exports every
function that include/fp8attn.h declares (no compute calls here)."""
import ctypes
import os
import re

from paper_2609_13031_b200 import api, build

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def declared_functions():
    names = []
    inc = os.path.join(ROOT, "include")
    for fn in sorted(os.listdir(inc)):
        if not fn.endswith(".h"):
            continue
        text = open(os.path.join(inc, fn)).read()
        text = re.sub(r"/\*.*?\*/", "", text, flags=re.S)
        names += re.findall(r"\b([a-z0-9_]+attn_[a-z0-9_]+)\s*\(", text)
    return sorted(set(names))


def test_library_builds_loads_and_exports_header_symbols():
    build.build_cuda()
    lib = ctypes.CDLL(api.LIB_PATH)
    names = declared_functions()
    assert set(api.EXPORTS) <= set(names)
    assert len(names) >= 7
    for n in names:
        assert hasattr(lib, n), n


def test_host_only_entry_points():
    api.load()
    assert api.status_string(0) == "ok"
    assert "timed out" in api.status_string(api.ERR_TIMEOUT)
    assert api.workspace_bytes(1, 8) >= 256 + 32
    assert api.workspace_bytes(4, 4) % 256 == 0
    assert api.workspace_bytes(0, 4) == 0


def test_host_step_plan_is_host_only_arithmetic():
    """Chunking of the host-to-host step: whole heads, at most 8 chunks, one chunk for small
    calls or on request; two buffer sets when pipelined, so the scratch shrinks with chunking."""
    api.load()
    c3 = (1, 8, 65536, 16384, 128)
    assert api.host_step_chunks(*c3) == 8 and api.host_step_chunks(*c3, api.HOST_ONE_CHUNK) == 1
    assert api.host_step_chunks(1, 2, 512, 128, 64) == 1                  # small: nothing to overlap
    assert api.host_step_chunks(4, 4, 262144, 65536, 64) == 8             # 16 heads, two per chunk
    assert api.host_step_chunks(1, 11, 8192, 1100, 128) == 6              # ragged last chunk
    assert api.host_step_chunks(1, 1, 1 << 20, 0, 64) == 1                # one head cannot be cut
    one = api.host_step_scratch_bytes(*c3, api.HOST_ONE_CHUNK)
    piped = api.host_step_scratch_bytes(*c3)
    per_head = (3 * 65536 + 16384) * 128 * (2 + 1) + (65536 + 16384) * 128 * 2   # inputs, codes, outputs
    assert one >= 8 * per_head and 2 * per_head <= piped < one / 2
    assert one % 256 == 0 and piped % 256 == 0
    assert api.host_step_scratch_bytes(1, 8, 0, 16, 64) == 0 and api.host_step_scratch_bytes(1, 8, 64, 16, 96) == 0


def test_quantizer_form_is_host_only_arithmetic():
    """On both sides of each line between a block per head (-1), one pass in stages and two passes."""
    api.load()
    both = api.QUERY_SCALE_FROM_ALL_ROWS
    for tensors, H, n, m, d, flags, stages in (
            (3, 8, 1024, 256, 64, 0, -1), (3, 8, 1025, 256, 64, 0, 1), (1, 8, 512, 0, 128, 0, -1), (1, 8, 513, 0, 128, 0, 1),
            (3, 8, 512, 512, 128, both, -1), (3, 8, 512, 513, 128, both, 0),
            (3, 8, 7500, 2048, 128, 0, 3), (3, 8, 8192, 2048, 128, 0, 0), (3, 2, 33203, 8300, 128, 0, 0), (3, 1, 33203, 8300, 128, 0, 3),
            (3, 4, 33000, 5000, 128, 0, 0), (3, 8, 44000, 1000, 128, 0, 24), (1, 8, 33203, 0, 128, 0, 0), (1, 8, 32768, 0, 128, 0, 4),
            (3, 8, 20011, 3001, 128, 0, 8), (3, 8, 20011, 3001, 128, both, 0), (3, 8, 65536, 16384, 128, both, 24),
            (3, 1, 65536, 0, 128, 0, 3), (3, 1, 65600, 0, 128, 0, 0),
            (3, 8, 8192, 2048, 128, api.QKV_TWO_LAUNCHES, 0), (3, 8, 8192, 2048, 128, api.SCALES_GIVEN, 0),
            (2, 8, 512, 0, 64, 0, 0), (3, 8, 512, 0, 96, 0, 0), (3, 0, 512, 0, 64, 0, 0), (3, 8, 0, 0, 64, 0, 0)):
        assert api.quantize_stages(tensors, 1, H, n, m, d, flags) == stages, (tensors, H, n, m, d, flags)


def test_tiles_per_cta_of_split_launches():
    """Both sides of the choice between two and three tiles for test rows against a table (d = 64)."""
    api.load()
    flags = api.SPLIT_TAIL | api.TEST_ROWS_ONLY
    for H, n, m, rows in ((8, 4096, 2048, 256), (8, 8192, 2048, 256), (8, 30011, 2048, 384), (4, 30011, 2048, 384),
                          (8, 131072, 700, 384), (8, 262144, 300, 384), (2, 131072, 300, 256), (16, 8192, 700, 256)):
        assert api.attention_rows_per_cta(1, H, n, m, 64, flags) == rows, (H, n, m)
    assert api.attention_rows_per_cta(1, 8, 30011, 2048, 64, api.TEST_ROWS_ONLY) == 256


def test_one_tile_gives_way_to_a_split_that_is_over_sooner():
    """Both sides of the choice between CTAs of one tile and the split of the keys."""
    api.load()
    test_rows = api.SPLIT_TAIL | api.TEST_ROWS_ONLY
    for H, n, m, d, flags, rows in (
            (49, 16000, 300, 64, test_rows, 384), (49, 4000, 300, 64, test_rows, 384), (40, 8000, 333, 64, test_rows, 384),
            (29, 8000, 600, 64, test_rows, 128), (49, 16000, 300, 128, test_rows, 128), (49, 1440, 300, 64, test_rows, 128),
            (8, 1930, 250, 64, api.SPLIT_TAIL, 128), (8, 1930, 250, 128, api.SPLIT_TAIL, 128), (1, 16200, 2600, 64, api.SPLIT_TAIL, 128),
            (16, 3000, 1000, 64, test_rows, 256), (8, 3000, 2300, 128, test_rows, 128), (16, 5000, 1000, 128, test_rows, 256),
            (4, 3500, 700, 64, api.SPLIT_TAIL, 256), (4, 4000, 200, 128, api.SPLIT_TAIL, 256),
            (40, 2000, 257, 64, test_rows, 128), (8, 2000, 1100, 128, test_rows, 256), (2, 16300, 129, 64, test_rows, 256),
            (8, 4096, 1000, 64, test_rows, 256), (8, 1920, 250, 64, api.SPLIT_TAIL, 128)):
        assert api.attention_rows_per_cta(1, H, n, m, d, flags) == rows, (H, n, m, d)
        assert api.attention_rows_per_cta(1, H, n, m, d, flags & ~api.SPLIT_TAIL) == 128, (H, n, m, d)


def test_dispatch_gate_matches_the_paper_constant():
    import os
    from helpers import read_golden_table
    gold = dict(read_golden_table(os.path.join(ROOT, "tests", "golden", "paper_constants.txt")))
    gate = int(float(gold["fp8_gate_train_rows"]))          # Method section: N > 8192
    assert api.GATE_TRAIN_ROWS == gate
    assert not api.gate_use_fp8(gate) and api.gate_use_fp8(gate + 1)
    assert not api.gate_use_fp8(1) and api.gate_use_fp8(1 << 20)


def test_argument_checks_run_on_the_host_before_anything_touches_a_gpu():
    """Every entry point validates its arguments first, so the error codes can be checked on
    a machine without a GPU.  Pointers here are fake, suitably aligned addresses: a call that
    fails validation must not dereference or launch anything."""
    import pytest
    import torch
    if torch.cuda.is_available():
        pytest.skip("fake pointers are only ever passed where no GPU could be reached")
    lib = api.load()
    P, WS = 0x10000, 0x20000                      # 16- and 256-byte aligned fake device addresses
    ws_bytes = api.workspace_bytes(1, 2)
    q = lambda *a: lib.fp8attn_quantize(*a)
    # shape and pointer checks of the quantizer
    assert q(P, 0, 2, 8, 64, None, P, P, WS, ws_bytes, None) == api.ERR_INVALID_ARG      # B = 0
    assert q(P, 1, 2, 8, 96, None, P, P, WS, ws_bytes, None) == api.ERR_UNSUPPORTED      # d = 96
    assert q(P, 1, 2, -1, 64, None, P, P, WS, ws_bytes, None) == api.ERR_INVALID_ARG     # rows < 0
    assert q(None, 1, 2, 8, 64, None, P, P, WS, ws_bytes, None) == api.ERR_INVALID_ARG   # no input
    assert q(P + 2, 1, 2, 8, 64, None, P, P, WS, ws_bytes, None) == api.ERR_INVALID_ARG  # misaligned
    assert q(P, 1, 2, 8, 64, None, P, None, WS, ws_bytes, None) == api.ERR_INVALID_ARG   # no scale at all
    assert q(P, 1, 2, 8, 64, None, P, P, None, ws_bytes, None) == api.ERR_WORKSPACE
    assert q(P, 1, 2, 8, 64, None, P, P, WS + 16, ws_bytes, None) == api.ERR_WORKSPACE   # misaligned
    assert q(P, 1, 2, 8, 64, None, P, P, WS, ws_bytes - 1, None) == api.ERR_WORKSPACE    # too small
    assert lib.fp8attn_quantize_ex(P, 1, 2, 8, 64, None, P, P, 0x40, WS, ws_bytes, None) == api.ERR_INVALID_ARG
    # the fused forward
    f = lambda *a: lib.fp8attn_icl_forward(*a)
    ok = [P, P, P, P, P, P, P, 1, 2, 8, 4, 64, 0.0, P, P, WS, ws_bytes, None]
    def bad(i, v):
        a = list(ok)
        a[i] = v
        return f(*a)
    assert bad(0, None) == api.ERR_INVALID_ARG         # train queries missing
    assert bad(1, None) == api.ERR_INVALID_ARG         # test queries missing although n_test > 0
    assert bad(4, None) == api.ERR_INVALID_ARG         # a scale missing
    assert bad(9, 0) == api.ERR_INVALID_ARG            # n_train = 0
    assert bad(10, -1) == api.ERR_INVALID_ARG          # n_test < 0
    assert bad(11, 256) == api.ERR_UNSUPPORTED         # head dimension
    assert bad(12, float("nan")) == api.ERR_INVALID_ARG
    assert bad(14, None) == api.ERR_INVALID_ARG        # test output missing
    assert bad(16, 0) == api.ERR_WORKSPACE
    # allocation-free quantizer: its own size limit
    assert lib.fp8attn_quantize_noalloc(P, 1, api.NOALLOC_MAX_HEADS + 1, 8, 64, None, P, P, None) == api.ERR_TOO_LARGE
    # arguments in order, but no GPU: the call reports it; nothing falls back to the CPU
    assert f(*ok) in (api.ERR_CUDA, api.ERR_UNSUPPORTED)
    assert q(P, 1, 2, 8, 64, None, P, P, WS, ws_bytes, None) in (api.ERR_CUDA, api.ERR_UNSUPPORTED)


def test_native_binding_refuses_what_the_call_does_not_take():
    """Without a GPU: the look at k, which comes first, and at what is no tensor at all.  What follows it needs tensors
    on a GPU: test_gpu_icl_attention_refusals.py."""
    import pytest
    import torch
    api.load()
    ok = torch.zeros((1, 1, 4, 64), dtype=torch.bfloat16)
    for args in ((ok, ok, ok, ok), (None, ok, ok, ok), (ok, ok, None, ok), (ok, ok, ok.view(1, 4, 64), ok)):
        with pytest.raises(AssertionError):
            api.icl_attention(*args, workspace=torch.zeros(4096, dtype=torch.uint8))
    with pytest.raises(TypeError):
        api.icl_attention(ok, 3, ok, ok, workspace=torch.zeros(4096, dtype=torch.uint8))


def test_only_icl_attention_needs_the_native_half(monkeypatch, tmp_path):
    """Another torch or interpreter, or a module that does not load: every other function works, and the one that
    needs it says why."""
    import sys
    import pytest
    import torch
    assert torch.__version__ in build.binding_path() and sys.implementation.cache_tag in build.binding_path()
    x = torch.zeros((1, 1, 4, 64), dtype=torch.bfloat16)
    for name, content, why in (("none.so", None, "not found"), ("broken.so", b"no library", "broken.so")):
        path = tmp_path / name
        if content is not None:
            path.write_bytes(content)
        monkeypatch.setattr(build, "binding_path", lambda: str(path))
        monkeypatch.setattr(api, "_native", None)
        monkeypatch.setattr(api, "_lib", None)
        assert api.status_string(0) == "ok" and api.workspace_bytes(1, 8) > 0
        with pytest.raises(RuntimeError, match=why):
            api.icl_attention(x, x, x, x, workspace=torch.zeros(4096, dtype=torch.uint8))
