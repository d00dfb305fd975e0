"""Host-only checks of the C ABI: the library loads without a GPU, exports every
function the header declares, sizes workspaces, and rejects bad arguments
before touching the device."""
import ctypes
import os
import re

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(scope="module")
def api():
    from paper_2412_03409_b200 import build
    build.build_library()
    from paper_2412_03409_b200 import api as _api
    return _api


def _declared_functions():
    text = open(os.path.join(ROOT, "include", "prefixkv.h")).read()
    text = re.sub(r"/\*.*?\*/", "", text, flags=re.S)
    return sorted(set(re.findall(r"\b(prefixkv_\w+)\s*\(", text)))


def test_header_functions_are_exported(api):
    names = _declared_functions()
    assert len(names) >= 8
    for n in names:
        assert hasattr(api.lib(), n), n
    assert set(api.EXPORTS) <= set(names)
    # the Python binding mirrors every compute entry point by name
    for n in names:
        if n != "prefixkv_last_cuda_error":
            assert hasattr(api, n), n


def test_workspace_sizes(api):
    import torch
    sh = api.make_shape(1, 32, 32, 128, 640, torch.bfloat16)
    per = 32 * 32 * 640 * 4
    assert api.prefixkv_workspace_bytes(sh, api.WS_SCORE) >= 2 * per
    assert api.prefixkv_workspace_bytes(sh, api.WS_COMPACT) >= 32 * 640 * 4
    assert api.prefixkv_workspace_bytes(sh, api.WS_DECODE) > 0
    assert api.prefixkv_workspace_bytes(sh, 99) == 0
    for bad in (api.make_shape(1, 2, 4, 48, 32, torch.float32),       # head_dim
                api.make_shape(1, 2, 4, 64, 16385, torch.float32),    # prompt too long
                api.make_shape(0, 2, 4, 64, 32, torch.float32)):      # empty batch
        assert api.prefixkv_workspace_bytes(bad, api.WS_SCORE) == 0


def test_null_and_range_arguments_rejected_on_host(api):
    import torch
    lib = api.lib()
    sh = api.make_shape(1, 2, 4, 64, 32, torch.float32)
    z = api.Strides(0, 0, 0, 0)
    assert lib.prefixkv_score(sh, None, z, None, z, None, None, None, None, 0, None) == api.PKV_ERR_INVALID_ARG
    assert lib.prefixkv_search(sh, None, None, 1e-6, 64, 0, 0, None, None, None, None, None, None,
                               None, 0, None) == api.PKV_ERR_INVALID_ARG
    if torch.cuda.is_available():
        return      # the cases below pass made-up non-null addresses: only where no launch can reach a GPU
    assert lib.prefixkv_search(sh, 16, 16, -1.0, 64, 0, 0, 16, 16, 16, 16, 16, 16, None, 0, None) == \
        api.PKV_ERR_INVALID_ARG                                    # negative tolerance
    assert lib.prefixkv_apply_lengths(sh, None, None, 0, None, None, None, None, None, 0, None) == \
        api.PKV_ERR_INVALID_ARG
    assert lib.prefixkv_compact(sh, None, z, None, z, None, None, None, None, None, None, 0, None) == \
        api.PKV_ERR_INVALID_ARG
    cache = api.CacheStruct(16, 16, 16, 16, 16, 10, 1, 0, None, None, None)
    assert lib.prefixkv_decode_attn(sh, ctypes.byref(cache), 16, 16, 16, 16, 1, 1, 16, 16, None, 0,
                                    None) == api.PKV_ERR_INVALID_ARG   # empty layer range
    assert lib.prefixkv_decode_attn(sh, ctypes.byref(cache), 16, 16, 16, 16, 0, 2, 16, 16, None, 0,
                                    None) == api.PKV_ERR_WORKSPACE     # no workspace
    odd = api.Strides(7, 7, 7, 7)                                      # rows not on 16 bytes
    assert lib.prefixkv_score(sh, 16, odd, 16, odd, 16, None, 16, 256, 1 << 30, None) == \
        api.PKV_ERR_INVALID_ARG
    assert lib.prefixkv_gini(sh, None, None, None) == api.PKV_ERR_INVALID_ARG


def test_the_decode_binding_is_this_interpreters(api, monkeypatch, tmp_path):
    """It carries the interpreter's suffix, is built again when what it is built from or with changes, and where there is no
    Python.h to build it with the call goes through ctypes."""
    import sysconfig

    import torch

    from paper_2412_03409_b200 import build
    assert build.CALL_PATH.endswith(sysconfig.get_config_var("EXT_SUFFIX")) and not build.call_is_stale()
    copy = tmp_path / os.path.basename(build.CALL_PATH)
    copy.write_bytes(open(build.CALL_PATH, "rb").read())
    monkeypatch.setattr(build, "CALL_PATH", str(copy))
    for src in (build.CALL_SRC, build.__file__):
        t = os.path.getmtime(src)
        os.utime(copy, (t + 1e6, t + 1e6))
        assert not build.call_is_stale()
        os.utime(copy, (t - 1, t - 1))
        assert build.call_is_stale()
    os.unlink(copy)
    with pytest.raises(ImportError):
        api._load_call()
    monkeypatch.setattr(build, "python_headers", lambda: False)
    build.build_call()
    by_ctypes = api._load_call()
    assert not copy.exists()
    sh = api.make_shape(1, 2, 4, 64, 32, torch.float32)
    cache = api.CacheStruct(None, None, None, None, None, 10, 1, 0, None, None, None)
    monkeypatch.setattr(api, "_stream", lambda: None)
    for call in (api._decode_attn, by_ctypes):
        if call is by_ctypes or torch.cuda.is_available():
            assert call(sh, cache, None, None, None, None, 0, 2, None, None, None) == api.PKV_ERR_INVALID_ARG


@pytest.mark.parametrize("heads,D,N,kept", [(1, 64, 128, False), (9999, 64, 129, True), (1820, 64, 1024, True), (1821, 64, 1024, False), (16, 64, 1025, True), (17, 64, 1025, False),
                                            (9, 64, 2048, True), (10, 64, 2048, False), (8, 64, 2049, False), (800, 128, 1024, True),
                                            (1, 128, 1025, False)])
def test_which_fp32_prompts_keep_their_logits(api, heads, D, N, kept):
    """By the workspace they ask for beyond the least: logits that leave the L2 cost more than a second pass."""
    import torch
    sh = api.make_shape(1, 1, heads, D, N, torch.float32)
    assert (api.prefixkv_workspace_bytes(sh, api.WS_SCORE) > api.prefixkv_workspace_bytes(sh, api.WS_SCORE_LEAST)) == kept


@pytest.mark.parametrize("B,L,H,D,N", [(1, 8, 16, 128, 777), (1, 32, 32, 128, 1024), (16, 24, 16, 64, 1024), (1, 1, 9, 64, 2048), (64, 40, 40, 128, 1000),
                                       (1, 2, 5000, 64, 1024), (16, 24, 16, 64, 2048)])
def test_kept_logits_take_bounded_memory(api, B, L, H, D, N):
    """Logits of 148 blocks and 128 MiB of part sums, however many heads there are; with the caller's log-sum-exp nothing but
    sums and normalisers of every query."""
    import torch
    sh, tiles = api.make_shape(B, L, H, D, N, torch.float32), (N + 127) // 128
    two = 2 * B * L * H * N * 4
    assert api.prefixkv_workspace_bytes(sh, api.WS_SCORE) <= max(two * 1.2, 148 * tiles * 65536 + (128 << 20)) + 1024
    assert two <= api.prefixkv_workspace_bytes(sh, api.WS_SCORE_LEAST) <= two * 1.2 + 1024
