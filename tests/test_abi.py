"""The C-ABI library builds, loads, and exports every function include/mlora.h declares (no GPU needed)."""
import ctypes
import os
import re

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(scope="module")
def libpath():
    from paper_2604_18655_b200 import build
    return build.build()


def declared_functions():
    text = open(os.path.join(ROOT, "include", "mlora.h")).read()
    text = re.sub(r"/\*.*?\*/", "", text, flags=re.S)
    return sorted(set(re.findall(r"\b(mlora_[a-z_0-9]+)\s*\(", text)))


def test_header_declares_the_main_calls():
    names = declared_functions()
    for f in ("mlora_create", "mlora_set_adapter", "mlora_prefill_shared", "mlora_decode_step", "mlora_verify_tree"):
        assert f in names


def test_library_exports_every_declared_symbol(libpath):
    lib = ctypes.CDLL(libpath)
    for name in declared_functions():
        assert hasattr(lib, name), f"{name} declared in mlora.h but not exported"


def test_binding_covers_every_declared_symbol(libpath):
    from paper_2604_18655_b200 import binding
    assert sorted(binding.EXPORTS) == declared_functions()
    binding.lib()


def test_host_side_argument_errors_need_no_gpu(libpath):
    from paper_2604_18655_b200 import binding as mb
    L = mb.lib()
    assert L.mlora_create(None, None) == -1
    assert b"null" in L.mlora_last_error(None)
    assert L.mlora_decode_step(None, 1, None, None, None, None) == -1
    assert L.mlora_destroy(None) == 0
    assert L.mlora_linear_workspace_bytes(None, 8, 16) == 0
    assert L.mlora_attention_workspace_bytes(8, 1, 32, 8, 128, 512, 65) > 0


def test_unsupported_rope_style_is_refused_on_the_host(libpath):
    """rope_style other than 0 (half-split pairs) is rejected before anything touches a device."""
    from paper_2604_18655_b200 import binding as mb
    L = mb.lib()
    d = mb.ModelDesc()
    d.n_layers, d.d_model, d.n_q_heads, d.n_kv_heads, d.head_dim, d.d_ffn = 1, 64, 1, 1, 64, 64
    d.group_size, d.max_tree, d.max_streams, d.max_prefix, d.max_suffix = 64, 1, 1, 1, 1
    arr = (ctypes.c_void_p * 8)(*([1] * 8))
    d.qweight, d.scales, d.rms_attn, d.rms_ffn = arr, arr, arr, arr
    d.rope_style = 1
    out = ctypes.c_void_p()
    assert L.mlora_create(ctypes.byref(d), ctypes.byref(out)) == -6
    assert b"rope_style" in L.mlora_last_error(None)


def test_projection_plan_waits_for_no_second_wave_of_clusters(libpath):
    """Host side of the tensor-core projection: four unpacking groups (one CTA an SM) only where all clusters run at once (15 of eight CTAs,
    33 of four on 148 SMs), never in a call of its own or with adapters; every tile has a use."""
    from paper_2604_18655_b200 import binding as mb
    resident, seen = {1: 148, 2: 148, 4: 132, 8: 120}, set()
    for K in (64, 512, 1408, 2048, 4096, 6144, 8192, 14336):
        for N in (16, 512, 1024, 1152, 2048, 2176, 2304, 3072, 4096, 11264, 14336):
            for M in (9, 33, 40, 64, 65, 100, 128, 129, 200, 256, 300, 700, 1999):
                for call in (0, 1, 2):
                    rows, split, groups = mb.mlora_debug_gemm_plan(M, K, N, call)
                    seen.add(rows)
                    ctas = -(-N // 128) * -(-M // rows) * split
                    if rows <= 128 and groups == 4:
                        assert call == 0 and ctas <= resident[split], (M, K, N, rows, split)
    assert seen == {32, 64, 96, 128, 192, 256}
    assert mb.mlora_debug_gemm_plan(64, 8192, 2048, 0)[2] == 2      # 16 clusters of eight
    with pytest.raises(mb.MloraError):
        mb.mlora_debug_gemm_plan(64, 100, 2048, 0)
