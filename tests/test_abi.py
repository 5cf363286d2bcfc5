"""The C-ABI library loads without a GPU and exports every symbol the header declares."""
import ctypes
import os
import re
import subprocess
import sys

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
HEADER = os.path.join(ROOT, "include", "attn_fp8.h")


@pytest.fixture(scope="module")
def lib_path():
    from paper_2609_37852_b200 import build
    return build.build()


def _declared_functions():
    text = open(HEADER).read()
    text = re.sub(r"/\*.*?\*/", "", text, flags=re.S)
    return sorted(set(re.findall(r"\b(attn_fp8_\w+)\s*\(", text)))


def test_header_declares_the_four_entry_points():
    names = _declared_functions()
    for n in ("attn_fp8_quantize", "attn_fp8_fwd", "attn_fp8_bwd_delta", "attn_fp8_bwd"):
        assert n in names


def test_library_exports_every_declared_symbol(lib_path):
    lib = ctypes.CDLL(lib_path)
    for name in _declared_functions():
        assert hasattr(lib, name), name


def test_binding_lists_the_same_symbols(lib_path):
    from paper_2609_37852_b200 import binding
    assert sorted(binding.EXPORTED_SYMBOLS) == _declared_functions()


def test_scale_offset_rule(lib_path):
    from paper_2609_37852_b200 import binding
    for n_blocks in (2, 4, 6, 8, 64):
        seen = set()
        for row in range(0, 256):
            for blk in range(n_blocks):
                want = ((row // 128) * ((n_blocks + 3) // 4) + blk // 4) * 512 + (row % 32) * 16 \
                    + ((row % 128) // 32) * 4 + blk % 4
                got = binding.attn_fp8_scale_offset(row, blk, n_blocks)
                assert got == want
                seen.add(got)
        assert len(seen) == 256 * n_blocks                      # a permutation: no two scales collide
    assert binding.attn_fp8_scale_bytes(2, 3, 256, 128) == 2 * 3 * 2 * 1 * 512
    assert binding.attn_fp8_scale_bytes(1, 1, 64, 256) == 1 * 2 * 512
    assert binding.attn_fp8_scale_bytes(1, 1, 192, 128) == 2 * 512


def test_unpack_scales_inverts_the_tiling(lib_path):
    import torch
    from paper_2609_37852_b200 import binding
    B, H, rows, cols = 1, 2, 256, 192
    nbytes = binding.attn_fp8_scale_bytes(B, H, rows, cols)
    flat = torch.zeros(nbytes, dtype=torch.uint8)
    plain = torch.randint(1, 255, (B, H, rows, cols // 32), dtype=torch.uint8)
    slab = nbytes // (B * H)
    for s in range(B * H):
        for r in range(rows):
            for k in range(cols // 32):
                flat[s * slab + binding.attn_fp8_scale_offset(r, k, cols // 32)] = plain[s // H, s % H, r, k]
    assert torch.equal(binding.unpack_scales(flat, B, H, rows, cols), plain)


def test_validation_errors_without_touching_a_gpu(lib_path):
    from paper_2609_37852_b200 import binding
    st = binding._lib.attn_fp8_quantize(None, 0, 1, 1, 128, 128, binding._QTensor(), None)
    assert st == 1 and "src" in binding.attn_fp8_last_error()
    st = binding._lib.attn_fp8_quantize(ctypes.c_void_p(16), 0, 1, 1, 100, 128, binding._QTensor(), None)
    assert st == 2
    st = binding._lib.attn_fp8_quantize(ctypes.c_void_p(8), 0, 1, 1, 128, 128, binding._QTensor(), None)
    assert st == 3
    p = binding.AttnParams(1, 128, 3, 2, 128, 128, True, 0.1).c_struct()
    q = binding._QTensor()
    st = binding._lib.attn_fp8_fwd(ctypes.byref(p), q, q, q, None, None, None, 0, None)
    assert st == 1 and "heads_q" in binding.attn_fp8_last_error()
    p = binding.AttnParams(1, 128, 4, 2, 96, 96, True, 0.1).c_struct()
    st = binding._lib.attn_fp8_fwd(ctypes.byref(p), q, q, q, None, None, None, 0, None)
    assert st == 2
    # more rows than the kernels' 32-bit row coordinates reach: refused before any launch
    p = binding.AttnParams(64, 1 << 20, 64, 8, 128, 128, True, 0.1).c_struct()
    st = binding._lib.attn_fp8_fwd(ctypes.byref(p), q, q, q, None, None, None, 0, None)
    assert st == 2 and "2^31" in binding.attn_fp8_last_error()


def test_batched_quantiser_and_workspace_validation_without_a_gpu(lib_path):
    """Argument checks of attn_fp8_quantize_batch and attn_fp8_workspace_init run before any device call."""
    from paper_2609_37852_b200 import binding
    lib = binding._lib
    fake = ctypes.c_void_p(4096)                                   # aligned, never dereferenced on these paths
    out = binding._QTensor(fake, fake, fake, fake)
    ok = binding._QuantizeJob(fake, binding.ATTN_SRC_BF16, 1, 1, 128, 128, out)
    jobs = (binding._QuantizeJob * 2)(ok, ok)
    assert lib.attn_fp8_quantize_batch(None, 1, fake, 256, None) == 1
    assert lib.attn_fp8_quantize_batch(jobs, 0, fake, 256, None) == 1
    assert lib.attn_fp8_quantize_batch(jobs, binding.ATTN_QUANTIZE_MAX_JOBS + 1, fake, 256, None) == 1
    jobs[1] = binding._QuantizeJob(fake, binding.ATTN_SRC_FP32, 1, 1, 128, 128, out)
    assert lib.attn_fp8_quantize_batch(jobs, 2, fake, 256, None) == 1 and "src_dtype" in binding.attn_fp8_last_error()
    jobs[1] = binding._QuantizeJob(fake, binding.ATTN_SRC_BF16, 1, 1, 192, 128, out)      # N not a multiple of 128
    assert lib.attn_fp8_quantize_batch(jobs, 2, fake, 256, None) == 2
    jobs[1] = binding._QuantizeJob(fake, binding.ATTN_SRC_BF16, 1, 1, 128, 128, binding._QTensor(fake, None, None, None))
    assert lib.attn_fp8_quantize_batch(jobs, 2, fake, 256, None) == 1      # codes without their scales
    assert lib.attn_fp8_workspace_init(None, 256, None) == 4
    assert lib.attn_fp8_workspace_init(fake, 16, None) == 4
    assert lib.attn_fp8_workspace_init(ctypes.c_void_p(4100), 256, None) == 3
    # a NULL workspace means the built-in scratch array of the current device: without a device the call
    # stops at the device check (ATTN_ERR_CUDA), with one it reads that array's status word
    import torch
    if not torch.cuda.is_available():
        assert lib.attn_fp8_read_status(None, None) == 6


@pytest.mark.parametrize("field,value", [
    ("batch", 2.0), ("batch", "2"), ("batch", np.int64(2)), ("batch", np.float32(2)), ("batch", 2 ** 32 + 2), ("batch", 2 ** 70),
    ("seqlen", 100.5), ("seqlen", True), ("heads_kv", np.uint8(3)), ("precision", 7.0), ("keys_valid", None), ("q_start", -128),
    ("causal", 1.0), ("causal", "1"), ("causal", "x"), ("causal", np.bool_(True)), ("causal", 2), ("causal", None),
    ("softmax_scale", "0.5"), ("softmax_scale", np.float16(0.5)), ("softmax_scale", 1), ("softmax_scale", None), ("softmax_scale", 1e300),
])
def test_parameters_are_taken_as_the_c_struct_takes_them(lib_path, field, value):
    """The marshalled call and the ctypes struct refuse the same values, and read the others alike."""
    from paper_2609_37852_b200 import binding
    p = binding.AttnParams(1, 256, 4, 2, 128, 128, True, 0.1)
    setattr(p, field, value)
    none, stream = binding.QTensor(shape=()), type("Stream", (), {"cuda_stream": 0})

    def outcome(call):
        try:
            return call(), binding.attn_fp8_last_error()
        except (TypeError, ValueError, OverflowError) as e:
            return type(e), None
    want = outcome(lambda: binding._lib.attn_fp8_fwd(ctypes.byref(p.c_struct()), *[none.c_struct()] * 3, None, None, None, 0, None))
    assert outcome(lambda: binding._marshal.fwd(p, none, none, none, None, None, None, stream)) == want


def test_a_module_of_another_torch_is_built_again_and_not_loaded(lib_path, monkeypatch):
    """The marshalling module holds torch's C++ interface: one compiled for another build is stale, and refused by name."""
    from paper_2609_37852_b200 import build
    assert build.marshal_built_for() == build.marshal_key()
    ran = []
    monkeypatch.setattr(build.subprocess, "run", lambda cmd, **kw: ran.append(cmd) or subprocess.CompletedProcess(cmd, 0, "", ""))
    build.build_marshal()
    assert not ran
    monkeypatch.setattr("torch.__version__", "0.0")
    build.build_marshal()
    assert len(ran) == 1
    r = subprocess.Popen([sys.executable, "-c", "import torch; torch.__version__ = '0.0'; import paper_2609_37852_b200.binding"],
                         cwd=ROOT, stderr=subprocess.PIPE, text=True)
    err = r.communicate(timeout=300)[1]
    assert r.returncode and "ImportError" in err and "built for" in err and "torch 0.0" in err
