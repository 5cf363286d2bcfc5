"""A context other than the first of its device: a second one beside it, and the one that follows a reset.

What the library keeps between calls and what belongs to a context (the shared-memory limit of a kernel, the address of the
built-in scratch array) must not be taken from one context into another.  The driver's own calls, without torch, in a
process of their own.
"""
import ctypes as C
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


class _QTensor(C.Structure):
    _fields_ = [(n, C.c_void_p) for n in ("row_codes", "row_scales", "col_codes", "col_scales")]


class _Job(C.Structure):
    _fields_ = [("src", C.c_void_p)] + [(n, C.c_int32) for n in ("dtype", "B", "H", "N", "d")] + [("out", _QTensor)]


def _calls():
    driver = C.CDLL("libcuda.so.1")
    lib = C.CDLL(os.path.join(ROOT, "paper_2609_37852_b200", "libattnfp8.so"))
    lib.attn_fp8_last_error.restype = C.c_char_p
    lib.attn_fp8_quantize_batch.argtypes = [C.POINTER(_Job), C.c_int32, C.c_void_p, C.c_size_t, C.c_void_p]

    def check(status):
        assert status == 0, (status, lib.attn_fp8_last_error())

    def alloc(n):
        p = C.c_uint64(0)
        check(driver.cuMemAlloc_v2(C.byref(p), C.c_size_t(n)))
        check(driver.cuMemsetD8_v2(p, C.c_ubyte(0), C.c_size_t(n)))
        return p.value

    def use():
        heads, n, d = 2, 256, 128                          # a launch with more shared memory than a kernel has by default
        elements = heads * n * d
        job = _Job(alloc(2 * elements), 0, 1, heads, n, d, _QTensor(alloc(elements), alloc(heads * 1024), alloc(elements), alloc(heads * 1024)))
        check(driver.cuCtxSynchronize())
        check(lib.attn_fp8_quantize_batch(C.byref(job), 1, alloc(256), 256, None))
        check(driver.cuCtxSynchronize())
        # the built-in array: a status written there by a kernel of this context and read back, once
        check(lib.attn_fp8_selftest_timeout(None, C.c_size_t(0), None))
        assert lib.attn_fp8_read_status(None, None) == 7
        check(lib.attn_fp8_read_status(None, None))

    dev, primary, second = C.c_int(0), C.c_void_p(), C.c_void_p()
    check(driver.cuInit(0))
    check(driver.cuDevicePrimaryCtxRetain(C.byref(primary), dev))
    check(driver.cuCtxSetCurrent(primary))
    use()
    check(driver.cuCtxCreate_v2(C.byref(second), 0, dev))
    use()
    check(driver.cuCtxSetCurrent(primary))
    use()
    check(driver.cuCtxDestroy_v2(second))
    check(driver.cuDevicePrimaryCtxReset_v2(dev))
    check(driver.cuDevicePrimaryCtxRetain(C.byref(primary), dev))
    check(driver.cuCtxSetCurrent(primary))
    use()


def test_calls_in_a_second_context_and_after_a_reset():
    r = subprocess.run([sys.executable, os.path.abspath(__file__)], capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stderr[-2000:]


if __name__ == "__main__":
    _calls()
