"""Host side of escape_cycles4_noalloc without a GPU: its translation unit
linked against a stand-in for the CUDA runtime that records the calls and
fails the one it is told to, and the device memory that it reserves."""
import ctypes
import os
import re
import subprocess

import pytest

from paper_1610_09411_gb300 import build as pb

FAKE = r"""
#include <stddef.h>
#include <string.h>
static char trace[256];
static int len, fail_at = -1, calls_of_kind[128];
static char fail_kind;
static int last_error;
static int call(char c) {
  if (len < 255) trace[len++] = c;
  int bad = c == fail_kind && calls_of_kind[(int)c]++ == fail_at;
  if (bad) last_error = 2;
  return bad ? 2 : 0;
}
#define OUT __attribute__((visibility("default")))
OUT void fake_reset(char kind, int at) {
  memset(trace, 0, sizeof trace); len = 0; memset(calls_of_kind, 0, sizeof calls_of_kind);
  fail_kind = kind; fail_at = at; last_error = 0;
}
OUT const char* fake_trace(void) { return trace; }
void* __cudaRegisterFatBinary(void* p) { return p; }
void __cudaRegisterFatBinaryEnd(void* p) { (void)p; }
void __cudaUnregisterFatBinary(void* p) { (void)p; }
void __cudaRegisterFunction(void) {}
void __cudaRegisterVar(void) {}
int __cudaGetKernel(void** k, const void* f) { *k = (void*)f; return 0; }
int __cudaPushCallConfiguration(void) { return 0; }
int __cudaPopCallConfiguration(void) { return 0; }
int __cudaLaunchKernel(void) { return call('K'); }
int cudaLaunchKernelExC(void) { return call('X'); }
int cudaDeviceGetAttribute(int* v) { *v = 4; return 0; }
int cudaFuncSetAttribute(void) { return call('A'); }
int cudaGetDevice(int* d) { *d = 0; return 0; }
int cudaGetLastError(void) { int e = last_error; last_error = 0; return e; }
int cudaGetSymbolAddress(void** p) { static char space[4096]; *p = space; return 0; }
int cudaMemcpyAsync(void* d, const void* s, size_t n) { (void)s; memset(d, 0, n); return call('C'); }
int cudaMemsetAsync(void) { return call('M'); }
int cudaStreamSynchronize(void) { return call('S'); }
"""
NOTE = "enum cudaError { cudaSuccess_ }; namespace esc { void note_cuda_error(cudaError) {} }\n"
SRC = os.path.join(pb.CSRC, "noalloc.cu")


def _nvcc(*args):
    try:
        cc = pb.nvcc()
    except RuntimeError:
        pytest.skip("no nvcc")
    r = subprocess.run([cc] + pb.ARCH + pb.NVCC_FLAGS + list(args), capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    return r.stdout + r.stderr


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    d = tmp_path_factory.mktemp("noalloc")
    obj, fake, note, so = (str(d / x) for x in ("noalloc.o", "fake.c", "note.cpp", "libnoalloc_host.so"))
    _nvcc("-c", SRC, "-o", obj)
    with open(fake, "w") as f:
        f.write(FAKE)
    with open(note, "w") as f:
        f.write(NOTE)
    # hidden: a CUDA runtime that the process has loaded must not take the calls
    subprocess.check_call(["gcc", "-O1", "-fPIC", "-fvisibility=hidden", "-w", "-c", fake, "-o", fake + ".o"])
    subprocess.check_call(["g++", "-O1", "-fPIC", "-c", note, "-o", note + ".o"])
    subprocess.check_call(["g++", "-shared", "-Wl,-Bsymbolic", "-o", so, obj, fake + ".o", note + ".o"])
    lib = ctypes.CDLL(so)
    lib.fake_trace.restype = ctypes.c_char_p
    lib.fake_reset.argtypes = [ctypes.c_char, ctypes.c_int]
    P = ctypes.c_void_p
    lib.escape_cycles4_noalloc.argtypes = [ctypes.c_int64, P, P, P, P, P]
    return lib


def _call(lib, kind, at):
    lib.fake_reset(kind.encode(), at)
    buf = (ctypes.c_uint64 * 64)()
    p = ctypes.addressof(buf)
    return lib.escape_cycles4_noalloc(10, p, p, p, p, None), lib.fake_trace().decode()


def test_calls_in_order(lib):
    status, trace = _call(lib, "-", 0)
    assert status == 0 and re.fullmatch(r"MA*KKXCS", trace)


@pytest.mark.parametrize("kind,at", [("K", 0), ("K", 1), ("X", 0), ("C", 0)])
def test_an_error_behind_queued_kernels_is_returned_after_they_end(lib, kind, at):
    status, trace = _call(lib, kind, at)
    assert status == 3                          # ECUDA
    assert "S" in trace[max(trace.rfind(c) for c in "KX"):]


def test_reserved_device_memory(tmp_path):
    """The header, an order key and a list entry per vertex; nothing unused."""
    out = _nvcc("-Xptxas", "-v", "-c", SRC, "-o", str(tmp_path / "noalloc.o"))
    gmem = [int(x) for x in re.findall(r"(\d+) bytes gmem", out)]
    assert gmem and max(gmem) <= 4 * (64 + 2 * 32768) + 1024
