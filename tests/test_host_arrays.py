"""What a host array of the C ABI is taken for, from the attributes CUDA reports of
its two ends (csrc/wb_pages.h, compiled for the host): only plain pageable memory
may be written by the host ahead of a copy; page-locked memory the GPU can address
is used in place; nothing is dereferenced to tell."""
import ctypes
import subprocess

import pytest

from paper_1701_07452_gb300 import _build

# cudaMemoryType
UNREGISTERED, HOST, DEVICE, MANAGED = 0, 1, 2, 3

SRC = r"""
#include "wb_pages.h"
extern "C" int host_array(int t0, unsigned long long d0, int t1, unsigned long long d1, unsigned long long span) {
  cudaPointerAttributes a = {}, b = {};
  a.type = (cudaMemoryType)t0;
  b.type = (cudaMemoryType)t1;
  a.devicePointer = (void*)d0;
  b.devicePointer = (void*)d1;
  const WbHostArray h = wb_host_array_of(a, b, span);
  return (h.plain ? 1 : 0) | (h.mapped ? 2 : 0) | (h.mapped && h.mapped != (void*)d0 ? 4 : 0);
}
extern "C" int touch(char* p, unsigned long long bytes) {
  wb_touch_pages(p, bytes);
  return (int)sysconf(_SC_PAGESIZE);
}
"""


@pytest.fixture(scope="module")
def pages(tmp_path_factory):
    d = tmp_path_factory.mktemp("pages")
    src, so = d / "pages.cu", d / "libpages.so"
    src.write_text(SRC)
    subprocess.run([_build.nvcc(), "-std=c++17", "-Xcompiler", "-fPIC", "-shared", "-I", _build.CSRC, str(src),
                    "-o", str(so)], check=True, capture_output=True)
    L = ctypes.CDLL(str(so))
    L.host_array.argtypes = [ctypes.c_int, ctypes.c_ulonglong, ctypes.c_int, ctypes.c_ulonglong, ctypes.c_ulonglong]
    L.touch.argtypes = [ctypes.c_void_p, ctypes.c_ulonglong]
    return L


PLAIN, MAPPED = 1, 2
AT = 0x7000_0000_0000  # an address nothing lives at


@pytest.mark.parametrize("t0,t1,want", [
    (UNREGISTERED, UNREGISTERED, PLAIN), (HOST, HOST, MAPPED), (DEVICE, DEVICE, 0), (MANAGED, MANAGED, 0),
    (UNREGISTERED, HOST, 0), (HOST, UNREGISTERED, 0), (UNREGISTERED, DEVICE, 0), (HOST, DEVICE, 0), (MANAGED, HOST, 0),
])
def test_kinds(pages, t0, t1, want):
    assert pages.host_array(t0, AT, t1, AT + 8000, 8000) == want


def test_page_locked_but_not_addressable_as_one_range(pages):
    """No device address, or two registrations that the GPU sees apart: neither."""
    assert pages.host_array(HOST, 0, HOST, AT + 8000, 8000) == 0
    assert pages.host_array(HOST, AT, HOST, 0, 8000) == 0
    assert pages.host_array(HOST, AT, HOST, AT + 9000, 8000) == 0
    assert pages.host_array(HOST, AT, HOST, AT - 8000, 8000) == 0


@pytest.mark.parametrize("at,size", [(0, 1), (8, 0), (4000, 200), (8, 3 * 65536), (65528, 65552)])
def test_touch_stays_inside(pages, at, size):
    buf = ctypes.create_string_buffer(b"\x11" * (5 * 65536), 5 * 65536)
    page = pages.touch(ctypes.addressof(buf) + at, size)
    raw = buf.raw
    assert set(raw[:at]) <= {0x11} and set(raw[at + size:]) <= {0x11}
    first = ctypes.addressof(buf) + at
    written = {(first + i) // page for i in range(size) if raw[at + i] == 0}
    assert size == 0 or written == set(range(first // page, (first + size - 1) // page + 1))
