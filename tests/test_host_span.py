"""Which host arrays the step kernel may access itself: the decision from what the driver reports, compiled for the CPU."""
import ctypes as C
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SOURCE = r"""
#include "host_span.cuh"
extern "C" uintptr_t span(int pinned, uintptr_t device, uintptr_t start, size_t size, uintptr_t host, size_t bytes, size_t align) {
  const marl::HostRange r = {pinned != 0, reinterpret_cast<const void*>(device), start, size};
  return reinterpret_cast<uintptr_t>(marl::kernel_span(r, reinterpret_cast<const void*>(host), bytes, align));
}
"""


@pytest.fixture(scope="module")
def span(tmp_path_factory):
    d = tmp_path_factory.mktemp("host_span")
    (d / "span.cpp").write_text(SOURCE)
    subprocess.check_call(["g++", "-std=c++17", "-O1", "-shared", "-fPIC", "-I", os.path.join(ROOT, "paper_2205_05248_b200", "csrc"),
                           "-o", str(d / "span.so"), str(d / "span.cpp")])
    fn = C.CDLL(str(d / "span.so")).span
    fn.restype = C.c_size_t
    fn.argtypes = [C.c_int] + [C.c_size_t] * 6
    return fn


H, D = 0x7F0000001000, 0x2000  # host and device address of a registration of 8 KB


@pytest.mark.parametrize("off,nbytes,align,ok", [
    (0, 8192, 16, True), (16, 8176, 16, True), (8191, 1, 1, True), (0, 1, 16, True),
    (0, 8193, 16, False), (16, 8192, 16, False), (8192, 1, 1, False), (-16, 64, 16, False),   # pinned in part, or beside it
    (4, 64, 16, False), (1, 4, 4, False), (4, 64, 4, True), (3, 9, 1, True),                  # alignment
    (16, 2**64 - 16, 16, False)])
def test_whole_and_aligned(span, off, nbytes, align, ok):
    assert span(1, D + off, H, 8192, H + off, nbytes, align) == (D + off if ok else 0)


def test_not_pinned_or_not_known(span):
    assert span(0, D, H, 8192, H, 64, 16) == 0       # pageable, device or managed memory
    assert span(1, 0, H, 8192, H, 64, 16) == 0       # not mapped
    assert span(1, D, H, 0, H, 64, 16) == 0          # the extent is not known
    assert span(1, D + 8, H, 8192, H, 64, 16) == 0   # mapped at another alignment
