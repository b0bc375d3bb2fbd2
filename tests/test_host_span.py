"""The rule for host buffers that kernels read where they lie (csrc/host_span.h): host arithmetic, compiled with the host
compiler and called with what the driver reports for page-locked, partly page-locked and pageable buffers."""
import ctypes as C
import shutil
import subprocess

import pytest

from paper_2511_22972_b200 import build

PAGE = 4096
BASE = 0x7f0000000000


@pytest.fixture(scope="module")
def rule(tmp_path_factory):
    cxx = shutil.which("g++")
    if not cxx:
        pytest.skip("no host compiler")
    d = tmp_path_factory.mktemp("span")
    (d / "span.cpp").write_text("""
#include "host_span.h"
extern "C" int in_place(unsigned type, uint64_t device, uint64_t start, size_t size, unsigned managed, uint64_t host, size_t bytes,
                        size_t element) {
  fly::HostSpan s; s.type = type; s.device = device; s.start = start; s.size = size; s.managed = managed;
  return fly::readable_in_place(s, (const void*)(uintptr_t)host, bytes, element);
}
""")
    subprocess.run([cxx, "-std=c++17", "-Wall", "-Wextra", "-Werror", "-shared", "-fPIC", "-I", build.CSRC, "-o", str(d / "span.so"),
                    str(d / "span.cpp")], check=True)
    fn = C.CDLL(str(d / "span.so")).in_place
    fn.argtypes = [C.c_uint, C.c_uint64, C.c_uint64, C.c_size_t, C.c_uint, C.c_uint64, C.c_size_t, C.c_size_t]
    return lambda host, size, start=BASE, type=1, device=None, managed=0, bytes=PAGE, element=2: bool(
        fn(type, host if device is None else device, start, size, managed, host, bytes, element))


def test_the_whole_buffer_has_to_lie_in_one_page_locked_range(rule):
    assert rule(BASE, PAGE) and rule(BASE, 16 * PAGE) and rule(BASE + 15 * PAGE, 16 * PAGE)
    assert not rule(BASE, PAGE - 1)                              # only the first part was registered
    assert not rule(BASE + 15 * PAGE + 2, 16 * PAGE)             # the last bytes lie outside
    assert not rule(BASE, PAGE, bytes=2 * PAGE)                  # two registrations side by side: the driver names the first
    assert not rule(BASE - 2, 16 * PAGE)
    assert not rule(BASE, 16 * PAGE, bytes=2 ** 64 - 1)


def test_other_memory_is_copied(rule):
    assert not rule(BASE, 0, start=0, type=0, device=0)          # pageable: the driver knows nothing
    assert not rule(BASE, 16 * PAGE, type=2)                     # device memory
    assert not rule(BASE, 16 * PAGE, managed=1)
    assert not rule(BASE, 16 * PAGE, device=BASE + 2 ** 40)      # registered under another address


@pytest.mark.parametrize("element", [2, 4])
def test_elements_off_their_alignment_are_copied(rule, element):
    for off in range(1, 9):
        assert rule(BASE + off, 16 * PAGE, element=element) == (off % element == 0)
