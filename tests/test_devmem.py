"""The library's device allocations and the memory it keeps for reuse, on the
CPU: the module compiled against a cudaMalloc and cudaFree that count bytes in
a device of 4 GiB."""
import ctypes
import os
import re
import subprocess

import pytest

from paper_2601_19911_gb300 import build, olap

CSRC = build.CSRC
GIB, MIB = 1 << 30, 1 << 20

FAKE = r"""
#include <cuda_runtime.h>
#include <cstdint>
#include <cstdlib>
#include <map>
#include "devmem.h"
static std::map<uintptr_t, size_t> live;
static uintptr_t next_at = 1 << 20;
static size_t used, limit = 4ull << 30;
static cudaError_t last;
extern "C" {
cudaError_t cudaMalloc(void** p, size_t n) {
    if (used + n > limit) return last = cudaErrorMemoryAllocation;
    used += n;
    *p = reinterpret_cast<void*>(next_at);
    live[next_at] = n;
    next_at += n + 4096;
    return cudaSuccess;
}
cudaError_t cudaFree(void* p) {
    auto it = live.find(reinterpret_cast<uintptr_t>(p));
    if (it == live.end()) abort();
    used -= it->second;
    live.erase(it);
    return cudaSuccess;
}
cudaError_t cudaGetLastError(void) { cudaError_t e = last; last = cudaSuccess; return e; }
size_t t_used() { return used; }
int t_sticky() { return last != cudaSuccess; }
void* t_alloc(size_t n) { void* p = nullptr; return olap::devmem::alloc(0, &p, n) == cudaSuccess ? p : nullptr; }
void* t_take(size_t n, size_t* cap) { void* p = nullptr; return olap::devmem::take(0, &p, n, cap) == cudaSuccess ? p : nullptr; }
void t_give(void* p, size_t cap) { olap::devmem::give(0, p, cap); }
uint64_t t_trim() { return olap::devmem::trim(0); }
void t_context(int up) { if (up) olap::devmem::context_created(0); else olap::devmem::context_gone(0); }
}
"""


@pytest.fixture()
def mem(tmp_path):
    (tmp_path / "fake.cpp").write_text(FAKE)
    so = str(tmp_path / "devmem.so")
    cuda = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(build.nvcc()))), "include")
    subprocess.run(["g++", "-std=c++17", "-shared", "-fPIC", "-Wl,-Bsymbolic", "-I", CSRC, "-I", cuda, str(tmp_path / "fake.cpp"),
                    os.path.join(CSRC, "devmem.cpp"), "-o", so], check=True)
    lib = ctypes.CDLL(so)
    for name in ("t_alloc", "t_take"):
        getattr(lib, name).restype = ctypes.c_void_p
    lib.t_used.restype = ctypes.c_size_t
    lib.t_trim.restype = ctypes.c_uint64
    lib.t_alloc.argtypes = [ctypes.c_size_t]
    lib.t_take.argtypes = [ctypes.c_size_t, ctypes.POINTER(ctypes.c_size_t)]
    lib.t_give.argtypes = [ctypes.c_void_p, ctypes.c_size_t]
    lib.t_context(1)
    return lib


def _take(mem, n):
    cap = ctypes.c_size_t()
    p = mem.t_take(n, ctypes.byref(cap))
    assert p and cap.value >= n
    return p, cap.value


def _keep(mem, *sizes):
    held = [_take(mem, n) for n in sizes]
    for p, cap in held:
        mem.t_give(p, cap)


def test_reuse_and_return_with_the_last_context(mem):
    p, cap = _take(mem, 100 * MIB)
    mem.t_give(p, cap)
    assert mem.t_used() == 100 * MIB
    q, cap2 = _take(mem, 80 * MIB)                 # within 1.5 times
    assert (q, cap2) == (p, cap)
    mem.t_context(1)
    mem.t_give(q, cap2)
    mem.t_context(0)
    assert mem.t_used() == 100 * MIB               # one context left
    mem.t_context(0)
    assert mem.t_used() == 0
    p, cap = _take(mem, MIB)
    mem.t_give(p, cap)                             # nobody left to keep it for
    assert mem.t_used() == 0


def test_failed_allocations_get_the_kept_memory(mem):
    _keep(mem, GIB, 900 * MIB)
    assert mem.t_used() == GIB + 900 * MIB
    assert mem.t_alloc(3 * GIB) and not mem.t_sticky()
    assert mem.t_used() == 3 * GIB
    assert not mem.t_alloc(2 * GIB)


def test_every_device_allocation_may_get_it():
    """No source file but this module calls cudaMalloc."""
    for src in build.sources():
        text = re.sub(r"//.*", "", open(src).read())
        calls = len(re.findall(r"\bcudaMalloc(?:Async|Managed|Pitch)?\s*\(", text))
        assert calls == (2 if src.endswith("devmem.cpp") else 0), src


def test_old_pieces_make_room(mem):
    """Pieces of a size that is no longer asked for do not stay for good."""
    _keep(mem, *[4096] * 8)                        # all places taken by small ones
    p, cap = _take(mem, 100 * MIB)
    mem.t_give(p, cap)
    assert _take(mem, 100 * MIB)[0] == p
    assert mem.t_used() == 7 * 4096 + 100 * MIB


def test_kept_memory_is_bounded(mem):
    _keep(mem, GIB, GIB, 100 * MIB)                # 2 GiB at most: the first one goes
    assert mem.t_used() == GIB + 100 * MIB
    _keep(mem, *[(10 + i * 40) * MIB for i in range(12)])
    assert mem.t_used() <= 2 * GIB
    p, cap = _take(mem, 3 * GIB)                   # too large to keep, and none goes for it
    used = mem.t_used() - cap
    mem.t_give(p, cap)
    assert mem.t_used() == used


def test_trim(mem):
    _keep(mem, GIB, 10 * MIB)
    assert mem.t_trim() == GIB + 10 * MIB
    assert mem.t_used() == 0 and mem.t_trim() == 0
    _keep(mem, MIB)                                # and keeping goes on
    assert mem.t_used() == MIB


def test_trim_of_a_bad_device():
    with pytest.raises(olap.OlapError) as ei:
        olap.device_trim(-1)
    assert ei.value.status in (olap.E_INVALID, olap.E_CUDA)
