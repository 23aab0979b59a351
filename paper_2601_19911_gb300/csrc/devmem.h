// Device memory of the library: allocations that first give back what is kept
// for reuse, and the pieces that join builds keep.
//
// A freed join table's memory is kept for the next table of about the same
// size, and the partition scratch of a large build for the next one: a
// table's cudaMalloc and cudaFree take 370 us at 134 MB, twice what building
// it takes.  Shared by the process's contexts and threads under one
// lock; at most KEEP_TOTAL per device and KEEP_BLOCKS pieces, the oldest making
// room for the newest; given back when the device's last context goes, when an
// allocation of the library fails for want of memory, and by olap_device_trim
// for the process's other allocators.  Contexts with a memory budget take no
// part.
#pragma once

#include <cuda_runtime.h>

#include <cstddef>
#include <cstdint>

namespace olap {
namespace devmem {
constexpr size_t KEEP_TOTAL = 2ull << 30;
constexpr int KEEP_BLOCKS = 8;
// cudaMalloc on the current device `dev`; gives the kept memory back and tries
// again when there is not enough.
cudaError_t alloc(int dev, void** p, size_t bytes);
template <typename T>
cudaError_t alloc(int dev, T** p, size_t bytes) {
    return alloc(dev, reinterpret_cast<void**>(p), bytes);
}
// A kept piece of bytes to 1.5 * bytes (+ 1 MiB), or a new one; *cap is its
// size.
cudaError_t take(int dev, void** p, size_t bytes, size_t* cap);
// Keep a piece (no work may use it any more), or free it.
void give(int dev, void* p, size_t cap);
// Free what is kept on `dev`, `dev` current; returns the bytes.
uint64_t trim(int dev);
// A context of `dev` was created / is going.
void context_created(int dev);
void context_gone(int dev);
}  // namespace devmem
}  // namespace olap
