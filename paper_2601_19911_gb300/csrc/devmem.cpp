#include "devmem.h"

#include <mutex>
#include <vector>

namespace olap {
namespace devmem {

namespace {

struct Piece {
    int dev;
    void* p;
    size_t cap;
};
std::mutex g_lock;
std::vector<Piece> g_kept;                                   // oldest first
int g_contexts[64] = {};

// Free the pieces of `dev`, `dev` current and g_lock held: a thread whose
// allocation failed meanwhile waits until they are free.
uint64_t give_back(int dev) {
    uint64_t bytes = 0;
    size_t w = 0;
    for (const Piece& x : g_kept) {
        if (x.dev == dev) {
            cudaFree(x.p);
            bytes += x.cap;
        } else {
            g_kept[w++] = x;
        }
    }
    g_kept.resize(w);
    return bytes;
}

}  // namespace

cudaError_t alloc(int dev, void** p, size_t bytes) {
    const cudaError_t e = cudaMalloc(p, bytes);
    if (e != cudaErrorMemoryAllocation) return e;
    cudaGetLastError();
    {
        std::lock_guard<std::mutex> guard(g_lock);
        give_back(dev);
    }
    return cudaMalloc(p, bytes);
}

cudaError_t take(int dev, void** p, size_t bytes, size_t* cap) {
    {
        std::lock_guard<std::mutex> guard(g_lock);
        size_t best = g_kept.size();
        for (size_t i = 0; i < g_kept.size(); ++i)
            if (g_kept[i].dev == dev && g_kept[i].cap >= bytes && g_kept[i].cap <= bytes + bytes / 2 + (1u << 20) &&
                (best == g_kept.size() || g_kept[i].cap < g_kept[best].cap))
                best = i;
        if (best < g_kept.size()) {
            *p = g_kept[best].p;
            *cap = g_kept[best].cap;
            g_kept.erase(g_kept.begin() + static_cast<std::ptrdiff_t>(best));
            return cudaSuccess;
        }
    }
    *cap = bytes;
    return alloc(dev, p, bytes);
}

void give(int dev, void* p, size_t cap) {
    std::lock_guard<std::mutex> guard(g_lock);
    if (dev < 0 || dev >= 64 || g_contexts[dev] == 0 || cap > KEEP_TOTAL) {
        cudaFree(p);
        return;
    }
    size_t held = cap;
    int pieces = 1;
    for (const Piece& x : g_kept)
        if (x.dev == dev) {
            held += x.cap;
            ++pieces;
        }
    size_t w = 0;
    for (const Piece& x : g_kept) {                          // the oldest make room
        if (x.dev == dev && (held > KEEP_TOTAL || pieces > KEEP_BLOCKS)) {
            cudaFree(x.p);
            held -= x.cap;
            --pieces;
        } else {
            g_kept[w++] = x;
        }
    }
    g_kept.resize(w);
    g_kept.push_back(Piece{dev, p, cap});
}

uint64_t trim(int dev) {
    std::lock_guard<std::mutex> guard(g_lock);
    return give_back(dev);
}

void context_created(int dev) {
    std::lock_guard<std::mutex> guard(g_lock);
    if (dev >= 0 && dev < 64) ++g_contexts[dev];
}

void context_gone(int dev) {
    std::lock_guard<std::mutex> guard(g_lock);
    if (dev >= 0 && dev < 64 && --g_contexts[dev] == 0) give_back(dev);
}

}  // namespace devmem
}  // namespace olap
