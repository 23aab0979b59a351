// Device side of the key-only hash join shared by the probe kernel and the
// batched executor: table constants, the fmix64 hash, the per-CTA staged
// output and the probe rounds.
#pragma once

#include <cstdint>

#include "common.cuh"

struct olap_join_table {
    olap_ctx* owner = nullptr;        // context whose budget counts this table (or NULL)
    int device = 0;
    ulonglong2* slots = nullptr;      // n_buckets * 2 slots
    uint64_t n_buckets = 0;
    uint32_t* side = nullptr;         // row-ids of build rows with the empty-marker key
    uint64_t n_side = 0;
    uint64_t n_build = 0;
    double load = 0.0;
    size_t bytes = 0;
    size_t cap = 0;                   // size of its memory when that may be kept for another table, else 0
    uint32_t* bloom = nullptr;        // blocked Bloom filter over the keys (NULL: none)
    uint64_t bloom_blocks = 0;        // 32-byte blocks, a power of two
    uint64_t chain_mask = 0;          // chains wrap within this many buckets + 1 (see join_block_build_kernel)
};

namespace olap {

constexpr uint64_t JN_EMPTY = ~0ull;
constexpr int JB_TPB = 256;
constexpr int JP_TPB = 256;
constexpr int JP_WARPS = JP_TPB / 32;
// Shape of the probe kernels, from a sweep (2^20-row table in L2 with 18 M
// probes / 2^24 rows with 30 M probes, partitioned / the same with Zipf
// probes, direct): 4 rows per lane on 16 warps per SM take 126 / 484 /
// 364 us; on 24 warps 142 / 519 / 455 us (spills, less L1); 8 rows 165 /
// 559 / 435 us.  A stage of 384 pairs flushes too often (the count word
// serialises: 128 / 596 us), one of 1280 takes the L1 the buckets use (690 us
// on the Zipf probes).
constexpr unsigned JP_WCAP = 640;           // pairs staged per warp
constexpr int JP_U = 4;                     // rows in flight per lane
constexpr int JP_CTAS = 2;                  // probe CTAs per SM
constexpr unsigned JP_PEND = 32 * JP_U + 32;  // probes per warp that walk on past their home bucket
constexpr int JP_WARP_SMEM = JP_WCAP * 8 + JP_PEND * 16;
constexpr int JP_SMEM = JP_WARPS * JP_WARP_SMEM;

struct JoinCtl {
    unsigned long long side_count;   // build rows with the empty-marker key
    unsigned long long side_fill;
    int err;
    int crowded;                     // a table block got more rows than it has room for
};

// Blocks of the table that are built in one CTA's shared memory.
constexpr int JT_BLOCK_LOG = 10;                       // 1024 buckets, 32 KB
constexpr uint64_t JT_BLOCK = 1ull << JT_BLOCK_LOG;

__device__ __forceinline__ uint64_t fmix64(uint64_t h) {
    h ^= h >> 33;
    h *= 0xff51afd7ed558ccdull;
    h ^= h >> 33;
    h *= 0xc4ceb9fe1a85ec53ull;
    h ^= h >> 33;
    return h;
}

// Streaming probe-side traffic (keys, row-ids, pairs) is read or written
// once: the .cs forms allocate its L2 lines evict-first, so the table's lines
// are what L2 keeps.
__device__ __forceinline__ uint64_t ld_stream_u64(const void* p) {
    uint64_t v;
    asm volatile("ld.global.cs.u64 %0, [%1];" : "=l"(v) : "l"(p));
    return v;
}
__device__ __forceinline__ uint32_t ld_stream_u32(const void* p) {
    uint32_t v;
    asm volatile("ld.global.cs.u32 %0, [%1];" : "=r"(v) : "l"(p));
    return v;
}
__device__ __forceinline__ void st_stream_pair(uint2* p, uint2 v) {
    asm volatile("st.global.cs.v2.u32 [%0], {%1, %2};" ::"l"(p), "r"(v.x), "r"(v.y) : "memory");
}

// Blocked Bloom filter (Putze, Sanders & Singler, "Cache-, hash- and
// space-efficient Bloom filters", WEA 2007): every key maps to one 32-byte
// block (one sector, one load) and sets one bit in each of the block's eight
// 32-bit words.  The filter blocks of the keys of one table block lie
// together, so that the CTA that builds the table block also fills them: the
// upper bits of the filter block are the table block's, the lower ones bits
// 40 and up of fmix64(key), which the table's bucket index (the low bits) does
// not use.  The eight bit positions are the upper 40 bits of that hash times an
// odd constant.
constexpr int BLOOM_WORDS = 8;

struct BloomView {
    const uint32_t* bits;             // NULL: no filter
    uint64_t mask;                    // table buckets - 1
    int block_log;                    // log2 buckets of a table block
    int per_log;                      // log2 filter blocks per table block
};
__device__ __forceinline__ uint64_t bloom_block(const BloomView& f, uint64_t h) {
    return (((h & f.mask) >> f.block_log) << f.per_log) | ((h >> 40) & ((1ull << f.per_log) - 1ull));
}
// The eight bit positions of a key with hash h, five bits each.
__device__ __forceinline__ uint64_t bloom_bits(uint64_t h) { return (h * 0x9E3779B97F4A7C15ull) >> 24; }
__device__ __forceinline__ uint32_t bloom_bit(uint64_t g, int w) {
    return 1u << static_cast<uint32_t>((g >> (5 * w)) & 31u);
}
// Whether `key` may be among the filter's keys (no false negatives).
__device__ __forceinline__ bool bloom_maybe(const BloomView& f, uint64_t key) {
    const uint64_t h = fmix64(key);
    const ulonglong2* p = reinterpret_cast<const ulonglong2*>(f.bits + bloom_block(f, h) * BLOOM_WORDS);
    uint64_t v[4];
    asm("ld.global.cg.v4.u64 {%0, %1, %2, %3}, [%4];" : "=l"(v[0]), "=l"(v[1]), "=l"(v[2]), "=l"(v[3]) : "l"(p));
    // bit s of word w, for all words at once: every word rotated by its five
    // bits (the shift itself drops the higher ones), the low bits combined
    const uint64_t g = bloom_bits(h);
    const uint32_t lo = static_cast<uint32_t>(g), hi = static_cast<uint32_t>(g >> 32);
    uint32_t all = 1u;
#pragma unroll
    for (int w = 0; w < BLOOM_WORDS; ++w) {
        const uint32_t x = static_cast<uint32_t>(v[w / 2] >> (32 * (w & 1)));
        const uint32_t at = 5 * w < 28 ? lo >> (5 * w) : 5 * w < 32 ? __funnelshift_r(lo, hi, 5 * w) : hi >> (5 * w - 32);
        all &= __funnelshift_r(x, x, at);
    }
    return all != 0;
}

// Device-side plan of one probe, written by its sampling stage: whether the
// Bloom pre-probe filters the rows (and how many it kept), and whether the
// probe skips the partition passes and reads its rows directly.  The stages
// after the sample read it, so the decision never travels through the host.
struct ProbeCtl {
    int active;                    // the pre-probe drops rows
    int direct;                    // the partition passes are skipped
    unsigned long long count;      // rows the pre-probe kept
    const int64_t* keys;           // with `redirect`: the rows the probe kernel reads
    const uint32_t* rowids;
    int redirect;
    int l1;                        // the probe's bucket reads go through L1
};

struct ProbeArgs {
    const int64_t* keys;
    const uint32_t* rowids;
    uint64_t n;
    const ulonglong2* slots;
    uint64_t mask;
    uint64_t chain_mask;
    const uint32_t* side;
    uint64_t n_side;
    uint2* out;
    uint64_t cap;
    unsigned long long* count;
};

// One 32-byte bucket {key0, row-id0 | pad, key1, row-id1 | pad} in a single
// 256-bit load; L2_ONLY bypasses L1 (ld.global.cg), else the read-only path
// through L1 (ld.global.nc).
struct Bucket {
    uint64_t k0, w0, k1, w1;          // w: row-id in the low 32 bits, further copies in the high 32
};

template <bool L2_ONLY>
__device__ __forceinline__ Bucket ld_bucket(const ulonglong2* slots, uint32_t b) {
    const ulonglong2* p = slots + static_cast<uint64_t>(b) * 2;
    Bucket v;
    if (L2_ONLY)
        asm("ld.global.cg.v4.u64 {%0, %1, %2, %3}, [%4];" : "=l"(v.k0), "=l"(v.w0), "=l"(v.k1), "=l"(v.w1) : "l"(p));
    else
        asm("ld.global.nc.v4.u64 {%0, %1, %2, %3}, [%4];" : "=l"(v.k0), "=l"(v.w0), "=l"(v.k1), "=l"(v.w1) : "l"(p));
    return v;
}

// Copy a warp's staged pairs to the output with one atomic on the global
// count (whole warp calls; cnt is warp-uniform).
__device__ __forceinline__ void warp_flush(const ProbeArgs& a, uint2* ws, unsigned& cnt) {
    if (cnt == 0) return;
    __syncwarp();
    const unsigned lane = threadIdx.x & 31u;
    unsigned long long g = 0;
    if (lane == 0) g = atomicAdd(a.count, static_cast<unsigned long long>(cnt));
    g = __shfl_sync(0xFFFFFFFFu, g, 0);
    // pairs past the capacity are only counted
    const uint64_t room = g < a.cap ? a.cap - g : 0;
    const unsigned n = room < cnt ? static_cast<unsigned>(room) : cnt;
    uint2* o = a.out + g;
    for (unsigned i = lane; i < n; i += 32) st_stream_pair(o + i, ws[i]);
    __syncwarp();
    cnt = 0;
}

// Stage one pair for every lane where m is set (whole warp calls; the caller
// has made room for 32).
__device__ __forceinline__ void warp_put(uint2* ws, unsigned& cnt, bool m, uint2 p) {
    const unsigned b = __ballot_sync(0xFFFFFFFFu, m);
    if (m) ws[cnt + __popc(b & ((1u << (threadIdx.x & 31u)) - 1u))] = p;
    cnt += __popc(b);
}

// Rows handed to the warps: chunks of consecutive rows from a counter (global
// for a whole probe, shared memory for one chunk of a batch item), so that
// warps stay busy to the end and a partitioned probe moves through its
// partitions in order, the whole grid on one table slice at a time.
struct RowQueue {
    unsigned long long* counter;  // next unclaimed row (zeroed before the launch)
    uint64_t n;
    uint32_t chunk;               // rows per take: 32, 64, ... JQ_CHUNK
};
constexpr uint32_t JQ_CHUNK = 512;

// Rows per take for n rows over `warps` warps: JQ_CHUNK (one atomic per 512
// rows) once every warp gets that many, fewer for small probes so that all
// warps take part (100,003 rows against a 2^20-row table: 37.9 -> 13.2 us,
// 10^6 rows 36 -> 18 us).
__device__ __forceinline__ uint32_t queue_chunk(uint64_t n, uint32_t warps) {
    uint32_t c = JQ_CHUNK;
    while (c > 32 && static_cast<uint64_t>(c) * warps > n) c >>= 1;
    return c;
}

struct RowRange {
    uint64_t b, e;
};
__device__ __forceinline__ RowRange take_chunk(const RowQueue& q) {
    unsigned long long g = 0;
    if ((threadIdx.x & 31u) == 0) g = atomicAdd(q.counter, static_cast<unsigned long long>(q.chunk));
    g = __shfl_sync(0xFFFFFFFFu, g, 0);
    return RowRange{min(static_cast<uint64_t>(g), q.n), min(static_cast<uint64_t>(g) + q.chunk, q.n)};
}

// One probe against one bucket (whole warp calls, with room for 64 pairs):
// stage the matches, and push the probe when its chain goes on.  A match
// whose slot counts no further copies of its key ends the walk, as does a
// bucket with a free slot.  An entry of `pend` holds the key, the row-id in
// the low half of y and the bucket to read in the high half.
__device__ __forceinline__ void probe_step(uint2* ws, unsigned& cnt, ulonglong2* pend, unsigned& np, bool real,
                                           const Bucket& v, uint64_t key, uint32_t rid, uint32_t bk, uint32_t cmask) {
    const bool m0 = real && v.k0 == key, m1 = real && v.k1 == key;
    const uint64_t w = m0 ? v.w0 : v.w1;
    warp_put(ws, cnt, m0 || m1, make_uint2(rid, static_cast<uint32_t>(w)));
    // (with both slots matching, slot 0 counts slot 1 as a further copy)
    const bool go = real && v.k1 != JN_EMPTY && !((m0 || m1) && (w >> 32) == 0);
    if (!__any_sync(0xFFFFFFFFu, go)) return;
    const bool both = m0 && m1;
    warp_put(ws, cnt, both, make_uint2(rid, static_cast<uint32_t>(v.w1)));
    const bool on = go && !(both && (v.w1 >> 32) == 0);
    const unsigned b = __ballot_sync(0xFFFFFFFFu, on);
    if (on)
        pend[np + __popc(b & ((1u << (threadIdx.x & 31u)) - 1u))] =
            make_ulonglong2(key, rid | (static_cast<uint64_t>((bk & ~cmask) | ((bk + 1u) & cmask)) << 32));
    np += __popc(b);
}

// One warp probes chunks of rows until the queue is empty, a tile of 32 *
// JP_U rows at a time: every lane has JP_U independent bucket loads in
// flight, and the next tile's keys are loaded while the current tile's
// buckets arrive.  The few probes whose chain goes on (a full home bucket
// without the key's last copy) are compacted in shared memory and walked 32
// at a time, so no lane waits for another's longer chain.  Bound by the
// bucket reads: L2-resident tables run at 143 G probes/s (103 G when every
// lane walked its chains itself, two rows at a time), a 2^24-row table with
// 30 M partitioned probes in 484 us for the whole call (648 us; 437 with the
// present partition passes), with 2^28 probes in 3.30 ms (4.26 ms).
template <bool L2_ONLY>
__device__ __forceinline__ void probe_rows(const ProbeArgs& a, const RowQueue& q, unsigned char* warp_smem) {
    uint2* ws = reinterpret_cast<uint2*>(warp_smem + JP_PEND * 16);
    ulonglong2* pend = reinterpret_cast<ulonglong2*>(warp_smem);
    const unsigned lane = threadIdx.x & 31u;
    const uint32_t mask = static_cast<uint32_t>(a.mask), cmask = static_cast<uint32_t>(a.chain_mask);
    constexpr unsigned TILE = 32u * JP_U;
    unsigned cnt = 0, np = 0;
    uint64_t key[JP_U];
    uint32_t rid[JP_U];
    auto load_tile = [&](const RowRange& r) {
        const int64_t* kp = a.keys + r.b + lane;
        const uint32_t* rp = a.rowids + r.b + lane;
        const uint32_t i0 = static_cast<uint32_t>(r.b) + lane;
        if (r.e - r.b >= TILE) {
#pragma unroll
            for (int j = 0; j < JP_U; ++j) key[j] = ld_stream_u64(kp + j * 32);
#pragma unroll
            for (int j = 0; j < JP_U; ++j) rid[j] = a.rowids ? ld_stream_u32(rp + j * 32) : i0 + j * 32;
        } else {
            const unsigned left = static_cast<unsigned>(r.e - r.b);
#pragma unroll
            for (int j = 0; j < JP_U; ++j) {
                const bool in = j * 32 + lane < left;
                key[j] = in ? ld_stream_u64(kp + j * 32) : JN_EMPTY;
                rid[j] = (in && a.rowids) ? ld_stream_u32(rp + j * 32) : i0 + j * 32;
            }
        }
    };
    auto drain = [&](unsigned keep) {           // walk pending probes while more than `keep` wait
        while (np > keep) {
            const unsigned take = min(np, 32u);
            np -= take;
            const bool act = lane < take;
            if (cnt > JP_WCAP - 64) warp_flush(a, ws, cnt);
            __syncwarp();
            const ulonglong2 p = pend[np + (act ? lane : 0u)];
            __syncwarp();
            const uint32_t bk = static_cast<uint32_t>(p.y >> 32);
            const Bucket v = ld_bucket<L2_ONLY>(a.slots, bk);
            probe_step(ws, cnt, pend, np, act, v, p.x, static_cast<uint32_t>(p.y), bk, cmask);
        }
    };
    RowRange r = take_chunk(q);
    load_tile(r);
    while (r.b < r.e) {
        Bucket v[JP_U];
        uint32_t bk[JP_U];
#pragma unroll
        for (int j = 0; j < JP_U; ++j) {
            bk[j] = static_cast<uint32_t>(fmix64(key[j])) & mask;
            v[j] = ld_bucket<L2_ONLY>(a.slots, bk[j]);
        }
        uint64_t ck[JP_U];
        uint32_t cr[JP_U];
        const unsigned rows = static_cast<unsigned>(min(r.e - r.b, static_cast<uint64_t>(TILE)));
#pragma unroll
        for (int j = 0; j < JP_U; ++j) {
            ck[j] = key[j];
            cr[j] = rid[j];
        }
        r.b += TILE;
        if (r.b >= r.e) r = take_chunk(q);
        load_tile(r);
        // Probe keys equal to the empty marker pair with every side-list row;
        // the warp emits them together, one such key at a time (rare).
        if (a.n_side) {
#pragma unroll
            for (int j = 0; j < JP_U; ++j) {
                unsigned sb = __ballot_sync(0xFFFFFFFFu, ck[j] == JN_EMPTY && j * 32 + lane < rows);
                while (sb) {
                    const int src = __ffs(sb) - 1;
                    sb &= sb - 1;
                    const uint32_t rr = __shfl_sync(0xFFFFFFFFu, cr[j], src);
                    for (uint64_t o0 = 0; o0 < a.n_side; o0 += 32) {
                        if (cnt > JP_WCAP - 32) warp_flush(a, ws, cnt);
                        const bool m = o0 + lane < a.n_side;
                        warp_put(ws, cnt, m, make_uint2(rr, m ? a.side[o0 + lane] : 0u));
                    }
                }
            }
        }
        if (cnt > JP_WCAP - 64 * JP_U) warp_flush(a, ws, cnt);
#pragma unroll
        for (int j = 0; j < JP_U; ++j)
            probe_step(ws, cnt, pend, np, ck[j] != JN_EMPTY, v[j], ck[j], cr[j], bk[j], cmask);
        drain(31u);
    }
    drain(0u);
    warp_flush(a, ws, cnt);
}

}  // namespace olap
