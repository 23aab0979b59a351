// Key-based hash join over key-only columns (Sec. III-B: "parallel probing
// using a key-only hash table"; pointers returned for late materialization,
// Sec. II-C).
//
// Table: open addressing, 16-byte slots {int64 key, row-id}, two slots per
// 32-byte bucket (one DRAM sector), linear probing over buckets.  A key goes
// to the first free slot at or after its home bucket, slot 0 before slot 1,
// so a bucket with a free slot ends every chain.  The empty marker is the key
// with all bits set; build rows carrying that key value live in a side list.
// Hash: the 64-bit finalizer of MurmurHash3 (fmix64, A. Appleby).
//
// Build: the rows are appended to the table blocks (1024 buckets) their home
// buckets lie in, and every block is then built in one CTA's shared memory:
// insertion, the count of further copies of its key along the chain in every
// slot (so a probe can stop at a key's last copy instead of walking on to the
// chain's end), and the block's part of the Bloom filter.  Chains wrap within
// their block.  A block with more rows than slots (thousands of copies of one
// key) sends the whole build to the general way: one CAS pass over the table,
// a pass over its chains, and chains that wrap at the table's end.
//
// Probe: every warp takes chunks of consecutive rows from a global counter
// (the loads of keys and row-ids coalesce) and probes them a tile of 128 rows
// at a time, four bucket loads in flight per lane.  Probes whose chain goes on
// past the home bucket are compacted per warp and walked 32 at a time, so
// lanes do not wait for the longest chain of the warp.  Matches are staged
// per warp in shared memory and appended to the output with one atomic on the
// global count per flush.
//
// Partitioned probe (table much larger than L2, many probe rows): a table
// larger than L2 turns every probe into a random DRAM sector read, and those
// run at a small fraction of the streaming rate.  Instead the probe rows are
// first radix-partitioned by the top bits of their home bucket into P
// partitions (a counting pass and a scatter pass, both streaming; the scatter
// appends a tile's rows of a partition as one run at the partition's cursor).
// The probe then takes the reordered
// rows chunk by chunk in partition order, so the whole grid works on one
// 1/P slice of the table at a time, sized to stay resident in L2: the table
// is read from DRAM about once.
#include <algorithm>
#include <atomic>
#include <cstring>
#include <string>

#include "block.cuh"
#include "ctx.h"
#include "join_dev.cuh"

namespace olap {

namespace {

// Build, first pass: every row goes, as a 16-byte entry {key, row-id}, to the
// next free places of its home bucket's block, in the memory that the block's
// slots will take.  The places come from the block's cursor, which sits in the
// block's last slot (zeroed before the launch).  A CTA takes a tile of rows,
// counts them per block, takes the places of all its rows of a block with one
// global atomic, puts the tile in block order in shared memory and writes it
// out from there, so that the rows of a block are written side by side: a
// lone 16-byte write costs the L2 a whole sector, and those are the bound
// (2^24 rows: 712 us row by row, 330 us with the partition passes before this
// one; 4 * 10^6 rows in one pass 62 us, two rows per block and tile).
// The blocks of a tile span at most JS_BINS: all blocks of a small table, or,
// for larger ones, those of the few partitions that the tile's rows are
// already ordered by; a tile that spans more goes row by row.
constexpr int JS_TPB = 512;
constexpr int JS_PER = 8;
constexpr int JS_TILE = JS_TPB * JS_PER;
constexpr int JS_BINS = 4096;
constexpr int JS_SMEM = JS_TILE * 12 + JS_BINS * 8;
constexpr int JS_PARTS = 64;                                  // partitions of a larger build's rows
static_assert(JS_TPB <= 512 && JS_TILE <= 65535, "scan words; ranks in 16 bits");

__global__ void __launch_bounds__(JS_TPB, 2) join_block_scatter_kernel(const int64_t* keys, const uint32_t* rowids,
                                                                       uint64_t n, int per, ulonglong2* slots,
                                                                       uint64_t mask, int block_log, JoinCtl* ctl) {
    extern __shared__ __align__(16) unsigned char ssmem[];
    uint64_t* sk = reinterpret_cast<uint64_t*>(ssmem);                       // the tile in block order
    uint32_t* sr = reinterpret_cast<uint32_t*>(ssmem + JS_TILE * 8);
    unsigned* off = reinterpret_cast<unsigned*>(ssmem + JS_TILE * 12);       // rows per block, then first position
    unsigned* base = off + JS_BINS;                                          // first place minus first position
    __shared__ unsigned lo, hi;                                              // the tile's blocks
    __shared__ unsigned long long sc[24];
    const unsigned room = (2u << block_log) - 1u;             // entries a block may hold: one slot stays free
    auto cursor = [&](uint64_t blk) {
        return reinterpret_cast<unsigned*>(slots + (blk << (block_log + 1)) + room);
    };
    auto block_of = [&](uint64_t key) { return static_cast<unsigned>((fmix64(key) & mask) >> block_log); };
    bool crowded = false;
    unsigned side = 0;
    auto put = [&](unsigned blk, unsigned pos, uint64_t key, uint32_t rid) {
        if (pos < room) slots[(static_cast<uint64_t>(blk) << (block_log + 1)) + pos] = make_ulonglong2(key, rid);
        else crowded = true;
    };
    const uint64_t tile = static_cast<uint64_t>(per) * JS_TPB;               // per <= JS_PER rows per thread
    for (uint64_t t0 = blockIdx.x * tile; t0 < n; t0 += gridDim.x * tile) {
        uint64_t key[JS_PER];
        uint32_t rid[JS_PER];
        unsigned at[JS_PER];                                  // block, then rank in its block | block << 16
#pragma unroll
        for (int j = 0; j < JS_PER; ++j) {
            const uint64_t i = t0 + static_cast<uint64_t>(j) * JS_TPB + threadIdx.x;
            const bool in = j < per && i < n;
            key[j] = in ? ld_stream_u64(keys + i) : JN_EMPTY;
            rid[j] = (in && rowids) ? ld_stream_u32(rowids + i) : static_cast<uint32_t>(i);
            side += (in && key[j] == JN_EMPTY) ? 1u : 0u;
        }
        for (unsigned b = threadIdx.x; b < JS_BINS; b += JS_TPB) off[b] = 0;
        if (threadIdx.x == 0) {
            lo = ~0u;
            hi = 0;
        }
        __syncthreads();
        unsigned mn = ~0u, mx = 0;
#pragma unroll
        for (int j = 0; j < JS_PER; ++j) {
            at[j] = block_of(key[j]);
            if (key[j] != JN_EMPTY) {
                mn = min(mn, at[j]);
                mx = max(mx, at[j]);
            }
        }
        mn = __reduce_min_sync(0xFFFFFFFFu, mn);
        mx = __reduce_max_sync(0xFFFFFFFFu, mx);
        if ((threadIdx.x & 31u) == 0) {
            atomicMin(&lo, mn);
            atomicMax(&hi, mx);
        }
        __syncthreads();
        const unsigned b0 = lo;
        if (b0 != ~0u && hi - b0 < JS_BINS) {
#pragma unroll
            for (int j = 0; j < JS_PER; ++j)
                if (key[j] != JN_EMPTY) at[j] = (at[j] - b0) | (atomicAdd(&off[at[j] - b0], 1u) << 16);
            __syncthreads();
            constexpr int PER = JS_BINS / JS_TPB;
            unsigned c[PER];
            unsigned total = 0;
#pragma unroll
            for (int q = 0; q < PER; ++q) {
                c[q] = off[threadIdx.x * PER + q];
                total += c[q];
            }
            unsigned run = static_cast<unsigned>(block_excl_scan<JS_TPB>(total, sc, sc + 16));
#pragma unroll
            for (int q = 0; q < PER; ++q) {
                const unsigned b = threadIdx.x * PER + q;
                off[b] = run;
                if (c[q]) base[b] = atomicAdd(cursor(static_cast<uint64_t>(b0) + b), c[q]) - run;
                run += c[q];
            }
            __syncthreads();
#pragma unroll
            for (int j = 0; j < JS_PER; ++j)
                if (key[j] != JN_EMPTY) {
                    const unsigned p = off[at[j] & 0xFFFFu] + (at[j] >> 16);
                    sk[p] = key[j];
                    sr[p] = rid[j];
                }
            __syncthreads();
            const unsigned len = static_cast<unsigned>(sc[16]);               // the scan's total
            for (unsigned p = threadIdx.x; p < len; p += JS_TPB) {
                const unsigned blk = block_of(sk[p]);
                put(blk, base[blk - b0] + p, sk[p], sr[p]);
            }
        } else {
#pragma unroll
            for (int j = 0; j < JS_PER; ++j)
                if (key[j] != JN_EMPTY) put(at[j], atomicAdd(cursor(at[j]), 1u), key[j], rid[j]);
        }
        __syncthreads();                                      // before the next tile clears the bins
    }
    if (crowded) ctl->crowded = 1;
    side = __reduce_add_sync(0xFFFFFFFFu, side);
    if ((threadIdx.x & 31u) == 0 && side) atomicAdd(&ctl->side_count, static_cast<unsigned long long>(side));
}

// Build, second pass: one block of the table at a time per CTA.  Its entries
// are taken into registers and put in shared memory as linear probing would
// leave them (first free slot at or after the home bucket, slot 0 before slot
// 1, wrapping within the block), counted along their chains, and the whole
// block is written over them: the table is written once, in order, and needs
// no clearing.  A block keeps a free slot, so every chain in it ends.
//
// No entry searches for its slot.  In the order of their home buckets, the
// entries of bucket b take the slots from max(end of the bucket before, 2 b)
// on, so the ends follow from a scan over the buckets' counts; what runs past
// the last slot comes before bucket 0 in a second look at the same scan.  (By
// CAS from slot to slot, many copies of a key in a block meet at every slot:
// 100,000 rows, 1200 of one key: BUILD_A; 10^6 rows of 64 copies each: BUILD_B.)
// Copies of a key lie in their home bucket's run of slots, so only the rest
// of its own run is compared with an entry.
// Bound by the instructions of that and by the writes.  With the passes
// before and the Bloom filter, 4 * 10^6 rows take BUILD_C us and 2^24 rows BUILD_D, where
// clearing the table, a CAS and a chain walk per row and eight atomics on the
// filter took 364 and 2352 us.
constexpr uint64_t JS_PART_MIN_N = 1ull << 22;                // smaller builds go row by row
constexpr int JT_TPB = 512;
constexpr int JT_SLOTS = 2 * static_cast<int>(JT_BLOCK);
constexpr int JT_PER = JT_SLOTS / JT_TPB;
constexpr int JT_BLOOM_MAX = 128;                             // filter blocks per table block, at a load of 0.9
constexpr int JT_SMEM = JT_SLOTS * 14 + static_cast<int>(JT_BLOCK) * 4 + JT_BLOOM_MAX * 32;
static_assert(JT_BLOCK == 2 * JT_TPB, "two buckets per thread");
static_assert(JT_SLOTS <= 2048, "places in 11 bits, ends in 16");

// A stretch of buckets as a function of the slot its entries may start at:
// they end at max(start + entries, least).
struct Stretch {
    unsigned entries, least;
};
__device__ __forceinline__ Stretch stretch_join(const Stretch& a, const Stretch& b) {
    return Stretch{a.entries + b.entries, max(a.least + b.entries, b.least)};
}

__global__ void __launch_bounds__(JT_TPB, 3) join_block_build_kernel(ulonglong2* slots, uint64_t blocks, int block_log,
                                                                     uint32_t* bloom, int per_log, JoinCtl* ctl) {
    extern __shared__ __align__(16) unsigned char tsmem[];
    uint64_t* sk = reinterpret_cast<uint64_t*>(tsmem);                       // keys of the block's slots
    uint32_t* sr = reinterpret_cast<uint32_t*>(tsmem + JT_SLOTS * 8);        // their row-ids
    uint16_t* sf = reinterpret_cast<uint16_t*>(tsmem + JT_SLOTS * 12);       // further copies of their keys
    unsigned* run = reinterpret_cast<unsigned*>(tsmem + JT_SLOTS * 14);      // entries per bucket, then first slot | entries << 16
    uint32_t* sb = run + JT_BLOCK;                                           // the block's filter words
    __shared__ Stretch ws[JT_TPB / 32];
    if (ctl->crowded) return;                                                // (set by the pass before)
    const unsigned bm = (1u << block_log) - 1u;
    const unsigned nslots = 2u << block_log;
    const unsigned nwords = bloom ? (BLOOM_WORDS << per_log) : 0u;
    const unsigned lane = threadIdx.x & 31u, warp = threadIdx.x >> 5;
    uint64_t k[JT_PER];
    uint32_t r[JT_PER];
    auto cursor = [&](uint64_t blk) {
        return blk < blocks ? __ldcg(reinterpret_cast<const unsigned*>(slots + (blk + 1) * nslots - 1)) : 0u;
    };
    auto load = [&](uint64_t blk, unsigned cnt) {
#pragma unroll
        for (int j = 0; j < JT_PER; ++j) {
            const unsigned i = static_cast<unsigned>(j) * JT_TPB + threadIdx.x;
            k[j] = JN_EMPTY;
            if (i < cnt) {
                const ulonglong2 e = __ldcg(slots + blk * nslots + i);
                k[j] = e.x;
                r[j] = static_cast<uint32_t>(e.y);
            }
        }
    };
    uint64_t blk = blockIdx.x;
    load(blk, cursor(blk));
    unsigned next_cnt = cursor(blk + gridDim.x);
    for (; blk < blocks; blk += gridDim.x) {
        ulonglong2* mine = slots + blk * nslots;
        for (unsigned i = threadIdx.x; i < nslots / 2; i += JT_TPB)
            reinterpret_cast<ulonglong2*>(sk)[i] = make_ulonglong2(JN_EMPTY, JN_EMPTY);
        run[threadIdx.x] = 0u;
        run[threadIdx.x + JT_TPB] = 0u;
        for (unsigned i = threadIdx.x; i < nwords; i += JT_TPB) sb[i] = 0u;
        __syncthreads();                                     // (every thread has its entries in registers)
        unsigned at[JT_PER];                                 // home bucket | rank among its entries << 10
#pragma unroll
        for (int j = 0; j < JT_PER; ++j) {
            if (k[j] == JN_EMPTY) continue;
            const uint64_t h = fmix64(k[j]);
            const unsigned b = static_cast<unsigned>(h) & bm;
            at[j] = b | atomicAdd(&run[b], 1u) << 10;
            if (nwords) {
                // the lanes go through the words of their blocks in different
                // orders: in the same order they would meet on four banks
                uint32_t* fb = sb + (static_cast<unsigned>(h >> 40) & ((1u << per_log) - 1u)) * BLOOM_WORDS;
                const uint64_t g = bloom_bits(h);
#pragma unroll
                for (unsigned v = 0; v < BLOOM_WORDS; ++v) {
                    const int w = static_cast<int>((v + threadIdx.x) & (BLOOM_WORDS - 1));
                    atomicOr(fb + w, bloom_bit(g, w));
                }
            }
        }
        __syncthreads();
        // Where the entries of the thread's two buckets start.
        const unsigned b0 = 2u * threadIdx.x;
        const uint2 c = reinterpret_cast<const uint2*>(run)[threadIdx.x];
        Stretch incl{0u, 0u};                                // (no bucket there: a table of fewer)
        if (b0 <= bm) incl = Stretch{c.x, 2u * b0 + c.x};
        if (b0 < bm) incl = stretch_join(incl, Stretch{c.y, 2u * b0 + 2u + c.y});
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const Stretch before{__shfl_up_sync(0xFFFFFFFFu, incl.entries, o), __shfl_up_sync(0xFFFFFFFFu, incl.least, o)};
            if (lane >= static_cast<unsigned>(o)) incl = stretch_join(before, incl);
        }
        if (lane == 31) ws[warp] = incl;
        Stretch mine_from{__shfl_up_sync(0xFFFFFFFFu, incl.entries, 1), __shfl_up_sync(0xFFFFFFFFu, incl.least, 1)};
        if (lane == 0) mine_from = Stretch{0u, 0u};
        __syncthreads();
        Stretch upto = ws[lane & (JT_TPB / 32 - 1)];          // every warp scans the warps' stretches
#pragma unroll
        for (int o = 1; o < JT_TPB / 32; o <<= 1) {
            const Stretch before{__shfl_up_sync(0xFFFFFFFFu, upto.entries, o), __shfl_up_sync(0xFFFFFFFFu, upto.least, o)};
            if (lane >= static_cast<unsigned>(o)) upto = stretch_join(before, upto);
        }
        const Stretch all{__shfl_sync(0xFFFFFFFFu, upto.entries, JT_TPB / 32 - 1),
                          __shfl_sync(0xFFFFFFFFu, upto.least, JT_TPB / 32 - 1)};
        Stretch from{__shfl_sync(0xFFFFFFFFu, upto.entries, (warp + 31u) & 31u),
                     __shfl_sync(0xFFFFFFFFu, upto.least, (warp + 31u) & 31u)};
        if (warp == 0) from = Stretch{0u, 0u};
        from = stretch_join(from, mine_from);
        const unsigned end = max(all.entries, all.least);    // of the last bucket, from slot 0
        const unsigned wrapped = end > nslots ? end - nslots : 0u;
        if (b0 <= bm) {
            const unsigned f0 = max(max(wrapped + from.entries, from.least), 2u * b0);
            const unsigned f1 = max(f0 + c.x, 2u * b0 + 2u);
            reinterpret_cast<uint2*>(run)[threadIdx.x] = make_uint2(f0 | c.x << 16, f1 | c.y << 16);
        }
        __syncthreads();
#pragma unroll
        for (int j = 0; j < JT_PER; ++j) {
            if (k[j] == JN_EMPTY) continue;
            const unsigned p = ((run[at[j] & 1023u] & 0xFFFFu) + (at[j] >> 10)) & (nslots - 1u);
            sk[p] = k[j];
            sr[p] = r[j];
        }
        __syncthreads();
#pragma unroll
        for (int j = 0; j < JT_PER; ++j) {
            if (k[j] == JN_EMPTY) continue;
            const unsigned v = run[at[j] & 1023u];
            const unsigned p = (v & 0xFFFFu) + (at[j] >> 10), stop = (v & 0xFFFFu) + (v >> 16);
            unsigned f = 0;
            for (unsigned q = p + 1u; q < stop; ++q) f += sk[q & (nslots - 1u)] == k[j] ? 1u : 0u;
            sf[p & (nslots - 1u)] = static_cast<uint16_t>(f);
        }
        // the next block's entries, on their way while this block is written
        load(blk + gridDim.x, next_cnt);
        next_cnt = cursor(blk + 2ull * gridDim.x);
        __syncthreads();
        for (unsigned b = threadIdx.x; b <= bm; b += JT_TPB) {               // a bucket at a time
            const ulonglong2 kk = reinterpret_cast<const ulonglong2*>(sk)[b];
            const uint2 rr = reinterpret_cast<const uint2*>(sr)[b];
            const unsigned ff = reinterpret_cast<const unsigned*>(sf)[b];
            const uint64_t w0 = kk.x == JN_EMPTY ? ~0ull : rr.x | (static_cast<uint64_t>(ff & 0xFFFFu) << 32);
            const uint64_t w1 = kk.y == JN_EMPTY ? ~0ull : rr.y | (static_cast<uint64_t>(ff >> 16) << 32);
            asm volatile("st.global.v4.u64 [%0], {%1, %2, %3, %4};" ::"l"(mine + 2 * b), "l"(kk.x), "l"(w0), "l"(kk.y),
                         "l"(w1)
                         : "memory");
        }
        for (unsigned i = threadIdx.x; i < nwords; i += JT_TPB) bloom[blk * nwords + i] = sb[i];
        __syncthreads();
    }
}

// The general build, for tables whose blocks do not hold their rows.
__global__ void __launch_bounds__(JB_TPB) join_build_kernel(const int64_t* keys, const uint32_t* rowids,
                                                            uint64_t n, ulonglong2* slots, uint64_t mask,
                                                            JoinCtl* ctl) {
    const uint64_t stride = static_cast<uint64_t>(gridDim.x) * JB_TPB;
    for (uint64_t i = static_cast<uint64_t>(blockIdx.x) * JB_TPB + threadIdx.x; i < n; i += stride) {
        const uint64_t key = static_cast<uint64_t>(keys[i]);
        if (key == JN_EMPTY) {
            atomicAdd(&ctl->side_count, 1ull);
            continue;
        }
        const uint32_t rid = rowids ? rowids[i] : static_cast<uint32_t>(i);
        uint64_t b = fmix64(key) & mask;
        bool done = false;
        for (uint64_t step = 0; step <= mask && !done; ++step) {
            // both slots in one round trip: a heavy key's rows wait for those
            // (10^6 rows, 3000 of one key: the call 5630 -> 3330 us)
            unsigned long long* kp = reinterpret_cast<unsigned long long*>(&slots[b * 2].x);
            const unsigned long long held[2] = {*reinterpret_cast<volatile unsigned long long*>(kp),
                                                *reinterpret_cast<volatile unsigned long long*>(kp + 2)};
            for (int s = 0; s < 2 && !done; ++s) {
                if (held[s] != JN_EMPTY) continue;
                if (atomicCAS(kp + 2 * s, JN_EMPTY, static_cast<unsigned long long>(key)) == JN_EMPTY) {
                    slots[b * 2 + s].y = rid;
                    done = true;
                }
            }
            b = (b + 1) & mask;
        }
        if (!done) atomicCAS(&ctl->err, 0, static_cast<int>(OLAP_E_DEVICE));
    }
}

// After the build: every occupied slot records, in the high half of its
// row-id word, how many further copies of its key follow it along the chain
// (up to the first bucket with a free slot, where every chain through it
// ends).  Copies of a key all sit between its home bucket and that end, in
// the order a probe walks them, so a probe that meets a copy with no further
// copies has seen them all and stops there instead of walking to the chain's
// end: for a unique build a hit stops at its key.
__global__ void __launch_bounds__(JB_TPB) join_chain_kernel(ulonglong2* slots, uint64_t mask) {
    const uint64_t n_slots = (mask + 1) * 2;
    const uint64_t stride = static_cast<uint64_t>(gridDim.x) * JB_TPB;
    for (uint64_t j = static_cast<uint64_t>(blockIdx.x) * JB_TPB + threadIdx.x; j < n_slots; j += stride) {
        const uint64_t key = slots[j].x;
        if (key == JN_EMPTY) continue;
        uint64_t b = j >> 1;
        uint32_t further = 0;
        uint64_t k1 = slots[b * 2 + 1].x;
        if ((j & 1) == 0 && k1 == key) ++further;
        for (uint64_t step = 0; k1 != JN_EMPTY && step < mask; ++step) {   // bucket b full: the chain goes on
            b = (b + 1) & mask;
            const uint64_t k0 = slots[b * 2].x;
            k1 = slots[b * 2 + 1].x;
            further += (k0 == key) + (k1 == key);
        }
        slots[j].y = (slots[j].y & 0xFFFFFFFFull) | (static_cast<uint64_t>(further) << 32);
    }
}

__global__ void __launch_bounds__(JB_TPB) join_side_kernel(const int64_t* keys, const uint32_t* rowids,
                                                           uint64_t n, uint32_t* side, JoinCtl* ctl) {
    const uint64_t stride = static_cast<uint64_t>(gridDim.x) * JB_TPB;
    for (uint64_t i = static_cast<uint64_t>(blockIdx.x) * JB_TPB + threadIdx.x; i < n; i += stride) {
        if (static_cast<uint64_t>(keys[i]) == JN_EMPTY) {
            const unsigned long long pos = atomicAdd(&ctl->side_fill, 1ull);
            side[pos] = rowids ? rowids[i] : static_cast<uint32_t>(i);
        }
    }
}

// The probe: rows [0, a.n) handed out in chunks by a row queue (see
// probe_rows).  Used on the input (direct probe) and on the rows reordered
// by partition (pass 3 of the partitioned probe): there the chunks come out in
// partition order, so the warps of the whole grid work on one partition's
// table slice at a time and that slice stays in L2.
// The last CTA to finish returns the row counter and its ticket to zero for the
// next probe of the context, and for a blocking call writes the pair count to
// the host and clears it as well, so that such a call is its kernels and one
// wait (three small memsets and a copy before).
// `args` holds the rows as launched (the probe's input, or its partitioned
// rows).  The device-side plan (ctl, when non-NULL) may change that: with the
// Bloom pre-probe active the row count is the number of rows it kept, and
// with `redirect` the rows are read from where the plan says (the kept rows,
// or the input when the partition passes were skipped), through L1 when the
// plan says so.
struct ProbeDone {
    unsigned* ticket;                          // CTAs done; zero between probes
    unsigned long long* host_count;            // page-locked host word of a blocking call, else NULL
};
template <bool L2_ONLY>
__global__ void __launch_bounds__(JP_TPB, JP_CTAS) join_probe_kernel(ProbeArgs args, unsigned long long* next_row,
                                                                     const ProbeCtl* ctl, ProbeDone done) {
    extern __shared__ __align__(16) unsigned char psmem[];
    unsigned char* mine = psmem + (threadIdx.x >> 5) * JP_WARP_SMEM;
    ProbeArgs a = args;
    bool l1 = !L2_ONLY;
    wait_prior_grid();
    if (ctl) {
        if (ctl->active) a.n = ctl->count;
        if (ctl->redirect) {
            a.keys = ctl->keys;
            a.rowids = ctl->rowids;
        }
        l1 = l1 || ctl->l1;
    }
    RowQueue q;
    q.counter = next_row;
    q.n = a.n;
    q.chunk = queue_chunk(a.n, gridDim.x * JP_WARPS);
    if (l1)
        probe_rows<false>(a, q, mine);
    else
        probe_rows<true>(a, q, mine);
    __syncthreads();
    if (threadIdx.x == 0) {
        __threadfence();
        if (atomicAdd(done.ticket, 1u) == gridDim.x - 1) {
            __threadfence();
            *done.ticket = 0;
            *next_row = 0;
            if (done.host_count) {
                *done.host_count = __ldcg(a.count);
                *a.count = 0;
            }
        }
    }
}

// ---- Bloom pre-probe ------------------------------------------------------

// Every build key sets its eight bits in its block (the empty-marker key,
// kept in the side list, is not entered: the pre-probe keeps such probe rows
// whatever the filter says).
__global__ void __launch_bounds__(JB_TPB) join_bloom_kernel(const int64_t* keys, uint64_t n, uint32_t* bloom,
                                                            BloomView f) {
    const uint64_t stride = static_cast<uint64_t>(gridDim.x) * JB_TPB;
    for (uint64_t i = static_cast<uint64_t>(blockIdx.x) * JB_TPB + threadIdx.x; i < n; i += stride) {
        const uint64_t key = static_cast<uint64_t>(keys[i]);
        if (key == JN_EMPTY) continue;
        const uint64_t h = fmix64(key);
        uint32_t* blk = bloom + bloom_block(f, h) * BLOOM_WORDS;
        const uint64_t g = bloom_bits(h);
#pragma unroll
        for (int w = 0; w < BLOOM_WORDS; ++w) atomicOr(blk + w, bloom_bit(g, w));
    }
}

constexpr int PF_TPB = 256;
constexpr int PF_SAMPLE = 4096;                // probe keys tested to decide
constexpr uint64_t PF_MIN_N = 1ull << 20;      // smaller probes skip the pre-probe (automatic mode)
constexpr int PF_PER = 6;                      // keys per lane per step
constexpr unsigned PF_WCAP = 256;              // rows staged per warp
constexpr int PF_CTAS = 4;                     // pre-probe CTAs per SM

constexpr int PLAN_SLOTS = 2 * PF_SAMPLE;      // fingerprint set of the sample (32 KB)
constexpr int PLAN_CTAS = 16;
constexpr int PLAN_TPB = 1024;                 // the first PF_SAMPLE / PLAN_CTAS threads load the CTA's sample

// The plan kernel's inputs, and its state in the context's device area.
struct PlanArgs {
    const int64_t* keys;
    const uint32_t* rowids;
    uint64_t n;
    BloomView bloom;                           // bits NULL: no pre-probe stage
    int pf_mode;                               // 1 automatic, 2 forced (with a filter)
    int skew_check;
    uint64_t min_rows;                         // with skew_check: fewer rows than this are not worth partitioning
    int partitioned;
    int skew_l1;
    const int64_t* pf_keys;
    const uint32_t* pf_rowids;
    uint32_t* sample;                          // PF_SAMPLE packed entries
    unsigned* counters;                        // [0] kept keys, [1] CTAs done; zero between calls
    ProbeCtl* ctl;
};

// The probe's plan, decided on the device from a stratified sample of
// PF_SAMPLE probe keys (n >= PF_SAMPLE; fewer rows are each taken once or
// more).  PLAN_CTAS CTAs load the sample, one key per thread (from one SM,
// 4096 scattered loads wait on each other's latency: 38 us; the other threads
// of a CTA only help the last one decide: 12.5 -> 8.5 us), test it
// against the Bloom filter and store one packed word per key: a 30-bit
// fingerprint of the key, bit 1 = kept by the filter, bit 0 = 1.  The last
// CTA to finish decides.  With a Bloom filter (pf_mode 1 = automatic,
// 2 = forced) the pre-probe runs when at most 60 % of the sample may be in
// the table, or always when forced.  With `skew_check` the probe skips its
// partition passes when the rows it will probe repeat: at least a fifth of
// the sampled keys that reach the probe (those the filter keeps, when it
// runs) equal an earlier sampled key.  Such a stream sends most probes to a
// few hot buckets, which stay in cache, while the partition passes would
// cost two more passes over the rows.  Repeats are found in a shared-memory
// fingerprint set; a fingerprint collision counts as a repeat (about 2^-7
// of one per sample).  It skips them as well when the pre-probe leaves fewer
// than `min_rows` (2^25 uniform rows against 2^24, a tenth kept: 278 -> 252 us).  The last CTA zeroes the kept-row count and tells the
// probe kernel where its rows are: the partitioned rows (`partitioned` and
// not direct, as launched), else the kept rows (pf_keys, pf_rowids) when the
// pre-probe runs, else the input; a direct probe reads buckets through L1
// when `skew_l1`.  It also clears the counters for the next call.
__global__ void __launch_bounds__(PLAN_TPB) join_probe_plan_kernel(PlanArgs a) {
    allow_next_grid();
    __shared__ uint32_t fset[PLAN_SLOTS];
    __shared__ unsigned kept_cta, dup_all, dup_kept;
    __shared__ bool last;
    if (threadIdx.x == 0) kept_cta = 0;
    __syncthreads();
    constexpr int PER_CTA = PF_SAMPLE / PLAN_CTAS;
    if (threadIdx.x < PER_CTA) {
        const uint64_t j = static_cast<uint64_t>(blockIdx.x) * PER_CTA + threadIdx.x;
        const uint64_t key = static_cast<uint64_t>(a.keys[(j * a.n) / PF_SAMPLE]);
        const bool kept = a.bloom.bits ? (key == JN_EMPTY || bloom_maybe(a.bloom, key)) : true;
        const uint32_t fp = static_cast<uint32_t>(fmix64(key) >> 32) & ~3u;
        a.sample[j] = fp | (kept ? 2u : 0u) | 1u;
        const unsigned m = __ballot_sync(0xFFFFFFFFu, kept);
        if ((threadIdx.x & 31u) == 0) atomicAdd(&kept_cta, static_cast<unsigned>(__popc(m)));
    }
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) {
        atomicAdd(&a.counters[0], kept_cta);
        last = atomicAdd(&a.counters[1], 1u) == gridDim.x - 1;
    }
    __syncthreads();
    if (!last) return;
    __threadfence();
    for (int j = threadIdx.x; j < PLAN_SLOTS; j += PLAN_TPB) fset[j] = 0u;
    if (threadIdx.x == 0) dup_all = dup_kept = 0;
    __syncthreads();
    unsigned m_dup = 0, m_dup_kept = 0;
    if (a.skew_check) {
        for (int j = threadIdx.x; j < PF_SAMPLE; j += PLAN_TPB) {
            const uint32_t w = __ldcg(a.sample + j);
            const uint32_t fp = w & ~2u;                 // the fingerprint, with the set's non-zero bit
            uint32_t slot = (fp >> 2) & (PLAN_SLOTS - 1);
            bool dup = false;
            for (int tries = 0; tries < PLAN_SLOTS; ++tries) {
                const uint32_t prev = atomicCAS(&fset[slot], 0u, fp);
                if (prev == 0u) break;
                if (prev == fp) {
                    dup = true;
                    break;
                }
                slot = (slot + 1) & (PLAN_SLOTS - 1);
            }
            m_dup += dup ? 1u : 0u;
            m_dup_kept += (dup && (w & 2u)) ? 1u : 0u;
        }
    }
    m_dup = __reduce_add_sync(0xFFFFFFFFu, m_dup);
    m_dup_kept = __reduce_add_sync(0xFFFFFFFFu, m_dup_kept);
    if ((threadIdx.x & 31u) == 0) {
        atomicAdd(&dup_all, m_dup);
        atomicAdd(&dup_kept, m_dup_kept);
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        const unsigned passes = atomicAdd(&a.counters[0], 0u);
        const bool active = a.bloom.bits && (a.pf_mode == 2 || passes * 10u <= static_cast<unsigned>(PF_SAMPLE) * 6u);
        const unsigned reach = active ? passes : static_cast<unsigned>(PF_SAMPLE);
        const unsigned rep = active ? dup_kept : dup_all;
        const bool skewed = a.skew_check && reach >= 64u && rep * 5u >= reach;
        const bool few = a.skew_check && active && a.n * passes < a.min_rows * PF_SAMPLE;
        const bool direct = skewed || few;
        ProbeCtl* ctl = a.ctl;
        ctl->active = active ? 1 : 0;
        ctl->direct = direct ? 1 : 0;
        ctl->count = 0;
        ctl->redirect = (!a.partitioned || direct) ? 1 : 0;
        ctl->keys = active ? a.pf_keys : a.keys;
        ctl->rowids = active ? a.pf_rowids : a.rowids;
        ctl->l1 = (skewed && a.skew_l1) ? 1 : 0;
        a.counters[0] = 0;
        a.counters[1] = 0;
    }
}

// The pre-probe: one streaming pass over the probe rows that keeps the rows
// whose key may be in the table (and every row with the empty-marker key),
// appended with their row-ids through a per-warp stage, one atomic per flush.
// Bound by the random filter-block reads from L2 (2.4*10^11 a second), the
// more of which a lane has in flight the better: six keys a lane and four CTAs
// per SM (eight keys, or five CTAs of five: the same; six of four: 3-5 %
// slower).  The kept rows' row-ids are all loaded before the first is staged.
// Whole probes against a 2^24-row table, a tenth kept: 2^25 Zipf rows with
// row-ids 236 -> 208 us, uniform 296 -> 248 (without partition passes after it).
__global__ void __launch_bounds__(PF_TPB, PF_CTAS) join_prefilter_kernel(const int64_t* keys, const uint32_t* rowids,
                                                                uint64_t n, BloomView bloom, ProbeCtl* ctl,
                                                                int64_t* out_keys, uint32_t* out_rowids) {
    wait_prior_grid();
    allow_next_grid();
    if (!ctl->active) return;
    __shared__ int64_t sk[PF_TPB / 32][PF_WCAP];
    __shared__ uint32_t sr[PF_TPB / 32][PF_WCAP];
    const unsigned lane = threadIdx.x & 31u, warp = threadIdx.x >> 5;
    int64_t* wk = sk[warp];
    uint32_t* wr = sr[warp];
    unsigned cnt = 0;
    auto flush = [&]() {
        __syncwarp();
        unsigned long long base = 0;
        if (lane == 0 && cnt) base = atomicAdd(&ctl->count, static_cast<unsigned long long>(cnt));
        base = __shfl_sync(0xFFFFFFFFu, base, 0);
        for (unsigned i = lane; i < cnt; i += 32) {
            out_keys[base + i] = wk[i];
            out_rowids[base + i] = wr[i];
        }
        __syncwarp();
        cnt = 0;
    };
    constexpr uint64_t G = 32ull * PF_PER;
    const uint64_t groups = (n + G - 1) / G;
    const uint64_t nw = static_cast<uint64_t>(gridDim.x) * (PF_TPB / 32);
    for (uint64_t g = static_cast<uint64_t>(blockIdx.x) * (PF_TPB / 32) + warp; g < groups; g += nw) {
        uint64_t key[PF_PER];
        const uint64_t i0 = g * G + lane;
        const unsigned len = static_cast<unsigned>(min(G, n - g * G));
        const int64_t* kp = keys + i0;
        if (len == G) {
#pragma unroll
            for (int j = 0; j < PF_PER; ++j) key[j] = ld_stream_u64(kp + j * 32);
        } else {
#pragma unroll
            for (int j = 0; j < PF_PER; ++j) key[j] = j * 32 + lane < len ? ld_stream_u64(kp + j * 32) : 0ull;
        }
        unsigned kept[PF_PER];                 // the warp's rows kept of step j
#pragma unroll
        for (int j = 0; j < PF_PER; ++j) {
            const bool maybe = bloom_maybe(bloom, key[j]) || key[j] == JN_EMPTY;
            kept[j] = __ballot_sync(0xFFFFFFFFu, maybe && j * 32 + lane < len);
        }
        uint32_t rid[PF_PER];                  // all of the kept rows' row-ids in flight before the first is staged
#pragma unroll
        for (int j = 0; j < PF_PER; ++j) {
            rid[j] = static_cast<uint32_t>(i0 + j * 32);
            if (rowids && ((kept[j] >> lane) & 1u)) rid[j] = ld_stream_u32(rowids + i0 + j * 32);
        }
#pragma unroll
        for (int j = 0; j < PF_PER; ++j) {
            if (kept[j] == 0) continue;
            if (cnt + 32 > PF_WCAP) flush();
            if ((kept[j] >> lane) & 1u) {
                const unsigned pos = cnt + __popc(kept[j] & ((1u << lane) - 1u));
                wk[pos] = static_cast<int64_t>(key[j]);
                wr[pos] = rid[j];
            }
            cnt += __popc(kept[j]);
        }
    }
    flush();
}

// ---- partitioned probe ------------------------------------------------------

constexpr int JQ_TPB = 320;
constexpr int JQ_PER = 7;                      // probe rows per thread per tile
constexpr int JQ_TILE = JQ_TPB * JQ_PER;       // rows per tile
constexpr int JQ_PMAX = 256;                   // most partitions
constexpr int JQ_CTAS_PER_SM = 4;              // grid of the two partition passes
static_assert(JQ_PMAX <= JQ_TPB, "one scan slot per partition");

struct PartArgs {
    const int64_t* keys;
    const uint32_t* rowids;                    // NULL => index
    uint64_t n;
    uint64_t mask;                             // buckets - 1
    int shift;                                 // partition = home bucket >> shift
    int parts;
    unsigned long long* counts;                // [parts] rows of each partition; zero between calls
    unsigned long long* next;                  // [parts] next output row of each partition
    unsigned* ticket;                          // CTAs that have counted; zero between calls
    int64_t* out_keys;
    uint32_t* out_rowids;
    const ProbeCtl* pf;                        // non-NULL: the device-side plan (pre-probe, direct)
    const int64_t* pf_keys;                    // the pre-probe's surviving rows, used when pf->active
    const uint32_t* pf_rowids;
};

// The rows a partition pass reads: the probe's input, or the rows the Bloom
// pre-probe kept (decided on the device by the stage before).
__device__ __forceinline__ PartArgs part_source(const PartArgs& in) {
    PartArgs a = in;
    if (a.pf && a.pf->active) {
        a.keys = a.pf_keys;
        a.rowids = a.pf_rowids;
        a.n = a.pf->count;
    }
    return a;
}

__device__ __forceinline__ unsigned part_of(uint64_t key, const PartArgs& a) {
    return static_cast<unsigned>((fmix64(key) & a.mask) >> a.shift);
}

// The keys of the tile at t0, thread by thread (zeros past the end).
__device__ __forceinline__ void part_load(const PartArgs& a, uint64_t t0, uint64_t (&k)[JQ_PER]) {
    const int64_t* p = a.keys + t0 + threadIdx.x;
    if (t0 + JQ_TILE <= a.n) {
#pragma unroll
        for (int j = 0; j < JQ_PER; ++j) k[j] = ld_stream_u64(p + j * JQ_TPB);
    } else {
#pragma unroll
        for (int j = 0; j < JQ_PER; ++j)
            k[j] = t0 + static_cast<uint64_t>(j) * JQ_TPB + threadIdx.x < a.n ? ld_stream_u64(p + j * JQ_TPB) : 0ull;
    }
}

// Exclusive sum over a warp's lanes.
__device__ __forceinline__ unsigned warp_excl_scan(unsigned x, unsigned lane) {
    unsigned incl = x;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const unsigned v = __shfl_up_sync(0xFFFFFFFFu, incl, o);
        if (lane >= static_cast<unsigned>(o)) incl += v;
    }
    return incl - x;
}

// Pass 1: rows of each partition; the last CTA to finish turns the totals into
// the partitions' first output rows.  As many CTAs as fit: it waits for its
// loads (3*10^7 rows 43 us, 5.6 TB/s).
__global__ void __launch_bounds__(JQ_TPB) join_part_count_kernel(PartArgs args) {
    wait_prior_grid();
    allow_next_grid();
    if (args.pf && args.pf->direct) return;
    const PartArgs a = part_source(args);
    __shared__ unsigned h[JQ_PMAX];
    for (int p = threadIdx.x; p < a.parts; p += JQ_TPB) h[p] = 0;
    __syncthreads();
    const uint64_t stride = static_cast<uint64_t>(gridDim.x) * JQ_TILE;
    for (uint64_t t0 = static_cast<uint64_t>(blockIdx.x) * JQ_TILE; t0 < a.n; t0 += stride) {
        uint64_t k[JQ_PER];
        part_load(a, t0, k);
        const unsigned len = static_cast<unsigned>(min(static_cast<uint64_t>(JQ_TILE), a.n - t0));
#pragma unroll
        for (int j = 0; j < JQ_PER; ++j)
            if (j * JQ_TPB + threadIdx.x < len) atomicAdd(&h[part_of(k[j], a)], 1u);
    }
    __syncthreads();
    const int p = threadIdx.x;
    if (p < a.parts && h[p]) atomicAdd(&a.counts[p], static_cast<unsigned long long>(h[p]));
    __shared__ unsigned long long wsum[JQ_TPB / 32];
    __shared__ unsigned long long total;
    __shared__ bool last;
    __threadfence();
    __syncthreads();
    if (p == 0) last = atomicAdd(a.ticket, 1u) == gridDim.x - 1;
    __syncthreads();
    if (!last) return;
    __threadfence();
    const unsigned long long c = p < a.parts ? __ldcg(a.counts + p) : 0ull;
    const unsigned long long start = block_excl_scan<JQ_TPB>(c, wsum, &total);
    if (p < a.parts) {
        a.next[p] = start;
        a.counts[p] = 0;
    }
    if (p == 0) *a.ticket = 0;
}

// Pass 2: each row to its partition, a tile at a time, reordered in shared
// memory so that the tile's rows of a partition are one contiguous run, at a
// place taken from the partition's cursor.  All CTAs append at the same few
// places (one per partition), so the runs' ragged ends meet in L2 and DRAM
// sees whole pages; rows of a partition keep no order.  The keys of the CTA's
// next tile are loaded while the current one is reordered.  A shared atomic
// per row gives its rank in the tile; then every warp scans the tile's counts
// for itself (NP partitions a lane, for up to 32 * NP) and takes the runs'
// starts from its lanes, so a tile needs two CTA barriers: counts complete,
// and reordered.  The counts alternate between two arrays (the other one is
// zeroed between the barriers), and the next tile cannot overwrite the reorder
// buffer before every thread has passed its first barrier, which it reaches
// only after writing this tile out.  Bound by shared memory: the scattered
// stores of the reorder and the atomics collide in its banks (L1 at 75 %).
// 3*10^7 rows into 32 partitions: 128 us, 163 with a region of its own for
// every CTA, one scanning warp and three barriers; the whole probe of a
// 2^24-row table 477 -> 437 us, 8*10^6 rows against 4*10^6 175 -> 139.  (Ranks
// by ballots instead of shared atomics: 557.)  Tiles of 320 x 7 rows, four
// CTAs: 256 x 8 444, 384 x 6 453, 512 x 6 464.
template <int NP>
__global__ void __launch_bounds__(JQ_TPB, JQ_CTAS_PER_SM) join_part_scatter_kernel(PartArgs args) {
    wait_prior_grid();
    allow_next_grid();
    if (args.pf && args.pf->direct) return;
    const PartArgs a = part_source(args);
    constexpr int WIDTH = 32 * NP;
    __shared__ unsigned h[2][WIDTH];
    __shared__ unsigned long long tbase[WIDTH];          // output row of the tile's run, less its start
    __shared__ int64_t sk[JQ_TILE];
    __shared__ uint32_t sr[JQ_TILE];
    __shared__ uint8_t sp[JQ_TILE];
    if (threadIdx.x < WIDTH) h[0][threadIdx.x] = 0;
    __syncthreads();
    const unsigned lane = threadIdx.x & 31u;
    const uint64_t stride = static_cast<uint64_t>(gridDim.x) * JQ_TILE;
    uint64_t kc[JQ_PER];
    const uint64_t first = static_cast<uint64_t>(blockIdx.x) * JQ_TILE;
    if (first < a.n) part_load(a, first, kc);
    int cur = 0;
    for (uint64_t t0 = first; t0 < a.n; t0 += stride, cur ^= 1) {
        uint64_t kn[JQ_PER];
        if (t0 + stride < a.n) part_load(a, t0 + stride, kn);
        const unsigned len = static_cast<unsigned>(min(static_cast<uint64_t>(JQ_TILE), a.n - t0));
        unsigned pr[JQ_PER];                   // partition | rank in the tile << 8
#pragma unroll
        for (int j = 0; j < JQ_PER; ++j) {
            const unsigned q = part_of(kc[j], a);
            pr[j] = j * JQ_TPB + threadIdx.x < len ? (q | (atomicAdd(&h[cur][q], 1u) << 8)) : 0u;
        }
        __syncthreads();
        // partitions lane + 32 * i: where their runs start in the tile
        unsigned off[NP], below = 0;
#pragma unroll
        for (int i = 0; i < NP; ++i) {
            const unsigned c = h[cur][lane + 32 * i];
            off[i] = below + warp_excl_scan(c, lane);
            if (i + 1 < NP) below = __shfl_sync(0xFFFFFFFFu, off[i] + c, 31);
            if (threadIdx.x < 32) {
                if (c) tbase[lane + 32 * i] = atomicAdd(&a.next[lane + 32 * i], static_cast<unsigned long long>(c)) - off[i];
                h[cur ^ 1][lane + 32 * i] = 0;
            }
        }
#pragma unroll
        for (int j = 0; j < JQ_PER; ++j) {
            const unsigned i = j * JQ_TPB + threadIdx.x;
            const unsigned q = pr[j] & 0xFFu;
            unsigned pos = __shfl_sync(0xFFFFFFFFu, off[0], q & 31u);
#pragma unroll
            for (int b = 1; b < NP; ++b) {
                const unsigned v = __shfl_sync(0xFFFFFFFFu, off[b], q & 31u);
                if (q >> 5 == static_cast<unsigned>(b)) pos = v;
            }
            pos += pr[j] >> 8;
            if (i < len) {
                sk[pos] = static_cast<int64_t>(kc[j]);
                sr[pos] = a.rowids ? ld_stream_u32(a.rowids + t0 + i) : static_cast<uint32_t>(t0 + i);
                sp[pos] = static_cast<uint8_t>(q);
            }
        }
        __syncthreads();
#pragma unroll
        for (int j = 0; j < JQ_PER; ++j) {
            const unsigned i = j * JQ_TPB + threadIdx.x;
            if (i < len) {
                const unsigned long long dst = tbase[sp[i]] + i;
                a.out_keys[dst] = sk[i];
                a.out_rowids[dst] = sr[i];
            }
        }
#pragma unroll
        for (int j = 0; j < JQ_PER; ++j) kc[j] = kn[j];
    }
}

// The scatter pass for a number of partitions.
void (*part_scatter(int parts))(PartArgs) {
    return parts <= 32 ? join_part_scatter_kernel<1> : parts <= 64 ? join_part_scatter_kernel<2> : join_part_scatter_kernel<8>;
}

uint64_t next_pow2(uint64_t x) {
    uint64_t p = 1;
    while (p < x) p <<= 1;
    return p;
}

template <typename K>
bool probe_kernel_setup(K kernel, int* per_sm) {
    int per = 0;
    if (cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, JP_SMEM) != cudaSuccess ||
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, kernel, JP_TPB, JP_SMEM) != cudaSuccess)
        return false;
    *per_sm = std::min(*per_sm, per);
    return true;
}

int probe_grid(int device) {
    static std::atomic<int> cached[64] = {};
    if (device < 0 || device >= 64) return 0;
    if (const int c = cached[device].load()) return c;
    int sms = 0, per = 1 << 20;
    if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, device) != cudaSuccess) return 0;
    if (!probe_kernel_setup(join_probe_kernel<false>, &per) || !probe_kernel_setup(join_probe_kernel<true>, &per))
        return 0;
    cached[device].store(sms * std::max(1, per));
    return cached[device].load();
}

// Resident CTAs of the two block build kernels.
int block_build_grid(int device, int* scatter) {
    static std::atomic<int> cached[64] = {};                  // build | scatter << 16
    if (device < 0 || device >= 64) return 0;
    int c = cached[device].load();
    if (!c) {
        int sms = 0, per = 0, per_s = 0;
        if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, device) != cudaSuccess ||
            cudaFuncSetAttribute(join_block_build_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, JT_SMEM) !=
                cudaSuccess ||
            cudaFuncSetAttribute(join_block_scatter_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, JS_SMEM) !=
                cudaSuccess ||
            cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, join_block_build_kernel, JT_TPB, JT_SMEM) !=
                cudaSuccess ||
            cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_s, join_block_scatter_kernel, JS_TPB, JS_SMEM) !=
                cudaSuccess)
            return 0;
        c = sms * std::max(1, per) | (sms * std::max(1, per_s)) << 16;
        cached[device].store(c);
    }
    *scatter = c >> 16;
    return c & 0xFFFF;
}

size_t align256(size_t x) { return (x + 255) & ~static_cast<size_t>(255); }

// Grids of the two partition passes: the CTAs that stay resident.
struct PartGrids {
    unsigned count, scatter;
};
PartGrids part_grids(int device, int sms) {
    static std::atomic<int> cached[64] = {};                  // per SM: count | scatter << 16
    if (device < 0 || device >= 64) return {0, 0};
    int c = cached[device].load();
    if (!c) {
        int per_c = 0, per_s = JQ_CTAS_PER_SM;
        if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_c, join_part_count_kernel, JQ_TPB, 0) != cudaSuccess)
            return {0, 0};
        for (int parts : {32, 64, JQ_PMAX}) {
            int p = 0;
            if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&p, part_scatter(parts), JQ_TPB, 0) != cudaSuccess)
                return {0, 0};
            per_s = std::min(per_s, p);
        }
        c = std::max(1, per_c) | std::max(1, per_s) << 16;
        cached[device].store(c);
    }
    return {static_cast<unsigned>(sms * (c & 0xFFFF)), static_cast<unsigned>(sms * (c >> 16))};
}

}  // namespace

// Rows from which on the partition passes may pay: a quarter of the table's
// buckets (the plan kernel tests the rows its pre-probe leaves against it).
static uint64_t part_min_rows(const olap_join_table* t) { return t->n_buckets / 4; }

// Partitions the probe of `n` rows against `t` uses (1 = direct probe).
int probe_parts(const olap_ctx* ctx, const olap_join_table* t, uint64_t n) {
    const int opt = ctx->opts.join_partitions;
    uint64_t parts = 1;
    if (opt >= 2) {
        parts = static_cast<uint64_t>(opt);
    } else if (opt == 0) {
        const uint64_t tb = t->n_buckets * 32;
        const uint64_t l2 = ctx->l2_bytes ? ctx->l2_bytes : (64ull << 20);
        // worth it when the table is well above L2 and there are rows enough
        if (tb > l2 / 2 && n >= part_min_rows(t)) parts = next_pow2((tb + l2 / 4 - 1) / (l2 / 4));
    }
    parts = std::min<uint64_t>(parts, static_cast<uint64_t>(JQ_PMAX));
    parts = std::min<uint64_t>(parts, t->n_buckets);
    return static_cast<int>(std::max<uint64_t>(parts, 1));
}

// log2 of a table block's buckets (smaller tables are one block) and of its
// Bloom filter blocks.
static int log2_of(uint64_t x) {
    int l = 0;
    while ((1ull << l) < x) ++l;
    return l;
}
static int table_block_log(uint64_t n_buckets) { return std::min(JT_BLOCK_LOG, log2_of(n_buckets)); }
static BloomView bloom_view(const olap_join_table* t) {
    const int bl = table_block_log(t->n_buckets);
    return BloomView{t->bloom, t->n_buckets - 1, bl, log2_of(t->bloom_blocks) - (log2_of(t->n_buckets) - bl)};
}

// Whether a probe of n rows against t runs the Bloom pre-probe stage (its
// sample still decides on the device whether rows are dropped).
bool probe_prefilter(const olap_ctx* ctx, const olap_join_table* t, uint64_t n) {
    if (!t->bloom || n == 0) return false;
    const int opt = ctx->opts.join_prefilter;
    return opt == OLAP_PREFILTER_ON || (opt == OLAP_PREFILTER_AUTO && n >= PF_MIN_N);
}

// Partition scratch: [partitioned keys | row-ids]; then, with the pre-probe,
// [kept keys | kept row-ids].  The probe's device-side plan and the partitions'
// counts live in the context's small device area.
size_t probe_part_bytes(uint64_t n, int parts) { return parts <= 1 ? 0 : align256(n * 8) + align256(n * 4); }

size_t probe_scratch_bytes(const olap_ctx* ctx, const olap_join_table* t, uint64_t n) {
    const size_t pb = probe_part_bytes(n, probe_parts(ctx, t, n));
    if (!probe_prefilter(ctx, t, n)) return pb;
    return pb + align256(n * 8) + align256(n * 4);
}

// The partition passes over n rows by the top bits of their home bucket, into
// `rows` (probe_part_bytes), with PART_COUNT_BYTES at `counts`, zero before the
// first call.
constexpr size_t PART_COUNT_BYTES = 2 * JQ_PMAX * 8 + 256;
static PartArgs part_args(void* rows, void* counts, const int64_t* keys, const uint32_t* rowids, uint64_t n,
                          uint64_t n_buckets, int parts) {
    unsigned char* m = static_cast<unsigned char*>(rows);
    PartArgs q{};
    q.keys = keys;
    q.rowids = rowids;
    q.n = n;
    q.mask = n_buckets - 1;
    q.shift = 0;
    while ((n_buckets >> q.shift) > static_cast<uint64_t>(parts)) ++q.shift;
    q.parts = parts;
    q.out_keys = reinterpret_cast<int64_t*>(m);
    q.out_rowids = reinterpret_cast<uint32_t*>(m + align256(n * 8));
    q.counts = static_cast<unsigned long long*>(counts);
    q.next = q.counts + JQ_PMAX;
    q.ticket = reinterpret_cast<unsigned*>(q.next + JQ_PMAX);
    return q;
}

}  // namespace olap


using namespace olap;

namespace {

// With host_count the count word is the context's own (zero between probes),
// and the probe leaves the count in *host_count; else the count goes to d_count.
olap_status probe_enqueue(olap_ctx* ctx, const olap_join_table* t, const int64_t* d_keys, const uint32_t* d_rowids,
                          uint64_t n, olap_pair* d_out, uint64_t capacity, uint64_t* d_count, uint64_t* host_count,
                          cudaStream_t s) {
    cudaError_t e = cudaSuccess;
    if (host_count) {
        *host_count = 0;
        d_count = static_cast<uint64_t*>(ctx->aux);
    } else if ((e = cudaMemsetAsync(d_count, 0, sizeof(uint64_t), s)) != cudaSuccess) {
        return cuda_fail(ctx, e, "probe count reset");
    }
    if (n == 0) {
        ctx->last_probe_parts = 1;
        ctx->last_probe_n = 0;
        ctx->last_probe_pf = nullptr;
        return OLAP_OK;
    }
    const int grid = probe_grid(ctx->device);
    if (grid <= 0) return fail(ctx, OLAP_E_CUDA, "probe kernel occupancy query failed");
    ProbeArgs a;
    a.keys = d_keys;
    a.rowids = d_rowids;
    a.n = n;
    a.slots = t->slots;
    a.mask = t->n_buckets - 1;
    a.chain_mask = t->chain_mask;
    a.side = t->side;
    a.n_side = t->n_side;
    a.out = reinterpret_cast<uint2*>(d_out);
    a.cap = capacity;
    a.count = reinterpret_cast<unsigned long long*>(d_count);
    const int parts = probe_parts(ctx, t, n);
    const bool pre = probe_prefilter(ctx, t, n);
    // the sample may still turn an automatically partitioned probe direct
    const bool skew_check = parts > 1 && ctx->opts.join_partitions == 0;
    PartArgs q{};
    PartGrids qg{};
    ProbeCtl* pf = nullptr;
    int64_t* pf_keys = nullptr;
    uint32_t* pf_rowids = nullptr;
    if (parts > 1 || pre) {
        olap_status st = ensure_part(ctx, probe_scratch_bytes(ctx, t, n));
        if (st != OLAP_OK) return st;
    }
    if (pre || skew_check) pf = reinterpret_cast<ProbeCtl*>(static_cast<unsigned char*>(ctx->aux) + 1024);
    if (pre) {
        unsigned char* m = static_cast<unsigned char*>(ctx->part) + probe_part_bytes(n, parts);
        pf_keys = reinterpret_cast<int64_t*>(m);
        pf_rowids = reinterpret_cast<uint32_t*>(m + align256(n * 8));
        if (m + align256(n * 8) + align256(n * 4) > static_cast<unsigned char*>(ctx->part) + ctx->part_bytes)
            return fail(ctx, OLAP_E_INVALID, "probe pre-filter scratch too small");
    }
    if (parts > 1) {
        qg = part_grids(ctx->device, ctx->sm_count);
        if (qg.count == 0) return fail(ctx, OLAP_E_CUDA, "partition kernel occupancy query failed");
        q = part_args(ctx->part, static_cast<unsigned char*>(ctx->aux) + 4096, d_keys, d_rowids, n, t->n_buckets, parts);
        if (probe_part_bytes(n, parts) > ctx->part_bytes)
            return fail(ctx, OLAP_E_INVALID, "probe partition scratch too small");
        q.pf = pf;
        q.pf_keys = pf_keys;
        q.pf_rowids = pf_rowids;
    }
    ctx->last_probe_parts = parts;
    ctx->last_probe_n = n;
    ctx->last_probe_pf = pf;
    ctx->probe_timed = ctx->time_kernels;
    if (ctx->time_kernels && (e = cudaEventRecord(ctx->kev[4], s)) != cudaSuccess)
        return cuda_fail(ctx, e, "timing event");
    // the row queue's counter, in the context's small device area
    unsigned long long* next_row = reinterpret_cast<unsigned long long*>(static_cast<unsigned char*>(ctx->aux) + 256);
    const ProbeDone done{reinterpret_cast<unsigned*>(next_row + 1), reinterpret_cast<unsigned long long*>(host_count)};
    ProbeArgs pa = a;
    const BloomView bloom = pre ? bloom_view(t) : BloomView{nullptr, 0, 0, 0};
    if (pf) {
        const int pf_mode = pre ? (ctx->opts.join_prefilter == OLAP_PREFILTER_ON ? 2 : 1) : 0;
        const int skew_l1 = ctx->opts.join_bucket_loads == OLAP_LOADS_AUTO ? 1 : 0;
        PlanArgs pl;
        pl.keys = d_keys;
        pl.rowids = d_rowids;
        pl.n = n;
        pl.bloom = bloom;
        pl.pf_mode = pf_mode;
        pl.skew_check = skew_check ? 1 : 0;
        pl.min_rows = part_min_rows(t);
        pl.partitioned = parts > 1 ? 1 : 0;
        pl.skew_l1 = skew_l1;
        pl.pf_keys = pf_keys;
        pl.pf_rowids = pf_rowids;
        pl.sample = reinterpret_cast<uint32_t*>(static_cast<unsigned char*>(ctx->aux) + 16384);
        pl.counters = reinterpret_cast<unsigned*>(static_cast<unsigned char*>(ctx->aux) + 1536);
        pl.ctl = pf;
        join_probe_plan_kernel<<<PLAN_CTAS, PLAN_TPB, 0, s>>>(pl);
    }
    if (pre)
        launch_after(join_prefilter_kernel, static_cast<unsigned>(ctx->sm_count * PF_CTAS), PF_TPB, 0, s, true, d_keys,
                     d_rowids, n, bloom, static_cast<ProbeCtl*>(pf), pf_keys, pf_rowids);
    if (parts > 1) {
        // (the first kernel of the chain follows whatever the stream holds)
        launch_after(join_part_count_kernel, qg.count, JQ_TPB, 0, s, pf != nullptr, q);
        launch_after(part_scatter(parts), qg.scatter, JQ_TPB, 0, s, true, q);
        pa.keys = q.out_keys;
        pa.rowids = q.out_rowids;
    }
    const bool after = pf || parts > 1;
    if (ctx->opts.join_bucket_loads == OLAP_LOADS_L1)
        launch_after(join_probe_kernel<false>, static_cast<unsigned>(grid), JP_TPB, JP_SMEM, s, after, pa, next_row,
                     static_cast<const ProbeCtl*>(pf), done);
    else
        launch_after(join_probe_kernel<true>, static_cast<unsigned>(grid), JP_TPB, JP_SMEM, s, after, pa, next_row,
                     static_cast<const ProbeCtl*>(pf), done);
    e = cudaGetLastError();
    // [plan,] [filter,] [count, scatter,] probe
    if (e == cudaSuccess) ctx->launches += (pf ? 1 : 0) + (pre ? 1 : 0) + (parts > 1 ? 2 : 0) + 1;
    if (e == cudaSuccess && ctx->time_kernels) e = cudaEventRecord(ctx->kev[5], s);
    return e == cudaSuccess ? OLAP_OK : cuda_fail(ctx, e, "probe launch");
}

olap_status check_join_table(olap_ctx* ctx, const olap_join_table* t) {
    if (!t || !t->slots) return fail(ctx, OLAP_E_INVALID, "join table is NULL or freed");
    if (t->device != ctx->device) return fail(ctx, OLAP_E_INVALID, "join table lives on another device");
    return OLAP_OK;
}

}  // namespace

extern "C" {

olap_status olap_join_build(olap_ctx* ctx, const int64_t* keys, const uint32_t* rowids, olap_mem where, uint64_t n,
                            double load_factor, olap_join_table** out) {
    if (!ctx) return OLAP_E_INVALID;
    ctx->last_error.clear();
    if (!out) return fail(ctx, OLAP_E_INVALID, "out is NULL");
    *out = nullptr;
    if (where < OLAP_MEM_HOST || where > OLAP_MEM_DEVICE) return fail(ctx, OLAP_E_INVALID, "bad memory kind");
    if (n && !keys) return fail(ctx, OLAP_E_INVALID, "keys is NULL");
    if (!rowids && n > (1ull << 32)) return fail(ctx, OLAP_E_INVALID, "implicit row-ids need n <= 2^32");
    if (reinterpret_cast<uintptr_t>(keys) % 8) return fail(ctx, OLAP_E_INVALID, "keys misaligned");
    double load = load_factor > 0.0 ? load_factor : (ctx->opts.load_factor > 0.0 ? ctx->opts.load_factor : 0.5);
    if (!(load > 0.0 && load <= 0.9)) return fail(ctx, OLAP_E_INVALID, "load factor must be in (0, 0.9]");
    cudaError_t e = cudaSetDevice(ctx->device);
    if (e != cudaSuccess) return cuda_fail(ctx, e, "set device");

    const uint64_t want_slots = static_cast<uint64_t>(static_cast<double>(n) / load) + 2;
    const uint64_t buckets = next_pow2((want_slots + 1) / 2);
    if (buckets > (1ull << 32)) return fail(ctx, OLAP_E_NOMEM, "join table: more than 2^32 buckets");
    const size_t slot_bytes = buckets * 32;
    // Bloom filter for the pre-probe: about 16 bits per build row, for tables
    // well above L2 (automatic) or every table with rows (forced on).
    const uint64_t l2 = ctx->l2_bytes ? ctx->l2_bytes : (64ull << 20);
    const bool with_bloom = n && (ctx->opts.join_prefilter == OLAP_PREFILTER_ON ||
                                  (ctx->opts.join_prefilter == OLAP_PREFILTER_AUTO && slot_bytes > l2 / 2));
    const int block_log = table_block_log(buckets);
    const uint64_t blocks = buckets >> block_log;
    const uint64_t bloom_blocks = with_bloom ? std::max(next_pow2((n + 15) / 16), blocks) : 0;
    const size_t bytes = slot_bytes + 256 + bloom_blocks * 32;
    if (!within_budget(ctx, bytes)) return fail(ctx, OLAP_E_NOMEM, "join table: device memory budget exceeded");

    // Key-only input: build keys (and row-ids) to the device.
    const int64_t* dk = keys;
    const uint32_t* dr = rowids;
    if (where != OLAP_MEM_DEVICE && n) {
        const size_t kb = (n * 8 + 255) & ~static_cast<size_t>(255);
        olap_status st = ensure_dev_in(ctx, kb + (rowids ? n * 4 : 0));
        if (st != OLAP_OK) return st;
        st = copy_h2d(ctx, ctx->dev_in, keys, n * 8, where);
        if (st != OLAP_OK) return st;
        dk = static_cast<const int64_t*>(ctx->dev_in);
        if (rowids) {
            dr = reinterpret_cast<const uint32_t*>(static_cast<unsigned char*>(ctx->dev_in) + kb);
            st = copy_h2d(ctx, const_cast<uint32_t*>(dr), rowids, n * 4, where);
            if (st != OLAP_OK) return st;
        }
    }

    olap_join_table* t = new olap_join_table();
    t->device = ctx->device;
    t->n_buckets = buckets;
    t->n_build = n;
    t->load = load;
    void* mem = nullptr;
    const bool keep = ctx->opts.mem_budget_bytes == 0;
    e = keep ? devmem::take(ctx->device, &mem, bytes, &t->cap) : devmem::alloc(ctx->device, &mem, bytes);
    if (e != cudaSuccess) {
        cudaGetLastError();
        delete t;
        return cuda_fail(ctx, e, "join table allocation");
    }
    t->slots = static_cast<ulonglong2*>(mem);
    t->bytes = bytes;
    ctx->table_bytes += bytes;                               // counted from here on: the scratch below is checked beside it
    // Partition scratch of a large build, for the time of the build.
    void* part = nullptr;
    size_t part_cap = 0;
    JoinCtl* jc = reinterpret_cast<JoinCtl*>(static_cast<unsigned char*>(mem) + slot_bytes);
    auto drop_part = [&]() {                                 // (no work uses it any more)
        if (part && keep) devmem::give(ctx->device, part, part_cap);
        else if (part) cudaFree(part);
        part = nullptr;
    };
    auto bail = [&](olap_status st) {
        cudaStreamSynchronize(ctx->stream);                  // launched passes may still write it
        drop_part();
        ctx->table_bytes -= bytes;
        cudaFree(mem);
        delete t;
        return st;
    };
    if (bloom_blocks) {
        t->bloom = reinterpret_cast<uint32_t*>(static_cast<unsigned char*>(mem) + slot_bytes + 256);
        t->bloom_blocks = bloom_blocks;
    }
    // Two passes over table blocks; the general build when there are no rows or
    // when a block turned out crowded.
    const int grid = ctx->sm_count * 8;
    const int per_log = bloom_blocks ? log2_of(bloom_blocks) - log2_of(blocks) : 0;
    bool general = n == 0;
    JoinCtl hc{};
    auto read_ctl = [&]() -> olap_status {
        e = cudaMemcpyAsync(ctx->host_status, jc, sizeof(hc), cudaMemcpyDeviceToHost, ctx->stream);
        if (e == cudaSuccess) e = cudaStreamSynchronize(ctx->stream);
        if (e != cudaSuccess) return cuda_fail(ctx, e, "join build");
        std::memcpy(&hc, ctx->host_status, sizeof(hc));
        return OLAP_OK;
    };
    e = cudaMemsetAsync(jc, 0, sizeof(JoinCtl), ctx->stream);
    if (e != cudaSuccess) return bail(cuda_fail(ctx, e, "join table init"));
    if (!general) {
        const size_t pitch = 32ull << block_log;
        int sgrid = 0;
        const int bgrid = block_build_grid(ctx->device, &sgrid);
        if (bgrid <= 0) return bail(fail(ctx, OLAP_E_CUDA, "block build kernel set-up failed"));
        // the blocks' cursors, in their last slots
        e = cudaMemset2DAsync(static_cast<unsigned char*>(mem) + pitch - 16, pitch, 0, 16, blocks, ctx->stream);
        if (e != cudaSuccess) return bail(cuda_fail(ctx, e, "join table init"));
        // More blocks than a tile counts: the rows are first ordered by the
        // upper bits of their block (the probe's partition passes), when there
        // is room for that; without it the first pass goes row by row.
        const int64_t* bk = dk;
        const uint32_t* br = dr;
        if (blocks > static_cast<uint64_t>(JS_BINS) && n >= JS_PART_MIN_N) {
            const PartGrids pg = part_grids(ctx->device, ctx->sm_count);
            const size_t pb = probe_part_bytes(n, JS_PARTS), want = pb + PART_COUNT_BYTES;
            if (pg.count && within_budget(ctx, want)) {
                e = keep ? devmem::take(ctx->device, &part, want, &part_cap) : devmem::alloc(ctx->device, &part, want);
                if (e != cudaSuccess) {
                    cudaGetLastError();
                    part = nullptr;
                }
            }
            if (part) {
                void* counts = static_cast<unsigned char*>(part) + pb;
                e = cudaMemsetAsync(counts, 0, PART_COUNT_BYTES, ctx->stream);
                if (e != cudaSuccess) return bail(cuda_fail(ctx, e, "partition counts"));
                const PartArgs q = part_args(part, counts, dk, dr, n, buckets, JS_PARTS);
                launch_after(join_part_count_kernel, pg.count, JQ_TPB, 0, ctx->stream, false, q);
                launch_after(part_scatter(JS_PARTS), pg.scatter, JQ_TPB, 0, ctx->stream, true, q);
                ctx->launches += 2;
                bk = q.out_keys;
                br = q.out_rowids;
            }
        }
        const uint64_t threads = static_cast<uint64_t>(sgrid) * JS_TPB;
        const int per = static_cast<int>(std::min<uint64_t>((n + threads - 1) / threads, JS_PER));
        const uint64_t tiles = (n + static_cast<uint64_t>(per) * JS_TPB - 1) / (static_cast<uint64_t>(per) * JS_TPB);
        join_block_scatter_kernel<<<static_cast<unsigned>(std::min<uint64_t>(tiles, sgrid)), JS_TPB, JS_SMEM,
                                    ctx->stream>>>(bk, br, n, per, t->slots, buckets - 1, block_log, jc);
        join_block_build_kernel<<<static_cast<unsigned>(std::min<uint64_t>(blocks, bgrid)), JT_TPB, JT_SMEM,
                                  ctx->stream>>>(t->slots, blocks, block_log, t->bloom, per_log, jc);
        e = cudaGetLastError();
        if (e != cudaSuccess) return bail(cuda_fail(ctx, e, "build launch"));
        ctx->launches += 2;
        olap_status st = read_ctl();
        if (st != OLAP_OK) return bail(st);
        drop_part();
        t->chain_mask = (1ull << block_log) - 1;
        general = hc.crowded != 0;
    }
    if (general) {
        t->chain_mask = buckets - 1;
        e = cudaMemsetAsync(mem, 0xFF, slot_bytes, ctx->stream);
        if (e == cudaSuccess) e = cudaMemsetAsync(jc, 0, sizeof(JoinCtl), ctx->stream);
        if (e == cudaSuccess && bloom_blocks) e = cudaMemsetAsync(t->bloom, 0, bloom_blocks * 32, ctx->stream);
        if (e != cudaSuccess) return bail(cuda_fail(ctx, e, "join table init"));
        if (n) {
            join_build_kernel<<<grid, JB_TPB, 0, ctx->stream>>>(dk, dr, n, t->slots, buckets - 1, jc);
            join_chain_kernel<<<grid, JB_TPB, 0, ctx->stream>>>(t->slots, buckets - 1);
            if (bloom_blocks) join_bloom_kernel<<<grid, JB_TPB, 0, ctx->stream>>>(dk, n, t->bloom, bloom_view(t));
            e = cudaGetLastError();
            if (e != cudaSuccess) return bail(cuda_fail(ctx, e, "build launch"));
            ctx->launches += bloom_blocks ? 3 : 2;
        }
        olap_status st = read_ctl();
        if (st != OLAP_OK) return bail(st);
    }
    if (hc.err) return bail(fail(ctx, static_cast<olap_status>(hc.err), "join build: table full"));
    if (hc.side_count) {
        e = devmem::alloc(ctx->device, reinterpret_cast<void**>(&t->side), hc.side_count * 4);
        if (e != cudaSuccess) {
            cudaGetLastError();
            return bail(cuda_fail(ctx, e, "join side list allocation"));
        }
        join_side_kernel<<<ctx->sm_count * 4, JB_TPB, 0, ctx->stream>>>(dk, dr, n, t->side, jc);
        e = cudaGetLastError();
        if (e == cudaSuccess) ctx->launches += 1;
        if (e == cudaSuccess) e = cudaStreamSynchronize(ctx->stream);
        if (e != cudaSuccess) {
            cudaFree(t->side);
            return bail(cuda_fail(ctx, e, "join side list"));
        }
        t->n_side = hc.side_count;
        t->bytes += hc.side_count * 4;
        ctx->table_bytes += hc.side_count * 4;
    }
    ctx->tables.insert(t);
    t->owner = ctx;
    *out = t;
    return OLAP_OK;
}

olap_status olap_join_probe_async(olap_ctx* ctx, const olap_join_table* table, const int64_t* d_keys,
                                  const uint32_t* d_rowids, uint64_t n, olap_pair* d_out, uint64_t capacity,
                                  uint64_t* d_count, void* stream) {
    if (!ctx) return OLAP_E_INVALID;
    ctx->last_error.clear();
    olap_status st = check_join_table(ctx, table);
    if (st != OLAP_OK) return st;
    if (!d_count) return fail(ctx, OLAP_E_INVALID, "d_count is NULL");
    if (n && !d_keys) return fail(ctx, OLAP_E_INVALID, "keys is NULL");
    if (capacity && !d_out) return fail(ctx, OLAP_E_INVALID, "out is NULL");
    if (!d_rowids && n > (1ull << 32)) return fail(ctx, OLAP_E_INVALID, "implicit row-ids need n <= 2^32");
    cudaStream_t s = stream ? static_cast<cudaStream_t>(stream) : ctx->stream;
    return probe_enqueue(ctx, table, d_keys, d_rowids, n, d_out, capacity, d_count, nullptr, s);
}

olap_status olap_join_probe(olap_ctx* ctx, const olap_join_table* table, const int64_t* keys,
                            const uint32_t* rowids, olap_mem where, uint64_t n, olap_pair* out, olap_mem out_where,
                            uint64_t capacity, uint64_t* out_count) {
    if (!ctx) return OLAP_E_INVALID;
    ctx->last_error.clear();
    if (!out_count) return fail(ctx, OLAP_E_INVALID, "out_count is NULL");
    *out_count = 0;
    olap_status st = check_join_table(ctx, table);
    if (st != OLAP_OK) return st;
    if (where < OLAP_MEM_HOST || where > OLAP_MEM_DEVICE || out_where < OLAP_MEM_HOST ||
        out_where > OLAP_MEM_DEVICE)
        return fail(ctx, OLAP_E_INVALID, "bad memory kind");
    if (n && !keys) return fail(ctx, OLAP_E_INVALID, "keys is NULL");
    if (capacity && !out) return fail(ctx, OLAP_E_INVALID, "out is NULL");
    if (!rowids && n > (1ull << 32)) return fail(ctx, OLAP_E_INVALID, "implicit row-ids need n <= 2^32");
    if (reinterpret_cast<uintptr_t>(keys) % 8) return fail(ctx, OLAP_E_INVALID, "keys misaligned");
    cudaError_t e = cudaSetDevice(ctx->device);
    if (e != cudaSuccess) return cuda_fail(ctx, e, "set device");

    const int64_t* dk = keys;
    const uint32_t* dr = rowids;
    if (where != OLAP_MEM_DEVICE && n) {
        const size_t kb = (n * 8 + 255) & ~static_cast<size_t>(255);
        st = ensure_dev_in(ctx, kb + (rowids ? n * 4 : 0));
        if (st != OLAP_OK) return st;
        st = copy_h2d(ctx, ctx->dev_in, keys, n * 8, where);
        if (st != OLAP_OK) return st;
        dk = static_cast<const int64_t*>(ctx->dev_in);
        if (rowids) {
            dr = reinterpret_cast<const uint32_t*>(static_cast<unsigned char*>(ctx->dev_in) + kb);
            st = copy_h2d(ctx, const_cast<uint32_t*>(dr), rowids, n * 4, where);
            if (st != OLAP_OK) return st;
        }
    }
    olap_pair* dout = out;
    if (out_where != OLAP_MEM_DEVICE) {
        st = ensure_dev_out(ctx, capacity * 8);
        if (st != OLAP_OK) return st;
        dout = static_cast<olap_pair*>(ctx->dev_out);
    }
    uint64_t* hcount = reinterpret_cast<uint64_t*>(ctx->host_status + 8);
    st = probe_enqueue(ctx, table, dk, dr, n, dout, capacity, nullptr, hcount, ctx->stream);
    if (st != OLAP_OK) return st;
    e = cudaStreamSynchronize(ctx->stream);
    if (e != cudaSuccess) return cuda_fail(ctx, e, "join probe");
    const uint64_t cnt = *reinterpret_cast<volatile uint64_t*>(hcount);
    *out_count = cnt;
    if (cnt > capacity) return fail(ctx, OLAP_E_OVERFLOW, "join probe: output capacity too small");
    if (out_where != OLAP_MEM_DEVICE && cnt) {
        st = copy_d2h(ctx, out, dout, cnt * 8, out_where);
        if (st != OLAP_OK) return st;
        e = cudaStreamSynchronize(ctx->stream);
        if (e != cudaSuccess) return cuda_fail(ctx, e, "join result copy");
    }
    return OLAP_OK;
}

olap_status olap_join_probe_partitions(olap_ctx* ctx, const olap_join_table* table, uint64_t n, int* parts) {
    if (!ctx) return OLAP_E_INVALID;
    ctx->last_error.clear();
    if (!parts) return fail(ctx, OLAP_E_INVALID, "parts is NULL");
    olap_status st = check_join_table(ctx, table);
    if (st != OLAP_OK) return st;
    *parts = probe_parts(ctx, table, n);
    return OLAP_OK;
}

olap_status olap_join_probe_info_last(olap_ctx* ctx, int* parts, int* prefiltered, uint64_t* rows_probed) {
    if (!ctx) return OLAP_E_INVALID;
    ctx->last_error.clear();
    if (!parts || !prefiltered || !rows_probed) return fail(ctx, OLAP_E_INVALID, "NULL output");
    if (ctx->last_probe_parts == 0) return fail(ctx, OLAP_E_INVALID, "no probe has run on this context");
    *parts = ctx->last_probe_parts;
    *prefiltered = 0;
    *rows_probed = ctx->last_probe_n;
    cudaError_t e = cudaStreamSynchronize(ctx->stream);
    if (e != cudaSuccess) return cuda_fail(ctx, e, "probe info");
    if (ctx->last_probe_pf) {
        ProbeCtl c;
        e = cudaMemcpy(&c, ctx->last_probe_pf, sizeof(c), cudaMemcpyDeviceToHost);
        if (e != cudaSuccess) return cuda_fail(ctx, e, "probe info");
        if (c.active) {
            *prefiltered = 1;
            *rows_probed = c.count;
        }
        if (c.direct) *parts = 1;
    }
    return OLAP_OK;
}

olap_status olap_join_table_info(const olap_join_table* t, uint64_t* n_build, uint64_t* n_buckets, uint64_t* n_side,
                                 uint64_t* bloom_bytes) {
    if (!t || !t->slots) return OLAP_E_INVALID;
    if (n_build) *n_build = t->n_build;
    if (n_buckets) *n_buckets = t->n_buckets;
    if (n_side) *n_side = t->n_side;
    if (bloom_bytes) *bloom_bytes = t->bloom_blocks * 32;
    return OLAP_OK;
}

void olap_join_free(olap_join_table* t) {
    if (!t) return;
    if (t->owner) {
        t->owner->table_bytes -= t->bytes;
        t->owner->tables.erase(t);
    }
    int cur = 0;
    cudaGetDevice(&cur);
    cudaSetDevice(t->device);
    cudaDeviceSynchronize();
    if (t->slots && t->cap) devmem::give(t->device, t->slots, t->cap);
    else if (t->slots) cudaFree(t->slots);
    if (t->side) cudaFree(t->side);
    t->slots = nullptr;
    t->side = nullptr;
    cudaSetDevice(cur);
    delete t;
}

}  // extern "C"

void detach_tables(olap_ctx* ctx) {
    for (olap_join_table* t : ctx->tables) t->owner = nullptr;
    ctx->tables.clear();
}
