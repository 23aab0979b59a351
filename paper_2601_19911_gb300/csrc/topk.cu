// Top-K selection over key-only (key, row-id) columns: ORDER BY key LIMIT K
// (Sec. III-A, "partial selection (or radix-based selection)", returning the
// row pointers of the Top-K rows in order).
//
// A few thousand keys take one launch (topk_local_kernel).  Otherwise three
// launches on one stream, the second one up to 2^21 keys part of the third:
//   0. topk_prepare_kernel zeroes the control block and, when N is large and
//      K is small against N, reads a stratified sample of 8192 keys (16 CTAs,
//      one key per thread) and finds the sample's r-th best entry by a radix
//      select in the last CTA to finish; r is chosen so that, with high
//      probability, at least K keys but not many more fall at or below it.
//   1. topk_filter_regs_kernel (default) or topk_filter_bulk_kernel (TMA
//      bulk copies into a shared-memory ring): the only full pass over the
//      keys, run only when there is a sample.  32-byte streaming loads, one
//      compare per key against the threshold in the key's own bit domain,
//      and every key that passes is appended (per-warp staging, one global
//      atomic per flush) to a candidate buffer with its row-id -- or only
//      counted, when the sample shows ties that would not fit there.
//   Phases 2-4 are one cooperative launch (topk_select_kernel) whose CTAs
//   meet at bounded grid barriers.  Its source is the candidate buffer when
//   the sample worked (at least K candidates, no overflow) and the full
//   input otherwise (no sample, or a misjudged one).
//   2. Refine: every pass cuts the current interval of the composite (rank
//      word, row-id) order into up to 4096 equal bins (a shared-memory
//      histogram with __match_any_sync aggregation, merged into a global
//      one); every CTA then scans it and goes on with the same bin, until the
//      bin that holds the K-th entry has at most 4096 entries.
//   3. Split: entries below the interval are selected; entries in it go to a
//      small buffer that is ranked to take the remaining count.
//   4. Put the K survivors in (rank word, row-id) order -- by counting smaller
//      entries when K <= 4096; else spread over 4096 equal bins of their
//      interval (or between 2047 sorted splitters when those crowd) and ranked
//      within their bin; tile sorts plus merge-path rounds when both fail --
//      and write keys (original bits, by the inverse transform) and row-ids.
// A column in host memory is read by the pass itself (topk_filter_host_kernel).
#include <algorithm>
#include <atomic>
#include <cmath>
#include <mutex>

#include "block.cuh"
#include "topk.cuh"

namespace olap {

namespace {

__device__ __forceinline__ unsigned long long gtimer() {
    unsigned long long t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

struct Elem {
    uint64_t r;
    uint32_t rid;
};

// Rank word of a two-column key: c0's 32-bit rank above c1's.
__device__ __forceinline__ uint64_t pair_rank(uint32_t b0, uint32_t b1, const TopkArgs& a) {
    return rank_key(b0, a.kind, a.desc) | (rank_key(b1, a.kind2, a.desc2) >> 32);
}

// Key bits of row i of the column at `keys` (a.keys, or a.host_keys).
__device__ __forceinline__ uint64_t key_bits(const TopkArgs& a, const void* keys, uint64_t i) {
    return a.w4 ? static_cast<uint64_t>(static_cast<const uint32_t*>(keys)[i]) : static_cast<const uint64_t*>(keys)[i];
}

__device__ __forceinline__ uint64_t input_rank(const TopkArgs& a, uint64_t i) {
    if (a.pair) return pair_rank(static_cast<const uint32_t*>(a.keys)[i], static_cast<const uint32_t*>(a.keys2)[i], a);
    return rank_key(key_bits(a, a.keys, i), a.kind, a.desc);
}
__device__ __forceinline__ uint32_t input_rowid(const TopkArgs& a, uint64_t i) {
    return a.rowids ? a.rowids[i] : static_cast<uint32_t>(i);
}
__device__ __forceinline__ Elem load_input(const TopkArgs& a, uint64_t i) { return Elem{input_rank(a, i), input_rowid(a, i)}; }

__device__ __forceinline__ Elem load_src(const TopkArgs& a, bool cand, uint64_t i) {
    if (cand) return Elem{__ldcg(a.cand_r + i), __ldcg(a.cand_rid + i)};
    return load_input(a, i);
}

__device__ __forceinline__ void write_result(const TopkArgs& a, uint64_t i, uint64_t r, uint32_t rid) {
    if (a.pair) {
        static_cast<uint32_t*>(a.out_keys)[i] = static_cast<uint32_t>(unrank_key(r & 0xFFFFFFFF00000000ull, a.kind, a.desc));
        static_cast<uint32_t*>(a.out_keys2)[i] = static_cast<uint32_t>(unrank_key(r << 32, a.kind2, a.desc2));
    } else if (a.w4)
        static_cast<uint32_t*>(a.out_keys)[i] = static_cast<uint32_t>(unrank_key(r, a.kind, a.desc));
    else
        static_cast<uint64_t*>(a.out_keys)[i] = unrank_key(r, a.kind, a.desc);
    a.out_rowids[i] = rid;
}

__device__ __forceinline__ uint32_t max_rowid(const TopkArgs& a) {
    return a.rowids ? 0xFFFFFFFFu : static_cast<uint32_t>(a.n - 1);
}
// (a 4-byte key's rank words are multiples of 2^32)
__device__ __forceinline__ uint64_t max_rank(const TopkArgs& a) { return a.w4 ? 0xFFFFFFFF00000000ull : ~0ull; }
// Bin b of the interval.
__device__ __forceinline__ Range range_narrow(const TopkArgs& a, const Range& g, int sh, unsigned b) {
    Range o = g;
    const uint64_t w = (1ull << sh) - 1ull;
    if (g.rlo != g.rhi) {
        o.rlo = g.rlo + (static_cast<uint64_t>(b) << sh);
        o.rhi = g.rhi - o.rlo < w ? g.rhi : o.rlo + w;
        if (a.w4) {
            o.rlo = (o.rlo + 0xFFFFFFFFull) & 0xFFFFFFFF00000000ull;
            o.rhi &= 0xFFFFFFFF00000000ull;
        }
        o.ilo = 0;
        o.ihi = max_rowid(a);
    } else {
        o.ilo = g.ilo + (b << sh);
        o.ihi = g.ihi - o.ilo < w ? g.ihi : o.ilo + static_cast<uint32_t>(w);
    }
    return o;
}
// The interval spanned by folded minima and maxima (fold_add).
__device__ __forceinline__ Range range_of(const TopkArgs& a, const unsigned long long* mm) {
    Range o{__ldcg(mm + 0), __ldcg(mm + 1), 0u, max_rowid(a)};
    if (o.rlo == o.rhi) {
        o.ilo = static_cast<uint32_t>(__ldcg(mm + 2));
        o.ihi = static_cast<uint32_t>(__ldcg(mm + 3));
    }
    return o;
}

// Minimum and maximum of rank words and of row-ids, folded per thread, then
// over the CTA into four global words (one atomic each: same-address atomics
// serialise in L2).
struct Fold {
    uint64_t rmin, rmax;
    uint32_t imin, imax;
};
__device__ __forceinline__ Fold fold_none() { return Fold{~0ull, 0ull, ~0u, 0u}; }
__device__ __forceinline__ void fold_add(Fold& f, uint64_t r, uint32_t rid) {
    f.rmin = min(f.rmin, r);
    f.rmax = max(f.rmax, r);
    f.imin = min(f.imin, rid);
    f.imax = max(f.imax, rid);
}
template <int TPB>
__device__ __forceinline__ Fold fold_cta(Fold f) {            // thread 0 gets the CTA's fold
    __shared__ Fold s_f[TPB / 32];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        f.rmin = min(f.rmin, __shfl_xor_sync(0xFFFFFFFFu, f.rmin, o));
        f.rmax = max(f.rmax, __shfl_xor_sync(0xFFFFFFFFu, f.rmax, o));
    }
    f.imin = __reduce_min_sync(0xFFFFFFFFu, f.imin);
    f.imax = __reduce_max_sync(0xFFFFFFFFu, f.imax);
    if ((threadIdx.x & 31u) == 0) s_f[threadIdx.x >> 5] = f;
    __syncthreads();
    if (threadIdx.x == 0)
        for (int w = 1; w < TPB / 32; ++w) {
            f.rmin = min(f.rmin, s_f[w].rmin);
            f.rmax = max(f.rmax, s_f[w].rmax);
            f.imin = min(f.imin, s_f[w].imin);
            f.imax = max(f.imax, s_f[w].imax);
        }
    __syncthreads();
    return f;
}
template <int TPB>
__device__ __forceinline__ void fold_merge(const Fold& mine, unsigned long long* dst) {
    const Fold f = fold_cta<TPB>(mine);
    if (threadIdx.x == 0 && f.rmin <= f.rmax) {
        atomicMin(dst + 0, static_cast<unsigned long long>(f.rmin));
        atomicMax(dst + 1, static_cast<unsigned long long>(f.rmax));
        atomicMin(dst + 2, static_cast<unsigned long long>(f.imin));
        atomicMax(dst + 3, static_cast<unsigned long long>(f.imax));
    }
}
__device__ __forceinline__ void fold_reset(unsigned long long* mm) {
    mm[0] = mm[2] = ~0ull;
    mm[1] = mm[3] = 0ull;
}

// Prepare kernel: a threshold rank word for the streaming pass from a
// stratified sample of TK_SAMPLE keys (sample j is key (j * n) / TK_SAMPLE +
// (n / TK_SAMPLE) / 2).  The prepare CTAs load it together, one key per
// thread, into a.samples -- from one SM, 8192 scattered loads wait on each
// other's DRAM latency -- and the last CTA to finish runs this radix select
// with a.digit-bit digits on the sample held in registers; it stops as soon as
// the chosen bucket's upper edge has between r and r + 8 samples at or
// below it, which for spread-out keys is after the first digit.  The
// threshold is the largest of those samples.  With the smallest of them it
// also fixes the interval of the select's fused first pass (see fuse_range):
// four times their spread below the threshold, or the threshold alone when
// they are all equal.  When so many samples tie that the candidates would not
// fit their buffer, the streaming pass is told to count only (count_pass).
__device__ void sample_threshold(const TopkArgs& a, unsigned* sh, unsigned long long* sc) {
    uint64_t s[TK_SPT];
#pragma unroll
    for (int j = 0; j < TK_SPT; ++j) s[j] = __ldcg(a.samples + static_cast<uint64_t>(j) * TK_TPB + threadIdx.x);
    const int kb = a.w4 ? 32 : 64;
    const unsigned long long r = a.sample_rank;
    uint64_t prefix = 0, edge = 0;
    unsigned long long rem = r, cum = 0, upto = 0;           // upto: samples up to the edge
    for (int L = 0; L < kb; L += a.digit) {
        const int d = min(a.digit, kb - L);
        for (int b = threadIdx.x; b < TK_BINS; b += TK_TPB) sh[b] = 0;
        __syncthreads();
#pragma unroll
        for (int j = 0; j < TK_SPT; ++j) {
            const bool match = (L == 0) || (((s[j] ^ prefix) >> (64 - L)) == 0);
            if (match) atomicAdd(&sh[static_cast<unsigned>((s[j] << L) >> (64 - d))], 1u);
        }
        __syncthreads();
        const Pick pk = pick_bucket<TK_TPB>(sh, rem, sc);
        prefix |= static_cast<uint64_t>(pk.b) << (64 - L - d);
        rem -= pk.below;
        cum += pk.below;
        edge = prefix | ((1ull << (64 - L - d)) - 1ull);
        upto = cum + pk.in_b;
        if (upto <= r + 8) break;
    }
    // The filter may be launched now (the other CTAs are gone), not before: its
    // first loads, 20 MB over the GPU, keep this CTA's own loads and
    // instruction fetches waiting (2^26 float32 keys: 14 us for the sample
    // with the filter launched at its start, 7 so).
    allow_next_grid();
    __shared__ unsigned long long lo, hi;                    // of the samples up to the edge, mostly few
    if (threadIdx.x == 0) {
        lo = ~0ull;
        hi = 0;
    }
    __syncthreads();
    uint64_t mn = ~0ull, mx = 0;
    if (upto <= 64) {
#pragma unroll
        for (int j = 0; j < TK_SPT; ++j)
            if (s[j] <= edge) {
                atomicMin(&lo, static_cast<unsigned long long>(s[j]));
                atomicMax(&hi, static_cast<unsigned long long>(s[j]));
            }
    } else {                                                 // ties: lane by lane they would wait for each other
#pragma unroll
        for (int j = 0; j < TK_SPT; ++j)
            if (s[j] <= edge) {
                mn = min(mn, s[j]);
                mx = max(mx, s[j]);
            }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            mn = min(mn, __shfl_xor_sync(0xFFFFFFFFu, mn, o));
            mx = max(mx, __shfl_xor_sync(0xFFFFFFFFu, mx, o));
        }
        if ((threadIdx.x & 31u) == 0) {
            atomicMin(&lo, static_cast<unsigned long long>(mn));
            atomicMax(&hi, static_cast<unsigned long long>(mx));
        }
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        const uint64_t t = hi, d = hi - lo;
        a.ctl->thresh = t;
        a.ctl->fbase = d >= t / 4 ? (d ? 0ull : t) : t - 4 * d;
        a.ctl->count_only = a.fuse && !a.host_keys && 4 * upto * a.n > 5 * a.cand_cap * TK_SAMPLE;
        a.ctl->ts[1] = gtimer();
    }
}

// Hits of the streaming pass are staged per warp in shared memory and
// flushed to the global candidate buffer WS_CAP at a time: one atomic on the
// global count per flush instead of one per warp-vector with a hit (a single
// global counter hit by every SM serialises in L2), and coalesced writes.
struct FuseRange {
    Range g;
    int sh;
    int count_only;
};
__device__ __forceinline__ FuseRange fuse_range(const TopkArgs& a) {
    FuseRange f;
    f.g = Range{__ldcg(&a.ctl->fbase), __ldcg(&a.ctl->thresh), 0u, max_rowid(a)};
    f.count_only = __ldcg(&a.ctl->count_only);
    f.sh = range_shift(f.g, a.digit);
    return f;
}

constexpr int WS_CAP = 256;
struct WarpStage {
    uint64_t* w;          // WS_CAP words (shared): the keys' bits, or the rank words of two-column keys
    uint32_t* idx;        // WS_CAP key indices (shared)
    unsigned count;       // entries held (the same in every lane)
    unsigned* hist;       // the CTA's histogram of the fused first pass (shared; NULL without one)
    const FuseRange* fr;  // its interval (shared)
};
constexpr int WS_BYTES = WS_CAP * 12;
// Rank word of a staged word, as three masks: the map of rank_key without
// branches (floats flip the magnitude of negatives, signed types the sign bit,
// DESC complements; 4-byte keys lie in the upper half; two-column words are
// ranks already).  Ranked as they leave the stage, in one loop, not as they
// enter it, in one of the filter's 16 unrolled places.
struct RankMask {
    uint64_t flip, fixed;
    int up;
};
__device__ __forceinline__ RankMask rank_mask(const TopkArgs& a) {
    RankMask m{0ull, 0ull, 0};
    if (a.pair) return m;
    const uint64_t all = a.w4 ? 0xFFFFFFFF00000000ull : ~0ull;
    if (a.kind == OLAP_KEY_F32 || a.kind == OLAP_KEY_F64) m.flip = all & ~SIGN64;
    if (a.kind != OLAP_KEY_U32 && a.kind != OLAP_KEY_U64) m.fixed = SIGN64;
    if (a.desc) m.fixed ^= all;
    m.up = a.w4 ? 32 : 0;
    return m;
}
__device__ __forceinline__ uint64_t staged_rank(const RankMask& m, uint64_t w) {
    const uint64_t v = w << m.up;
    return v ^ (static_cast<uint64_t>(static_cast<int64_t>(v) >> 63) & m.flip) ^ m.fixed;
}
constexpr int FUSE_BYTES = (TK_BINS + 4) * 4;     // the histogram, its count of entries below, 16-byte units

__device__ __forceinline__ WarpStage warp_stage(unsigned char* base, unsigned* hist, const FuseRange* fr) {
    const unsigned w = threadIdx.x >> 5;
    unsigned char* p = base + static_cast<size_t>(w) * WS_BYTES;
    return WarpStage{reinterpret_cast<uint64_t*>(p), reinterpret_cast<uint32_t*>(p + WS_CAP * 8), 0u, hist, fr};
}

// The select's first refine pass, folded into the streaming filter (the
// register and two-column filters).  Every candidate already passes through
// a warp stage; as it leaves, its bin of the interval [fbase, threshold] is
// counted in a CTA histogram in shared memory, which the CTA adds to the
// select's pass-0 histogram when it is done.  The select then starts at the
// bin pick, one pass over the candidates and one grid barrier sooner.  The
// interval comes from the sampled keys at or below the threshold, so it fits
// keys that cluster (doubles of one magnitude) and, when those samples are
// all equal, bins the ties by row-id.  2^26 rows ordered by a 1024-value
// column and a second one: one pass instead of three over the candidates, the
// select 29 -> 11.6 us.  Candidates below the interval are counted in one
// more word.

template <int TPB>
__device__ __forceinline__ void fuse_init(unsigned* hist) {
    for (int b = threadIdx.x; b <= TK_BINS; b += TPB) hist[b] = 0;
    __syncthreads();
}

__device__ __forceinline__ void fuse_add(unsigned* hist, const FuseRange& f, uint64_t r, uint32_t rid) {
    atomicAdd(&hist[r < f.g.rlo ? TK_BINS : range_bin(f.g, f.sh, r, rid)], 1u);
}

// Whole CTA, after its last candidate: add the CTA's counts to the pass-0
// histogram (non-zero bins only).
template <int TPB>
__device__ __forceinline__ void fuse_merge(const TopkArgs& a, const unsigned* hist) {
    __syncthreads();
    for (int b = threadIdx.x; b < TK_BINS; b += TPB)
        if (hist[b]) atomicAdd(&a.ghist[b], hist[b]);
    if (threadIdx.x == 0 && hist[TK_BINS]) atomicAdd(&a.ctl->flow, static_cast<unsigned long long>(hist[TK_BINS]));
}

// Move the warp's staged hits to the candidate buffer (all 32 lanes call).
__device__ __forceinline__ void stage_flush_plain(const TopkArgs& a, WarpStage& ws) {
    if (ws.count == 0) return;
    __syncwarp();
    const unsigned lane = threadIdx.x & 31u;
    unsigned long long base = 0;
    if (lane == 0) base = atomicAdd(&a.ctl->cand_count, static_cast<unsigned long long>(ws.count));
    base = __shfl_sync(0xFFFFFFFFu, base, 0);
    const RankMask m = rank_mask(a);
    for (unsigned j = lane; j < ws.count; j += 32) {
        const unsigned long long pos = base + j;
        if (pos < a.cand_cap) {
            const uint32_t idx = ws.idx[j];
            a.cand_r[pos] = staged_rank(m, ws.w[j]);
            a.cand_rid[pos] = a.rowids ? a.rowids[idx] : idx;
        }
    }
    __syncwarp();
    ws.count = 0;
}

// The same, also counting the hits for the fused first pass.
__device__ __forceinline__ void stage_write_fused(const TopkArgs& a, const WarpStage& ws, unsigned long long base) {
    const FuseRange f = *ws.fr;
    const RankMask m = rank_mask(a);
    for (unsigned j = threadIdx.x & 31u; j < ws.count; j += 32) {
        const unsigned long long pos = base + j;
        const uint32_t idx = ws.idx[j];
        const uint64_t r = staged_rank(m, ws.w[j]);
        const uint32_t rid = a.rowids ? a.rowids[idx] : idx;
        if (pos < a.cand_cap) {
            a.cand_r[pos] = r;
            a.cand_rid[pos] = rid;
        }
        fuse_add(ws.hist, f, r, rid);
    }
}
__device__ __forceinline__ void stage_flush_fused(const TopkArgs& a, const WarpStage& ws) {
    __syncwarp();
    unsigned long long base = 0;
    if ((threadIdx.x & 31u) == 0) base = atomicAdd(&a.ctl->cand_count, static_cast<unsigned long long>(ws.count));
    base = __shfl_sync(0xFFFFFFFFu, base, 0);
    stage_write_fused(a, ws, base);
    __syncwarp();
}

template <bool FUSE = false>
__device__ __forceinline__ void stage_flush(const TopkArgs& a, WarpStage& ws) {
    if (!FUSE) {
        stage_flush_plain(a, ws);
        return;
    }
    if (ws.count == 0) return;
    stage_flush_fused(a, ws);
    ws.count = 0;
}

// Stage the hits of a warp-vector: bit e of `hit` set for the lane's element e
// of VEC, whose word to stage is word(e) and whose index is idx0 + e (all 32
// lanes call).  Most vectors that get here have one or two hits in all, so the
// elements without any are skipped by one warp-wide OR.
template <int VEC, bool FUSE, typename WordOf>
__device__ __forceinline__ void stage_hits(const TopkArgs& a, unsigned hit, uint64_t idx0, WarpStage& ws, WordOf word) {
    const unsigned lt = (1u << (threadIdx.x & 31u)) - 1u;
    const unsigned any = __reduce_or_sync(0xFFFFFFFFu, hit);
    const unsigned total = __reduce_add_sync(0xFFFFFFFFu, static_cast<unsigned>(__popc(hit)));
    if (ws.count + total > WS_CAP) stage_flush<FUSE>(a, ws);
    unsigned before = ws.count;
#pragma unroll
    for (int e = 0; e < VEC; ++e) {
        if (!((any >> e) & 1u)) continue;
        const bool h = (hit >> e) & 1u;
        const unsigned bal = __ballot_sync(0xFFFFFFFFu, h);
        if (h) {
            const unsigned pos = before + __popc(bal & lt);
            ws.w[pos] = word(e);
            ws.idx[pos] = static_cast<uint32_t>(idx0 + e);
        }
        before += __popc(bal);
    }
    ws.count = before;
}

// Test the keys of one vector of NW 32-bit words (keys idx0 ...) against the
// threshold and stage the hits.  Called by all 32 lanes of a warp together.
template <bool W4, int NW, bool FUSE>
__device__ __forceinline__ void filter_vector(const TopkArgs& a, const KeyLimit& lim, const uint32_t (&w)[NW],
                                              bool valid, uint64_t idx0, WarpStage& ws) {
    constexpr int VEC = W4 ? NW : NW / 2;
    auto key = [&](int e) {
        return W4 ? static_cast<uint64_t>(w[e]) : static_cast<uint64_t>(w[2 * e]) | (static_cast<uint64_t>(w[2 * e + 1]) << 32);
    };
    auto pass = [&](int e) { return W4 ? pass32(w[e], lim) : pass64(key(e), lim); };
    bool any = false;
#pragma unroll
    for (int e = 0; e < VEC; ++e) any = any | pass(e);
    if (!__any_sync(0xFFFFFFFFu, any && valid)) return;
    unsigned hit = 0;
#pragma unroll
    for (int e = 0; e < VEC; ++e) hit |= (valid && pass(e)) ? (1u << e) : 0u;
    stage_hits<VEC, FUSE>(a, hit, idx0, ws, key);
}

// The unaligned head [0, head) and ragged tail [tail0, n) of the keys: at
// most 14 keys, one per lane of warp 0 of CTA 0.
template <bool FUSE = false, bool COPY = false>
__device__ __forceinline__ void filter_ends(const TopkArgs& a, uint64_t t, uint64_t head, uint64_t tail0,
                                            WarpStage& ws) {
    if (blockIdx.x != 0 || threadIdx.x >= 32) return;
    const uint64_t rest = head + (a.n - tail0);
    const uint64_t j = threadIdx.x;
    const bool valid = j < rest;
    uint64_t idx = 0, r = ~0ull, word = 0;
    if (valid) {
        idx = j < head ? j : tail0 + (j - head);
        if (a.pair) {
            word = r = load_input(a, idx).r;
        } else {
            word = key_bits(a, COPY ? a.host_keys : a.keys, idx);
            r = rank_key(word, a.kind, a.desc);
            if (COPY && a.w4) static_cast<uint32_t*>(const_cast<void*>(a.keys))[idx] = static_cast<uint32_t>(word);
            else if (COPY) static_cast<uint64_t*>(const_cast<void*>(a.keys))[idx] = word;
        }
    }
    stage_hits<1, FUSE>(a, valid && r <= t ? 1u : 0u, idx, ws, [&](int) { return word; });
}

// The last hits of all warps of the CTA, with one atomic on the global count
// (one per warp is 4864 on one word at the end of the pass: 4 us).
template <int TPB>
__device__ __forceinline__ void cta_flush_fused(const TopkArgs& a, const WarpStage& ws) {
    __shared__ unsigned cnts[TPB / 32];
    __shared__ unsigned long long s_base;
    const unsigned lane = threadIdx.x & 31u, warp = threadIdx.x >> 5;
    if (lane == 0) cnts[warp] = ws.count;
    __syncthreads();
    unsigned before = 0, all = 0;
#pragma unroll
    for (int w = 0; w < TPB / 32; ++w) {
        if (w < static_cast<int>(warp)) before += cnts[w];
        all += cnts[w];
    }
    if (threadIdx.x == 0 && all) s_base = atomicAdd(&a.ctl->cand_count, static_cast<unsigned long long>(all));
    __syncthreads();
    if (all) stage_write_fused(a, ws, s_base + before);
}

// The streaming pass when the candidates would not fit (few distinct keys): no
// entry is stored, but all up to the threshold are counted as above, so the
// select reads the input with its first refine pass done.  K = 10, 2 * 10^6
// int64 keys of one value 95 -> 54 us (56 without a sample), of 12 values 101 ->
// 55 (75); 2^26 keys of one value 3226 -> 1545.
// A call: its code would lie in the way of the common path, which every launch
// fetches anew.
template <int TPB>
__device__ __noinline__ void count_pass(const TopkArgs& a, const FuseRange& f, unsigned* hist) {
    constexpr int U = 4;                       // loads in flight per thread
    const unsigned lane = threadIdx.x & 31u;
    const uint64_t stride = static_cast<uint64_t>(TPB) * gridDim.x;
    const bool ties = f.g.rlo == f.g.rhi;      // the bins are of row-ids
    unsigned hits = 0;
    for (uint64_t wb = static_cast<uint64_t>(blockIdx.x) * TPB + (threadIdx.x & ~31u); wb < a.n; wb += U * stride) {
        uint64_t r[U];
#pragma unroll
        for (int u = 0; u < U; ++u)
            if (wb + lane + u * stride < a.n) r[u] = input_rank(a, wb + lane + u * stride);
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const uint64_t i = wb + lane + u * stride;
            const bool in = i < a.n && r[u] <= f.g.rhi;
            unsigned bin = 0xFFFFFFFFu;
            if (in && r[u] < f.g.rlo) bin = TK_BINS;
            else if (in) bin = range_bin(f.g, f.sh, r[u], ties ? input_rowid(a, i) : 0u);
            const unsigned peers = __match_any_sync(0xFFFFFFFFu, bin);
            if (in && lane == static_cast<unsigned>(__ffs(peers) - 1))
                atomicAdd(&hist[bin], static_cast<unsigned>(__popc(peers)));
            hits += in ? 1u : 0u;
        }
    }
    __shared__ unsigned s_hits[TPB / 32];
    hits = __reduce_add_sync(0xFFFFFFFFu, hits);
    if (lane == 0) s_hits[threadIdx.x >> 5] = hits;
    __syncthreads();
    if (threadIdx.x == 0) {
        unsigned long long all = 0;
        for (int w = 0; w < TPB / 32; ++w) all += s_hits[w];
        if (all) atomicAdd(&a.ctl->cand_count, all);
    }
    fuse_merge<TPB>(a, hist);
}

// Phase 1: the single streaming pass.  Appends (rank word, row-id) of every
// key whose rank word is <= t; counts all of them.  Two 32-byte loads in
// flight per thread, tested in one comparison per key and one vote per 64
// bytes.  The first loads are issued before the threshold is known: the keys
// are complete (the prepare kernel has waited for everything before it), so
// only the threshold has to be waited for.  Bound by HBM: 2^28 int64 keys
// 313 -> 303 us (7.1 TB/s); 2 * 10^7 float32 keys, with the final flush by
// CTA, 24 -> 15 us of the kernel, most of it start and end.
template <bool W4>
struct FilterSpan {                            // the 32-byte vectors of the keys
    static constexpr int W = W4 ? 4 : 8;
    static constexpr int VEC = 32 / W;
    uint64_t head, nvec, tail0;
    const unsigned char* base;
    __device__ FilterSpan(const TopkArgs& a, const void* keys) {
        const uint64_t head0 = ((32 - (reinterpret_cast<uintptr_t>(keys) & 31)) & 31) / W;
        head = head0 < a.n ? head0 : a.n;
        nvec = (a.n - head) / VEC;
        tail0 = head + nvec * VEC;
        base = static_cast<const unsigned char*>(keys) + head * W;
    }
};

template <int TPB>
__device__ __forceinline__ void filter_load(const unsigned char* base, uint64_t end, uint64_t bb,
                                            uint32_t (&v)[TK_UNROLL][8]) {
#pragma unroll
    for (int u = 0; u < TK_UNROLL; ++u) {
        const uint64_t vi = bb + static_cast<uint64_t>(u) * TPB + threadIdx.x;
        ld_stream_words(base + (vi < end ? vi : 0) * 32, v[u]);
    }
}

// The steps of a CTA: PER vectors each while whole rounds of the grid
// remain; what is left after those is split evenly, so that no CTA has a
// round more than another.
struct FilterStep {
    uint64_t bb, end;                          // vectors of the current step
    uint64_t whole;                            // vectors of the whole rounds
    __device__ void split(uint64_t nvec, uint64_t per) {      // after the last whole round
        const uint64_t share = ((nvec - whole + gridDim.x - 1) / gridDim.x + 31) & ~31ull;
        bb = min(nvec, whole + share * blockIdx.x);
        end = min(nvec, bb + share);
    }
    __device__ void first(uint64_t nvec, uint64_t per) {
        whole = nvec / (per * gridDim.x) * (per * gridDim.x);
        bb = per * blockIdx.x;
        end = bb + per;
        if (bb >= whole) split(nvec, per);
    }
    __device__ void next(uint64_t nvec, uint64_t per) {
        if (bb >= whole) {
            bb = end;
            return;
        }
        bb += per * gridDim.x;
        end = bb + per;
        if (bb >= whole) split(nvec, per);
    }
};

template <bool W4, int TPB, int MODE, bool COPY>
__device__ __forceinline__ void filter_loop(const TopkArgs& a, const FilterSpan<W4>& sp, uint64_t lim, FilterStep st,
                                            uint32_t (&v)[TK_UNROLL][8], WarpStage& ws) {
    constexpr int VEC = FilterSpan<W4>::VEC;
    constexpr uint64_t PER = static_cast<uint64_t>(TPB) * TK_UNROLL;
    auto key = [&](int u, int e) {
        return W4 ? static_cast<uint64_t>(v[u][e])
                  : static_cast<uint64_t>(v[u][2 * e]) | (static_cast<uint64_t>(v[u][2 * e + 1]) << 32);
    };
    auto pass = [&](int u, int e) {
        return W4 ? key_pass<MODE, uint32_t, int32_t>(v[u][e], static_cast<uint32_t>(lim))
                  : key_pass<MODE, uint64_t, int64_t>(key(u, e), lim);
    };
    unsigned char* copy = COPY ? const_cast<unsigned char*>(static_cast<const unsigned char*>(a.keys)) + sp.head * sp.W
                               : nullptr;
    while (st.bb < st.end) {
        if (COPY) {
#pragma unroll
            for (int u = 0; u < TK_UNROLL; ++u) {
                const uint64_t vi = st.bb + static_cast<uint64_t>(u) * TPB + threadIdx.x;
                if (vi < st.end) st_words(copy + vi * 32, v[u]);
            }
        }
        bool any = false;
#pragma unroll
        for (int u = 0; u < TK_UNROLL; ++u)
#pragma unroll
            for (int e = 0; e < VEC; ++e) any = any | pass(u, e);
        if (__any_sync(0xFFFFFFFFu, any)) {
#pragma unroll
            for (int u = 0; u < TK_UNROLL; ++u) {
                const uint64_t vi = st.bb + static_cast<uint64_t>(u) * TPB + threadIdx.x;
                unsigned hit = 0;
#pragma unroll
                for (int e = 0; e < VEC; ++e) hit |= (vi < st.end && pass(u, e)) ? (1u << e) : 0u;
                if (__any_sync(0xFFFFFFFFu, hit != 0))
                    stage_hits<VEC, true>(a, hit, sp.head + vi * VEC, ws, [&](int e) { return key(u, e); });
            }
        }
        st.next(sp.nvec, PER);
        if (st.bb < st.end) filter_load<TPB>(sp.base, st.end, st.bb, v);
    }
}

template <bool W4, int TPB, bool COPY = false>
__device__ __forceinline__ void filter_pass(const TopkArgs& a, unsigned char* fsm) {
    unsigned* hist = reinterpret_cast<unsigned*>(fsm);
    __shared__ FuseRange s_fr;
    fuse_init<TPB>(hist);
    const FilterSpan<W4> sp(a, COPY ? a.host_keys : a.keys);
    FilterStep st;
    st.first(sp.nvec, static_cast<uint64_t>(TPB) * TK_UNROLL);
    uint32_t v[TK_UNROLL][8];
    if (st.bb < st.end) filter_load<TPB>(sp.base, st.end, st.bb, v);
    wait_prior_grid();
    allow_next_grid();
    if (threadIdx.x == 0) s_fr = fuse_range(a);
    __syncthreads();
    if (!COPY && s_fr.count_only) return count_pass<TPB>(a, s_fr, hist);
    const uint64_t t = s_fr.g.rhi;
    const KeyLimit kl = key_limit(t, a.kind, a.desc);
    uint64_t lim;
    int mode;
    if (W4) {
        uint32_t l32;
        mode = key_cmp<uint32_t>(kl.m32, kl.c32, &l32);
        lim = l32;
    } else {
        mode = key_cmp<uint64_t>(kl.m64, kl.c64, &lim);
    }
    WarpStage ws = warp_stage(fsm + FUSE_BYTES, hist, &s_fr);
    if (mode == CMP_GE_U) filter_loop<W4, TPB, CMP_GE_U, COPY>(a, sp, lim, st, v, ws);
    else if (mode == CMP_LE_U) filter_loop<W4, TPB, CMP_LE_U, COPY>(a, sp, lim, st, v, ws);
    else if (mode == CMP_GE_S) filter_loop<W4, TPB, CMP_GE_S, COPY>(a, sp, lim, st, v, ws);
    else filter_loop<W4, TPB, CMP_LE_S, COPY>(a, sp, lim, st, v, ws);
    filter_ends<true, COPY>(a, t, sp.head, sp.tail0, ws);
    cta_flush_fused<TPB>(a, ws);
    fuse_merge<TPB>(a, hist);
}

// The 32-bit order-preserving transform of one 4-byte key kind as two masks:
// rank = b ^ (sign-extended top bit of b & flip) ^ fixed.  float32 flips the
// magnitude of negatives and sets the sign bit of the others (IEEE
// totalOrder), int32 flips the sign bit, uint32 keeps the bits; DESC
// complements the result.  The same map as rank_key, without branches.
struct Rank32 {
    uint32_t flip, fixed;
};
__device__ __forceinline__ Rank32 rank32_of(int kind, bool desc) {
    Rank32 m;
    m.flip = kind == OLAP_KEY_F32 ? 0x7FFFFFFFu : 0u;
    m.fixed = (kind == OLAP_KEY_U32 ? 0u : 0x80000000u) ^ (desc ? 0xFFFFFFFFu : 0u);
    return m;
}
__device__ __forceinline__ uint32_t rank32(uint32_t b, Rank32 m) {
    return b ^ (static_cast<uint32_t>(static_cast<int32_t>(b) >> 31) & m.flip) ^ m.fixed;
}

// Phase 1 for a two-column key: both columns streamed with vector loads when
// they share their alignment (a scalar head and tail around the vectors; 32
// bytes of each column per load, 16 when they share only that), else row by
// row; every row whose composite rank word is <= t is appended.  A warp reads
// the second column only where one of its rows passes on the first, or along
// with the first when that was so in its last three steps (few distinct first
// keys): 2^26 rows, 1024 distinct first keys 85 -> 67 us, four 84 (94 when
// always read late).
template <int TPB, int NW>
__device__ void filter_pass_pair_vec(const TopkArgs& a, uint64_t t, WarpStage& ws) {
    constexpr int U = 8 / NW;                  // 32 bytes of each column in flight per thread
    constexpr int VB = NW * 4;
    const uint64_t n = a.n;
    const Rank32 m0 = rank32_of(a.kind, a.desc), m1 = rank32_of(a.kind2, a.desc2);
    const uint32_t t0 = static_cast<uint32_t>(t >> 32);
    const uintptr_t a0 = reinterpret_cast<uintptr_t>(a.keys);
    const uint64_t head0 = ((VB - (a0 & (VB - 1))) & (VB - 1)) / 4;
    const uint64_t head = head0 < n ? head0 : n;
    const uint64_t nvec = (n - head) / NW;
    const uint64_t tail0 = head + nvec * NW;
    const unsigned char* v0 = static_cast<const unsigned char*>(a.keys) + head * 4;
    const unsigned char* v1 = static_cast<const unsigned char*>(a.keys2) + head * 4;
    const uint64_t per_block = static_cast<uint64_t>(TPB) * U;
    const uint64_t stride = per_block * gridDim.x;
    unsigned recent = 0;                       // whether a row passed on the first column, step by step
    for (uint64_t bb = per_block * blockIdx.x; bb < nvec; bb += stride) {
        uint32_t x0[U][NW], x1[U][NW];
        const bool both = (recent & 7u) == 7u;
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const uint64_t vi = bb + static_cast<uint64_t>(u) * TPB + threadIdx.x;
            const uint64_t at = (vi < nvec ? vi : 0) * VB;
            ld_stream_words(v0 + at, x0[u]);
            if (both) ld_stream_words(v1 + at, x1[u]);
        }
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const uint64_t vi = bb + static_cast<uint64_t>(u) * TPB + threadIdx.x;
            bool any = false;
#pragma unroll
            for (int e = 0; e < NW; ++e) any = any | (rank32(x0[u][e], m0) <= t0);
            any = __any_sync(0xFFFFFFFFu, any);
            recent = recent << 1 | (any ? 1u : 0u);
            if (!any) continue;
            if (!both) ld_stream_words(v1 + (vi < nvec ? vi : 0) * VB, x1[u]);
            auto rank = [&](int e) { return (static_cast<uint64_t>(rank32(x0[u][e], m0)) << 32) | rank32(x1[u][e], m1); };
            unsigned hit = 0;
#pragma unroll
            for (int e = 0; e < NW; ++e) hit |= (vi < nvec && rank(e) <= t) ? (1u << e) : 0u;
            if (!__any_sync(0xFFFFFFFFu, hit != 0)) continue;
            stage_hits<NW, true>(a, hit, head + vi * NW, ws, rank);
        }
    }
    filter_ends<true>(a, t, head, tail0, ws);
}

template <int TPB>
__device__ __forceinline__ void filter_pass_pair(const TopkArgs& a, unsigned char* fsm) {
    unsigned* hist = reinterpret_cast<unsigned*>(fsm);
    __shared__ FuseRange s_fr;
    fuse_init<TPB>(hist);
    wait_prior_grid();
    allow_next_grid();
    if (threadIdx.x == 0) s_fr = fuse_range(a);
    __syncthreads();
    if (s_fr.count_only) return count_pass<TPB>(a, s_fr, hist);
    const uint64_t t = s_fr.g.rhi;
    const uint64_t n = a.n;
    const uintptr_t off = reinterpret_cast<uintptr_t>(a.keys) ^ reinterpret_cast<uintptr_t>(a.keys2);
    WarpStage ws = warp_stage(fsm + FUSE_BYTES, hist, &s_fr);
    if ((off & 31) == 0) {
        filter_pass_pair_vec<TPB, 8>(a, t, ws);
    } else if ((off & 15) == 0) {
        filter_pass_pair_vec<TPB, 4>(a, t, ws);
    } else {
    const unsigned lane = threadIdx.x & 31u;
    const uint64_t stride = static_cast<uint64_t>(TPB) * gridDim.x;
    for (uint64_t wb = static_cast<uint64_t>(blockIdx.x) * TPB + (threadIdx.x & ~31u); wb < n; wb += stride) {
        const uint64_t i = wb + lane;
        uint64_t r = ~0ull;
        if (i < n) r = pair_rank(static_cast<const uint32_t*>(a.keys)[i], static_cast<const uint32_t*>(a.keys2)[i], a);
        const bool hit = i < n && r <= t;
        if (!__any_sync(0xFFFFFFFFu, hit)) continue;
        stage_hits<1, true>(a, hit ? 1u : 0u, i, ws, [&](int) { return r; });
    }
    }
    cta_flush_fused<TPB>(a, ws);
    fuse_merge<TPB>(a, hist);
}

// Issue the bulk copy of the tile at byte offset `off` of the key body into
// ring slot `s` (the last tile of the body may be short).
__device__ __forceinline__ void issue_tile(unsigned char* smem, uint64_t* full, const unsigned char* vbase,
                                           uint64_t body, uint64_t off, uint32_t s, uint32_t tile,
                                           uint64_t policy) {
    const uint64_t left = body - off;
    const uint32_t bytes = static_cast<uint32_t>(left < tile ? left : tile);
    mbar_arrive_expect_tx(&full[s], bytes);
    bulk_g2s(smem + static_cast<size_t>(s) * tile, vbase + off, bytes, &full[s], policy);
}

// Phase 1, bulk-copy flavour: each CTA streams its tiles (tile i of the
// grid-interleaved order) through a ring of `stages` shared-memory slots.
// Thread 0 issues cp.async.bulk copies; a slot's "full" mbarrier completes
// when its bytes land, and its "empty" mbarrier when every warp has read it,
// after which thread 0 refills it.  No CTA-wide barrier per tile.  Returns
// false if a copy never landed (bounded waits).
template <bool W4, int TPB>
__device__ bool filter_pass_bulk(const TopkArgs& a, uint64_t t, unsigned char* smem) {
    constexpr int W = W4 ? 4 : 8;
    constexpr int VEC = 16 / W;
    constexpr unsigned NWARPS = TPB / 32;
    const uint32_t tile = static_cast<uint32_t>(a.tile_bytes);
    const uint32_t stages = static_cast<uint32_t>(a.stages);
    const uint64_t n = a.n;
    const uintptr_t addr = reinterpret_cast<uintptr_t>(a.keys);
    const uint64_t head0 = ((16 - (addr & 15)) & 15) / W;
    const uint64_t head = head0 < n ? head0 : n;
    const uint64_t nvec = (n - head) / VEC;
    const uint64_t tail0 = head + nvec * VEC;
    const unsigned char* vbase = static_cast<const unsigned char*>(a.keys) + head * W;
    const uint64_t body = nvec * 16;
    const uint64_t ntiles = (body + tile - 1) / tile;
    const uint64_t my_n = blockIdx.x < ntiles ? (ntiles - 1 - blockIdx.x) / gridDim.x + 1 : 0;
    const KeyLimit lim = key_limit(t, a.kind, a.desc);
    uint64_t* full = reinterpret_cast<uint64_t*>(smem + static_cast<size_t>(tile) * stages);
    uint64_t* empty = full + TK_MAX_STAGES;
    WarpStage ws = warp_stage(reinterpret_cast<unsigned char*>(empty + TK_MAX_STAGES), nullptr, nullptr);
    const uint64_t step = static_cast<uint64_t>(gridDim.x) * tile;       // bytes between my tiles

    if (threadIdx.x == 0) {
        for (uint32_t s = 0; s < stages; ++s) {
            mbar_init(&full[s], 1);
            mbar_init(&empty[s], NWARPS);
        }
        mbar_fence_init();
    }
    __syncthreads();
    const uint64_t policy = l2_evict_first_policy();
    uint64_t off = static_cast<uint64_t>(blockIdx.x) * tile;
    uint64_t issued = 0;                                   // tiles issued (thread 0)
    if (threadIdx.x == 0) {
        const uint32_t pre = static_cast<uint32_t>(my_n < stages ? my_n : stages);
        for (uint32_t s = 0; s < pre; ++s) issue_tile(smem, full, vbase, body, off + s * step, s, tile, policy);
        issued = pre;
    }
    const uint64_t refill = static_cast<uint64_t>(stages) * step;
    const unsigned lane = threadIdx.x & 31u;
    uint32_t s = 0, par = 0;
    bool ok = true;
    for (uint64_t i = 0; i < my_n; ++i) {
        if (!mbar_wait(&full[s], par)) {
            ok = false;
            break;
        }
        const uint64_t left = body - off;
        const uint32_t nv = static_cast<uint32_t>((left < tile ? left : tile) / 16);
        const unsigned char* st = smem + static_cast<size_t>(s) * tile;
        const uint64_t idx_base = head + (off / 16) * VEC;
        for (uint32_t vb = 0; vb < tile / 16; vb += TPB) {
            const uint32_t v = vb + threadIdx.x;
            const bool valid = v < nv;
            uint4 x = make_uint4(0xFFFFFFFFu, 0xFFFFFFFFu, 0xFFFFFFFFu, 0xFFFFFFFFu);
            if (valid) x = ld_shared_v4(st + v * 16);
            const uint32_t xw[4] = {x.x, x.y, x.z, x.w};
            filter_vector<W4, 4, false>(a, lim, xw, valid, idx_base + static_cast<uint64_t>(v) * VEC, ws);
        }
        __syncwarp();
        if (lane == 0) mbar_arrive(&empty[s]);
        if (threadIdx.x == 0 && i + stages < my_n) {
            if (!mbar_wait(&empty[s], par)) {
                ok = false;
                break;
            }
            fence_proxy_async_smem();
            issue_tile(smem, full, vbase, body, off + refill, s, tile, policy);
            ++issued;
        }
        off += step;
        if (++s == stages) {
            s = 0;
            par ^= 1u;
        }
    }
    filter_ends(a, t, head, tail0, ws);
    stage_flush(a, ws);
    if (!__syncthreads_and(ok)) {
        // Let the copies this CTA issued land before leaving.  Only the last
        // `stages` issued tiles can still be in flight (every earlier fill of
        // a slot was consumed before the slot was refilled).
        if (threadIdx.x == 0) {
            const uint64_t first = issued > stages ? issued - stages : 0;
            for (uint64_t q = first; q < issued; ++q)
                mbar_wait(&full[q % stages], static_cast<uint32_t>((q / stages) & 1));
            atomicCAS(&a.ctl->err, 0, static_cast<int>(OLAP_E_TIMEOUT));
        }
        __syncthreads();
        return false;
    }
    return true;
}

// One refine pass: histogram of the bins of the entries in the interval,
// merged into `gh`, and the minima and maxima of those entries merged into
// `mm`.  `gz` and `mz` (the buffers of the pass after next) are reset by
// CTA 0.
__device__ void hist_pass(const TopkArgs& a, bool cand, uint64_t src_n, const Range& g, int shift, unsigned* gh,
                          unsigned* gz, unsigned* sh, unsigned long long* mm, unsigned long long* mz) {
    for (int b = threadIdx.x; b < TK_BINS; b += TK_TPB) sh[b] = 0;
    if (blockIdx.x == 0) {
        for (int b = threadIdx.x; b < TK_BINS; b += TK_TPB) gz[b] = 0;
        if (threadIdx.x == 0) fold_reset(mz);
    }
    __syncthreads();
    Fold acc = fold_none();
    const uint64_t stride = static_cast<uint64_t>(TK_TPB) * gridDim.x;
    const unsigned lane = threadIdx.x & 31u;
    for (uint64_t wb = static_cast<uint64_t>(blockIdx.x) * TK_TPB + (threadIdx.x & ~31u); wb < src_n;
         wb += stride) {
        const uint64_t i = wb + lane;
        unsigned bin = 0xFFFFFFFFu;
        if (i < src_n) {
            const Elem e = load_src(a, cand, i);
            if (range_cmp(g, e.r, e.rid) == 0) {
                bin = range_bin(g, shift, e.r, e.rid);
                fold_add(acc, e.r, e.rid);
            }
        }
        const unsigned peers = __match_any_sync(0xFFFFFFFFu, bin);
        if (bin != 0xFFFFFFFFu && lane == static_cast<unsigned>(__ffs(peers) - 1))
            atomicAdd(&sh[bin], static_cast<unsigned>(__popc(peers)));
    }
    fold_merge<TK_TPB>(acc, mm);
    for (int b = threadIdx.x; b < TK_BINS; b += TK_TPB)
        if (sh[b]) atomicAdd(&gh[b], sh[b]);
}

// Split: entries below the interval are selected (appended to out), entries
// in it go to the small buffer, or to out when all of them (or any `krem`
// identical ones) are taken.  Every entry is loaded one step ahead; `nx` is
// the thread's first candidate on the candidate path.
__device__ void split_pass(const TopkArgs& a, bool cand, uint64_t src_n, const Range& g, bool take_all,
                           uint64_t krem, Elem nx) {
    TopkCtl* ctl = a.ctl;
    const uint64_t stride = static_cast<uint64_t>(TK_TPB) * gridDim.x;
    const unsigned lane = threadIdx.x & 31u;
    const uint64_t eq_base = a.k - krem;
    unsigned long long* eq_ctr = take_all ? &ctl->eq_count : &ctl->small_count;
    const uint64_t i0 = static_cast<uint64_t>(blockIdx.x) * TK_TPB + threadIdx.x;
    if (!cand && i0 < src_n) nx = load_src(a, cand, i0);
    for (uint64_t wb = i0 - lane; wb < src_n; wb += stride) {
        const uint64_t i = wb + lane;
        int c = 1;
        const Elem e = nx;
        if (i < src_n) c = range_cmp(g, e.r, e.rid);
        if (i + stride < src_n) nx = load_src(a, cand, i + stride);
        const unsigned lt = __ballot_sync(0xFFFFFFFFu, c < 0);
        const unsigned eq = __ballot_sync(0xFFFFFFFFu, c == 0);
        if (lt) {
            unsigned long long base = 0;
            if (lane == 0) base = atomicAdd(&ctl->out_count, static_cast<unsigned long long>(__popc(lt)));
            base = __shfl_sync(0xFFFFFFFFu, base, 0);
            if (c < 0) {
                const uint64_t pos = base + __popc(lt & ((1u << lane) - 1u));
                a.out_r0[pos] = e.r;
                a.out_rid0[pos] = e.rid;
            }
        }
        if (eq) {
            unsigned long long base = 0;
            if (lane == 0) base = atomicAdd(eq_ctr, static_cast<unsigned long long>(__popc(eq)));
            base = __shfl_sync(0xFFFFFFFFu, base, 0);
            if (c == 0) {
                const uint64_t pos = base + __popc(eq & ((1u << lane) - 1u));
                if (take_all) {
                    if (pos < krem) {
                        a.out_r0[eq_base + pos] = e.r;
                        a.out_rid0[eq_base + pos] = e.rid;
                    }
                } else if (pos < TK_SMALL) {
                    a.small_r[pos] = e.r;
                    a.small_rid[pos] = e.rid;
                }
            }
        }
    }
}

// The same for the larger-K finish, which also wants the minima and maxima of
// the entries in out (merged into ctl->fin, so that it needs no pass of its
// own).  Nearly every warp has some of those, and an atomic each on one word
// is what such a pass then waits for (2^24 keys, K = 100,000: 97 us; with one
// atomic per CTA and step, between two barriers, 199).  So a warp stages its
// entries for out in shared memory and takes their places SPLIT_CAP at a time.
// SPLIT_U loads are in flight per thread.
constexpr int SPLIT_CAP = 256;
constexpr int SPLIT_U = 4;
static_assert(TK_TPB / 32 * SPLIT_CAP * 12 <= TK_SORT_SMEM, "the warps' stages");
static_assert(SPLIT_U * 32 <= SPLIT_CAP, "a step's entries fit an empty stage");
__device__ void split_pass_large(const TopkArgs& a, bool cand, uint64_t src_n, const Range& g, bool take_all,
                                 uint64_t krem, bool whole, Elem first, unsigned char* smem) {
    TopkCtl* ctl = a.ctl;
    const unsigned lane = threadIdx.x & 31u, warp = threadIdx.x >> 5, lt_mask = (1u << lane) - 1u;
    uint64_t* wr = reinterpret_cast<uint64_t*>(smem + warp * (SPLIT_CAP * 12));
    uint32_t* wrid = reinterpret_cast<uint32_t*>(wr + SPLIT_CAP);
    unsigned cnt = 0;                                        // staged entries of the warp
    Fold acc = fold_none();
    const uint64_t stride = static_cast<uint64_t>(TK_TPB) * gridDim.x;
    const uint64_t eq_base = a.k - krem;
    unsigned long long* eq_ctr = take_all ? &ctl->eq_count : &ctl->small_count;
    const int last = whole ? 0 : -1;                         // range_cmp of the entries that all go to out
    bool loaded = cand;                                      // `first` is the thread's first candidate
    auto write = [&](unsigned long long base) {
        __syncwarp();
        for (unsigned j = lane; j < cnt; j += 32) {
            a.out_r0[base + j] = wr[j];
            a.out_rid0[base + j] = wrid[j];
        }
        __syncwarp();
    };
    for (uint64_t wb = static_cast<uint64_t>(blockIdx.x) * TK_TPB + (threadIdx.x & ~31u); wb < src_n;
         wb += SPLIT_U * stride) {
        Elem e[SPLIT_U];
#pragma unroll
        for (int u = 0; u < SPLIT_U; ++u) {
            const uint64_t i = wb + lane + u * stride;
            if (u == 0 && loaded) e[u] = first;
            else if (i < src_n) e[u] = load_src(a, cand, i);
        }
        loaded = false;
        if (cnt + SPLIT_U * 32 > SPLIT_CAP) {
            unsigned long long base = 0;
            if (lane == 0) base = atomicAdd(&ctl->out_count, static_cast<unsigned long long>(cnt));
            write(__shfl_sync(0xFFFFFFFFu, base, 0));
            cnt = 0;
        }
#pragma unroll
        for (int u = 0; u < SPLIT_U; ++u) {
            const uint64_t i = wb + lane + u * stride;
            const int c = i < src_n ? range_cmp(g, e[u].r, e[u].rid) : 1;
            const unsigned lt = __ballot_sync(0xFFFFFFFFu, c <= last);
            if (c <= last) {
                const unsigned pos = cnt + __popc(lt & lt_mask);
                wr[pos] = e[u].r;
                wrid[pos] = e[u].rid;
                fold_add(acc, e[u].r, e[u].rid);
            }
            cnt += __popc(lt);
            const unsigned eq = __ballot_sync(0xFFFFFFFFu, c == 0 && last < 0);
            if (!eq) continue;
            unsigned long long base = 0;
            if (lane == 0) base = atomicAdd(eq_ctr, static_cast<unsigned long long>(__popc(eq)));
            base = __shfl_sync(0xFFFFFFFFu, base, 0);
            if (c != 0) continue;
            const uint64_t pos = base + __popc(eq & lt_mask);
            if (take_all) {
                if (pos < krem) {
                    a.out_r0[eq_base + pos] = e[u].r;
                    a.out_rid0[eq_base + pos] = e[u].rid;
                    fold_add(acc, e[u].r, e[u].rid);
                }
            } else if (pos < TK_SMALL) {
                a.small_r[pos] = e[u].r;
                a.small_rid[pos] = e[u].rid;
            }
        }
    }
    // what is left of all warps, with one atomic
    __shared__ unsigned s_cnt[TK_TPB / 32];
    __shared__ unsigned long long s_base;
    if (lane == 0) s_cnt[warp] = cnt;
    __syncthreads();
    unsigned before = 0, all = 0;
    for (unsigned w = 0; w < TK_TPB / 32; ++w) {
        if (w < warp) before += s_cnt[w];
        all += s_cnt[w];
    }
    if (threadIdx.x == 0 && all) s_base = atomicAdd(&ctl->out_count, static_cast<unsigned long long>(all));
    __syncthreads();
    if (all) write(s_base + before);
    fold_merge<TK_TPB>(acc, ctl->fin);
}

// Entries of [lo, hi) in shared memory that order before entry e of them
// (equal ones by position); whole warp calls and gets the count.
__device__ __forceinline__ unsigned warp_rank_of(const uint64_t* sr, const uint32_t* srid, int lo, int hi, int e) {
    const uint64_t er = sr[e];
    const uint32_t erid = srid[e];
    unsigned c = 0;
#pragma unroll 4
    for (int j = lo + static_cast<int>(threadIdx.x & 31u); j < hi; j += 32) rank_count(c, sr[j], srid[j], er, erid, j < e);
    return __reduce_add_sync(0xFFFFFFFFu, 0u - c);
}

// Rank a bin of m <= 32 * Q entries in one warp's registers (a lane holds
// entries lane, lane + 32, ...; the others come by shuffle) and write them
// from position o on.
template <int Q>
__device__ __forceinline__ void warp_rank_bin(const TopkArgs& a, uint64_t o, unsigned m) {
    const unsigned lane = threadIdx.x & 31u;
    uint64_t er[Q];
    uint32_t erid[Q];
    unsigned c[Q];
#pragma unroll
    for (int q = 0; q < Q; ++q) {
        const unsigned i = q * 32u + lane;
        er[q] = i < m ? __ldcg(a.out_r1 + o + i) : ~0ull;
        erid[q] = i < m ? __ldcg(a.out_rid1 + o + i) : ~0u;
        c[q] = 0;
    }
#pragma unroll
    for (int p = 0; p < Q; ++p) {
        const unsigned lim = m > p * 32u ? min(32u, m - p * 32u) : 0u;
        for (unsigned j = 0; j < lim; ++j) {
            const uint64_t jr = __shfl_sync(0xFFFFFFFFu, er[p], j);
            const uint32_t jrid = __shfl_sync(0xFFFFFFFFu, erid[p], j);
#pragma unroll
            for (int q = 0; q < Q; ++q) rank_count(c[q], jr, jrid, er[q], erid[q], p < q || (p == q && j < lane));
        }
    }
#pragma unroll
    for (int q = 0; q < Q; ++q)
        if (q * 32u + lane < m) write_result(a, o + (0u - c[q]), er[q], erid[q]);
}

// Merge-path split: how many of the first `diag` outputs of the merge of
// A[0, na) and B[0, nb) come from A (A wins ties, keeping the merge stable).
__device__ __forceinline__ uint64_t merge_path(const uint64_t* ar, const uint32_t* arid, uint64_t na,
                                               const uint64_t* br, const uint32_t* brid, uint64_t nb,
                                               uint64_t diag) {
    uint64_t lo = diag > nb ? diag - nb : 0;
    uint64_t hi = diag < na ? diag : na;
    while (lo < hi) {
        const uint64_t mid = (lo + hi) >> 1;
        const uint64_t j = diag - 1 - mid;
        if (!elem_less(__ldcg(br + j), __ldcg(brid + j), __ldcg(ar + mid), __ldcg(arid + mid))) lo = mid + 1;
        else hi = mid;
    }
    return lo;
}

// Early exit after an expired wait: CTA 0 publishes the device status, and a
// blocking call hears of every CTA.
__device__ __forceinline__ void report(const TopkArgs& a) {
    if (threadIdx.x != 0) return;
    raise_expiry(&a.ctl->err, a.host_err);
    if (blockIdx.x == 0 && a.dev_status) *a.dev_status = ld_volatile_i32(&a.ctl->err);
}

}  // namespace

// Kernel 1 of 3: reset the control block and the histograms (CTA 0, and all
// CTAs' shares), and on the sampled path load the sample and estimate the
// filter threshold (TK_PREP_CTAS CTAs; the last one to finish selects).
__global__ void __launch_bounds__(TK_TPB) topk_prepare_kernel(TopkArgs a) {
    __shared__ unsigned sh[TK_BINS];
    __shared__ unsigned long long sc[24];
    __shared__ int last;
    TopkCtl* ctl = a.ctl;
    wait_prior_grid();                    // the call before may still read the control block
    // (a host column's first loads take the link, not the sample's way: 3 * 10^6
    // page-locked keys 167 -> 162 us)
    if (a.host_keys) allow_next_grid();
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        ctl->ts[0] = gtimer();
        a.bar->count = 0;
        ctl->cand_count = 0;
        ctl->out_count = 0;
        ctl->eq_count = 0;
        ctl->small_count = 0;
        ctl->err = 0;
        ctl->path = a.use_sample ? 1 : 0;
        ctl->passes = 0;
        ctl->flow = 0;
        for (int s = 0; s < 3; ++s) fold_reset(ctl->mm[s]);
        fold_reset(ctl->fin);
    }
    for (int b = blockIdx.x * TK_TPB + threadIdx.x; b < 3 * TK_BINS; b += gridDim.x * TK_TPB) a.ghist[b] = 0;
    if (!a.use_sample) {
        allow_next_grid();
        if (threadIdx.x == 0) ctl->ts[1] = gtimer();
        return;
    }
    const uint64_t j = static_cast<uint64_t>(blockIdx.x) * TK_TPB + threadIdx.x;   // < TK_SAMPLE
    const uint64_t at = (j * a.n) / TK_SAMPLE + (a.n / TK_SAMPLE) / 2;
    a.samples[j] = a.host_keys ? rank_key(key_bits(a, a.host_keys, at), a.kind, a.desc) : load_input(a, at).r;
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) last = (atomicAdd(&a.bar->prep, 1u) + 1u) % gridDim.x == 0;
    __syncthreads();
    if (!last) return;
    __threadfence();
    sample_threshold(a, sh, sc);
}

// Kernel 2 of 3 (sampled path only): the single streaming pass over the keys,
// bulk-copy flavour.  Independent CTAs, several per SM.
template <bool W4>
__global__ void __launch_bounds__(TKF_TPB, 4) topk_filter_bulk_kernel(TopkArgs a) {
    extern __shared__ __align__(128) unsigned char fsmem[];
    wait_prior_grid();
    allow_next_grid();
    const uint64_t t = __ldcg(&a.ctl->thresh);
    filter_pass_bulk<W4, TKF_TPB>(a, t, fsmem);
}

// Kernel 2 of 3, register-load flavour (TPB threads; dynamic shared memory:
// the fused pass's histogram and the per-warp stages).
template <bool W4, int TPB>
__global__ void __launch_bounds__(TPB, 1024 / TPB) topk_filter_regs_kernel(const __grid_constant__ TopkArgs a) {
    extern __shared__ __align__(16) unsigned char fsm[];
    filter_pass<W4, TPB>(a, fsm);
}

// Kernel 2 of 3 for a column in host memory that the device reads itself: the
// same pass over the host column, which also leaves the copy in device memory
// (a.keys, at the same offset from a 32-byte boundary) that a misjudged
// sample's select reads.  Bound by the host link, which a kernel's loads fill
// as well as a DMA copy (2^31 bytes 10.16 against 10.15 ms, 24 MB 120 against
// 117 us): the filter's own pass over the copy goes, and the first loads are
// under way while the sample is ranked.  2^21.5 page-locked int64 keys 173 ->
// 157 us for the call, 2^24 710 -> 680, 2^28 10512 -> 10220.
template <bool W4>
__global__ void __launch_bounds__(TKR_TPB, 1) topk_filter_host_kernel(TopkArgs a) {
    extern __shared__ __align__(16) unsigned char fsm[];
    filter_pass<W4, TKR_TPB, true>(a, fsm);
}

// Kernel 2 of 3 for a two-column key (register loads of both columns).
template <int TPB>
__global__ void __launch_bounds__(TPB, 1024 / TPB) topk_filter_pair_kernel(const __grid_constant__ TopkArgs a) {
    extern __shared__ __align__(16) unsigned char fsm[];
    filter_pass_pair<TPB>(a, fsm);
}

// The select's finish for more survivors than one CTA's shared memory ranks.
__device__ void finish_large(const TopkArgs& a, unsigned char* smem, unsigned long long* sc,
                                          unsigned bar_target, int pass, bool take_all, uint64_t krem, uint64_t bcnt) {
    TopkCtl* ctl = a.ctl;
    unsigned* sh = reinterpret_cast<unsigned*>(smem);
    uint64_t* sr = reinterpret_cast<uint64_t*>(smem);
    uint32_t* srid = reinterpret_cast<uint32_t*>(smem + TK_RANK_MAX * 8);
    const bool stamp = blockIdx.x == 0 && threadIdx.x == 0;
    // Phase 4, larger K.  (a) The bucket entries (ns <= 4096) are ranked by
    // the grid as above and the first krem written at their final positions.
    // (b) The below entries are partitioned into bins -- a histogram, a scan,
    // a scatter into out_r1 -- and every bin is ranked and written at its
    // final positions.  The bins are first the 4096 equal ones of the interval
    // the entries span; when one of those holds more than TK_SMALL (a few
    // heavily tied keys), they are the gaps between 2047 of the entries, taken
    // evenly and sorted, with the entries equal to one of those
    // in bins of their own, which need no ranking: composites rarely tie, so
    // any distribution of keys splits (10^8 int32 keys of 1024 values,
    // K = 100,000: finish 222 -> 50 us).  More entries than such bins can
    // take, or an unlucky choice, fall back to tile sorts and merge-path rounds.
    {
        const uint64_t nb = take_all ? a.k : a.k - krem;
        const int nsi = take_all ? 0 : static_cast<int>(bcnt);
        const unsigned lane = threadIdx.x & 31u;
        const int nwarps = static_cast<int>(gridDim.x) * (TK_TPB / 32);
        const int gw = static_cast<int>(blockIdx.x) * (TK_TPB / 32) + static_cast<int>(threadIdx.x >> 5);
        if (nsi > 0) {
            for (int i = threadIdx.x; i < nsi; i += TK_TPB) {
                sr[i] = __ldcg(a.small_r + i);
                srid[i] = __ldcg(a.small_rid + i);
            }
            __syncthreads();
            for (int e = gw; e < nsi; e += nwarps) {
                const unsigned c = warp_rank_of(sr, srid, 0, nsi, e);
                if (lane == 0 && c < krem) write_result(a, nb + c, sr[e], srid[e]);
            }
            __syncthreads();
        }
        // One partition with the given bins: 1 done, 0 a bin too large, -1 a
        // wait expired.  ph: clean; pc: zeroed here for the cursors; `pure`:
        // odd bins hold identical entries; `most`: entries of a bin.
        auto partition = [&](auto bin, unsigned* ph, unsigned* pc, bool pure, unsigned most) -> int {
            for (int b = threadIdx.x; b < TK_BINS; b += TK_TPB) sh[b] = 0;
            if (blockIdx.x == 0)
                for (int b = threadIdx.x; b < TK_BINS; b += TK_TPB) pc[b] = 0;
            __syncthreads();
            const uint64_t gstride = static_cast<uint64_t>(TK_TPB) * gridDim.x;
            for (uint64_t wb = static_cast<uint64_t>(blockIdx.x) * TK_TPB + (threadIdx.x & ~31u); wb < nb;
                 wb += gstride) {
                const uint64_t i = wb + lane;
                unsigned dig = 0xFFFFFFFFu;
                if (i < nb) dig = bin(__ldcg(a.out_r0 + i), __ldcg(a.out_rid0 + i));
                const unsigned peers = __match_any_sync(0xFFFFFFFFu, dig);
                if (dig != 0xFFFFFFFFu && lane == static_cast<unsigned>(__ffs(peers) - 1))
                    atomicAdd(&sh[dig], static_cast<unsigned>(__popc(peers)));
            }
            __syncthreads();
            for (int b = threadIdx.x; b < TK_BINS; b += TK_TPB)
                if (sh[b]) atomicAdd(&ph[b], sh[b]);
            if (!grid_sync(a.bar, &ctl->err, bar_target)) return -1;
            // Scan of the partition histogram (every CTA), largest bin.
            constexpr int PER = TK_BINS / TK_TPB;
            unsigned v[PER];
            unsigned long long local = 0;
            unsigned mx = 0;
            pick_load_global<TK_TPB>(ph, v);
#pragma unroll
            for (int j = 0; j < PER; ++j) {
                local += v[j];
                if (!(pure && (j & 1))) mx = max(mx, v[j]);
            }
            unsigned* off = sh;                              // exclusive offsets per bin
            unsigned long long run = block_excl_scan<TK_TPB>(local, sc, sc + 16);
#pragma unroll
            for (int j = 0; j < PER; ++j) {
                off[threadIdx.x * PER + j] = static_cast<unsigned>(run);
                run += v[j];
            }
            if (!__syncthreads_and(mx <= most)) return 0;
            // Scatter the below entries into bin order (out_r1).
            for (uint64_t i = static_cast<uint64_t>(blockIdx.x) * TK_TPB + threadIdx.x; i < nb; i += gstride) {
                const uint64_t er = __ldcg(a.out_r0 + i);
                const uint32_t erid = __ldcg(a.out_rid0 + i);
                const unsigned d = bin(er, erid);
                const unsigned pos = off[d] + atomicAdd(&pc[d], 1u);
                a.out_r1[pos] = er;
                a.out_rid1[pos] = erid;
            }
            if (!grid_sync(a.bar, &ctl->err, bar_target)) return -1;
            // Bins of at most 128 entries: one warp each, in registers.
            // (`pure`: pairs of bins, so that the warps and CTAs share the even
            // ones evenly; grids are even)
            auto size = [&](int b) { return (b + 1 < TK_BINS ? off[b + 1] : static_cast<unsigned>(nb)) - off[b]; };
            const int each = pure ? 2 : 1;
            for (int b = gw * each; b < TK_BINS; b += nwarps * each) {
                if (pure) {                                  // the identical entries after bin b
                    const unsigned o = off[b + 1], same = size(b + 1);
                    for (unsigned i = lane; i < same; i += 32)
                        write_result(a, o + i, __ldcg(a.out_r1 + o + i), __ldcg(a.out_rid1 + o + i));
                }
                const unsigned m = size(b), o = off[b];
                if (m == 0 || m > 128) continue;
                if (m <= 32) warp_rank_bin<1>(a, o, m);
                else if (m <= 64) warp_rank_bin<2>(a, o, m);
                else warp_rank_bin<4>(a, o, m);
            }
            // Larger bins: one CTA each, in shared memory, one or two threads
            // an entry that go through the bin together (a warp an entry, as
            // for the small buffer, spends most of its time on the sums: 2^24
            // uniform int64 keys, K = 10^6 the call 647 -> 522 us).
            uint64_t* br = reinterpret_cast<uint64_t*>(smem + TK_BINS * 4);
            uint32_t* brid = reinterpret_cast<uint32_t*>(smem + TK_BINS * 4 + TK_SMALL * 8);
            for (int b = static_cast<int>(blockIdx.x) * each; b < TK_BINS; b += static_cast<int>(gridDim.x) * each) {
                const unsigned m = size(b);
                if (m <= 128) continue;
                const unsigned o = off[b];
                for (unsigned i = threadIdx.x; i < m; i += TK_TPB) {
                    br[i] = __ldcg(a.out_r1 + o + i);
                    brid[i] = __ldcg(a.out_rid1 + o + i);
                }
                __syncthreads();
                const unsigned two = m <= TK_TPB / 2 ? 1u : 0u;
                for (unsigned e0 = 0; e0 < m; e0 += TK_TPB >> two) {
                    const unsigned e = e0 + (threadIdx.x >> two);
                    const unsigned at = e < m ? e : 0u;
                    const uint64_t er = br[at];
                    const uint32_t erid = brid[at];
                    unsigned c = 0;
#pragma unroll 4
                    for (unsigned j = threadIdx.x & two; j < m; j += 1u + two) rank_count(c, br[j], brid[j], er, erid, j < at);
                    if (two) c += __shfl_xor_sync(0xFFFFFFFFu, c, 1);
                    if (e < m && !(threadIdx.x & two)) write_result(a, o + (0u - c), er, erid);
                }
                __syncthreads();
            }
            return 1;
        };
        unsigned* hb[3];                                     // the three histograms; hb[0] is clean
        for (int j = 0; j < 3; ++j) hb[j] = a.ghist + ((pass + j) % 3) * TK_BINS;
        const Range pr = range_of(a, ctl->fin);
        const int psh = range_shift(pr, a.digit);
        const bool splits = nb <= TK_SPLIT_MAX;
        int done = partition([&](uint64_t r, uint32_t rid) { return range_bin(pr, psh, r, rid); }, hb[0], hb[1], false,
                             splits ? TK_BIN_EVEN : TK_BIN_MAX);
        if (done == 0 && splits) {
            uint64_t* pr_r = reinterpret_cast<uint64_t*>(smem + TK_BINS * 4 + TK_SMALL * 12);
            uint32_t* pr_rid = reinterpret_cast<uint32_t*>(smem + TK_BINS * 4 + TK_SMALL * 12 + (TK_SPLITTERS + 1) * 8);
            for (int j = threadIdx.x; j < TK_SPLITTERS; j += TK_TPB) {
                const uint64_t i = static_cast<uint64_t>(j) * nb / TK_SPLITTERS;
                pr_r[j] = __ldcg(a.out_r0 + i);
                pr_rid[j] = __ldcg(a.out_rid0 + i);
            }
            __syncthreads();
            // sorted by the grid: every warp ranks some (in one CTA a bitonic
            // sort of 2047 takes 50 us), in out_r1, which is free until the entries
            // are scattered; every CTA has read them in order before that
            for (int e = gw; e < TK_SPLITTERS; e += nwarps) {
                const unsigned c = warp_rank_of(pr_r, pr_rid, 0, TK_SPLITTERS, e);
                if (lane == 0) {
                    a.out_r1[c] = pr_r[e];
                    a.out_rid1[c] = pr_rid[e];
                }
            }
            if (!grid_sync(a.bar, &ctl->err, bar_target)) return report(a);
            for (int j = threadIdx.x; j < TK_SPLITTERS; j += TK_TPB) {
                pr_r[j] = __ldcg(a.out_r1 + j);
                pr_rid[j] = __ldcg(a.out_rid1 + j);
            }
            __syncthreads();
            auto gap = [&](uint64_t r, uint32_t rid) {       // 2 * splitters below, + 1 when equal to the next
                int lo = 0;
#pragma unroll
                for (int w = (TK_SPLITTERS + 1) / 2; w > 0; w >>= 1)
                    if (elem_less(pr_r[lo + w - 1], pr_rid[lo + w - 1], r, rid)) lo += w;
                const bool eq = lo < TK_SPLITTERS && pr_r[lo] == r && pr_rid[lo] == rid;
                return static_cast<unsigned>(2 * lo + (eq ? 1 : 0));
            };
            done = partition(gap, hb[1], hb[2], true, TK_BIN_MAX);
        }
        if (done < 0) return report(a);
        if (done) {
            if (stamp) {
                ctl->ts[7] = gtimer();
                ctl->ts[8] = ctl->ts[7];
                ctl->ts[6] = ctl->ts[7];
                if (a.dev_status) *a.dev_status = ld_volatile_i32(&ctl->err);
            }
            return;
        }
        // The bucket entries are already written; sort the below entries with
        // the merge path (k below plus krem written above).
    }

    // Phase 4, fallback: CTA 0 finishes the bucket, then a grid merge sort.
    if (blockIdx.x == 0) {
        if (!take_all) {
            const int cnt = static_cast<int>(bcnt);
            for (int i = threadIdx.x; i < cnt; i += TK_TPB) {
                sr[i] = __ldcg(a.small_r + i);
                srid[i] = __ldcg(a.small_rid + i);
            }
            __syncthreads();
            block_sort<TK_TPB>(sr, srid, cnt);
            const uint64_t base = a.k - krem;
            for (uint64_t i = threadIdx.x; i < krem; i += TK_TPB) {
                a.out_r0[base + i] = sr[i];
                a.out_rid0[base + i] = srid[i];
            }
            __syncthreads();
        }
        if (stamp) {
            ctl->ts[7] = gtimer();
            ctl->ts[8] = ctl->ts[7];
        }
    }
    if (!grid_sync(a.bar, &ctl->err, bar_target)) return report(a);

    // Tiles of TK_SMALL sorted, then merge-path rounds.
    const uint64_t k = a.k;
    const uint64_t ntiles = (k + TK_SMALL - 1) / TK_SMALL;
    for (uint64_t tIdx = blockIdx.x; tIdx < ntiles; tIdx += gridDim.x) {
        const uint64_t lo = tIdx * TK_SMALL;
        const int cnt = static_cast<int>(k - lo < TK_SMALL ? k - lo : TK_SMALL);
        for (int i = threadIdx.x; i < cnt; i += TK_TPB) {
            sr[i] = __ldcg(a.out_r0 + lo + i);
            srid[i] = __ldcg(a.out_rid0 + lo + i);
        }
        __syncthreads();
        block_sort<TK_TPB>(sr, srid, cnt);
        for (int i = threadIdx.x; i < cnt; i += TK_TPB) {
            a.out_r0[lo + i] = sr[i];
            a.out_rid0[lo + i] = srid[i];
        }
        __syncthreads();
    }
    if (!grid_sync(a.bar, &ctl->err, bar_target)) return report(a);
    uint64_t* src_r = a.out_r0;
    uint32_t* src_rid = a.out_rid0;
    uint64_t* dst_r = a.out_r1;
    uint32_t* dst_rid = a.out_rid1;
    constexpr uint64_t E = 8;
    const uint64_t nthreads = static_cast<uint64_t>(gridDim.x) * TK_TPB;
    const uint64_t gtid = static_cast<uint64_t>(blockIdx.x) * TK_TPB + threadIdx.x;
    for (uint64_t w = TK_SMALL; w < k; w *= 2) {
        const uint64_t ntasks = (k + E - 1) / E;
        for (uint64_t task = gtid; task < ntasks; task += nthreads) {
            const uint64_t o = task * E;
            const uint64_t base = (o / (2 * w)) * (2 * w);
            const uint64_t a0 = base, a1 = min(base + w, k);
            const uint64_t b0 = a1, b1 = min(base + 2 * w, k);
            const uint64_t na = a1 - a0, nb = b1 - b0;
            const uint64_t diag = o - base;
            uint64_t i = merge_path(src_r + a0, src_rid + a0, na, src_r + b0, src_rid + b0, nb, diag);
            uint64_t j = diag - i;
            const uint64_t end = min(o + E, b1);
            uint64_t ar = 0, br = 0;
            uint32_t arid = 0, brid = 0;
            if (i < na) { ar = __ldcg(src_r + a0 + i); arid = __ldcg(src_rid + a0 + i); }
            if (j < nb) { br = __ldcg(src_r + b0 + j); brid = __ldcg(src_rid + b0 + j); }
            for (uint64_t q = o; q < end; ++q) {
                const bool takeA = i < na && (j >= nb || !elem_less(br, brid, ar, arid));
                if (takeA) {
                    dst_r[q] = ar;
                    dst_rid[q] = arid;
                    ++i;
                    if (i < na) { ar = __ldcg(src_r + a0 + i); arid = __ldcg(src_rid + a0 + i); }
                } else {
                    dst_r[q] = br;
                    dst_rid[q] = brid;
                    ++j;
                    if (j < nb) { br = __ldcg(src_r + b0 + j); brid = __ldcg(src_rid + b0 + j); }
                }
            }
        }
        if (!grid_sync(a.bar, &ctl->err, bar_target)) return report(a);
        uint64_t* tr = src_r; src_r = dst_r; dst_r = tr;
        uint32_t* ti = src_rid; src_rid = dst_rid; dst_rid = ti;
    }
    for (uint64_t i = gtid; i < k; i += nthreads) write_result(a, i, __ldcg(src_r + i), __ldcg(src_rid + i));
    if (gtid == 0 && a.dev_status) *a.dev_status = ld_volatile_i32(&ctl->err);
    if (gtid == 0) ctl->ts[6] = gtimer();
}

// Kernel 3 of 3 (cooperative): refine, split, finish and sort.  For inputs of
// at most TK_DIRECT_N keys with a sample it also makes the streaming pass (a
// filter kernel of its own costs a launch and its end more than a few
// megabytes take to read), and a grid barrier stands where the filter kernel
// ended: 2^20 float64 keys, K = 100, 29 us with refine passes over the input,
// 23 us so.
// LARGE: for K above TK_SMALL.  A smaller K always fits the ranked finish, and its
// kernel goes without the code of the larger one, which each call would fetch
// past (2^24 int64 keys, K = 1: the call 46 -> 43 us).
enum SelectFilter { SEL_NONE = 0, SEL_W8 = 1, SEL_W4 = 2, SEL_PAIR = 3 };
template <int FILTER, bool LARGE>
__global__ void __launch_bounds__(TK_TPB, 2) topk_select_kernel(const __grid_constant__ TopkArgs a) {
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ unsigned long long sc[24];
    TopkCtl* ctl = a.ctl;
    unsigned* sh = reinterpret_cast<unsigned*>(smem);
    uint64_t* sr = reinterpret_cast<uint64_t*>(smem);
    uint32_t* srid = reinterpret_cast<uint32_t*>(smem + TK_RANK_MAX * 8);

    unsigned bar_target = 0;                                 // of the grid barriers
    if (FILTER == SEL_NONE) {
        wait_prior_grid();
        allow_next_grid();
    } else {
        if (FILTER == SEL_W8) filter_pass<false, TK_TPB>(a, smem);
        if (FILTER == SEL_W4) filter_pass<true, TK_TPB>(a, smem);
        if (FILTER == SEL_PAIR) filter_pass_pair<TK_TPB>(a, smem);
        if (!grid_sync(a.bar, &ctl->err, bar_target)) return report(a);
    }
    const bool stamp = blockIdx.x == 0 && threadIdx.x == 0;
    if (stamp) ctl->ts[2] = gtimer();
    // Source of the selection: the candidates of the streaming pass when the
    // sample judged well (at least k of them, all stored), else the input.
    // Either way, with k or more entries up to the threshold the fused
    // histogram holds them all.  (count_only is never set without it.)
    bool cand = false, counted = false;
    uint64_t src_n = a.n, upto = a.n;                        // entries up to the threshold, or all
    uint64_t low = 0;                                        // candidates below the fused interval
    FuseRange fr{};
    unsigned hv0[TK_BINS / TK_TPB];                          // the thread's bins of the fused pass
    Elem first{0, 0};                                        // the thread's first candidate
    if (a.use_sample) {
        // all that the first steps need, in one round trip to L2
        const int err = __ldcg(&ctl->err);
        const uint64_t cnt = __ldcg(&ctl->cand_count);
        fr = fuse_range(a);
        low = __ldcg(&ctl->flow);
        pick_load_global<TK_TPB>(a.ghist, hv0);
        const uint64_t i0 = static_cast<uint64_t>(blockIdx.x) * TK_TPB + threadIdx.x;
        if (i0 < a.cand_cap) first = Elem{__ldcg(a.cand_r + i0), __ldcg(a.cand_rid + i0)};
        if (err != 0) return report(a);
        counted = a.fuse && cnt >= a.k;
        cand = cnt >= a.k && cnt <= a.cand_cap && !fr.count_only;
        if (cand) src_n = cnt;
        if (cand || counted) upto = cnt;
        if (stamp) ctl->path = cand ? 1 : 2;
    }
    const unsigned long long use_ts3 = stamp ? gtimer() : 0ull;

    // Phase 2: refine the interval that holds the K-th entry, at or below the
    // threshold when k entries are.
    Range g{0ull, cand || counted ? fr.g.rhi : max_rank(a), 0u, max_rowid(a)};
    uint64_t krem = a.k, bcnt = upto;
    int pass = 0, npass = 0;
    // With the filter's fused first pass, pass 0's histogram is ready; when
    // fewer than k entries are counted in it, the passes start at buffer 1
    // (clean) and pass 2 clears buffer 0 before pass 3 uses it.
    bool ready = counted;
    if (a.fuse && !counted) pass = 1;
    if (ready && bcnt > TK_SMALL && krem < bcnt) {
        if (low >= a.k) {
            g.rhi = fr.g.rlo - 1;
            if (a.w4) g.rhi &= 0xFFFFFFFF00000000ull;
            bcnt = low;
        } else {
            const Pick pk = pick_loaded<TK_TPB>(hv0, a.k - low, sc);
            krem = a.k - low - pk.below;
            bcnt = pk.in_b;
            g = range_narrow(a, fr.g, fr.sh, pk.b);
        }
        ready = false;
        ++pass;
        ++npass;
    }
    while (bcnt > TK_SMALL && !range_point(g) && krem < bcnt) {
        const int shift = range_shift(g, a.digit);
        unsigned* gh = a.ghist + (pass % 3) * TK_BINS;
        unsigned* gz = a.ghist + ((pass + 1) % 3) * TK_BINS;
        unsigned long long* mm = ctl->mm[pass % 3];
        hist_pass(a, cand, src_n, g, shift, gh, gz, sh, mm, ctl->mm[(pass + 1) % 3]);
        if (!grid_sync(a.bar, &ctl->err, bar_target)) return report(a);
        ++npass;
        unsigned hv[TK_BINS / TK_TPB];
        pick_load_global<TK_TPB>(gh, hv);
        const Pick pk = pick_loaded<TK_TPB>(hv, krem, sc);
        // every entry of the interval in one bin: go on with the interval that
        // their minima and maxima span
        const bool whole = pk.below == 0 && pk.in_b == bcnt;
        krem -= pk.below;
        bcnt = pk.in_b;
        g = whole ? range_of(a, mm) : range_narrow(a, g, shift, pk.b);
        ++pass;
    }
    // The buffer at pass % 3 must be clean for the finish: when the fused
    // pass-0 histogram was never consumed, buffer 1 (zeroed by prepare) is.
    if (ready) pass = 1;
    if (stamp) {
        ctl->passes = npass;
        ctl->ts[3] = use_ts3;
        ctl->ts[4] = gtimer();
    }

    // Phase 3: split around the interval.
    const bool take_all = (krem == bcnt) || range_point(g);
    // the larger-K finish wants the span of the entries split writes out
    const bool large = (take_all ? a.k : a.k - krem) + (take_all ? 0 : bcnt) > TK_RANK_MAX;
    if (LARGE && large)
        split_pass_large(a, cand, src_n, g, take_all, krem, krem == bcnt, first, smem);
    else
        split_pass(a, cand, src_n, g, take_all, krem, first);
    if (!grid_sync(a.bar, &ctl->err, bar_target)) return report(a);
    if (stamp) ctl->ts[5] = gtimer();

    // Phase 4, survivors that fit one CTA's shared memory (every K <= 4096):
    // each warp of the grid takes survivors one at a time and computes its
    // final position as its rank -- the number of entries of its own set
    // that order before it (equal entries by position), so ranks are
    // distinct.  The "below" entries precede every bucket entry;
    // a bucket entry is kept when its rank within the bucket is below krem.
    {
        const uint64_t nb = take_all ? a.k : a.k - krem;     // out_r0[0, nb)
        const uint64_t ns = take_all ? 0 : bcnt;             // small buffer
        if (!LARGE || nb + ns <= TK_RANK_MAX) {
            const int nbi = static_cast<int>(nb), nsi = static_cast<int>(ns);
            for (int i = threadIdx.x; i < nbi; i += TK_TPB) {
                sr[i] = __ldcg(a.out_r0 + i);
                srid[i] = __ldcg(a.out_rid0 + i);
            }
            for (int i = threadIdx.x; i < nsi; i += TK_TPB) {
                sr[nbi + i] = __ldcg(a.small_r + i);
                srid[nbi + i] = __ldcg(a.small_rid + i);
            }
            __syncthreads();
            if (stamp) ctl->ts[7] = gtimer();
            const unsigned lane = threadIdx.x & 31u;
            const int nwarps = static_cast<int>(gridDim.x) * (TK_TPB / 32);
            const int gw = static_cast<int>(blockIdx.x) * (TK_TPB / 32) + static_cast<int>(threadIdx.x >> 5);
            for (int e = gw; e < nbi + nsi; e += nwarps) {
                const bool below = e < nbi;
                const unsigned c = warp_rank_of(sr, srid, below ? 0 : nbi, below ? nbi : nbi + nsi, e);
                if (lane == 0) {
                    if (below) write_result(a, c, sr[e], srid[e]);
                    else if (c < krem) write_result(a, nb + c, sr[e], srid[e]);
                }
            }
            if (stamp) {
                ctl->ts[8] = gtimer();
                ctl->ts[6] = ctl->ts[8];
                if (a.dev_status) *a.dev_status = ld_volatile_i32(&ctl->err);
            }
            return;
        }
    }

    if (LARGE) finish_large(a, smem, sc, bar_target, pass, take_all, krem, bcnt);
}

// The whole Top-K of a small input, in one launch without a control block or
// a grid barrier: every CTA loads all n keys into shared memory, finds the
// interval of the K-th entry by refine passes of its own over them (the same
// in every CTA), lists the entries below it and in it, and ranks the entries
// whose index falls to it among those.  Bound by latency: the loads, three
// barriers a pass, and a launch less than the general path's two (TK_LOCAL_N
// has both sides).
__global__ void __launch_bounds__(TKL_TPB, 1) topk_local_kernel(TopkArgs a) {
    extern __shared__ __align__(16) unsigned char smem[];
    unsigned* hist = reinterpret_cast<unsigned*>(smem);                      // then the two lists
    uint16_t* list = reinterpret_cast<uint16_t*>(smem);                      // below from the front, the rest after
    uint64_t* sr = reinterpret_cast<uint64_t*>(smem + TK_BINS * 4);
    uint32_t* srid = reinterpret_cast<uint32_t*>(smem + TK_BINS * 4 + a.n * 8);
    __shared__ unsigned long long sc[24];
    __shared__ unsigned long long mm[4];
    __shared__ unsigned n_below, n_eq;
    const int n = static_cast<int>(a.n);
    const unsigned lane = threadIdx.x & 31u, warp = threadIdx.x >> 5;
    wait_prior_grid();
    allow_next_grid();
    unsigned long long t0 = 0;
    if (blockIdx.x == 0 && threadIdx.x == 0) t0 = gtimer();
    auto span = [&](const Fold& mine) {                      // minima and maxima over the CTA, in mm
        if (threadIdx.x == 0) fold_reset(mm);
        __syncthreads();
        Fold f = mine;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            f.rmin = min(f.rmin, __shfl_xor_sync(0xFFFFFFFFu, f.rmin, o));
            f.rmax = max(f.rmax, __shfl_xor_sync(0xFFFFFFFFu, f.rmax, o));
        }
        f.imin = __reduce_min_sync(0xFFFFFFFFu, f.imin);
        f.imax = __reduce_max_sync(0xFFFFFFFFu, f.imax);
        if (lane == 0 && f.rmin <= f.rmax) {
            atomicMin(&mm[0], static_cast<unsigned long long>(f.rmin));
            atomicMax(&mm[1], static_cast<unsigned long long>(f.rmax));
            atomicMin(&mm[2], static_cast<unsigned long long>(f.imin));
            atomicMax(&mm[3], static_cast<unsigned long long>(f.imax));
        }
        __syncthreads();
        Range g{mm[0], mm[1], 0u, max_rowid(a)};
        if (g.rlo == g.rhi) {
            g.ilo = static_cast<uint32_t>(mm[2]);
            g.ihi = static_cast<uint32_t>(mm[3]);
        }
        __syncthreads();
        return g;
    };
    Fold all = fold_none();
#pragma unroll 4
    for (int i = threadIdx.x; i < n; i += TKL_TPB) {
        const Elem e = load_input(a, i);
        sr[i] = e.r;
        srid[i] = e.rid;
        fold_add(all, e.r, e.rid);
    }
    Range g = span(all);
    uint64_t krem = a.k, bcnt = a.n;
    // Down to a bin that costs less to rank than another pass.
    while (bcnt > 64 && !range_point(g) && krem < bcnt) {
        const int shift = range_shift(g, TK_DIG);
        for (int b = threadIdx.x; b < TK_BINS; b += TKL_TPB) hist[b] = 0;
        __syncthreads();
        for (int i = threadIdx.x; i < n; i += TKL_TPB) {
            const uint64_t r = sr[i];
            const uint32_t rid = srid[i];
            if (range_cmp(g, r, rid) == 0) atomicAdd(&hist[range_bin(g, shift, r, rid)], 1u);
        }
        __syncthreads();
        const Pick pk = pick_bucket<TKL_TPB>(hist, krem, sc);
        const bool whole = pk.below == 0 && pk.in_b == bcnt;
        krem -= pk.below;
        bcnt = pk.in_b;
        if (whole) {
            Fold f = fold_none();
            for (int i = threadIdx.x; i < n; i += TKL_TPB)
                if (range_cmp(g, sr[i], srid[i]) == 0) fold_add(f, sr[i], srid[i]);
            const Range narrow = span(f);
            // (an interval that does not shrink is cut like any other)
            const bool same = narrow.rlo == g.rlo && narrow.rhi == g.rhi && narrow.ilo == g.ilo && narrow.ihi == g.ihi;
            g = same ? range_narrow(a, g, shift, pk.b) : narrow;
        } else {
            g = range_narrow(a, g, shift, pk.b);
        }
    }
    // The lists: fewer than K entries below the interval, and in it at most 64
    // or, when all of it is taken, the rest of the K.  Identical entries (one
    // key and row-id) are not ranked: krem copies are written.
    const bool point = range_point(g);
    const unsigned nb = static_cast<unsigned>(a.k - krem);
    if (threadIdx.x == 0) n_below = n_eq = 0;
    __syncthreads();                                         // (the histogram has been read)
    for (int i = threadIdx.x; i < n; i += TKL_TPB) {
        const int c = range_cmp(g, sr[i], srid[i]);
        if (c < 0) list[atomicAdd(&n_below, 1u)] = static_cast<uint16_t>(i);
        else if (c == 0 && !point) list[nb + atomicAdd(&n_eq, 1u)] = static_cast<uint16_t>(i);
    }
    if (point && blockIdx.x == 0)
        for (unsigned t = threadIdx.x; t < krem; t += TKL_TPB) write_result(a, nb + t, g.rlo, g.ilo);
    __syncthreads();
    const unsigned total = static_cast<unsigned>(bcnt);
    const int last = point ? -1 : 0;                         // range_cmp of the entries to rank
    // entry i falls to warp i mod (warps of the grid)
    const int nw = static_cast<int>(gridDim.x) * (TKL_TPB / 32);
    const int gw = static_cast<int>(warp * gridDim.x + blockIdx.x);
    for (int base = gw; base < n; base += 32 * nw) {
        const int i = base + nw * static_cast<int>(lane);
        const int c = i < n ? range_cmp(g, sr[i], srid[i]) : 1;
        unsigned todo = __ballot_sync(0xFFFFFFFFu, c <= last);
        while (todo) {
            const int src = __ffs(todo) - 1;
            todo &= todo - 1;
            const int e = base + nw * src;
            const bool below = __shfl_sync(0xFFFFFFFFu, c, src) < 0;
            const uint64_t er = sr[e];
            const uint32_t erid = srid[e];
            unsigned cnt = 0;
            const uint16_t* l = below ? list : list + nb;
            const unsigned len = below ? nb : total;
            for (unsigned j = lane; j < len; j += 32) {
                const int x = l[j];
                rank_count(cnt, sr[x], srid[x], er, erid, x < e);
            }
            const unsigned rank = __reduce_add_sync(0xFFFFFFFFu, 0u - cnt);
            if (lane == 0) {
                if (below) write_result(a, rank, er, erid);
                else if (rank < krem) write_result(a, nb + rank, er, erid);
            }
        }
    }
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        const unsigned long long t1 = gtimer();
        a.ctl->err = 0;
        a.ctl->path = 0;
        a.ctl->passes = 0;
        a.ctl->cand_count = 0;
        for (int j = 0; j < 6; ++j) a.ctl->ts[j] = t0;
        for (int j = 6; j < 9; ++j) a.ctl->ts[j] = t1;
        if (a.dev_status) *a.dev_status = OLAP_OK;
    }
}

// ---------------------------------------------------------------------------
// Host side.
// ---------------------------------------------------------------------------
TopkPlan topk_plan(uint64_t n, uint64_t k) {
    TopkPlan p{0, 0, 0, 0};
    if (n <= TK_LOCAL_N && k <= TK_LOCAL_K && n * k <= TK_LOCAL_NK) {
        p.local = 1;
        return p;
    }
    if (n > TK_SAMPLE_N && k <= n / 256) {
        const double lam = static_cast<double>(k) * TK_SAMPLE / static_cast<double>(n);
        double r = std::ceil(lam + 4.0 * std::sqrt(lam)) + 3.0;
        if (r > TK_SAMPLE) r = TK_SAMPLE;
        p.use_sample = n > TK_DIRECT_N ? TK_SAMPLE_FILTER : TK_SAMPLE_INLINE;
        p.sample_rank = static_cast<unsigned>(r);
        const uint64_t stratum = (n + TK_SAMPLE - 1) / TK_SAMPLE;
        uint64_t cap = 2 * (static_cast<uint64_t>(r) + 8) * stratum;
        cap = std::max<uint64_t>(cap, k + TK_SMALL);
        cap = (cap + 1023) & ~1023ull;
        p.cand_cap = std::min<uint64_t>(cap, n);
    }
    return p;
}

TopkPlan topk_plan_call(const TopkArgs& a) {
    TopkPlan p = topk_plan(a.n, a.k);
    if (!p.local) return p;
    const size_t wide = a.pair || a.w4 ? 4 : 8;
    struct Span {
        const void* p;
        size_t bytes;
    };
    const Span in[] = {{a.keys, a.n * wide}, {a.keys2, a.n * 4}, {a.rowids, a.n * 4}};
    const Span out[] = {{a.out_keys, a.k * wide}, {a.out_keys2, a.k * 4}, {a.out_rowids, a.k * 4}, {a.dev_status, 4}};
    for (const Span& i : in)
        for (const Span& o : out) {
            const uintptr_t x = reinterpret_cast<uintptr_t>(i.p), y = reinterpret_cast<uintptr_t>(o.p);
            if (x && y && x < y + o.bytes && y < x + i.bytes) p.local = 0;
        }
    return p;
}

static size_t up256(size_t x) { return (x + 255) & ~static_cast<size_t>(255); }

size_t topk_scratch_bytes(const TopkPlan& p, uint64_t k) {
    size_t b = up256(sizeof(TopkCtl)) + up256(sizeof(GridBar)) + up256(3 * TK_BINS * 4);
    if (p.use_sample) b += up256(TK_SAMPLE * 8);
    b += up256(p.cand_cap * 8) + up256(p.cand_cap * 4);
    b += up256(TK_SMALL * 8) + up256(TK_SMALL * 4);
    const uint64_t kk = std::max<uint64_t>(k, 1);
    b += up256(kk * 8) + up256(kk * 4);
    if (k > TK_SMALL) b += up256(kk * 8) + up256(kk * 4);
    return b;
}

void topk_carve(TopkArgs& a, const TopkPlan& p, void* base) {
    unsigned char* c = static_cast<unsigned char*>(base);
    auto take = [&](size_t bytes) {
        void* r = c;
        c += up256(bytes);
        return r;
    };
    // The grid barrier comes first so that it keeps its place (and its
    // zeroed state) whatever the other buffer sizes are.
    a.bar = static_cast<GridBar*>(take(sizeof(GridBar)));
    a.ctl = static_cast<TopkCtl*>(take(sizeof(TopkCtl)));
    a.ghist = static_cast<unsigned*>(take(3 * TK_BINS * 4));
    a.small_r = static_cast<uint64_t*>(take(TK_SMALL * 8));
    a.small_rid = static_cast<uint32_t*>(take(TK_SMALL * 4));
    a.cand_cap = p.cand_cap;
    a.cand_r = static_cast<uint64_t*>(take(p.cand_cap * 8));
    a.cand_rid = static_cast<uint32_t*>(take(p.cand_cap * 4));
    const uint64_t kk = std::max<uint64_t>(a.k, 1);
    a.out_r0 = static_cast<uint64_t*>(take(kk * 8));
    a.out_rid0 = static_cast<uint32_t*>(take(kk * 4));
    if (a.k > TK_SMALL) {
        a.out_r1 = static_cast<uint64_t*>(take(kk * 8));
        a.out_rid1 = static_cast<uint32_t*>(take(kk * 4));
    } else {
        a.out_r1 = nullptr;
        a.out_rid1 = nullptr;
    }
    a.samples = p.use_sample ? static_cast<uint64_t*>(take(TK_SAMPLE * 8)) : nullptr;
    a.local = p.local;
    a.use_sample = p.use_sample;
    a.sample_rank = p.sample_rank;
    a.filter = TK_FILTER_BULK;
}

// Dynamic shared bytes the filter kernel may use, per device; set once, under
// g_attr_lock, by the first thread that needs the kernels' attributes there.
static std::atomic<int> g_smem_limit[64] = {};
static std::mutex g_attr_lock;

// Dynamic shared memory of a register filter with tpb threads.
static int regs_smem(int tpb) { return FUSE_BYTES + tpb / 32 * WS_BYTES; }
static_assert(FUSE_BYTES + TK_TPB / 32 * WS_BYTES <= TK_SORT_SMEM, "the select's own streaming pass");

static bool set_kernel_attrs(int device) {
    if (g_smem_limit[device].load()) return true;
    std::lock_guard<std::mutex> guard(g_attr_lock);
    if (g_smem_limit[device].load()) return true;
    // Opt-in limit per block, less the filter kernel's static shared memory.
    int optin = 0;
    cudaFuncAttributes fa;
    if (cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, device) != cudaSuccess ||
        cudaFuncGetAttributes(&fa, topk_filter_bulk_kernel<false>) != cudaSuccess)
        return false;
    const int lim = std::min<int>(optin - static_cast<int>(fa.sharedSizeBytes) - 256, TK_SMEM_MAX);
    bool ok = true;
    auto opt_in = [&](auto fn, int bytes) {
        ok = ok && cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes) == cudaSuccess;
    };
    opt_in(topk_filter_bulk_kernel<false>, lim);
    opt_in(topk_filter_bulk_kernel<true>, lim);
    opt_in(topk_filter_regs_kernel<false, 256>, regs_smem(256));
    opt_in(topk_filter_regs_kernel<true, 256>, regs_smem(256));
    opt_in(topk_filter_pair_kernel<256>, regs_smem(256));
    opt_in(topk_filter_regs_kernel<false, 512>, regs_smem(512));
    opt_in(topk_filter_regs_kernel<true, 512>, regs_smem(512));
    opt_in(topk_filter_pair_kernel<512>, regs_smem(512));
    opt_in(topk_filter_regs_kernel<false, 1024>, regs_smem(1024));
    opt_in(topk_filter_regs_kernel<true, 1024>, regs_smem(1024));
    opt_in(topk_filter_pair_kernel<1024>, regs_smem(1024));
    opt_in(topk_filter_host_kernel<false>, regs_smem(TKR_TPB));
    opt_in(topk_filter_host_kernel<true>, regs_smem(TKR_TPB));
    opt_in(topk_local_kernel, TKL_SMEM_MAX);
    opt_in(topk_select_kernel<SEL_NONE, false>, TK_SORT_SMEM);
    opt_in(topk_select_kernel<SEL_NONE, true>, TK_SORT_SMEM);
    opt_in(topk_select_kernel<SEL_W8, false>, TK_SORT_SMEM);
    opt_in(topk_select_kernel<SEL_W8, true>, TK_SORT_SMEM);
    opt_in(topk_select_kernel<SEL_W4, false>, TK_SORT_SMEM);
    opt_in(topk_select_kernel<SEL_W4, true>, TK_SORT_SMEM);
    opt_in(topk_select_kernel<SEL_PAIR, false>, TK_SORT_SMEM);
    opt_in(topk_select_kernel<SEL_PAIR, true>, TK_SORT_SMEM);
    if (!ok) return false;
    g_smem_limit[device].store(lim);
    return true;
}

bool topk_geometry(int device, int tile_bytes, int stages, int ctas_per_sm, int regs_tpb, TopkGeom* out) {
    TopkGeom g;
    g.regs_tpb = regs_tpb ? regs_tpb : TKR_TPB;
    if (g.regs_tpb != 256 && g.regs_tpb != 512 && g.regs_tpb != 1024) return false;
    g.tile_bytes = tile_bytes ? tile_bytes : TK_TILE_DEFAULT;
    g.stages = stages ? stages : TK_STAGES_DEFAULT;
    g.ctas_per_sm = ctas_per_sm ? ctas_per_sm : TK_CTAS_PER_SM_DEFAULT;
    if (g.tile_bytes < 16 * TKF_TPB || g.tile_bytes % (16 * TKF_TPB) || g.stages < 1 ||
        g.stages > TK_MAX_STAGES || g.ctas_per_sm < 1 || g.ctas_per_sm > 8)
        return false;
    if (device < 0 || device >= 64) return false;
    g.smem_bytes = g.tile_bytes * g.stages + 16 * TK_MAX_STAGES + (TKF_TPB / 32) * WS_BYTES;
    int sms = 0, per_sm = 0;
    if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, device) != cudaSuccess) return false;
    if (!set_kernel_attrs(device)) return false;
    if (g.smem_bytes > g_smem_limit[device].load()) return false;
    // Streaming filter: independent CTAs, capped at ctas_per_sm per SM.
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, topk_filter_bulk_kernel<false>, TKF_TPB,
                                                      g.smem_bytes) != cudaSuccess)
        return false;
    per_sm = std::min(per_sm, g.ctas_per_sm);
    if (per_sm < 1) return false;
    g.filter_grid = sms * per_sm;
    cudaError_t oe;
    const size_t rs = static_cast<size_t>(regs_smem(g.regs_tpb));
    if (g.regs_tpb == 256)
        oe = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, topk_filter_regs_kernel<false, 256>, 256, rs);
    else if (g.regs_tpb == 512)
        oe = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, topk_filter_regs_kernel<false, 512>, 512, rs);
    else
        oe = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, topk_filter_regs_kernel<false, 1024>, 1024, rs);
    if (oe != cudaSuccess) return false;
    g.regs_grid = sms * std::max(1, std::min(per_sm, 2048 / g.regs_tpb));
    // Cooperative select kernel: every CTA resident, two per SM at most.
    per_sm = 2;
    auto fits = [&](auto fn) {
        int per = 0;
        if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, fn, TK_TPB, TK_SORT_SMEM) != cudaSuccess) per = 0;
        per_sm = std::min(per_sm, per);
    };
    fits(topk_select_kernel<SEL_NONE, false>);
    fits(topk_select_kernel<SEL_NONE, true>);
    fits(topk_select_kernel<SEL_W8, false>);
    fits(topk_select_kernel<SEL_W8, true>);
    fits(topk_select_kernel<SEL_W4, false>);
    fits(topk_select_kernel<SEL_W4, true>);
    fits(topk_select_kernel<SEL_PAIR, false>);
    fits(topk_select_kernel<SEL_PAIR, true>);
    // Two CTAs per SM for the select in general; one per SM when it reads a
    // candidate list and finishes a small K: its grid barriers then dominate,
    // and half the arrivals take less time (measured, 2^28 keys, K = 1000:
    // select 22.6 -> 19.9 us; at K = 10^5 the merge-path finish wants both).
    if (per_sm < 1) return false;
    g.grid = sms * per_sm;
    g.grid_small = sms;
    *out = g;
    return true;
}

// One launch of a Top-K kernel: cooperative for the select, and with
// programmatic stream serialisation (the kernel waits in wait_prior_grid for
// the one before it).
static cudaError_t launch_kernel(void (*fn)(TopkArgs), unsigned grid, unsigned block, size_t smem,
                                 cudaStream_t stream, const TopkArgs& a, bool coop) {
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(block);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = stream;
    cudaLaunchAttribute at[2];
    unsigned na = 0;
    at[na].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[na].val.programmaticStreamSerializationAllowed = 1;
    ++na;
    if (coop) {
        at[na].id = cudaLaunchAttributeCooperative;
        at[na].val.cooperative = 1;
        ++na;
    }
    cfg.attrs = at;
    cfg.numAttrs = na;
    return cudaLaunchKernelEx(&cfg, fn, a);
}

template <bool LARGE>
static void (*select_kernel(int filter))(TopkArgs) {
    switch (filter) {
        case SEL_W8: return topk_select_kernel<SEL_W8, LARGE>;
        case SEL_W4: return topk_select_kernel<SEL_W4, LARGE>;
        case SEL_PAIR: return topk_select_kernel<SEL_PAIR, LARGE>;
        default: return topk_select_kernel<SEL_NONE, LARGE>;
    }
}

cudaError_t topk_launch(const TopkArgs& args, const TopkGeom& geom, cudaStream_t stream, cudaEvent_t* ev) {
    TopkArgs a = args;
    a.tile_bytes = geom.tile_bytes;
    a.stages = geom.stages;
    if (a.digit == 0) a.digit = TK_DIG;
    if (a.digit < TK_DIG_MIN || a.digit > TK_DIG) return cudaErrorInvalidValue;
    // the register and two-column filters fold the select's first pass
    a.fuse = a.use_sample == TK_SAMPLE_INLINE ||
                     (a.use_sample == TK_SAMPLE_FILTER && (a.pair || a.host_keys || a.filter == TK_FILTER_REGS))
                 ? 1
                 : 0;
    cudaError_t e;
    if (ev && (e = cudaEventRecord(ev[0], stream)) != cudaSuccess) return e;
    if (a.local) {
        if (ev && ((e = cudaEventRecord(ev[1], stream)) != cudaSuccess ||
                   (e = cudaEventRecord(ev[2], stream)) != cudaSuccess))
            return e;
        // a CTA for every 8 results: each reads the whole input, and ranking
        // is what they share
        const unsigned g = static_cast<unsigned>(std::min<uint64_t>(geom.grid_small, (a.k + 7) / 8));
        e = launch_kernel(topk_local_kernel, g, TKL_TPB, TK_BINS * 4 + a.n * 12, stream, a, false);
        if (e != cudaSuccess || !ev) return e;
        return cudaEventRecord(ev[3], stream);
    }
    e = launch_kernel(topk_prepare_kernel, a.use_sample ? TK_PREP_CTAS : 1, TK_TPB, 0, stream, a, false);
    if (e != cudaSuccess) return e;
    if (ev && (e = cudaEventRecord(ev[1], stream)) != cudaSuccess) return e;
    if (a.use_sample == TK_SAMPLE_FILTER) {
        void (*fn)(TopkArgs) = nullptr;
        unsigned grid = static_cast<unsigned>(geom.regs_grid), block = static_cast<unsigned>(geom.regs_tpb);
        size_t smem = static_cast<size_t>(regs_smem(geom.regs_tpb));
        if (a.host_keys) {
            fn = a.w4 ? topk_filter_host_kernel<true> : topk_filter_host_kernel<false>;
            grid = static_cast<unsigned>(geom.grid_small);   // one CTA per SM
            block = TKR_TPB;
            smem = static_cast<size_t>(regs_smem(TKR_TPB));
        } else if (a.pair) {
            fn = geom.regs_tpb == 256    ? topk_filter_pair_kernel<256>
                 : geom.regs_tpb == 1024 ? topk_filter_pair_kernel<1024>
                                         : topk_filter_pair_kernel<512>;
        } else if (a.filter == TK_FILTER_REGS) {
            if (geom.regs_tpb == 256)
                fn = a.w4 ? topk_filter_regs_kernel<true, 256> : topk_filter_regs_kernel<false, 256>;
            else if (geom.regs_tpb == 1024)
                fn = a.w4 ? topk_filter_regs_kernel<true, 1024> : topk_filter_regs_kernel<false, 1024>;
            else
                fn = a.w4 ? topk_filter_regs_kernel<true, 512> : topk_filter_regs_kernel<false, 512>;
        } else {
            fn = a.w4 ? topk_filter_bulk_kernel<true> : topk_filter_bulk_kernel<false>;
            grid = static_cast<unsigned>(geom.filter_grid);
            block = TKF_TPB;
            smem = geom.smem_bytes;
        }
        if ((e = launch_kernel(fn, grid, block, smem, stream, a, false)) != cudaSuccess) return e;
    }
    if (ev && (e = cudaEventRecord(ev[2], stream)) != cudaSuccess) return e;
    // (the direct path keeps both CTAs per SM: its passes read the input)
    const int sgrid = (a.use_sample && a.k <= static_cast<uint64_t>(TK_SMALL)) ? geom.grid_small : geom.grid;
    const int which = a.use_sample != TK_SAMPLE_INLINE ? SEL_NONE : a.pair ? SEL_PAIR : a.w4 ? SEL_W4 : SEL_W8;
    const bool large = a.k > static_cast<uint64_t>(TK_SMALL);
    void (*const sel)(TopkArgs) = large ? select_kernel<true>(which) : select_kernel<false>(which);
    e = launch_kernel(sel, static_cast<unsigned>(sgrid), TK_TPB, TK_SORT_SMEM, stream, a, true);
    if (e != cudaSuccess || !ev) return e;
    return cudaEventRecord(ev[3], stream);
}

}  // namespace olap
