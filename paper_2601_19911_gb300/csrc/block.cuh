// Block-level building blocks shared by the Top-K kernels (grid-wide and
// per-CTA): composite ordering, block scan, histogram bucket pick, shared
// memory bitonic sort, streaming loads and the key-domain threshold test.
#pragma once

#include <cstdint>

#include "common.cuh"

namespace olap {

constexpr int PICK_BINS = 4096;   // histogram bins of a 12-bit digit

// (ar, arid) orders before (br, brid): the borrow of the 96-bit difference.
// Written with comparisons the compiler branches on the rank words, and the
// lanes of a sort or a search diverge on every entry.
__device__ __forceinline__ bool elem_less(uint64_t ar, uint32_t arid, uint64_t br, uint32_t brid) {
    uint32_t less;
    asm("{\n .reg .u32 t;\n"
        " sub.cc.u32 t, %1, %2;\n"
        " subc.cc.u32 t, %3, %4;\n"
        " subc.cc.u32 t, %5, %6;\n"
        " subc.u32 %0, 0, 0;\n}"
        : "=r"(less)
        : "r"(arid), "r"(brid), "r"(static_cast<uint32_t>(ar)), "r"(static_cast<uint32_t>(br)),
          "r"(static_cast<uint32_t>(ar >> 32)), "r"(static_cast<uint32_t>(br >> 32)));
    return less != 0;
}

__device__ __forceinline__ uint4 ld_stream_v4(const void* p) {
    uint4 v;
    asm volatile("ld.global.cs.v4.u32 {%0, %1, %2, %3}, [%4];"
                 : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w)
                 : "l"(p));
    return v;
}

// One 32-byte streaming load (sm_100 and later): half as many load
// instructions and votes per byte as 16-byte ones.  Read-only pass over 2^31
// bytes, 64 bytes in flight per thread: 292.5 us, 315 us with 16-byte loads.
__device__ __forceinline__ void ld_stream_32(const void* p, uint32_t (&w)[8]) {
    uint64_t v[4];
    asm volatile("ld.global.cs.v4.u64 {%0, %1, %2, %3}, [%4];" : "=l"(v[0]), "=l"(v[1]), "=l"(v[2]), "=l"(v[3]) : "l"(p));
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        w[2 * j] = static_cast<uint32_t>(v[j]);
        w[2 * j + 1] = static_cast<uint32_t>(v[j] >> 32);
    }
}
// Programmatic dependent launch.  Every kernel of a call is launched while
// the one before it in the stream is still running, and waits here until that
// one has finished and its writes are visible.  A kernel launched without the
// attribute passes straight through.
__device__ __forceinline__ void wait_prior_grid() {
    asm volatile("griddepcontrol.wait;" ::: "memory");
}
// Lets the next kernel in the stream launch now (it still waits for this one
// to finish before it reads anything this one or an earlier one writes).
__device__ __forceinline__ void allow_next_grid() {
    asm volatile("griddepcontrol.launch_dependents;" :::);
}

// A launch in a chain of kernels; `after`: with programmatic stream
// serialisation behind the kernel before it.  Errors are left to
// cudaGetLastError.
template <typename... P>
inline void launch_after(void (*fn)(P...), unsigned grid, int block, size_t smem, cudaStream_t s, bool after, P... args) {
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(static_cast<unsigned>(block));
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute at;
    at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at.val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = &at;
    cfg.numAttrs = after ? 1 : 0;
    cudaLaunchKernelEx(&cfg, fn, args...);
}

// A 32-byte store (of the vector ld_stream_words loads); p 32-byte aligned.
__device__ __forceinline__ void st_words(void* p, const uint32_t (&w)[8]) {
    asm volatile("st.global.v4.u64 [%0], {%1, %2, %3, %4};" ::"l"(p),
                 "l"(static_cast<uint64_t>(w[0]) | (static_cast<uint64_t>(w[1]) << 32)),
                 "l"(static_cast<uint64_t>(w[2]) | (static_cast<uint64_t>(w[3]) << 32)),
                 "l"(static_cast<uint64_t>(w[4]) | (static_cast<uint64_t>(w[5]) << 32)),
                 "l"(static_cast<uint64_t>(w[6]) | (static_cast<uint64_t>(w[7]) << 32))
                 : "memory");
}
__device__ __forceinline__ void ld_stream_words(const void* p, uint32_t (&w)[8]) { ld_stream_32(p, w); }
__device__ __forceinline__ void ld_stream_words(const void* p, uint32_t (&w)[4]) {
    const uint4 v = ld_stream_v4(p);
    w[0] = v.x;
    w[1] = v.y;
    w[2] = v.z;
    w[3] = v.w;
}

// An interval of the composite (rank word, row-id) order: the entries with
// rlo <= r <= rhi when rlo < rhi (any row-id), else those with r == rlo and
// ilo <= row-id <= ihi.  A refine pass cuts it into at most 2^digit equal bins.
struct Range {
    uint64_t rlo, rhi;
    uint32_t ilo, ihi;
};
__device__ __forceinline__ bool range_point(const Range& g) { return g.rlo == g.rhi && g.ilo == g.ihi; }
// -1 below the interval, 0 in it, 1 above.
__device__ __forceinline__ int range_cmp(const Range& g, uint64_t r, uint32_t rid) {
    if (r < g.rlo) return -1;
    if (r > g.rhi) return 1;
    if (g.rlo != g.rhi) return 0;
    return rid < g.ilo ? -1 : (rid > g.ihi ? 1 : 0);
}
__device__ __forceinline__ int range_shift(const Range& g, int digit) {
    const int bits = g.rlo != g.rhi ? 64 - __clzll(static_cast<long long>(g.rhi - g.rlo))
                                    : 32 - __clz(static_cast<int>(g.ihi - g.ilo));
    return bits > digit ? bits - digit : 0;
}
__device__ __forceinline__ unsigned range_bin(const Range& g, int sh, uint64_t r, uint32_t rid) {
    return static_cast<unsigned>(g.rlo != g.rhi ? (r - g.rlo) >> sh : static_cast<uint64_t>((rid - g.ilo) >> sh));
}
// c -= 1 when entry j orders before entry e, or equals it and `ties`: the
// borrow of the 96-bit difference, five adds and no branch.  (Written with
// comparisons the compiler branches on the rank words, and lanes diverge on
// every entry.)
__device__ __forceinline__ void rank_count(unsigned& c, uint64_t jr, uint32_t jrid, uint64_t er, uint32_t erid,
                                           bool ties) {
    asm("{\n .reg .u32 t;\n"
        " sub.cc.u32 t, 0, %6;\n"
        " subc.cc.u32 t, %1, %2;\n"
        " subc.cc.u32 t, %3, %4;\n"
        " subc.cc.u32 t, %5, %7;\n"
        " subc.u32 %0, %0, 0;\n}"
        : "+r"(c)
        : "r"(jrid), "r"(erid), "r"(static_cast<uint32_t>(jr)), "r"(static_cast<uint32_t>(er)),
          "r"(static_cast<uint32_t>(jr >> 32)), "r"(ties ? 1u : 0u), "r"(static_cast<uint32_t>(er >> 32)));
}

// Block-wide exclusive scan over one value per thread (TPB threads; warp_sums
// holds a word per warp, and callers keep the total 16 words after it).
template <int TPB>
__device__ __forceinline__ unsigned long long block_excl_scan(unsigned long long v,
                                                              unsigned long long* warp_sums,
                                                              unsigned long long* total) {
    static_assert(TPB <= 512, "16 warp sums");
    const unsigned lane = threadIdx.x & 31u, warp = threadIdx.x >> 5;
    unsigned long long incl = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const unsigned long long t = __shfl_up_sync(0xFFFFFFFFu, incl, o);
        if (lane >= static_cast<unsigned>(o)) incl += t;
    }
    if (lane == 31) warp_sums[warp] = incl;
    __syncthreads();
    if (warp == 0) {
        constexpr int NW = TPB / 32;
        unsigned long long w = lane < NW ? warp_sums[lane] : 0ull;
        unsigned long long wi = w;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const unsigned long long t = __shfl_up_sync(0xFFFFFFFFu, wi, o);
            if (lane >= static_cast<unsigned>(o)) wi += t;
        }
        if (lane < NW) warp_sums[lane] = wi - w;
        if (lane == NW - 1) *total = wi;
    }
    __syncthreads();
    const unsigned long long r = warp_sums[warp] + incl - v;
    __syncthreads();
    return r;
}

// Find the bucket b of a PICK_BINS histogram where the running count first
// reaches `need` (1 <= need <= total).  Every thread gets b, the count below b
// and the count in b.
struct Pick {
    unsigned b;
    unsigned long long below;
    unsigned long long in_b;
};

// The thread's bins, PICK_BINS / TPB of them in order, are in v.  Counts sum
// to less than 2^32.  sc: 24 words of shared memory.
template <int TPB>
__device__ __forceinline__ Pick pick_loaded(const unsigned (&v)[PICK_BINS / TPB], unsigned long long need,
                                            unsigned long long* sc) {
    constexpr int PER = PICK_BINS / TPB, NW = TPB / 32;
    unsigned* warp_sums = reinterpret_cast<unsigned*>(sc);      // NW <= 32 entries
    unsigned* res = warp_sums + 32;                             // b, below, in_b
    const unsigned lane = threadIdx.x & 31u, warp = threadIdx.x >> 5;
    unsigned local = 0;
#pragma unroll
    for (int j = 0; j < PER; ++j) local += v[j];
    unsigned incl = local;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const unsigned t = __shfl_up_sync(0xFFFFFFFFu, incl, o);
        if (lane >= static_cast<unsigned>(o)) incl += t;
    }
    if (lane == 31) warp_sums[warp] = incl;
    __syncthreads();
    unsigned ws = lane < NW ? warp_sums[lane] : 0u;             // every warp scans the warps' sums
    const unsigned mine = ws;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const unsigned t = __shfl_up_sync(0xFFFFFFFFu, ws, o);
        if (lane >= static_cast<unsigned>(o)) ws += t;
    }
    const unsigned before = __shfl_sync(0xFFFFFFFFu, ws - mine, warp) + incl - local;
    const unsigned nd = static_cast<unsigned>(need);
    if (before < nd && nd <= before + local) {
        unsigned run = before;
#pragma unroll
        for (int j = 0; j < PER; ++j) {
            if (run < nd && nd <= run + v[j]) {
                res[0] = threadIdx.x * PER + j;
                res[1] = run;
                res[2] = v[j];
            }
            run += v[j];
        }
    }
    __syncthreads();
    const Pick p{res[0], res[1], res[2]};
    __syncthreads();
    return p;
}

// The thread's share of a histogram in global memory, read past L1.
template <int TPB>
__device__ __forceinline__ void pick_load_global(const unsigned* hist, unsigned (&v)[PICK_BINS / TPB]) {
    constexpr int PER = PICK_BINS / TPB;
    static_assert(PER % 4 == 0, "16-byte loads");
    const uint4* h = reinterpret_cast<const uint4*>(hist) + threadIdx.x * (PER / 4);
#pragma unroll
    for (int j = 0; j < PER / 4; ++j) {
        const uint4 x = __ldcg(h + j);
        v[4 * j] = x.x;
        v[4 * j + 1] = x.y;
        v[4 * j + 2] = x.z;
        v[4 * j + 3] = x.w;
    }
}
// A histogram in shared memory.
template <int TPB>
__device__ Pick pick_bucket(const unsigned* hist, unsigned long long need, unsigned long long* sc) {
    constexpr int PER = PICK_BINS / TPB;
    unsigned v[PER];
#pragma unroll
    for (int j = 0; j < PER; ++j) v[j] = hist[threadIdx.x * PER + j];
    return pick_loaded<TPB>(v, need, sc);
}

// Bitonic sort of `count` entries in shared memory (room for the next power of two), ascending
// by (r, rid); padded to a power of two with all-ones entries.
template <int TPB>
__device__ void block_sort(uint64_t* sr, uint32_t* srid, int count) {
    int m = 1;
    while (m < count) m <<= 1;
    for (int i = count + threadIdx.x; i < m; i += TPB) {
        sr[i] = ~0ull;
        srid[i] = ~0u;
    }
    __syncthreads();
    for (int size = 2; size <= m; size <<= 1) {
        for (int stride = size >> 1; stride > 0; stride >>= 1) {
            for (int t = threadIdx.x; t < (m >> 1); t += TPB) {
                const int lo = 2 * t - (t & (stride - 1));
                const int hi = lo + stride;
                const bool up = ((lo & size) == 0);
                const uint64_t a = sr[lo], b = sr[hi];
                const uint32_t ar = srid[lo], br = srid[hi];
                const bool swap = up ? elem_less(b, br, a, ar) : elem_less(a, ar, b, br);
                if (swap) {
                    sr[lo] = b;
                    sr[hi] = a;
                    srid[lo] = br;
                    srid[hi] = ar;
                }
            }
            __syncthreads();
        }
    }
}

// The threshold of the streaming pass moved into the key domain, so that a
// key is tested with one XOR and one unsigned comparison and no transform:
// `rank <= t` holds exactly when `(key ^ m) >= c` for the (m, c) below (m64 /
// c64 for 8-byte keys, m32 / c32 for 4-byte keys, whose rank is t's upper
// half t32 = t >> 32; the lower half of a 4-byte key's rank is zero).
//   signed integers: rank = key ^ SIGN (ASC) or its complement (DESC); the
//     signed key order is the unsigned order of key ^ SIGN, and "<=" becomes
//     ">=" on the complement.
//   unsigned integers: ASC  key <= t  <=>  ~key >= ~t;  DESC  ~key <= t  <=>  key >= ~t.
//   floats: with y = x ^ ((x >> (w-1)) & MAG) the signed image of totalOrder
//     (MAG = all bits but the sign) and L the signed limit on y, each of the
//     four cases (order x sign of L) is one unsigned comparison of x under a
//     fixed XOR mask:
//       DESC, L >= 0: y >= L  <=>  x ^ SIGN >= L ^ SIGN
//       DESC, L <  0: y >= L  <=>  ~x >= ~(L ^ MAG)
//       ASC,  L >= 0: y <= L  <=>  x ^ MAG >= L ^ MAG
//       ASC,  L <  0: y <= L  <=>  x >= L ^ MAG
//     (XOR with MAG reverses the signed order among negative values.)
struct KeyLimit {
    uint64_t m64, c64;
    uint32_t m32, c32;
};

template <typename U>
__device__ __forceinline__ void float_limit(U t, bool desc, U* m, U* c) {
    constexpr U SIGN = static_cast<U>(1) << (sizeof(U) * 8 - 1);
    constexpr U MAG = ~SIGN;
    const U uL = (desc ? static_cast<U>(~t) : t) ^ SIGN;          // signed limit on y, as bits
    const bool neg = (uL & SIGN) != 0;
    if (desc) {
        if (!neg) { *m = SIGN; *c = uL ^ SIGN; }
        else      { *m = static_cast<U>(~static_cast<U>(0)); *c = static_cast<U>(~(uL ^ MAG)); }
    } else {
        if (!neg) { *m = MAG; *c = uL ^ MAG; }
        else      { *m = 0;   *c = uL ^ MAG; }
    }
}

template <typename U>
__device__ __forceinline__ void int_limit(U t, bool desc, bool is_signed, U* m, U* c) {
    constexpr U SIGN = static_cast<U>(1) << (sizeof(U) * 8 - 1);
    if (is_signed) {
        const U lim = (desc ? static_cast<U>(~t) : t) ^ SIGN;      // signed limit on the key
        *m = desc ? SIGN : static_cast<U>(~SIGN);
        *c = lim ^ *m;
    } else {
        *m = desc ? static_cast<U>(0) : static_cast<U>(~static_cast<U>(0));
        *c = static_cast<U>(~t);
    }
}

__device__ __forceinline__ KeyLimit key_limit(uint64_t t, int kind, bool desc) {
    KeyLimit k{0, 0, 0, 0};
    const uint32_t t32 = static_cast<uint32_t>(t >> 32);
    switch (kind) {
        case OLAP_KEY_I64: int_limit<uint64_t>(t, desc, true, &k.m64, &k.c64); break;
        case OLAP_KEY_U64: int_limit<uint64_t>(t, desc, false, &k.m64, &k.c64); break;
        case OLAP_KEY_F64: float_limit<uint64_t>(t, desc, &k.m64, &k.c64); break;
        case OLAP_KEY_I32: int_limit<uint32_t>(t32, desc, true, &k.m32, &k.c32); break;
        case OLAP_KEY_U32: int_limit<uint32_t>(t32, desc, false, &k.m32, &k.c32); break;
        default: float_limit<uint32_t>(t32, desc, &k.m32, &k.c32); break;   // float32
    }
    return k;
}
// The same test as one comparison without the XOR: every limit above is x >= c
// or x <= c on the key's bits read as a signed or an unsigned integer.
enum KeyCmp { CMP_GE_U = 0, CMP_LE_U = 1, CMP_GE_S = 2, CMP_LE_S = 3 };
template <typename U>
__device__ __forceinline__ int key_cmp(U m, U c, U* lim) {
    constexpr U SIGN = static_cast<U>(1) << (sizeof(U) * 8 - 1);
    if (m == 0) { *lim = c; return CMP_GE_U; }
    if (m == static_cast<U>(~static_cast<U>(0))) { *lim = static_cast<U>(~c); return CMP_LE_U; }
    if (m == SIGN) { *lim = c ^ SIGN; return CMP_GE_S; }
    *lim = static_cast<U>(~c) ^ SIGN;                 // x ^ ~SIGN is the complement of x ^ SIGN
    return CMP_LE_S;
}
template <int MODE, typename U, typename S>
__device__ __forceinline__ bool key_pass(U x, U c) {
    if (MODE == CMP_GE_U) return x >= c;
    if (MODE == CMP_LE_U) return x <= c;
    if (MODE == CMP_GE_S) return static_cast<S>(x) >= static_cast<S>(c);
    return static_cast<S>(x) <= static_cast<S>(c);
}
__device__ __forceinline__ bool pass64(uint64_t bits, const KeyLimit& k) { return (bits ^ k.m64) >= k.c64; }
__device__ __forceinline__ bool pass32(uint32_t bits, const KeyLimit& k) { return (bits ^ k.m32) >= k.c32; }

}  // namespace olap
