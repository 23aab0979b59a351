// Top-K selection (ORDER BY key LIMIT K, Sec. III-A) on the GPU: launch
// arguments and host entry of the cooperative select kernel.
#pragma once

#include <cstdint>

#include "common.cuh"

namespace olap {

constexpr int TK_TPB = 512;               // threads per CTA
constexpr int TK_DIG = 12;                // default radix digit width (8..12; histograms hold 2^12 bins)
constexpr int TK_DIG_MIN = 8;
constexpr int TK_BINS = 1 << TK_DIG;
constexpr int TK_SMALL = 4096;            // entries one CTA sorts in shared memory
constexpr int TK_SAMPLE = 8192;           // sample size of the threshold estimate
constexpr int TK_SPT = TK_SAMPLE / TK_TPB;
constexpr int TK_PREP_CTAS = TK_SAMPLE / TK_TPB;   // prepare CTAs on the sampled path: one key per thread
constexpr int TK_UNROLL = 2;              // 32-byte loads in flight per thread (register filter)
constexpr uint64_t TK_DIRECT_N = 1ull << 21;   // at or below: no filter kernel of its own
// At or below: no sample, refine the input (float64 keys, K = 100, general path:
// 2^18 keys 21 against 22.5 us, 400,000 both 22.6, 2^19 24.6 against 22.5, 2^20
// 29 against 23-25).
constexpr uint64_t TK_SAMPLE_N = 3ull << 17;
// Few keys: every CTA holds the whole input in shared memory and works without
// the others (topk_local_kernel), up to TK_LOCAL_N keys, K = TK_LOCAL_K and
// n * K = TK_LOCAL_NK.  Device time against the general path, float64 keys:
// 1000 keys 4.5 against 7-9 us, 5000 keys 7.6 against 11.6, 10,007 keys 11 (K
// = 10) and 15 (K = 1000) against 12 and 16; past the line it loses: 16,000
// keys with K = 4000 37 against 25 us, 16,384 with K = 100 15 against 14.
constexpr uint64_t TK_LOCAL_N = 3ull << 12;
constexpr uint64_t TK_LOCAL_K = 4096;
constexpr uint64_t TK_LOCAL_NK = 1ull << 24;
constexpr int TKL_TPB = 1024;
constexpr int TKL_SMEM_MAX = TK_BINS * 4 + static_cast<int>(TK_LOCAL_N) * 12;
// Whether and where the sampled streaming pass runs: in a kernel of its own, or
// at the start of the select kernel.
enum { TK_SAMPLE_NONE = 0, TK_SAMPLE_FILTER = 1, TK_SAMPLE_INLINE = 2 };
constexpr int TK_RANK_MAX = 8192;         // survivors ranked in shared memory by the whole grid
constexpr int TK_SPLITTERS = 2047;        // splitters of the larger-K finish on tied keys (2^k - 1)
static_assert(TK_SPLITTERS <= TK_SMALL, "the splitters fit where K > TK_SMALL entries do");
// Entries they may split, about 128 per gap, which a warp ranks in registers
// (tied int64 keys, K = 250,000: the call 332 us, 452 with tile sorts and merges;
// 2 * 10^6 tied float32 keys, K = 400,000: 443 us by splitters, 326 by merges).
constexpr uint64_t TK_SPLIT_MAX = 2048ull * 128;
// Entries of a bin that the larger-K finish ranks in one CTA, all pairs of them:
// in equal bins where splitters may take their place (2 * 10^6 normal int64
// keys, K = 200,000: the call 139 us, 203 with splitters past 256; of 1024
// values, K = 20,000, bins of 1950 615 us, splitters 92), and otherwise.
constexpr unsigned TK_BIN_EVEN = 512;
constexpr unsigned TK_BIN_MAX = 1024;
constexpr int TK_SORT_SMEM = TK_RANK_MAX * 12;  // select kernel shared bytes (ranking / sort tile / histogram)
constexpr int TK_MAX_STAGES = 16;         // full + empty mbarrier pairs reserved after the ring
constexpr int TK_SMEM_MAX = 227 * 1024;   // opt-in shared memory per CTA
// The streaming filter runs as its own kernel: 256-thread CTAs, several per
// SM, each with a ring of bulk copies (default 16 KB x 3, four CTAs per SM);
// the register-load flavour uses CTAs of 256, 512 (default) or 1024 threads.
constexpr int TKF_TPB = 256;
constexpr int TKR_TPB = 512;
constexpr int TK_TILE_DEFAULT = 16384;
constexpr int TK_STAGES_DEFAULT = 3;
constexpr int TK_CTAS_PER_SM_DEFAULT = 4;

// Filter flavours: 32-byte register loads (the default), or bulk copies through
// a ring of shared-memory stages.
enum TopkFilter { TK_FILTER_REGS = 0, TK_FILTER_BULK = 1 };

// Device control block, zeroed by CTA 0 at the start of every launch.
struct TopkCtl {
    unsigned long long cand_count;   // filter: rank words <= threshold seen
    unsigned long long thresh;       // sample threshold (inclusive)
    unsigned long long fbase;        // the fused first pass bins [fbase, thresh]
    unsigned long long flow;         // candidates below fbase
    unsigned long long out_count;    // split: entries below the final prefix
    unsigned long long eq_count;     // split: prefix-equal entries taken wholesale
    unsigned long long small_count;  // split: prefix-equal entries kept for the finish
    int err;                         // olap_status of the device side
    int path;                        // 0 direct, 1 sampled candidates, 2 fallback
    int passes;                      // refine passes run
    int count_only;                  // the candidates would not fit: the streaming pass counts only
    // Minimum and maximum rank word, minimum and maximum row-id of the entries
    // a refine pass saw (three slots, by pass), and of the selected entries
    // before the finish partition.
    unsigned long long mm[3][4];
    unsigned long long fin[4];
    // %globaltimer stamps: prepare start, prepare end (sample done), select
    // start (filter done), source decided, refine done, split done, end,
    // small-buffer finish done, survivor sort done.
    unsigned long long ts[9];
};

struct TopkArgs {
    const void* keys;
    const void* host_keys;           // not NULL: the column in host memory, which the filter copies to keys
    const uint32_t* rowids;          // NULL => row-id = index
    uint64_t n;
    uint64_t k;                      // already min(k, n), > 0
    int kind;                        // olap_key_type
    int w4;                          // 4-byte keys (float32, int32, uint32)
    int desc;
    int local;                       // topk_local_kernel
    int use_sample;                  // TK_SAMPLE_NONE, _FILTER or _INLINE
    unsigned sample_rank;            // 1-based rank of the threshold in the sample
    int filter;                      // TopkFilter
    int fuse;                        // the filter folds the select's first radix pass (set at launch)
    int digit;                       // radix digit width, TK_DIG_MIN..TK_DIG (0 => TK_DIG)
    int tile_bytes;                  // bulk-copy size (multiple of 16 * TK_TPB)
    int stages;                      // copies in flight per CTA (<= TK_MAX_STAGES)
    TopkCtl* ctl;
    GridBar* bar;
    unsigned* ghist;                 // 3 x TK_BINS
    uint64_t* cand_r;
    uint32_t* cand_rid;
    uint64_t cand_cap;
    uint64_t* small_r;               // TK_SMALL
    uint32_t* small_rid;
    uint64_t* out_r0;                // k entries (selected, then sorted)
    uint32_t* out_rid0;
    uint64_t* out_r1;                // k entries, merge ping-pong (k > TK_SMALL)
    uint32_t* out_rid1;
    uint64_t* samples;               // TK_SAMPLE rank words of the sample (sampled path)
    void* out_keys;                  // caller's outputs (device)
    uint32_t* out_rowids;
    // Two-column key (ORDER BY c0, c1): keys / kind / desc describe c0 and
    // these c1; both columns are 4-byte kinds and the rank word is c0's rank
    // in the upper 32 bits and c1's in the lower 32 (w4 = 0).
    int pair;
    int kind2;
    int desc2;
    const void* keys2;
    void* out_keys2;
    int32_t* dev_status;             // optional status word, written by CTA 0
    int32_t* host_err;               // optional, zero before the call: the error of any CTA that gave up
};

// Plan of one Top-K call: which path and how much scratch it needs.
struct TopkPlan {
    int local;                       // topk_local_kernel
    int use_sample;
    unsigned sample_rank;
    uint64_t cand_cap;
};
TopkPlan topk_plan(uint64_t n, uint64_t k);
// The plan of a call whose columns, sizes and outputs are in `args`: as above,
// but not topk_local_kernel when an output lies over an input.  Its CTAs write
// while others may still load; every other path writes its results behind a
// grid barrier that follows the last read of the input, so results may take
// the place of the keys or row-ids they come from.  Needs the same scratch.
TopkPlan topk_plan_call(const TopkArgs& args);

// Bytes of device scratch a call with this plan needs (all buffers above).
size_t topk_scratch_bytes(const TopkPlan& p, uint64_t k);

// Carve the scratch buffers of `args` out of `base` (256-byte aligned pieces).
void topk_carve(TopkArgs& args, const TopkPlan& p, void* base);

// Launch geometry of one Top-K: the filter's copy ring (tile x stages), the
// filter grids and the cooperative select grid.
struct TopkGeom {
    int tile_bytes;
    int stages;
    int ctas_per_sm;       // filter CTAs per SM (cap)
    int smem_bytes;        // filter dynamic shared bytes: ring + mbarriers
    int grid;              // cooperative select kernel CTAs
    int grid_small;        // the same for a candidate-path select with k <= TK_SMALL (one CTA per SM)
    int filter_grid;       // bulk-copy filter CTAs
    int regs_grid;         // register-load filter CTAs
    int regs_tpb;          // register-load filter threads per CTA (256, 512, 1024)
};
// Fill in the geometry for the requested ring and register-filter block size
// on `device`; 0 values take the defaults.  Returns false if the ring does not
// fit, the block size is not one of 256/512/1024, or no CTA fits.
bool topk_geometry(int device, int tile_bytes, int stages, int ctas_per_sm, int regs_tpb, TopkGeom* out);

// Enqueue one Top-K: prepare (1 CTA, or TK_PREP_CTAS that load the sample),
// the streaming filter when the sampled path is taken, then the cooperative
// select kernel.  Returns the first CUDA
// launch error.
// ev (optional, 4 events): recorded before the prepare kernel and after the
// prepare, filter and select kernels (the filter pair is empty when the plan
// has no sample filter).
cudaError_t topk_launch(const TopkArgs& args, const TopkGeom& geom, cudaStream_t stream,
                        cudaEvent_t* ev = nullptr);

}  // namespace olap
