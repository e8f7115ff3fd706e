// sm_100a kernels of the mixed prefill-chunk + decode attention iteration.
//
//   sw_kv_append_kernel     scatter of this iteration's new K/V rows into their pages (Table 1, KV manager)
//   sw_mixed_attn_kernel    ONE persistent launch per iteration (Sec. 4.1).  Optionally it first writes the new K/V
//                           rows itself (the fused form of the append).  CTAs with chunk-prefill entries run them on
//                           the tensor cores (sw_prefill.cuh).  Every CTA then plans the split-KV decode units from
//                           the context lengths (without chunks, where line_form allows it: shares the pages out as a
//                           line instead, run_line); a warp's first unit is fixed by its index, further ones come from a
//                           shared counter; a unit streams its K/V pages with TMA into the warp's shared-memory ring
//                           and keeps an online softmax in registers; of the units of one (request, kv head) the one
//                           that drew the last ticket merges the partial results or, where there are many, the last
//                           ones one query-head row each.
#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include "sw_internal.h"
#include "sw_ptx.cuh"

namespace sw {
using namespace swptx;

// ---------------------------------------------------------------------------------------------------------------
// device status: first problem wins
// ---------------------------------------------------------------------------------------------------------------
__device__ __forceinline__ void report(int32_t* ctrl, int code, int site, int index) {
    if (atomicCAS(&ctrl[kCtrStatus], 0, code) == 0) ctrl[kCtrDetail] = (site << 24) | (index & 0xFFFFFF);
}

// ---------------------------------------------------------------------------------------------------------------
// KV append
// ---------------------------------------------------------------------------------------------------------------
// A warp takes 32 of the 16-byte pieces of a row's Hkv*D elements (of several rows where a row has fewer), of K and of V, and
// kAppendBatch times as many at once: what the append costs is its chain of latencies (position, page id, row, store), not its
// bytes.  `first` and `stride` spread the pieces over the calling warps.  (One piece per thread and pass, with 64-bit divisions,
// took 7.6-11 us of a launch with 2048 chunk rows.  With one row per warp, 8192 rows of 16 pieces made the fused launch of 8/2/64
// 151 us and that of 8/1/128 156 instead of 139 and 148.)
// (P is AppendParams or MixedParams: the fields have the same names; every index into the chunk arrays is a
// compile-time constant so that the kernel parameters stay in constant memory.)
constexpr int kAppendBatch = 4;   // in the fused launch, with 11 warps an SM; the stand-alone kernel has 32 of one part each
// (six: 2048 rows without a prefix 51.6 -> 50.7 us, but 64 contexts beside 512 tokens 62.8 -> 64.8)
template <bool kMulti, int kBatch, class P>
__device__ __forceinline__ void append_rows(const P& p, int head_dim, int first, int stride) {
    const int lane = threadIdx.x & 31;
    const int pieces_per_row = p.Hkv * head_dim / 8;
    const int per_row = (pieces_per_row + 31) / 32;   // warp-wide parts of a row
    const int rows_at_once = max(1, 32 / pieces_per_row), sub = lane / pieces_per_row, sub_lane = lane - sub * pieces_per_row;
    const int rows = p.C + p.n, total = (rows + rows_at_once - 1) / rows_at_once * per_row;
#pragma unroll 1
    for (int c0 = first; c0 < total; c0 += kBatch * stride) {
        uint4 k[kBatch], v[kBatch];
        int page[kBatch], slot[kBatch];   // slot: -1 = no such position in the list (reported)
#pragma unroll
        for (int b = 0; b < kBatch; ++b) {
            const int c = c0 + b * stride;
            slot[b] = -1;
            if (c >= total) break;
            const int part = c / per_row, row = part * rows_at_once + sub, piece = (c - part * per_row) * 32 + sub_lane;
            if (piece >= pieces_per_row || sub >= rows_at_once || row >= rows) continue;
            const int64_t src = ((int64_t)row * pieces_per_row + piece) * 8;
            k[b] = *reinterpret_cast<const uint4*>(p.k_new + src);
            v[b] = *reinterpret_cast<const uint4*>(p.v_new + src);
            unsigned pos;
            const int32_t* pages;
            int npages;
            if (row < p.C) {
                // the chunk this row belongs to: the last one that starts at or before it
                int cP = p.cP[0], cRow0 = 0, page0 = 0, page1 = p.num_prefill_pages;
#pragma unroll
                for (int j = 0; j < kMaxChunks; ++j)
                    if (kMulti && j < p.nchunks && row >= p.cRow0[j]) {
                        cP = p.cP[j];
                        cRow0 = p.cRow0[j];
                        page0 = p.cPage0[j];
                        page1 = p.cPage0[j + 1];
                    }
                pos = (unsigned)cP + (unsigned)(row - cRow0);
                pages = p.prefill_pages + page0;
                npages = page1 - page0;
            } else {
                const int i = row - p.C;
                const int len = p.decode_kv_len[i];
                pos = len < 1 ? 0xffffffffu : (unsigned)len - 1;
                const int beg = p.decode_page_indptr[i];
                pages = p.decode_pages + beg;
                npages = p.decode_page_indptr[i + 1] - beg;
            }
            const int pi = (int)(pos / kPageSize);
            if (pi < npages) {
                slot[b] = (int)(pos % kPageSize);
                page[b] = pages[pi];
            } else {
                report(p.ctrl, SW_ERR_OUT_OF_RANGE, kSiteAppendLen, row);
            }
        }
#pragma unroll
        for (int b = 0; b < kBatch; ++b) {
            const int c = c0 + b * stride;
            if (c >= total) break;
            if (slot[b] < 0) continue;
            const int part = c / per_row, e0 = ((c - part * per_row) * 32 + sub_lane) * 8;   // element offset inside the row's [Hkv][D]
            if (page[b] < 0 || page[b] >= p.num_pages) {
                report(p.ctrl, SW_ERR_OUT_OF_RANGE, kSiteAppendPage, part * rows_at_once + sub);
                continue;
            }
            const int64_t block = ((int64_t)page[b] * 2 * p.Hkv + e0 / head_dim) * kPageSize + slot[b];   // K; V is Hkv blocks further
            *reinterpret_cast<uint4*>(p.pool + block * head_dim + e0 % head_dim) = k[b];
            *reinterpret_cast<uint4*>(p.pool + (block + (int64_t)p.Hkv * kPageSize) * head_dim + e0 % head_dim) = v[b];
        }
    }
}

constexpr int kAppendThreads = 256, kAppendBlocksPerSm = 4;
__global__ void __launch_bounds__(kAppendThreads, kAppendBlocksPerSm) sw_kv_append_kernel(const AppendParams p) {
    // launched with programmatic stream serialization: it may start while the previous kernel (the attention of
    // the previous iteration, possibly still reading this pool) drains; nothing is touched before this wait
    grid_launch_dependents();
    grid_dependency_wait();
    append_rows<true, 1>(p, p.D, (int)(blockIdx.x * (blockDim.x / 32) + threadIdx.x / 32), (int)(gridDim.x * (blockDim.x / 32)));
}

cudaError_t launch_kv_append(const AppendParams& p, int num_sms, cudaStream_t stream) {
    const int pieces_per_row = p.Hkv * p.D / 8, rows_at_once = pieces_per_row < 32 ? 32 / pieces_per_row : 1;
    const int64_t total = (int64_t)((p.C + p.n + rows_at_once - 1) / rows_at_once) * ((pieces_per_row + 31) / 32);   // warp-wide parts
    if (total == 0) return cudaSuccess;
    const int threads = kAppendThreads;
    int64_t blocks = (total + threads / 32 - 1) / (threads / 32);
    // The grid is resident at once, so that the launch after this one is released at once too.  (Four parts a warp and grids of eight
    // blocks per SM: 3000 rows of 32/8/128 5.5 us instead of 5.2, 8192 10.7 instead of 10.3.  Eight blocks of 32 registers are as
    // fast alone and 1 us slower with the attention launch behind them, 461 rows 20.2 instead of 19.3 us.)
    if (blocks > (int64_t)num_sms * kAppendBlocksPerSm) blocks = (int64_t)num_sms * kAppendBlocksPerSm;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)blocks);
    cfg.blockDim = dim3(threads);
    cfg.dynamicSmemBytes = 0;
    cfg.stream = stream;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, sw_kv_append_kernel, p);
}

// Fused launches with chunks (append and attention in one kernel): every CTA writes its share of the new K/V rows at the
// start of the kernel and then adds one to a counter.  A page that can hold one of those rows (the last page of a decode
// request; the chunk's own keys) is not fetched before the counter shows every CTA's share.  The grid is one CTA per SM,
// so all CTAs are resident and the wait is short; it is bounded all the same.  Whole-warp call; false when the wait ran
// out.  (Fused decode-only launches need no counter, see load_new_row.)
__device__ __forceinline__ bool wait_append(const MixedParams& p, uint32_t set_addr) {
    if (!p.append_first) return true;
    int ok = 1;
    if ((threadIdx.x & 31) == 0) {
        const int32_t* counters = p.ctrl + lds_s32(set_addr);
        const long long t0 = clock64();
        while (ld_acquire_gpu(&counters[kSetAppend]) < (int)gridDim.x) {
            if (clock64() - t0 > kWaitBudgetCycles) {
                ok = 0;
                break;
            }
            __nanosleep(64);
        }
    }
    ok = __shfl_sync(0xffffffffu, ok, 0);
    fence_proxy_async_global();  // the rows were written with plain stores and are read through TMA
    return ok != 0;
}

// ---------------------------------------------------------------------------------------------------------------
// mixed attention: shared-memory plan
// ---------------------------------------------------------------------------------------------------------------
constexpr int kPageHashBits = 2048;   // buckets of the hash that tells pages with one writer from pages that may have several

// Words of the CTA's scratch from kMiscAt on: TMEM base, abort flag, the two tiles' ticket flags, the next entries (two, by the parity
// of the current one), where the launch's counters start (words into ctrl), and whether no decode unit is left for the CTA.
constexpr int kMiscAt = 32;
enum MiscWord { kMiscTmem = 0, kMiscAbort = 1, kMiscFlags = 2, kMiscNext = 5, kMiscSet = 7, kMiscNoUnits = 8 };

template <int D>
struct Geo {
    static constexpr int kHalves = D / 64;                    // 128-byte swizzled column blocks per row
    static constexpr int kBlockBytes = kPageSize * 128;       // one [16 tokens][64 elems] swizzled block
    static constexpr int kStageBytes = 2 * kHalves * kBlockBytes;  // K then V of one (page, kv head)
    static constexpr int kStages = 2;                          // page buffers in flight per warp (four at head size 64 gain nothing)
    static constexpr int kRingBytes = kWarps * kStages * kStageBytes;
    static constexpr int kBarOffset = kRingBytes;                              // kWarps*kStages mbarriers
    static constexpr int kPfBarOffset = kBarOffset + kWarps * kStages * 8;     // barriers of the prefill tiles
    static constexpr int kLastBarOffset = kPfBarOffset + 31 * 8;               // barrier: the list of last pages is there
    static constexpr int kPlanOffset = kPfBarOffset + 32 * 8;                  // int32 unit_prefix[kMaxDecode+1]
    static constexpr int kLenOffset = kPlanOffset + (kMaxDecode + 1) * 4 + 12;  // int32 kv_len[kMaxDecode]
    static constexpr int kIndptrOffset = kLenOffset + kMaxDecode * 4;           // int32 page_indptr[kMaxDecode+1]
    static constexpr int kLastOffset = kIndptrOffset + (kMaxDecode + 1) * 4 + 12; // int32 id of request i's last page
    static constexpr int kMiscOffset = kLastOffset + kMaxDecode * 4;              // scan scratch, TMEM base, abort flag
    static constexpr int kSetOffset = kMiscOffset + (kMiscAt + kMiscSet) * 4;      // where this launch's counters start (words into ctrl)
    static constexpr int kSharedOffset = kMiscOffset + 768;   // after 64 ints scan scratch and flags, the plan's counters, the chunk table:
    static constexpr int kSmemBytes = kSharedOffset + 2 * kPageHashBits / 8;      // two bit sets over hashed last pages
};

// From this many units of a request on, its last g units share the merge.  A merge of groups of eight by one warp takes two splits a
// round trip, of groups of four four: sharing it from eight units on instead of 24 took 64 contexts of 2000-20000 tokens of 32/4/128
// from 242 to 225 us, 128 of 8/1/128 from 136 to 123, 97 of them beside 423 tokens from 55 to 48; at head size 64, whose pages are
// half as long, 40 of 8/2/64 beside 700 tokens from 61 to 57.  (Groups of four at head size 128: 20 contexts of 20000 tokens of 32/8/128
// 263 -> 252, but 64 log-normal ones beside 256 tokens 143.7 -> 145.5; groups of two: 4/2/64 in place of 8/2/64 56 -> 58.)
__device__ __forceinline__ constexpr int wide_merge_splits(int head_dim, int g) { return g == 8 || (g == 4 && head_dim == 64) ? 8 : 24; }
constexpr int kOneRoundMaxPages = 48;  // longest unit (pages) for which one round of units is planned
constexpr int kPlanCounters = 8;       // shared counters of the plan's block sums, zeroed in the kernel prologue
// When the CTAs of a single wave of prefill entries turn to decode units: a fixed start-up plus the time of the longest
// entry's 128-key steps (MixedParams::step_us each, with the other CTAs streaming decode pages at the same time); the
// decode units stream one (page, kv head) stage per MixedParams::stage_us meanwhile.  Both figures come from the
// device's clocks (see sw_create).
constexpr float kLateBaseUs = 1.0f;
constexpr int kMinEarlyCtas = 64;  // CTAs whose rings of page copies keep the memory system busy on their own
constexpr int kMinLateCtas = 24;   // fewer late CTAs than this: their delay is not worth units of two sizes

// Decode-only launches run without units where they can: the stages (pages of one KV head) of all requests lie in a line, KV head by KV
// head and request by request, and every CTA gets an equal stretch of it, every warp an equal part of that.  So all warps stream the
// same number of pages, and the results of a (request, KV head) pair that lies on several warps meet in shared memory: what goes
// through global memory is one partial result per CTA that a pair reaches beyond, not one per warp.
// Per launch of 32/8/128, units -> line: one context of 8192 tokens 18.1 -> 15.4 us (33.5 MB: 2.2 TB/s), of 32768 38.7 -> 29.7, 16
// of 256-2048 22.1 -> 21.4, 64 of those 57.9 -> 54.4, 8 of 200-400 12.7 -> 11.0, 16 of 8192 90.5 -> 85.6, four of 49152 (55 pages a warp, which
// were two rounds of units) 139.7 -> 123.0 (6.5 TB/s), 128 log-normal ones 256 -> 249.1 (6.8 TB/s), 16 of 32k-131k 775 -> 760
// (7.1 TB/s); 20 of 256-4096 tokens of 16/4/64 18.7 -> 16.1.  What is left: 4 us to the first copies, CTAs that end up to 15 % apart (the
// SMs' rates differ), 2-4 us of merges.
// A CTA whose SM another kernel holds has its stretch for good; when it comes, the others have ended and it has their bandwidth: beside one
// held SM the launches above take 1.13 to 1.4 times as long, with units they took 1.06 (16 of 32k-131k, four rounds) to 1.6.
// (Beside chunk-prefill entries units stay: shares fixed by an estimate of when the late CTAs come were slower as often as faster, 16
// contexts of 256-2048 beside 300 tokens 26.4 -> 31.8 us, 40 of 256-8192 of 16/4/64 beside 700 42.2 -> 40.1.)
constexpr int kLineMaxStages = 0x7fffff00;   // 16 TB at head size 128
// Where no pair is longer than a few stages, none is cut: the boundaries of warps and CTAs move to the nearest end of a pair, there are as many
// CTAs as pairs, and nothing is merged.  `Few' is eight (what a unit has at least) and three times a warp's share of the line, up
// to 24 (at head size 64, where a partial result is half as long, 20).  Cut -> whole, us of 32/8/128: 16 contexts of 16-64 tokens 11.1 -> 8.9, 100 of
// 16-100 16.9 -> 12.3, 256 of 16-60 22.0 -> 17.9, 400 of 16-200 42.6 -> 38.4, 48 of 130-200 16.8 -> 14.5, 128 of 16-320 26.3 -> 22.5, 430 of
// 100-380 78.7 -> 77.0; of 8/2/64 256 of 16-60 11.6 -> 9.0, 400 of 16-200 17.9 -> 15.7; but 430 of 100-380 21.9 -> 22.8, hence the
// 20.  (Whole pairs beside cut ones gain nothing: 48 of 16-400 17.5 -> 18.3 and more.  32 of 81, which stretches of 12 pages cut at
// ends of pairs only: 9.0 -> 9.7.)
constexpr int kLineWhole = 8;
__device__ __forceinline__ constexpr int line_whole_max(int head_dim) { return head_dim == 64 ? 20 : 24; }
constexpr int kLineMaxDecode = 432;
constexpr int kLineGroups = kWarps + 1, kLineWords = 4, kLineTable = 88;   // (where launches with chunks keep their table)
static_assert((kLineTable + kLineGroups * kLineWords + 1) * 4 <= 768, "the table of the line lies in the CTA's scratch");
// Up to 432 requests, whose lengths, offsets, first stages and last pages take 1732 bytes of the four arrays of the plan; what is left
// of each holds three partial results (O of the group, m, l) of at most 2 KB + 64 bytes.
constexpr int kLineGroupElems = 512, kStashBytes = kLineGroupElems * 4 + 2 * kMaxGroup * 4, kStashesPerArray = 3, kPlanArrays = 4;
constexpr int kLineArrayBytes = ((kLineMaxDecode + 1) * 4 + 15) / 16 * 16;
static_assert(kPlanArrays * kStashesPerArray >= kWarps, "one partial result per warp");
static_assert(kLineArrayBytes + 15 + kStashesPerArray * kStashBytes <= kMaxDecode * 4, "behind an array's first entries lie its partial results");
static_assert(kLineGroupElems * 4 + 2 * kMaxGroup * 4 <= Geo<64>::kStageBytes, "a partial result fits a page buffer");
static_assert(kMaxCtas <= kTargetItems, "the line has a slot for every CTA and every (request, KV head) pair");
inline bool line_form(const MixedParams& p, int head_dim) {   // on the host
    return p.n <= kLineMaxDecode && p.group * head_dim <= kLineGroupElems;
}
struct Line {
    const int* len;     // shared-memory copies of the context lengths and page-list offsets
    const int* indptr;
    const int* prefix;  // stages before a request's, of one KV head
    int stages;         // of one KV head
    int total;          // of all KV heads
    int ctas;           // that share the line, in steps of 2^shift stages
    int coarse, shift;  // steps: 2^23 at most
    bool whole;         // no (request, KV head) pair is cut
};
struct Plan {
    const int* len;     // shared-memory copies of the context lengths and page-list offsets
    const int* indptr;
    bool two_sizes;     // large units handed out by index to the early CTAs, small ones pulled by the late CTAs only
    int total_items;    // units of all requests, times the KV heads
};

// Block-wide exclusive scan of one value per thread (kThreads threads): a warp scan, one barrier, then every thread
// adds up the warps before its own.  scratch: kWarps ints nobody has touched since the last barrier; one use only.
__device__ __forceinline__ int block_exclusive_scan(int v, int* scratch, int* total) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    int inc = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        int t = __shfl_up_sync(0xffffffffu, inc, o);
        if (lane >= o) inc += t;
    }
    if (lane == 31) scratch[warp] = inc;
    __syncthreads();
    int before = 0, all = 0;
#pragma unroll
    for (int w = 0; w < kWarps; ++w) {
        const int t = scratch[w];
        all += t;
        if (w < warp) before += t;
    }
    *total = all;
    return before + inc - v;
}

// Block-wide sum of one value per thread: a warp reduction, one shared-memory add per warp, one barrier.  ctr is a
// counter that was zero before the previous barrier; one use only.
__device__ __forceinline__ int block_sum(int v, int* ctr) {
    const int w = __reduce_add_sync(0xffffffffu, v);
    if ((threadIdx.x & 31) == 0 && w != 0) atomicAdd(ctr, w);
    __syncthreads();
    return *reinterpret_cast<volatile int*>(ctr);
}

constexpr int kLongPages = 512;   // from this many pages on a context is not cut into units of half the smallest size
// One-class unit size: pages per unit when `warps_per_head` warps share `total_pages`.  Small batches are
// latency-bound: one round of units, as many as there are warps, gets every warp streaming at once.  Large batches are
// bandwidth-bound: a few rounds of smaller units shorten the tail.  Every request adds at most one ragged unit per
// head, hence the "- n".
__device__ __forceinline__ int plan_split_pages(const MixedParams& p, int total_pages, bool any_long, int warps_per_head) {
    const int one_round = (total_pages + warps_per_head - 1) / warps_per_head;  // pages per unit if run in one round
    const int rounds = one_round <= kOneRoundMaxPages ? 1 : (one_round <= 160 ? 2 : 4);
    int units_target = max(1, rounds * warps_per_head - p.n);
    units_target = min(units_target, max(1, p.target_items / p.Hkv));
    // Where the batch is at most 16 stages per SM its time is the chain of a unit's pages, and units of half the smallest size
    // are faster although more of them are merged: one 1024-token context 14.8 -> 12.5 us, one of 4096 16.0 -> 14.9, four of 256-2048
    // 15.6 -> 13.9 (8192 tokens, 28 stages per SM: 18.3 -> 20.1).  Not for contexts of up to eight pages (one unit of the usual
    // size, which needs no merge), unless there are four of them or fewer: 32 of 81 tokens, 8/2/64, 12.3 us split and 10.6 whole, one
    // of 128, 32/8/128, 10.6 and 12.2.  And not where a context would be cut into 128 units or more, whose merge is the longer chain: one
    // of 32768 tokens, 8/1/128, 33.5 us and 25.8, one of 16384, 8/2/64, 21.9 and 19.7 (8192: 17.0 and 16.8).
    const bool small = total_pages >= p.small_from && total_pages <= p.small_to && !any_long;
    return max((total_pages + units_target - 1) / units_target, kMinSplitTokens / kPageSize / (small ? 2 : 1));
}

// CTAs that start with chunk-prefill work turn to decode units later than the others.
struct LateJoin {
    int ctas;   // how many CTAs (0 = none, gridDim.x = all: both plan like a decode-only launch)
    float us;   // estimated delay of their first decode unit relative to the other CTAs' first
};

// Every CTA derives the same plan from the context lengths: no host planning, no extra launch.
//
// When some CTAs join late the plan may have two unit sizes (plan.two_sizes).  The decode phase is bandwidth-bound, so
// by the time the late CTAs arrive the others have streamed about late.us * pages_per_us pages; what is left then is
// shared evenly among all warps.  The first requests are cut into large units (streamed share + even share), one for
// each warp of the early CTAs and handed out by index; the remaining requests are cut into small units (the even
// share), which only the warps of the late CTAs pull from the counter.  Both counts are made to fit the warps that
// run them, so that no warp starts a second unit.  If the early warps are nearly done by the time the late ones arrive,
// the plan is sized for the early warps alone; if the early CTAs are few, their head start is small or there are many
// requests per warp, it falls back to units of one size pulled by everybody.
__device__ __forceinline__ Plan make_plan(const MixedParams& p, int* unit_prefix, int* len_s, int* indptr_s, int* scratch,
                                          LateJoin late, float pages_per_us) {
    Plan plan;
    plan.len = len_s;
    plan.indptr = indptr_s;
    plan.two_sizes = false;
    const int per_thread = (p.n + kThreads - 1) / kThreads;
    const int beg = min(p.n, (int)threadIdx.x * per_thread);
    const int end = min(p.n, beg + per_thread);
    // total context in pages (fits an int: n <= 2048 requests of < 2^27 pages)
    int pages_local = 0;
    bool long_local = false;
    for (int i = beg; i < end; ++i) {
        const int len = p.decode_kv_len[i];
        const int pg = len > 0 ? (len + kPageSize - 1) / kPageSize : 0;
        pages_local += pg;
        long_local |= pg >= kLongPages;
        len_s[i] = len;                              // the units read these from shared memory later
        indptr_s[i] = p.decode_page_indptr[i];
    }
    if (threadIdx.x == 0 && p.n > 0) indptr_s[p.n] = p.decode_page_indptr[p.n];
    int* ctr = scratch + 64;  // kPlanCounters counters zeroed in the kernel prologue, one per block sum
    int pages_before = 0;
    const int warp_pages = __reduce_add_sync(0xffffffffu, pages_local);
    if ((threadIdx.x & 31) == 0 && warp_pages != 0) atomicAdd(ctr, warp_pages);
    const bool any_long = __syncthreads_or(long_local);   // (the barrier of the sum, see block_sum)
    const int total_pages = *reinterpret_cast<volatile int*>(ctr++);

    const int G = (int)gridDim.x;
    constexpr int kMinPages = kMinSplitTokens / kPageSize;
    int split_a = 0, split_b = 0;  // pages per unit of the first requests / of the rest
    int a_pages = 0x7fffffff;      // requests whose pages start below this (per head) are cut with split_a
    if (late.ctas <= 0 || late.ctas >= G) {
        split_a = split_b = plan_split_pages(p, total_pages, any_long, max(1, G * kWarps / p.Hkv));
    } else {
        const float early = (float)((G - late.ctas) * kWarps), all = (float)(G * kWarps);
        const float pages = (float)total_pages * p.Hkv;
        const float streamed = fminf(pages, pages_per_us * late.us);
        const float even = (pages - streamed) / all;
        // units and pages (per head) of the early warps and of the late ones; a request adds about half a ragged unit
        const float a_units = early / p.Hkv, b_units = (all - early) / p.Hkv;
        const float a_share = fminf((float)total_pages, a_units * (streamed / early + even));
        const float b_share = (float)total_pages - a_share;
        const float a_ragged = 0.6f * p.n * a_share / fmaxf(1.f, (float)total_pages);
        const float b_ragged = 0.6f * p.n - a_ragged;
        if (G - late.ctas < kMinEarlyCtas || late.ctas < kMinLateCtas || streamed < 0.25f * pages) {
            // Too few early CTAs to keep the memory system busy on their own (the estimate of what they stream would
            // not hold), or a head start that is small next to the whole phase: one unit size, every warp pulls.
            split_a = split_b = plan_split_pages(p, total_pages, any_long, max(1, G * kWarps / p.Hkv));
        } else if (pages - streamed < (float)(late.ctas * kWarps * kMinPages)) {
            split_a = split_b = plan_split_pages(p, total_pages, any_long, max(1, (G - late.ctas) * kWarps / p.Hkv));
        } else if (a_ragged > 0.25f * a_units || b_ragged > 0.25f * b_units) {
            // too many requests per warp for one even unit each: units pulled by every warp balance better
            split_a = split_b = plan_split_pages(p, total_pages, any_long, max(1, G * kWarps / p.Hkv));
        } else {
            split_a = max(kMinPages, (int)ceilf(a_share / (a_units - a_ragged)));
            split_b = max(kMinPages, (int)ceilf(b_share / (b_units - b_ragged)));
            a_pages = (int)a_share;
            plan.two_sizes = true;
        }
    }
    if (plan.two_sizes) {
        int unused;
        pages_before = block_exclusive_scan(pages_local, scratch + 16, &unused);
        // count the units of either size and grow the size until they fit their warps (the estimates are rarely off)
        const int a_units = (G - late.ctas) * kWarps / p.Hkv, b_units = late.ctas * kWarps / p.Hkv;
        for (int pass = 0; pass < (kPlanCounters - 1) / 2; ++pass) {
            int cnt_a = 0, cnt_b = 0, before = pages_before;
            for (int i = beg; i < end; ++i) {
                const int pg = len_s[i] > 0 ? (len_s[i] + kPageSize - 1) / kPageSize : 0;
                if (before < a_pages) cnt_a += (pg + split_a - 1) / split_a; else cnt_b += (pg + split_b - 1) / split_b;
                before += pg;
            }
            const int total_a = block_sum(cnt_a, ctr++);
            const int total_b = block_sum(cnt_b, ctr++);
            if (total_a <= a_units && total_b <= b_units) break;
            if (total_a > a_units) split_a = (int)(((int64_t)split_a * total_a + a_units - 1) / a_units) + 1;
            if (total_b > b_units) split_b = (int)(((int64_t)split_b * total_b + b_units - 1) / b_units) + 1;
        }
    }
    int units_local = 0;
    for (int i = beg; i < end; ++i) {
        const int len = len_s[i];
        const int pg = len > 0 ? (len + kPageSize - 1) / kPageSize : 0;
        const int split = pages_before < a_pages ? split_a : split_b;
        units_local += (pg + split - 1) / split;
        pages_before += pg;
    }
    pages_before -= pages_local;
    int total_units = 0;
    int run = block_exclusive_scan(units_local, scratch, &total_units);
    for (int i = beg; i < end; ++i) {
        unit_prefix[i] = run;
        const int len = len_s[i];
        const int pg = len > 0 ? (len + kPageSize - 1) / kPageSize : 0;
        const int split = pages_before < a_pages ? split_a : split_b;
        run += (pg + split - 1) / split;
        pages_before += pg;
    }
    if (threadIdx.x == 0) unit_prefix[p.n] = total_units;
    __syncthreads();
    plan.total_items = total_units * p.Hkv;
    return plan;
}

// The line of a decode-only launch.  A request whose page list ends before its context has no stages in it, and no output.
template <int D>
__device__ __forceinline__ Line make_line(const MixedParams& p, int* prefix, int* len_s, int* indptr_s, int* scratch) {
    const int per_thread = (p.n + kThreads - 1) / kThreads;
    const int first = min(p.n, (int)threadIdx.x * per_thread), last = min(p.n, first + per_thread);
    auto stages_of = [&](int len, int listed) {
        const int pages = len > 0 ? (len - 1) / kPageSize + 1 : 0;
        return pages <= listed ? pages : 0;
    };
    int here = 0;
    for (int i = first; i < last; ++i) {
        const int len = p.decode_kv_len[i], at = p.decode_page_indptr[i], listed = p.decode_page_indptr[i + 1] - at;
        len_s[i] = len;
        indptr_s[i] = at;
        prefix[i] = stages_of(len, listed);
        here += prefix[i];
        if (i == p.n - 1) indptr_s[p.n] = at + listed;
        if (len > 0 && prefix[i] == 0 && blockIdx.x == 0) report(p.ctrl, SW_ERR_OUT_OF_RANGE, kSiteAttnLen, p.C + i);
    }
    Line line;
    line.len = len_s;
    line.indptr = indptr_s;
    line.prefix = prefix;
    int before = block_exclusive_scan(here, scratch + 16, &line.stages);
    if (line.stages < 0 || (int64_t)line.stages * p.Hkv > kLineMaxStages) {
        if (blockIdx.x == 0 && threadIdx.x == 0) report(p.ctrl, SW_ERR_WORKSPACE, kSiteScratch, line.stages);
        line.stages = 0;
    }
    const int few = min(line_whole_max(D), kLineWhole + line.stages * p.Hkv / ((int)gridDim.x * 4));
    bool longer = false;
    for (int i = first; i < last; ++i) {
        const int stages = prefix[i];
        longer |= stages > few;
        prefix[i] = before;
        before += stages;
    }
    if (threadIdx.x == 0) prefix[p.n] = line.stages;
    if (threadIdx.x == 32) scratch[kLineTable + kLineGroups * kLineWords] = 0;
    line.total = line.stages * p.Hkv;
    line.ctas = line.total / kWarps;
    line.whole = __syncthreads_or(longer) == 0;
    if (line.whole) line.ctas = max(line.ctas, p.n * p.Hkv);
    line.ctas = max(1, min((int)gridDim.x, line.ctas));
    line.shift = max(0, 9 - __clz(line.total));
    line.coarse = ((line.total - 1) >> line.shift) + 1;
    return line;
}

// ---------------------------------------------------------------------------------------------------------------
// one split-KV unit on one warp
// ---------------------------------------------------------------------------------------------------------------
struct Unit {
    int q_row;          // row of q / out
    int kvh;            // KV head
    int len;            // keys attended by this row in total
    int t_begin, t_end; // this unit's key range
    int nsplit;         // units of this (row, kv head); 1 = write the result directly
    int split;          // index among them
    int ticket;         // ticket slot (decode request * Hkv + kvh)
    int slot;           // partial-result slot
    const int32_t* pages;
};

template <int D>
struct WarpRing {
    uint32_t buf;   // shared address of this warp's first stage
    uint32_t bar;   // shared address of this warp's first mbarrier
    uint32_t it;    // pages consumed so far (stage = it % stages, parity = (it / stages) & 1)
};

// Lane 0 arms the stage's barrier and fetches the page with one copy: the head's K blocks, then its V blocks.
template <int D>
__device__ __forceinline__ void issue_page(const CUtensorMap* kvp_map, const WarpRing<D>& ring, uint32_t issue_it, int page,
                                           int kvh) {
    if ((threadIdx.x & 31) == 0) {
        const uint32_t stage = issue_it % Geo<D>::kStages;
        const uint32_t bar = ring.bar + stage * 8;
        mbar_arrive_expect_tx(bar, Geo<D>::kStageBytes);
        // a decode page is read once: evict-first keeps it from pushing the chunk's K/V tiles out of L2
        tma_load_5d_hint(ring.buf + stage * Geo<D>::kStageBytes, kvp_map, bar, 0, 0, 0, 2 * page, kvh, l2_policy_evict_first());
    }
}

// Merge of the splits of one (request, kv head), rows [row0, row0 + nrows) of the group (all of them, or one row when several
// units share the merge).  J splits at a time: lane j fetches (m, l) of split j while all lanes fetch their four (two) columns
// of the J partial outputs, so a merge of up to J splits costs one round trip to L2; it is the round trips (about a
// microsecond each) that a merge consists of: with eight at a time instead of sixteen a 32768-token context of one query head per KV
// head took 32.8 us per launch instead of 25.6 (4/4/64) and 43.8 instead of 38.1 (8/8/128).  G >= nrows is a compile-time bound:
// rows beyond the group read row 0 with weight zero, which keeps the loops free of branches.  Slots of the splits are Hkv apart.
template <int D, int G, int J = (G >= 8 ? 2 : (G == 4 ? 4 : (G == 2 ? 8 : 16)))>
__device__ __forceinline__ void merge_splits(const MixedParams& p, const Unit& u, int row0, int nrows) {
    constexpr int V = D / 32;                 // output columns per lane
    const int lane = threadIdx.x & 31;
    const int g = p.group;
    const int slot0 = u.slot - u.split * p.Hkv;
    const int ns = u.nsplit;
    const float* ml0 = p.part_ml + (int64_t)slot0 * (2 * kMaxGroup) + row0;  // split s: + s * ml_stride
    const int64_t ml_stride = (int64_t)p.Hkv * (2 * kMaxGroup);
    const float* po0 = p.part_o + ((int64_t)slot0 * g + row0) * D + lane * V;  // split s, row r: + s * po_stride + r * D
    const int64_t po_stride = (int64_t)p.Hkv * g * D;
    float m_all[G], l_all[G], acc[G][V];
#pragma unroll
    for (int r = 0; r < G; ++r) {
        m_all[r] = -INFINITY;
        l_all[r] = 0.f;
#pragma unroll
        for (int v = 0; v < V; ++v) acc[r][v] = 0.f;
    }
#pragma unroll 1
    for (int s0 = 0; s0 < ns; s0 += J) {
        float x[J][G][V];
#pragma unroll
        for (int j = 0; j < J; ++j) {
            const float* src = po0 + min(s0 + j, ns - 1) * po_stride;
#pragma unroll
            for (int r = 0; r < G; ++r) {
                const float* row = src + (r < nrows ? r : 0) * D;
                if constexpr (V == 4) {
                    const float4 t = __ldcg(reinterpret_cast<const float4*>(row));
                    x[j][r][0] = t.x, x[j][r][1] = t.y, x[j][r][2] = t.z, x[j][r][3] = t.w;
                } else {
                    const float2 t = __ldcg(reinterpret_cast<const float2*>(row));
                    x[j][r][0] = t.x, x[j][r][1] = t.y;
                }
            }
        }
        const bool live = lane < J && s0 + lane < ns;
        const float* ml = ml0 + min(s0 + (lane < J ? lane : 0), ns - 1) * ml_stride;
        float w[G];
#pragma unroll
        for (int r = 0; r < G; ++r) {
            float ms = __ldcg(ml + (r < nrows ? r : 0));
            const float ls = __ldcg(ml + kMaxGroup + (r < nrows ? r : 0));
            if (!live) ms = -INFINITY;
            float mw = fmaxf(ms, m_all[r]);   // over lanes 0 .. J-1
#pragma unroll
            for (int o2 = J / 2; o2 > 0; o2 >>= 1) mw = fmaxf(mw, __shfl_xor_sync(0xffffffffu, mw, o2));
            mw = __shfl_sync(0xffffffffu, mw, 0);
            w[r] = ms == -INFINITY ? 0.f : fast_exp2((ms - mw) * p.sm_scale_log2);
            float lw = w[r] * ls;
            if (!live) lw = 0.f;
#pragma unroll
            for (int o2 = J / 2; o2 > 0; o2 >>= 1) lw += __shfl_xor_sync(0xffffffffu, lw, o2);
            lw = __shfl_sync(0xffffffffu, lw, 0);
            const float a = m_all[r] == -INFINITY ? 0.f : fast_exp2((m_all[r] - mw) * p.sm_scale_log2);
            l_all[r] = l_all[r] * a + lw;
            m_all[r] = mw;
#pragma unroll
            for (int v = 0; v < V; ++v) acc[r][v] *= a;
        }
#pragma unroll
        for (int j = 0; j < J; ++j)
#pragma unroll
            for (int r = 0; r < G; ++r) {
                const float wj = __shfl_sync(0xffffffffu, w[r], j);   // zero past the last split
#pragma unroll
                for (int v = 0; v < V; ++v) acc[r][v] = fmaf(wj, x[j][r][v], acc[r][v]);
            }
    }
#pragma unroll
    for (int r = 0; r < G; ++r) {
        if (r < nrows) {
            const float inv = 1.f / l_all[r];
            const int hd = u.kvh * g + row0 + r;
            __nv_bfloat16* dst = p.out + ((int64_t)u.q_row * p.Hq + hd) * D + lane * V;
            if constexpr (V == 4) {
                *reinterpret_cast<uint2*>(dst) = make_uint2(pack_bf16x2(acc[r][0] * inv, acc[r][1] * inv),
                                                            pack_bf16x2(acc[r][2] * inv, acc[r][3] * inv));
            } else {
                *reinterpret_cast<uint32_t*>(dst) = pack_bf16x2(acc[r][0] * inv, acc[r][1] * inv);
            }
            if (p.lse && lane == 0) p.lse[(int64_t)u.q_row * p.Hq + hd] = m_all[r] * p.sm_scale + __logf(l_all[r]);
        }
    }
}

// The new row of a (request, KV head) pair as 16-byte pieces: lanes 0 .. D/8-1 hold K, the next D/8 hold V.
//
// Fused decode-only launches: the new row of a request is written into its last page by the units that reach that page (one
// per KV head), and, since the page's copy may have been made before, into the copy as well.  Requests that share their last
// page (drafts of one sequence, say) find each other's new rows through the list of last pages.  Nobody waits for anybody.
// (Appending first and counting the shares, as launches with chunks do, puts 3.5 us before the first page copy and makes the
// units that reach a last page wait up to 6 us for the counter.  Measured with the units spread over the SMs and the shared
// merge of small batches: one 8192-token context 23.5 -> 18.4 us per launch, 16 contexts of 256-2048 tokens 25.3 -> 22.4 us.)
template <int D>
__device__ __forceinline__ uint4 load_new_row(const MixedParams& p, int i, int kvh) {
    const int lane = threadIdx.x & 31;
    if (lane >= D / 4) return make_uint4(0u, 0u, 0u, 0u);
    const __nv_bfloat16* src = lane < D / 8 ? p.k_new : p.v_new;
    return *reinterpret_cast<const uint4*>(src + ((int64_t)i * p.Hkv + kvh) * D + (lane % (D / 8)) * 8);
}
template <int D>
__device__ __forceinline__ void patch_row(uint32_t buf, int slot, uint4 v) {
    const int lane = threadIdx.x & 31, chunk = lane % (D / 8);
    if (lane < D / 4)
        sts_v4(buf + (lane / (D / 8)) * (Geo<D>::kHalves * Geo<D>::kBlockBytes) + (chunk >> 3) * Geo<D>::kBlockBytes + slot * 128 +
                   (((chunk & 7) ^ (slot & 7)) << 4), v.x, v.y, v.z, v.w);
}
__device__ __forceinline__ unsigned page_hash(int page) { return ((unsigned)page * 2654435761u) >> 21; }
static_assert(kPageHashBits == 1 << (32 - 21), "the hash has as many values as there are buckets");
// All new rows of the page in buffer `buf`, the last one of request i.  A request whose last page lies outside the pool has id -1 in
// the list and reads page 0: it shares that page with nobody.  (Requests of length 0 and less have id -1 too, and no row at all: a
// search for -1 would find them and write in front of the buffer.)
template <int D>
__device__ __forceinline__ void patch_page(const MixedParams& p, uint32_t smem, uint32_t buf, int i, int kvh, int valid, uint4 own) {
    const int lane = threadIdx.x & 31;
    const int page = lds_s32(smem + Geo<D>::kLastOffset + i * 4);
    const unsigned h = page_hash(page);
    const bool several = page >= 0 && (lds_s32(smem + Geo<D>::kSharedOffset + (kPageHashBits + h) / 32 * 4) >> (h & 31) & 1);
#pragma unroll 1
    for (int j0 = 0; several && j0 < p.n; j0 += 32) {
        const int j = j0 + lane;
        bool hit = false;
        if (j < p.n && j != i && lds_s32(smem + Geo<D>::kLastOffset + j * 4) == page)
            hit = (lds_s32(smem + Geo<D>::kLenOffset + j * 4) - 1) % kPageSize + 1 < valid;
        unsigned found = __ballot_sync(0xffffffffu, hit);
        while (found) {
            const int other = j0 + __ffs(found) - 1;
            found &= found - 1;
            patch_row<D>(buf, (lds_s32(smem + Geo<D>::kLenOffset + other * 4) - 1) % kPageSize, load_new_row<D>(p, other, kvh));
        }
    }
    patch_row<D>(buf, valid - 1, own);
    if (page >= 0 && lane < D / 4) {
        const int64_t block = ((int64_t)page * 2 + lane / (D / 8)) * p.Hkv + kvh;
        *reinterpret_cast<uint4*>(p.pool + (block * kPageSize + valid - 1) * D + (lane % (D / 8)) * 8) = own;
    }
    __syncwarp();
}

// Shared merges (requests cut into many units): the calling unit, whose partial result is written, publishes it and learns which
// query-head rows it has to merge, as a bit mask (0: none; -1: the bounded wait expired).  One lane calls it.  merge_row: the unit's
// own row, -1 if it has none.
//
// A merger may only wait for units that run: one that has not started may be waiting for this merger's SM (another kernel can
// hold an SM for as long as it likes, and two launches of this one can each hold a part of the SMs), or for its warp.  So every
// unit counts itself in `started` when it begins, and a merger that finds units missing hands its row over and leaves; the unit
// that publishes last, after which nobody has to wait, merges the rows that were handed over before.
// `ready`: the low half counts the units that have published and then, once those are all, the rows that are merged; bit 16 + r:
// row r is handed over.
constexpr int kPublished = 0xffff;
constexpr long long kPatienceCycles = 20000;   // ten microseconds: the CTAs of a launch start within two or three of each other
__device__ __forceinline__ int rows_to_merge(int32_t* ready, const int32_t* started, int nsplit, int merge_row) {
    const int own = merge_row < 0 ? 0 : 1 << merge_row;
    const int before = atomicAdd(ready, 1);
    if ((before & kPublished) == nsplit - 1) {
        __threadfence();
        return own | before >> 16;
    }
    if (own == 0) return 0;
    const long long t0 = clock64();
    while ((ld_acquire_gpu(ready) & kPublished) < nsplit) {
        const long long waited = clock64() - t0;
        if (waited > kWaitBudgetCycles) return -1;
        if (waited > kPatienceCycles && ld_relaxed_gpu(started) < nsplit) {
            if ((atomicOr(ready, own << 16) & kPublished) < nsplit) return 0;
            __threadfence();   // the others have started and published meanwhile: the last one did not see it
            return own;
        }
        __nanosleep(64);
    }
    return own;
}

// A decode unit's queries as B fragments of Q^T: the lane holds head lane / 4, elements 2 (lane % 4) + {0, 1} (+ 8) of every 16.
template <int D>
__device__ __forceinline__ void load_query(const MixedParams& p, int q_row, int kvh, uint32_t (&qb)[D / 16][2]) {
    const int lane = threadIdx.x & 31;
    const uint32_t* src = reinterpret_cast<const uint32_t*>(p.q + ((int64_t)q_row * p.Hq + kvh * p.group + (lane >> 2)) * D + (lane & 3) * 2);
    const bool live = (lane >> 2) < p.group;
#pragma unroll
    for (int ks = 0; ks < D / 16; ++ks) {
        qb[ks][0] = live ? src[ks * 8] : 0u;
        qb[ks][1] = live ? src[ks * 8 + 4] : 0u;
    }
}

// O^T of the keys so far: columns 16 t + lane / 4 (+ 8) of heads 2 (lane % 4) + {0, 1}; m of those two heads; l over the lane's own keys.
template <int D>
struct DecodeState {
    float o[D / 16][4];
    float m0, m1, l0, l1;
    __device__ __forceinline__ void clear() {
#pragma unroll
        for (int i = 0; i < D / 16; ++i) o[i][0] = o[i][1] = o[i][2] = o[i][3] = 0.f;
        m0 = m1 = -INFINITY;
        l0 = l1 = 0.f;
    }
};

// One page (K and V of a head at sK, `valid` keys of it attended) on one warp.
//
// The products are transposed: the 16 rows of an mma.m16n8k16 are keys (of S = K Q^T) or output columns (of O^T = V^T P^T) and
// its 8 columns are the query heads of the group (columns past the group are zero queries), half the instructions of the form
// with the heads as rows, which would be padded to 16.
template <int D>
__device__ __forceinline__ void attend_page(const MixedParams& p, uint32_t sK, int valid, const uint32_t (&qb)[D / 16][2], DecodeState<D>& st) {
    constexpr int KS = D / 16;  // k-slices of K Q^T; also 16-column tiles of O
    const int lane = threadIdx.x & 31;
    // Per-lane offsets of the ldmatrix rows: the four 8x8 matrices are keys 0-7 / 8-15 of one 8-element block, then of the next
    // (K), or the two blocks of keys 0-7, then of keys 8-15 (V, transposed).  In the 128-byte swizzle 16-byte chunk c of row r
    // lies at c ^ (r % 8), so a step of two chunks flips address bits 5 and 6.
    const uint32_t k_addr = sK + (lane & 15) * 128 + (((lane >> 4) ^ (lane & 7)) << 4);
    const uint32_t v_addr = sK + Geo<D>::kHalves * Geo<D>::kBlockBytes + ((lane & 7) + ((lane >> 4) << 3)) * 128 +
                            ((((lane >> 3) & 1) ^ (lane & 7)) << 4);
    // S^T = K Q^T for 16 keys, in two chains
    float s[4] = {0.f, 0.f, 0.f, 0.f}, s2[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
    for (int ks = 0; ks < KS; ++ks) {
        uint32_t a0, a1, a2, a3;
        ldmatrix_x4((k_addr ^ ((ks & 3) * 32)) + (ks >> 2) * Geo<D>::kBlockBytes, a0, a1, a2, a3);
        mma_bf16_16816(ks & 1 ? s2 : s, a0, a1, a2, a3, qb[ks][0], qb[ks][1]);
    }
    // the lane's keys are lane / 4 and lane / 4 + 8; keys past the context are masked
    const bool ok0 = (lane >> 2) < valid, ok1 = (lane >> 2) + 8 < valid;
    s[0] = ok0 ? s[0] + s2[0] : -INFINITY;
    s[1] = ok0 ? s[1] + s2[1] : -INFINITY;
    s[2] = ok1 ? s[2] + s2[2] : -INFINITY;
    s[3] = ok1 ? s[3] + s2[3] : -INFINITY;
    float mx0 = fmaxf(s[0], s[2]), mx1 = fmaxf(s[1], s[3]);
#pragma unroll
    for (int w = 4; w < 32; w <<= 1) {
        mx0 = fmaxf(mx0, __shfl_xor_sync(0xffffffffu, mx0, w));
        mx1 = fmaxf(mx1, __shfl_xor_sync(0xffffffffu, mx1, w));
    }
    mx0 = fmaxf(st.m0, mx0);
    mx1 = fmaxf(st.m1, mx1);
    const float c0 = fast_exp2((st.m0 - mx0) * p.sm_scale_log2), c1 = fast_exp2((st.m1 - mx1) * p.sm_scale_log2);
    st.m0 = mx0;
    st.m1 = mx1;
    const float b0 = mx0 * p.sm_scale_log2, b1 = mx1 * p.sm_scale_log2;
    s[0] = fast_exp2(fmaf(s[0], p.sm_scale_log2, -b0));
    s[1] = fast_exp2(fmaf(s[1], p.sm_scale_log2, -b1));
    s[2] = fast_exp2(fmaf(s[2], p.sm_scale_log2, -b0));
    s[3] = fast_exp2(fmaf(s[3], p.sm_scale_log2, -b1));
    st.l0 = st.l0 * c0 + (s[0] + s[2]);
    st.l1 = st.l1 * c1 + (s[1] + s[3]);
#pragma unroll
    for (int i = 0; i < KS; ++i) {
        st.o[i][0] *= c0;
        st.o[i][1] *= c1;
        st.o[i][2] *= c0;
        st.o[i][3] *= c1;
    }
    // P^T [keys][heads] as the B operand: keys along the fragment's registers, so the 8x8 blocks are transposed
    const uint32_t p0 = movmatrix_trans(pack_bf16x2(s[0], s[1])), p1 = movmatrix_trans(pack_bf16x2(s[2], s[3]));

    // the unwritten slots of a partly filled last page hold whatever the pool held: zero those V rows so that
    // 0 * garbage cannot produce NaN
    if (valid < kPageSize) {
        __syncwarp();
        const int dead_rows = kPageSize - valid;
        for (int c = lane; c < dead_rows * (D / 8); c += 32) {
            const int row_i = valid + c / (D / 8);
            const int chunk = c % (D / 8);
            sts_v4(sK + (Geo<D>::kHalves + (chunk >> 3)) * Geo<D>::kBlockBytes + row_i * 128 + (((chunk & 7) ^ (row_i & 7)) << 4),
                   0u, 0u, 0u, 0u);
        }
        __syncwarp();
    }

    // O^T += V^T P^T
#pragma unroll
    for (int dn = 0; dn < KS; ++dn) {
        uint32_t a0, a1, a2, a3;
        ldmatrix_x4_trans((v_addr ^ ((dn & 3) * 32)) + (dn >> 2) * Geo<D>::kBlockBytes, a0, a1, a2, a3);
        mma_bf16_16816(st.o[dn], a0, a1, a2, a3, p0, p1);
    }
}

// The end of a unit: the row sums over the keys of all lanes, then O through shared memory, so that rows leave in whole lines:
// O[head][D] with the 32-byte groups of a row rotated by half the head (the lanes' four head pairs then fall on different banks).
template <int D>
__device__ __forceinline__ void stage_result(uint32_t dst, int g, DecodeState<D>& st) {
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int w = 4; w < 32; w <<= 1) {
        st.l0 += __shfl_xor_sync(0xffffffffu, st.l0, w);
        st.l1 += __shfl_xor_sync(0xffffffffu, st.l1, w);
    }
    const int h = (lane & 3) * 2;
    const uint32_t addr = dst + (h * D + (lane >> 2)) * 4;
#pragma unroll
    for (int t = 0; t < D / 16; ++t) {
        const uint32_t a0 = addr + ((16 * t) ^ (h * 4)) * 4, a1 = addr + ((16 * t + 8) ^ (h * 4)) * 4;
        if (h < g) {
            sts_f32(a0, st.o[t][0]);
            sts_f32(a1, st.o[t][2]);
        }
        if (h + 1 < g) {
            sts_f32(a0 + D * 4, st.o[t][1]);
            sts_f32(a1 + D * 4, st.o[t][3]);
        }
    }
    __syncwarp();
}
// Output rows of a (request, KV head) pair that one unit did alone, from the staged result.
template <int D>
__device__ __forceinline__ void write_rows(const MixedParams& p, uint32_t src, int q_row, int kvh, const DecodeState<D>& st) {
    constexpr int kRowLanes = D / 4;   // lanes that hold a row, four columns each
    const int lane = threadIdx.x & 31, g = p.group, col = (lane % kRowLanes) * 4;
    for (int r0 = 0; r0 < g; r0 += 32 / kRowLanes) {
        const int r = r0 + lane / kRowLanes;
        const float ma = __shfl_sync(0xffffffffu, st.m0, r >> 1), mb = __shfl_sync(0xffffffffu, st.m1, r >> 1);
        const float la = __shfl_sync(0xffffffffu, st.l0, r >> 1), lb = __shfl_sync(0xffffffffu, st.l1, r >> 1);
        if (r < g) {
            const float4 x = lds_f4(src + (r * D + (col ^ ((r >> 1) * 8))) * 4);
            const float inv = 1.f / (r & 1 ? lb : la);
            const int head = kvh * g + r;
            *reinterpret_cast<uint2*>(p.out + ((int64_t)q_row * p.Hq + head) * D + col) =
                make_uint2(pack_bf16x2(x.x * inv, x.y * inv), pack_bf16x2(x.z * inv, x.w * inv));
            if (p.lse && col == 0) p.lse[(int64_t)q_row * p.Hq + head] = (r & 1 ? mb : ma) * p.sm_scale + __logf(r & 1 ? lb : la);
        }
    }
}

// Runs one unit; returns false if a bounded wait expired.  kAlone: of a launch without chunk rows, whose new rows are written here;
// with chunks they are written before.
template <int D, bool kAlone>
__device__ bool run_unit(const CUtensorMap* kvp_map, const MixedParams& p, const Unit& u, WarpRing<D>& ring, uint32_t smem,
                         int32_t* work, int fixed_items, bool pulls, bool resident, int& next_item) {
    constexpr int kStages = Geo<D>::kStages;
    const int lane = threadIdx.x & 31;
    const int g = p.group;

    uint32_t qb[D / 16][2];
    load_query<D>(p, u.q_row, u.kvh, qb);
    DecodeState<D> st;
    st.clear();

    const int pg0 = u.t_begin / kPageSize;
    const int pg1 = (u.t_end + kPageSize - 1) / kPageSize;
    const int npg = pg1 - pg0;

    int ids = 0;
    int issued = 0;
    bool append_timeout = false;
    const uint32_t it0 = ring.it;  // ring position of this unit's first page
    auto issue_next = [&]() {
        if ((issued & 31) == 0) {
            const int pi = pg0 + issued + lane;
            ids = pi < pg1 ? u.pages[pi] : 0;
        }
        int page = __shfl_sync(0xffffffffu, ids, issued & 31);
        if (page < 0 || (int64_t)page >= p.num_pages) {
            // a bad id never reaches the copy engine: the problem is reported and page 0 is fetched in its place, so
            // the barrier still receives the bytes it expects
            if (lane == 0) report(p.ctrl, SW_ERR_OUT_OF_RANGE, kSiteAttnPage, u.q_row);
            page = 0;
        }
        // the request's last page holds the row this iteration appends
        if (!kAlone && p.append_first && (pg0 + issued + 1) * kPageSize >= u.len && !wait_append(p, smem + Geo<D>::kSetOffset)) {
            if (lane == 0) report(p.ctrl, SW_ERR_DEVICE_TIMEOUT, kSiteWait, u.q_row);
            append_timeout = true;
        }
        issue_page<D>(kvp_map, ring, it0 + issued, page, u.kvh);
        ++issued;
    };
    for (int k = 0; k < kStages && k < npg; ++k) issue_next();
    // Once this unit's last page is on its way the following unit is claimed from the shared counter: the counter's
    // round trip hides behind the last pages, and no warp hoards a unit while others are still idle.
    // With the claim the unit draws its ticket among the units of its (request, kv head): the last ticket makes it
    // the one that merges.  Both answers are read at the end of the unit, when they have long arrived.
    // A request cut into many units (wide_merge_splits or more; g where every unit of the launch has a warp of its own, `resident`)
    // has g mergers per kv head, fixed in advance: its last g units, one query-head row each (units of one request and head are
    // Hkv apart in the order in which SMs take them, so the mergers sit on different SMs).  They claim their next unit after
    // the merge.  What they wait for: see rows_to_merge.
    const bool wide = g > 1 && u.nsplit >= (resident ? g : wide_merge_splits(D, g));
    const int merge_row = wide && u.nsplit - 1 - u.split < g ? u.nsplit - 1 - u.split : -1;
    if (wide && lane == 0) atomicAdd(&p.tickets[u.ticket], 1);   // started
    bool claimed = merge_row >= 0;
    int ticket = 0;  // lane 0
    auto claim_next = [&]() {
        if (!claimed && issued >= npg) {
            claimed = true;
            if (lane == 0) {
                next_item = pulls ? fixed_items + atomicAdd(work, 1) : 0x7fffffff;
                if (u.nsplit > 1 && !wide) ticket = atomicAdd(&p.tickets[u.ticket], 1);
            }
        }
    };
    claim_next();

    uint32_t sK = 0;
    for (int k = 0; k < npg; ++k) {
        if (append_timeout) return false;
        const uint32_t stage = ring.it % kStages;
        const uint32_t parity = (ring.it / kStages) & 1;
        sK = ring.buf + stage * Geo<D>::kStageBytes;
        const int valid = u.len - (pg0 + k) * kPageSize;   // keys of this page that are attended (16 or more: all)
        const bool patched = kAlone && p.append_last && valid <= kPageSize;
        uint4 row;
        if (patched) row = load_new_row<D>(p, u.q_row, u.kvh);   // (no chunk rows: q_row is the request)
        if (!mbar_wait(ring.bar + stage * 8, parity)) {
            report(p.ctrl, SW_ERR_DEVICE_TIMEOUT, kSiteWait, u.q_row);
            return false;
        }
        if (patched) {
            if (!mbar_wait(smem + Geo<D>::kLastBarOffset, 0)) {
                report(p.ctrl, SW_ERR_DEVICE_TIMEOUT, kSiteWait, u.q_row);
                return false;
            }
            __syncwarp();
            patch_page<D>(p, smem, sK, u.q_row, u.kvh, valid, row);
        }

        attend_page<D>(p, sK, valid, qb, st);
        ring.it += 1;
        __syncwarp();  // every lane is done reading this stage before it is refilled
        if (issued < npg) issue_next();
        claim_next();
    }

    stage_result<D>(sK, g, st);
    constexpr int kRowLanes = D / 4;   // lanes that hold a row, four columns each
    const int col = (lane % kRowLanes) * 4;
    if (u.nsplit == 1) {
        write_rows<D>(p, sK, u.q_row, u.kvh, st);
        fence_proxy_async_smem();  // the buffer was written with plain stores and is refilled by the copy engine
        __syncwarp();
        return true;
    }

    // Partial result -> scratch.  The units that did not draw the last ticket publish it (fence, then one more on the
    // `ready` counter, without waiting for anything); the one that did waits until the others have and merges.  It is
    // usually the last to finish, so its wait is short, and no fence or ticket round trip sits between its last page
    // and the merge.
    for (int r = lane / kRowLanes; r < g; r += 32 / kRowLanes)
        *reinterpret_cast<float4*>(p.part_o + ((int64_t)u.slot * g + r) * D + col) = lds_f4(sK + (r * D + (col ^ ((r >> 1) * 8))) * 4);
    if (lane < 4) {
        float* ml = p.part_ml + (int64_t)u.slot * (2 * kMaxGroup) + lane * 2;
        if (lane * 2 < g) ml[0] = st.m0, ml[kMaxGroup] = st.l0;
        if (lane * 2 + 1 < g) ml[1] = st.m1, ml[kMaxGroup + 1] = st.l1;
    }
    fence_proxy_async_smem();  // the buffer was written with plain stores and is refilled by the copy engine
    __syncwarp();
    if (wide) {
        // Many splits (one long context cut for all the warps): a single warp would load their partial outputs a few
        // at a time.  Every unit publishes its partial result; g of the request's last units then merge one row of
        // the group each.  The last merger to finish re-arms the counters.
        __threadfence();
        __syncwarp();
        int rows = 0;
        if (lane == 0) rows = rows_to_merge(&p.ready[u.ticket], &p.tickets[u.ticket], u.nsplit, merge_row);
        rows = __shfl_sync(0xffffffffu, rows, 0);
        if (rows < 0) {
            if (lane == 0) report(p.ctrl, SW_ERR_DEVICE_TIMEOUT, kSiteWait, u.q_row);
            return false;
        }
        const int merged = __popc(rows);
        for (; rows != 0; rows &= rows - 1) merge_splits<D, 1>(p, u, __ffs(rows) - 1, 1);
        if (lane == 0) {
            if (merged > 0 && (atomicAdd(&p.ready[u.ticket], merged) & kPublished) + merged == u.nsplit + g) {
                p.ready[u.ticket] = 0;      // ready for the next launch
                p.tickets[u.ticket] = 0;
            }
            if (merge_row >= 0) next_item = pulls ? fixed_items + atomicAdd(work, 1) : 0x7fffffff;
        }
        return true;
    }
    ticket = __shfl_sync(0xffffffffu, ticket, 0);
    const bool merger = ticket == u.nsplit - 1;
    if (!merger) {
        __threadfence();
        __syncwarp();
        if (lane == 0) atomicAdd(&p.ready[u.ticket], 1);
        return true;
    }
    // last ticket: merge all splits of this (request, kv head) once the others are published
    __syncwarp();  // this warp's own partial result, written above by all lanes, is ordered before the loads below
    int ok = 1;
    if (lane == 0) {
        const long long t0 = clock64();
        while (ld_acquire_gpu(&p.ready[u.ticket]) < u.nsplit - 1) {
            if (clock64() - t0 > kWaitBudgetCycles) {
                ok = 0;
                break;
            }
            __nanosleep(64);
        }
        p.tickets[u.ticket] = 0;  // ready for the next launch
        p.ready[u.ticket] = 0;
    }
    ok = __shfl_sync(0xffffffffu, ok, 0);
    if (!ok) {
        if (lane == 0) report(p.ctrl, SW_ERR_DEVICE_TIMEOUT, kSiteWait, u.q_row);
        return false;
    }
    switch (g) {
        case 1: merge_splits<D, 1>(p, u, 0, 1); break;
        case 2: merge_splits<D, 2>(p, u, 0, 2); break;
        case 4: merge_splits<D, 4>(p, u, 0, 4); break;
        default: merge_splits<D, kMaxGroup>(p, u, 0, g); break;
    }
    return true;
}

// The requests' last pages, which fused decode-only launches write, by id; whole CTA.  Only warps with a request wait for the load.
template <int D>
__device__ __forceinline__ void list_last_pages(const MixedParams& p, const int* lens, const int* indptr, uint32_t smem, unsigned* sets) {
    for (int i = threadIdx.x; i < p.n; i += kThreads) {
        const int len = lens[i], pi = (len - 1) / kPageSize;
        int id = -1;
        if (len < 1 || pi >= indptr[i + 1] - indptr[i]) {
            if (blockIdx.x == 0) report(p.ctrl, SW_ERR_OUT_OF_RANGE, kSiteAppendLen, i);
        } else {
            id = p.decode_pages[indptr[i] + pi];
            if (id < 0 || (int64_t)id >= p.num_pages) {
                if (blockIdx.x == 0) report(p.ctrl, SW_ERR_OUT_OF_RANGE, kSiteAppendPage, i);
                id = -1;
            }
        }
        sts_s32(smem + Geo<D>::kLastOffset + i * 4, id);
        // first request in its bucket: marked in the first set; any other: the bucket is marked in the second
        const unsigned h = page_hash(id), bit = 1u << (h & 31);
        if (atomicOr(&sets[h / 32], bit) & bit) atomicOr(&sets[(kPageHashBits + h) / 32], bit);
    }
    __syncwarp();
    if ((threadIdx.x & 31) == 0) mbar_arrive(smem + Geo<D>::kLastBarOffset);
}

// The line of stages (see line_form): CTA `cta` of line.ctas streams its stretch and merges.
//
// Position x of the line is page x % stages, in the order of the requests, of KV head x / stages.  CTA c has [c T / C, (c + 1) T / C) of the T
// stages, its warp w the same share of those.  (Lines of 2^23 stages and more are shared out in steps of 2^shift stages, so that
// positions times CTAs fit 32 bits.  This arithmetic stands in a chain of instructions that are executed once, and fetched for it: with
// shares that need no product, and 64-bit divisions, one 8192-token context took 16.6 us instead of 15.1.)
//
// Page copies run ahead of the (request, KV head) pair that is being worked on.  A pair that begins and ends in the warp is finished
// by it (all are where none is cut: line.whole).  Any other leaves a partial result in shared memory, in the warp's first page buffer if
// it is the last thing the warp does and in the plan's unused space otherwise; when all warps are done, warps merge the pairs row by
// row.  A pair that goes on beyond the CTA is published (slots of a pair's CTAs follow one another) and merged by the CTA that publishes
// last, so nobody waits for another CTA.  If a wait expires, the warp ends (its own copies awaited) and the CTA merges and publishes
// nothing: the launch is reported, and the pairs that it did not finish keep what their rows held before.
template <int D>
__device__ __forceinline__ void run_line(const CUtensorMap* kvp_map, const MixedParams& p, const Line& line, int* scratch,
                                         unsigned* sets, uint32_t smem, int cta) {
    constexpr int kStages = Geo<D>::kStages, V = D / 32;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int g = p.group, C = line.ctas;
    auto cta_begin = [&](int c) { return min(line.total, c * line.coarse / C << line.shift); };
    auto cta_of = [&](int x) { return (((x >> line.shift) + 1) * C - 1) / line.coarse; };
    const int X0 = cta_begin(min(cta, C)), X1 = cta_begin(min(cta + 1, C));
    const unsigned L = X1 - X0;
    auto warp_begin = [&](int w) { return X0 + (int)(w * L / kWarps); };
    const int* prefix = line.prefix;
    auto ring_of = [&](int w) { return smem + w * kStages * Geo<D>::kStageBytes; };
    auto stash_of = [&](int w) {   // array w / 3 of the plan, behind its first kLineMaxDecode + 1 words
        const int at = w < 6 ? (w < 3 ? Geo<D>::kPlanOffset : Geo<D>::kLenOffset) : (w < 9 ? Geo<D>::kIndptrOffset : Geo<D>::kLastOffset);
        return smem + ((at + 15) & ~15) + kLineArrayBytes + (w % kStashesPerArray) * kStashBytes;
    };
    // (head, request, page) of a position
    auto locate = [&](int x, int& kvh, int& i) {
        kvh = x / line.stages;
        const int rem = x - kvh * line.stages;
        int lo = 0, hi = p.n;  // largest i with prefix[i] <= rem
        while (hi - lo > 1) {
            const int mid = (lo + hi) >> 1;
            if (prefix[mid] <= rem) lo = mid; else hi = mid;
        }
        i = lo;
        return rem - prefix[lo];
    };
    int* table = scratch + kLineTable;   // pairs that are merged; their number behind them
    WarpRing<D> ring;
    ring.buf = ring_of(warp);
    ring.bar = smem + Geo<D>::kBarOffset + warp * kStages * 8;
    ring.it = 0;
    int x0 = warp_begin(warp), x1 = warp_begin(warp + 1);
    if (line.whole) {
        int x = lane == 0 ? x0 : x1, kvh, i;
        if (x < line.total) {
            const int page = locate(x, kvh, i), pages = prefix[i + 1] - prefix[i];
            x += 2 * page < pages ? -page : pages - page;
        }
        x0 = __shfl_sync(0xffffffffu, x, 0);
        x1 = __shfl_sync(0xffffffffu, x, 1);
    }
    const int total = x1 - x0;
    int id = 0, head = 0, issued = 0;   // lane l: page id and KV head of stage x0 + 32 n + l
    auto issue_next = [&]() {
        if ((issued & 31) == 0) {
            const int x = x0 + issued + lane;
            id = 0;
            if (x < x1) {
                int i;
                const int page = locate(x, head, i);
                id = p.decode_pages[line.indptr[i] + page];
                if (id < 0 || (int64_t)id >= p.num_pages) {   // never reaches the copy engine
                    report(p.ctrl, SW_ERR_OUT_OF_RANGE, kSiteAttnPage, p.C + i);
                    id = 0;
                }
            }
        }
        issue_page<D>(kvp_map, ring, issued, __shfl_sync(0xffffffffu, id, issued & 31), __shfl_sync(0xffffffffu, head, issued & 31));
        ++issued;
    };
    for (int k = 0; k < kStages && k < total; ++k) issue_next();
    if (p.append_last) list_last_pages<D>(p, line.len, line.indptr, smem, sets);   // after the first copies are on their way
    bool expired = false;
    auto wait = [&](uint32_t bar, uint32_t parity) {
        return mbar_test_wait(bar, parity) || (p.line_wait_cycles > 0 && mbar_wait(bar, parity, p.line_wait_cycles));
    };
#pragma unroll 1
    for (int x = x0; x < x1;) {
        int kvh, i;
        const int page = locate(x, kvh, i), pages = prefix[i + 1] - prefix[i];
        const int a = x - page, b = a + pages, end = min(b, x1);   // the pair's stretch of the line; where the warp's part of it ends
        const bool alone = a >= x0 && b <= x1;
        uint32_t qb[D / 16][2];
        load_query<D>(p, p.C + i, kvh, qb);
        DecodeState<D> st;
        st.clear();
        uint32_t sK = 0;
        int valid = line.len[i] - page * kPageSize;   // keys from the page on
#pragma unroll 1
        for (; x < end; ++x, valid -= kPageSize) {
            const uint32_t stage = ring.it % kStages, parity = (ring.it / kStages) & 1;
            sK = ring.buf + stage * Geo<D>::kStageBytes;
            const bool patched = p.append_last && valid <= kPageSize;
            uint4 row;
            if (patched) row = load_new_row<D>(p, i, kvh);
            expired = !wait(ring.bar + stage * 8, parity) || (patched && !wait(smem + Geo<D>::kLastBarOffset, 0));
            if (__any_sync(0xffffffffu, expired)) {
                expired = true;
                break;
            }
            if (patched) patch_page<D>(p, smem, sK, i, kvh, valid, row);
            attend_page<D>(p, sK, valid, qb, st);
            ring.it += 1;
            __syncwarp();  // every lane is done reading this stage before it is refilled
            if (x + 1 < end && issued < total) issue_next();
        }
        if (expired) {
            report(p.ctrl, SW_ERR_DEVICE_TIMEOUT, kSiteWait, p.C + i);
#pragma unroll 1
            for (; ring.it < (uint32_t)issued; ++ring.it) mbar_wait(ring.bar + ring.it % kStages * 8, (ring.it / kStages) & 1);
            break;
        }
        const uint32_t keep = alone ? sK : (end == x1 ? ring.buf : stash_of(warp));
        stage_result<D>(keep, g, st);
        if (alone) {
            write_rows<D>(p, keep, p.C + i, kvh, st);
        } else {
            if (lane < 4) {   // m and l of the group behind O
                sts_f32(keep + (g * D + 2 * lane) * 4, st.m0);
                sts_f32(keep + (g * D + 2 * lane + 1) * 4, st.m1);
                sts_f32(keep + (g * D + kMaxGroup + 2 * lane) * 4, st.l0);
                sts_f32(keep + (g * D + kMaxGroup + 2 * lane + 1) * 4, st.l1);
            }
            if (lane == 0 && max(a, x0) == max(a, X0)) {   // the pair's first warp in this CTA
                const int lb = min(b, X1), wb = ((lb - X0) * kWarps - 1u) / L, ca = cta_of(a), cb = cta_of(b - 1);
                int* e = table + atomicAdd(table + kLineGroups * kLineWords, 1) * kLineWords;
                e[0] = i * p.Hkv + kvh;
                e[1] = warp | wb << 8 | (lb == warp_begin(wb + 1) ? 1 << 16 : 0);
                e[2] = ca;
                e[3] = cb - ca + 1;
            }
        }
        // The pair's last page buffer was written with plain stores (the new row, zeroed rows of V, the result), wherever the result
        // went, and is refilled by the copy engine.
        fence_proxy_async_smem();
        __syncwarp();
        if (issued < total) issue_next();
    }
    if (__syncthreads_or(expired)) return;
    const int lg = 31 - __clz(g), tasks = *reinterpret_cast<volatile int*>(table + kLineGroups * kLineWords) << lg;
    bool beyond = false;   // some pair goes on in another CTA
#pragma unroll 1
    for (int t = lane; t < tasks; t += 32) beyond |= table[(t >> lg) * kLineWords + 3] > 1;
    beyond = __any_sync(0xffffffffu, beyond);
    auto finish_row = [&](int pair, int row, float m, float l, const float (&acc)[V]) {
        const int i = pair / p.Hkv, kvh = pair - i * p.Hkv;
        const float inv = 1.f / l;
        const int64_t out_row = (int64_t)(p.C + i) * p.Hq + kvh * g + row;
        uint32_t* dst = reinterpret_cast<uint32_t*>(p.out + out_row * D + lane * V);
#pragma unroll
        for (int v = 0; v < V; v += 2) dst[v / 2] = pack_bf16x2(acc[v] * inv, acc[v + 1] * inv);
        if (p.lse && lane == 0) p.lse[out_row] = m * p.sm_scale + __logf(l);
    };
#pragma unroll 1
    for (int t = warp; t < tasks; t += kWarps) {
        const int* e = table + (t >> lg) * kLineWords;
        const int pair = e[0], row = t & (g - 1), wa = e[1] & 0xff, wb = e[1] >> 8 & 0xff;
        const int w = min(wa + lane, wb);
        const bool live = wa + lane <= wb && warp_begin(w) < warp_begin(w + 1);
        const uint32_t at = w < wb || (e[1] >> 16) != 0 ? ring_of(w) : stash_of(w);
        const float ms = live ? lds_f32(at + (g * D + row) * 4) : -INFINITY;
        float mw = ms, lw = live ? lds_f32(at + (g * D + kMaxGroup + row) * 4) : 0.f;
#pragma unroll
        for (int o = 8; o > 0; o >>= 1) mw = fmaxf(mw, __shfl_xor_sync(0xffffffffu, mw, o));   // (kWarps <= 16)
        const float wgt = ms == -INFINITY ? 0.f : fast_exp2((ms - mw) * p.sm_scale_log2);
        lw *= wgt;
#pragma unroll
        for (int o = 8; o > 0; o >>= 1) lw += __shfl_xor_sync(0xffffffffu, lw, o);
        mw = __shfl_sync(0xffffffffu, mw, 0);
        lw = __shfl_sync(0xffffffffu, lw, 0);
        float acc[V];
#pragma unroll
        for (int v = 0; v < V; ++v) acc[v] = 0.f;
        const uint32_t col = (row * D + ((lane * V) ^ ((row >> 1) * 8))) * 4;
#pragma unroll 2
        for (int j = 0; j <= wb - wa; ++j) {
            const float wj = __shfl_sync(0xffffffffu, wgt, j);
            const uint32_t src = __shfl_sync(0xffffffffu, at, j) + col;
            if (wj == 0.f) continue;   // (warps without a stage among them: their buffers hold anything)
#pragma unroll
            for (int v = 0; v < V; v += 2) {
                const float2 y = lds_f2(src + v * 4);
                acc[v] = fmaf(wj, y.x, acc[v]);
                acc[v + 1] = fmaf(wj, y.y, acc[v + 1]);
            }
        }
        if (e[3] == 1) {
            finish_row(pair, row, mw, lw, acc);
        } else {
            const int slot = cta + (pair % p.Hkv) * p.n + pair / p.Hkv;
            float2* dst = reinterpret_cast<float2*>(p.part_o + ((int64_t)slot * g + row) * D + lane * V);
#pragma unroll
            for (int v = 0; v < V; v += 2) dst[v / 2] = make_float2(acc[v], acc[v + 1]);
            if (lane == 0) {
                p.part_ml[(int64_t)slot * (2 * kMaxGroup) + row] = mw;
                p.part_ml[(int64_t)slot * (2 * kMaxGroup) + kMaxGroup + row] = lw;
            }
        }
    }
    if (!beyond) return;
    __syncthreads();
    if (threadIdx.x < kLineGroups && threadIdx.x << lg < tasks) {
        int* e = table + threadIdx.x * kLineWords;
        if (e[3] > 1) {
            __threadfence();
            const bool last = atomicAdd(&p.tickets[e[0]], 1) == e[3] - 1;
            if (last) p.tickets[e[0]] = 0;   // ready for the next launch
            __threadfence();
            e[1] = last;
        }
    }
    __syncthreads();
#pragma unroll 1
    for (int t = warp; t < tasks; t += kWarps) {
        const int* e = table + (t >> lg) * kLineWords;
        if (e[3] == 1 || e[1] == 0) continue;
        const int pair = e[0], row = t & (g - 1), ns = e[3], slot0 = e[2] + (pair % p.Hkv) * p.n + pair / p.Hkv;
        const float* ml = p.part_ml + (int64_t)slot0 * (2 * kMaxGroup) + row;
        const float2* po = reinterpret_cast<const float2*>(p.part_o + ((int64_t)slot0 * g + row) * D + lane * V);
        float m = -INFINITY, l = 0.f, acc[V];
#pragma unroll
        for (int v = 0; v < V; ++v) acc[v] = 0.f;
        // 32 partial results at a time, lane j holding m and l of the j-th; eight of O in flight
#pragma unroll 1
        for (int s0 = 0; s0 < ns; s0 += 32) {
            const int here = min(32, ns - s0);
            const float ms = lane < here ? __ldcg(ml + (s0 + lane) * (2 * kMaxGroup)) : -INFINITY;
            const float ls = lane < here ? __ldcg(ml + (s0 + lane) * (2 * kMaxGroup) + kMaxGroup) : 0.f;
            float wgt = 0.f;
#pragma unroll 1
            for (int j0 = 0; j0 < here; j0 += 8) {
                float2 y[8][V / 2];
#pragma unroll
                for (int j = 0; j < 8; ++j)
#pragma unroll
                    for (int v = 0; v < V / 2; ++v) y[j][v] = __ldcg(po + (int64_t)(s0 + min(j0 + j, here - 1)) * (g * D / 2) + v);
                if (j0 == 0) {
                    float mw = fmaxf(m, ms);
#pragma unroll
                    for (int o = 16; o > 0; o >>= 1) mw = fmaxf(mw, __shfl_xor_sync(0xffffffffu, mw, o));
                    wgt = ms == -INFINITY ? 0.f : fast_exp2((ms - mw) * p.sm_scale_log2);
                    float lw = wgt * ls;
#pragma unroll
                    for (int o = 16; o > 0; o >>= 1) lw += __shfl_xor_sync(0xffffffffu, lw, o);
                    const float f = m == -INFINITY ? 0.f : fast_exp2((m - mw) * p.sm_scale_log2);
                    l = l * f + lw;
                    m = mw;
#pragma unroll
                    for (int v = 0; v < V; ++v) acc[v] *= f;
                }
#pragma unroll
                for (int j = 0; j < 8; ++j) {
                    const float wj = j0 + j < here ? __shfl_sync(0xffffffffu, wgt, j0 + j) : 0.f;
#pragma unroll
                    for (int v = 0; v < V; v += 2) {
                        acc[v] = fmaf(wj, y[j][v / 2].x, acc[v]);
                        acc[v + 1] = fmaf(wj, y[j][v / 2].y, acc[v + 1]);
                    }
                }
            }
        }
        finish_row(pair, row, m, l, acc);
    }
}

}  // namespace sw
#include "sw_prefill.cuh"
namespace sw {

// ---------------------------------------------------------------------------------------------------------------
// the persistent kernel
// ---------------------------------------------------------------------------------------------------------------
// Forms of the kernel, chosen by the host: iterations with one prefill chunk, whose descriptors are then plain kernel parameters; with
// several (descriptors looked up per work item); without any, where the decodes may be worked off as a line (line_form), and the others.
// A form has only the code that it needs: with the line's code in the kernel of one chunk, the small mixed launch of 8/2/64 took 13.6 us
// and 64 contexts beside 512 tokens 63.7, with kernels of their own 13.2 and 62.5; 20 contexts of 8/1/128, worked off as units, take
// 16.8 us in a kernel of their own and 21.6 beside the line's code (18.3 with all in one).
enum Form { kOneChunk, kSeveralChunks, kLine, kUnits };
template <int D, Form kForm>
__global__ void __launch_bounds__(kThreads, 1) sw_mixed_attn_kernel(const __grid_constant__ CUtensorMap kv_map,
                                                                       const __grid_constant__ CUtensorMap kvp_map,
                                                                    const __grid_constant__ CUtensorMap q_map,
                                                                    const __grid_constant__ CUtensorMap out_map,
                                                                    const MixedParams p) {
    static_assert(PfGeo<D>::kBytes <= Geo<D>::kRingBytes, "prefill tiles must fit the region shared with the decode ring");
    extern __shared__ uint8_t smem_raw[];
    const uint32_t raw = smem_u32(smem_raw);
    const uint32_t base = (raw + 1023u) & ~1023u;
    uint8_t* smem = smem_raw + (base - raw);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;

    int* unit_prefix = reinterpret_cast<int*>(smem + Geo<D>::kPlanOffset);
    int* scratch = reinterpret_cast<int*>(smem + Geo<D>::kMiscOffset);

    constexpr bool kMulti = kForm == kSeveralChunks, tensor_prefill = kMulti || kForm == kOneChunk;
    unsigned* sets = reinterpret_cast<unsigned*>(smem + Geo<D>::kSharedOffset);   // of hashed last pages
    volatile int* misc = reinterpret_cast<volatile int*>(scratch + kMiscAt);
    if (threadIdx.x >= 32 && threadIdx.x < 32 + kPlanCounters) scratch[64 + threadIdx.x - 32] = 0;  // block-sum counters
    if (threadIdx.x < kWarps * Geo<D>::kStages) {
        mbar_init(base + Geo<D>::kBarOffset + threadIdx.x * 8, 1);
        fence_mbar_init();
    }
    if (threadIdx.x >= 128 && threadIdx.x < 128 + 2 * kPageHashBits / 32)
        sets[threadIdx.x - 128] = 0;
    if (threadIdx.x == 96) {
        tma_prefetch_desc(&kvp_map);
        mbar_init(base + Geo<D>::kLastBarOffset, kWarps);
        if constexpr (tensor_prefill) {
            tma_prefetch_desc(&kv_map);
            tma_prefetch_desc(&q_map);
            tma_prefetch_desc(&out_map);
            pf_init_barriers(base + Geo<D>::kPfBarOffset);
        }
        misc[kMiscTmem] = 0;
        misc[kMiscAbort] = 0;
        misc[kMiscNoUnits] = 0;
        fence_mbar_init();
    }
    // The plan of the chunk-prefill phase and, with several chunks, their descriptors go to shared memory: the roles look them
    // up instead of carrying them in registers.  It depends on the decode page count, which an earlier kernel may have written,
    // so it is made after the wait below; the table of several chunks (a microsecond) is filled here for the usual case, that
    // every CTA takes entries, and filled again after the wait where that turns out otherwise.
    if constexpr (kMulti) {
        if (warp == 2) pf_fill_chunk_table(p, scratch + kChunkTable, (int)gridDim.x);
    }
    // Everything above touched only shared memory and kernel parameters.  From here on the kernel reads what earlier
    // kernels of the stream wrote (the pool after the KV append, q, the page tables): wait for them to finish.
    grid_dependency_wait();
    grid_launch_dependents();
    // Counters come in two sets that launches use in turn, so that no CTA has to wait at its end to find out whether it is
    // the last one: every CTA counts itself once when it ends (modulo two grids), hence a launch that reads between 0 and
    // grid - 1 uses set 0, one that reads more uses set 1, and it clears the other one for the launch after it.
    const int set = ld_relaxed_gpu(&p.ctrl[kCtrArrived]) >= (int)gridDim.x ? 1 : 0;
    int32_t* counters = p.ctrl + kCtrSets + set * kSetWords;
    if (threadIdx.x == 0) misc[kMiscSet] = kCtrSets + set * kSetWords;
    if (blockIdx.x == 0 && threadIdx.x < kSetWords) p.ctrl[kCtrSets + (set ^ 1) * kSetWords + threadIdx.x] = 0;
    if (tensor_prefill && warp == 2) {
        if constexpr (kMulti) {
            __syncwarp();
            const int ctas = pf_table_ctas(p, scratch + kChunkTable);
            __syncwarp();
            if (ctas != (int)gridDim.x) pf_fill_chunk_table(p, scratch + kChunkTable, ctas);
        } else {
            pf_fill_plan(p, scratch + kChunkTable);
        }
        __syncwarp();
    }
    if (tensor_prefill && p.append_first) {
        // fused launch with chunks: this CTA's share of the new K/V rows (the planning warp has none), then its mark on the
        // counter the readers wait for
        if (warp != 2)
            append_rows<kMulti, kAppendBatch>(p, D, (int)blockIdx.x * (kWarps - 1) + warp - (warp > 2), (int)gridDim.x * (kWarps - 1));
        fence_proxy_async_global();
        __threadfence();
        __syncthreads();
        if (threadIdx.x == 0) atomicAdd(&counters[kSetAppend], 1);
    }
    __syncthreads();

    // chunk-prefill tiles first (long, tensor-bound); the decode units below fill the tail
    // The first prefill entry of a CTA is its own index and the first decode unit of a warp is fixed as well: neither
    // waits for a counter.  CTAs that start with prefill work take all their decode units from the counter.
    int prefill_ctas = 0;
    LateJoin late{0, 0.f};
    if constexpr (tensor_prefill) {
        const PfPlan pplan = pf_make_plan(base + Geo<D>::kMiscOffset + kChunkTable * 4);
        prefill_ctas = min(pplan.n_entries, pplan.ctas);
        late.ctas = prefill_ctas;
        late.us = kLateBaseUs + p.step_us * ((pplan.longest + pplan.pieces - 1) / pplan.pieces);
        if (pplan.n_items >= pplan.ctas)  // whole rounds: the prefill CTAs share all items' steps
            late.us = kLateBaseUs + p.step_us * (0.5f * (float)(pplan.longest + pplan.shortest) * (float)pplan.n_items / (float)pplan.ctas);
        if (kMulti && pplan.end_steps > 0) late.us = kLateBaseUs + p.step_us * (float)pplan.end_steps;
        const int first_entry = blockIdx.x;
        if (first_entry < prefill_ctas) {  // CTA-uniform: this CTA has prefill work
            if (warp == 1) {
                tmem_alloc(smem_u32(const_cast<int*>(&misc[kMiscTmem])), 512);
                tmem_relinquish();
            }
            tc_fence_before_sync();
            __syncthreads();
            tc_fence_after_sync();
            PfShared sh;
            sh.smem = base;
            sh.bars = base + Geo<D>::kPfBarOffset;
            sh.tmem = (uint32_t)misc[kMiscTmem];
            sh.abort_flag = &misc[kMiscAbort];
            PfScratch scr;
            scr.ml = p.pf_ml;
            scr.o = p.pf_o;
            scr.tickets = p.pf_tickets;
            scr.flags = &misc[kMiscFlags];
            prefill_phase<D, kMulti>(&kv_map, &q_map, &out_map, p, sh, pplan, scr, first_entry, &misc[kMiscNext]);
            tc_fence_before_sync();
            __syncthreads();
            if (warp == 1) tmem_dealloc(sh.tmem, 512);
        }
        __syncthreads();
    }
    if (p.n == 0 || misc[kMiscNoUnits]) {   // no decode units, or none left for this CTA
        if (threadIdx.x == 0) atomicInc(reinterpret_cast<unsigned*>(&p.ctrl[kCtrArrived]), 2 * gridDim.x - 1);
        return;
    }

    int* lens = reinterpret_cast<int*>(smem + Geo<D>::kLenOffset);
    int* indptr = reinterpret_cast<int*>(smem + Geo<D>::kIndptrOffset);
    if constexpr (kForm == kLine) {
        const Line line = make_line<D>(p, unit_prefix, lens, indptr, scratch);
        run_line<D>(&kvp_map, p, line, scratch, sets, base, (int)blockIdx.x);
        if (threadIdx.x == 0) atomicInc(reinterpret_cast<unsigned*>(&p.ctrl[kCtrArrived]), 2 * gridDim.x - 1);
        return;
    }
    const Plan plan = make_plan(p, unit_prefix, lens, indptr, scratch, late, p.stages_per_us);
    if ((int)blockIdx.x == prefill_ctas && threadIdx.x == 0) atomicExch(p.ctrl + misc[kMiscSet] + kSetItems, plan.total_items + 1);
    if (plan.total_items > p.max_items) {
        if (threadIdx.x == 0) report(p.ctrl, SW_ERR_WORKSPACE, kSiteScratch, plan.total_items);
    } else {
        if (!tensor_prefill && p.append_last) list_last_pages<D>(p, plan.len, plan.indptr, base, sets);
        int32_t* work = p.ctrl + lds_s32(base + Geo<D>::kSetOffset) + kSetWork;
        WarpRing<D> ring;
        ring.buf = base + warp * Geo<D>::kStages * Geo<D>::kStageBytes;
        ring.bar = base + Geo<D>::kBarOffset + warp * Geo<D>::kStages * 8;
        ring.it = 0;
        const int fixed_items = ((int)gridDim.x - prefill_ctas) * kWarps;  // units handed out without the counter
        const bool resident = plan.total_items <= fixed_items;   // every unit has a warp of its own in a CTA that starts with units
        // With two unit sizes the early CTAs run their one large unit each and leave the counter to the late CTAs; where every unit
        // has a warp of its own the counter has none to give (asking it costs a merger 0.7 us at its end).
        const bool pulls = !resident && (!plan.two_sizes || (int)blockIdx.x < prefill_ctas);
        // neighbouring units go to different SMs: a batch with fewer units than warps is spread over all of them
        int item = warp * ((int)gridDim.x - prefill_ctas) + (int)blockIdx.x - prefill_ctas;
        if ((int)blockIdx.x < prefill_ctas) {
            if (lane == 0) item = fixed_items + atomicAdd(work, 1);
            item = __shfl_sync(0xffffffffu, item, 0);
        }
        while (item < plan.total_items) {
            int next_item = 0;  // lane 0: claimed inside run_unit
            Unit u;
            bool ok = true;
            {
                const int di = item;
                const int unit = di / p.Hkv;
                u.kvh = di % p.Hkv;
                int lo = 0, hi = p.n;  // largest i with unit_prefix[i] <= unit
                while (hi - lo > 1) {
                    const int mid = (lo + hi) >> 1;
                    if (unit_prefix[mid] <= unit) lo = mid; else hi = mid;
                }
                const int i = lo;
                u.q_row = p.C + i;
                u.len = plan.len[i];
                u.split = unit - unit_prefix[i];
                u.nsplit = unit_prefix[i + 1] - unit_prefix[i];
                // the request's pages are shared out evenly among its units (no ragged last unit)
                const int req_pages = (u.len + kPageSize - 1) / kPageSize;
                const int unit_pages = (req_pages + u.nsplit - 1) / u.nsplit;
                u.t_begin = min(u.len, u.split * unit_pages * kPageSize);
                u.t_end = min(u.len, u.t_begin + unit_pages * kPageSize);
                u.ticket = i * p.Hkv + u.kvh;
                u.slot = di;
                const int beg = plan.indptr[i];
                u.pages = p.decode_pages + beg;
                ok = (u.len + kPageSize - 1) / kPageSize <= plan.indptr[i + 1] - beg;
            }
            if (!ok) {
                if (lane == 0) {
                    report(p.ctrl, SW_ERR_OUT_OF_RANGE, kSiteAttnLen, u.q_row);
                    next_item = pulls ? fixed_items + atomicAdd(work, 1) : 0x7fffffff;
                }
            } else if (!run_unit<D, !tensor_prefill>(&kvp_map, p, u, ring, base, work, fixed_items, pulls, resident, next_item)) {
                break;
            }
            item = __shfl_sync(0xffffffffu, next_item, 0);
        }
    }

    __syncthreads();
    if (threadIdx.x == 0) atomicInc(reinterpret_cast<unsigned*>(&p.ctrl[kCtrArrived]), 2 * gridDim.x - 1);
}

// Self-test of the bounded wait: one warp waits on a barrier that nothing will ever complete; the wait must give up
// after `budget_cycles`, record SW_ERR_DEVICE_TIMEOUT in the status word and let the kernel end normally.
__global__ void sw_selftest_wait_kernel(int32_t* ctrl, long long budget_cycles) {
    __shared__ __align__(8) unsigned long long bar;
    const uint32_t addr = smem_u32(&bar);
    if (threadIdx.x == 0) {
        mbar_init(addr, 1);
        fence_mbar_init();
    }
    __syncwarp();
    if (!mbar_wait(addr, 0, budget_cycles) && threadIdx.x == 0) report(ctrl, SW_ERR_DEVICE_TIMEOUT, kSiteWait, 0xABCD);
}

cudaError_t launch_selftest_wait(int32_t* ctrl, long long budget_cycles, cudaStream_t stream) {
    sw_selftest_wait_kernel<<<1, 32, 0, stream>>>(ctrl, budget_cycles);
    return cudaGetLastError();
}

// 226.7 KB at head size 128, 288 bytes below what a CTA may have
static_assert(Geo<128>::kSmemBytes + 1024 <= 227 * 1024 && Geo<64>::kSmemBytes + 1024 <= 227 * 1024, "shared memory of a CTA");
size_t mixed_attn_smem_bytes(int head_dim) {
    return (head_dim == 64 ? Geo<64>::kSmemBytes : Geo<128>::kSmemBytes) + 1024;
}

template <int D, class F>
cudaError_t for_each_form(F f) {
    cudaError_t e = f(sw_mixed_attn_kernel<D, kOneChunk>);
    if (e == cudaSuccess) e = f(sw_mixed_attn_kernel<D, kSeveralChunks>);
    if (e == cudaSuccess) e = f(sw_mixed_attn_kernel<D, kLine>);
    return e == cudaSuccess ? f(sw_mixed_attn_kernel<D, kUnits>) : e;
}
template <class F>
cudaError_t for_each_form(int head_dim, F f) { return head_dim == 64 ? for_each_form<64>(f) : for_each_form<128>(f); }
cudaError_t configure_kernels(int head_dim) {
    const int bytes = (int)mixed_attn_smem_bytes(head_dim);
    return for_each_form(head_dim, [&](auto* kernel) { return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes); });
}

// CTAs of the persistent kernel that one SM can hold at a time (the smallest figure of all forms).  The fused launch
// makes CTAs wait for one another's share of the KV append, which is only safe when the whole grid is resident.
cudaError_t mixed_attn_resident_ctas_per_sm(int head_dim, int* out) {
    const size_t bytes = mixed_attn_smem_bytes(head_dim);
    *out = 1 << 30;
    return for_each_form(head_dim, [&](auto* kernel) {
        int n = 0;
        const cudaError_t e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, kernel, kThreads, bytes);
        *out = n < *out ? n : *out;
        return e;
    });
}

cudaError_t launch_mixed_attn(int head_dim, const KvMaps& kv_maps, const CUtensorMap& q_map, const CUtensorMap& out_map,
                              const MixedParams& p,
                              int num_sms, cudaStream_t stream) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)num_sms);
    cfg.blockDim = dim3(kThreads);
    cfg.dynamicSmemBytes = mixed_attn_smem_bytes(head_dim);
    cfg.stream = stream;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;  // prologue overlaps the previous kernel's tail
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    auto launch = [&](auto* kernel) { return cudaLaunchKernelEx(&cfg, kernel, kv_maps.half, kv_maps.page, q_map, out_map, p); };
    auto form = [&](auto* one, auto* several, auto* line, auto* units) {
        return p.nchunks > 1 ? launch(several) : (p.nchunks == 1 ? launch(one) : (line_form(p, head_dim) ? launch(line) : launch(units)));
    };
    if (head_dim == 64)
        return form(sw_mixed_attn_kernel<64, kOneChunk>, sw_mixed_attn_kernel<64, kSeveralChunks>, sw_mixed_attn_kernel<64, kLine>,
                    sw_mixed_attn_kernel<64, kUnits>);
    return form(sw_mixed_attn_kernel<128, kOneChunk>, sw_mixed_attn_kernel<128, kSeveralChunks>, sw_mixed_attn_kernel<128, kLine>,
                sw_mixed_attn_kernel<128, kUnits>);
}

}  // namespace sw
