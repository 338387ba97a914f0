// Short decode calls: one thread-block cluster per (sequence, KV head) unit does everything, in one launch.
//
// The chain of kernels that serves long calls (seer_gate.cu, seer_decode.cu) spends, on a short one, most of its
// time between its parts: lists through global memory, a schedule over all units, partial results published with
// a fence and a ticket and read back by the last CTA.  Here the S CTAs (S = 1 .. 16) of a unit's cluster share
// the unit from its first byte to its output:
//   1. gate (GATE): the unit's gate query, spread over the cluster's warps, into every CTA's shared memory; the
//      scores of each CTA's keys into every CTA's; every CTA selects for itself, and keeps the listed tiles that it
//      reads (tile t belongs to CTA t mod S); meanwhile the producer warps compress the block that has just filled,
//      if one has;
//      list (!GATE, several query tokens): the CTA reads its tiles' numbers from the caller's list, or counts them off (dense);
//   2. tiles: one producer warp keeps a ring of three 64-token K/V stages in flight; eight consumer warps, two
//      groups of four, take alternate tiles, a warp 16 tokens (the same tensor-core steps as decode_kernel);
//   3. combine: the warps' partials meet in shared memory, the CTA's go, a slice of the channels each, to the
//      cluster's CTAs, which write their slice of the output.
// Nothing between the steps leaves the SMs.  What one CTA stores into another's shared memory (queries, scores, partials)
// carries its own completion: the store counts its bytes down on an mbarrier of the receiver, which knows how many there
// will be.  A CTA thus waits for what it reads and for nothing else.  The cluster's hardware barrier, whose release first
// waits for all of a thread's stores to be acknowledged, is used twice: before the first of these stores, and at the end,
// so that no CTA leaves while one is under way.
#include <cooperative_groups.h>

#include <cstring>
#include <type_traits>

#include "seer_cluster.cuh"

namespace cg = cooperative_groups;

namespace seer {

namespace {

constexpr int kCodes = 256;                                // tile (or gathered block) numbers that a CTA holds
constexpr int kListed = 8192;                              // most scored blocks of a list
constexpr int kBins = 1024;                                // histogram of the selection
constexpr int kFew = 2048;                                 // candidates that its short list holds
constexpr int kMergeStride = 132;                          // floats per row of a warp's partial (bank spread)
constexpr int kKeyTile = 16;                               // keys are dealt to the cluster's warps in tiles of 16
constexpr int kMaxQLen = 8;
constexpr int kKeySlots = 32;                              // most key tiles that a CTA has asked for at a time (a lane each)

// Two sizes.  NW = 8 worker warps (gate, consumers, combine) and a ring of three stages: two CTAs per SM, up to 16
// rows (8 without MULTI).  NW = 16 and five stages: one CTA per SM, up to 32 rows.
template <int NW, bool MULTI>
struct Size {
    static constexpr int kWorkers = 32 * NW, kThreads = kWorkers + 32;     // ... and the producer warp
    static constexpr int kStages = NW == 8 ? 3 : 5, kGroups = NW / 4;
    static constexpr int kRows = !MULTI ? 8 : NW == 8 ? 16 : 32;
    static constexpr int kArrivals = kStages * kGroups;
};

template <int NW, bool MULTI>
struct __align__(1024) StepSmem {
    using Z = Size<NW, MULTI>;
    // K/V ring.  Before the first tile is asked for, the gate's: the scores of the unit (up to kStepMaxBlocks) at its
    // beginning, GateScratch at its end, compressed keys on their way between them.  After the last tile: the warps' partials.
    unsigned char ring[Z::kStages * kStageBytes];
    // what the cluster's CTAs send after their last tile (a fast one while this one still selects: memory that is its own
    // from the moment on that this CTA has sent its scores)
    union {
        __align__(16) float recv_o[Z::kRows * kHeadDim];   // [source CTA][row][this CTA's slice of the channels]
        double sums[NW][16][MULTI ? kMaxQLen : 1];         // before that: partial sums of the gate query: [warp][row][token]
    };
    float2 recv_ml[kMaxS][Z::kRows];                       // [source CTA][row]: max, sum
    float2 warp_ml[NW][8];
    // Tile n arrives in stage n % kStages and is announced on full[n % kArrivals].  The consumer groups that share a
    // tile's rows take all of one residue of the tile numbers, at their own pace, and every barrier belongs to one
    // residue, so its groups follow all of its phases.  (With a barrier per stage a group would miss the others' phases
    // and could take one that is two back for the one that it waits for.)
    uint64_t full[Z::kArrivals], empty[Z::kStages];
    uint64_t key_full[kKeySlots];
    uint64_t got_query, got_scores, got_feat, got_parts;   // bytes from the cluster's CTAs
    int meta[Z::kArrivals];                                // tokens from the tile's first row on (blocks of 16 or 32 tokens: per block, 8 bits each)
    int codes[kCodes];                                     // GATE: this CTA's tiles: 64-token tile numbers, or the gathered blocks
    // selection
    int warp_tot[NW];
    float warp_red[NW];
    uint32_t warp_min[NW], warp_max[NW];                   // ... and of a warp's candidates
    uint32_t list_key[32];
    int list_j[32];
    __align__(16) float feat[3 * kHeadDim];                // pooled features of the block that has just filled
    __align__(16) float feat_own[3][16];                   // those of 16 channels, on their way to the cluster's CTAs
    uint32_t pre_min, pre_max;                             // smallest and largest key of a candidate
    uint32_t prefix;
    int rem, bin_cnt, list_n, tile_n, few_n, last_eq, no_list;
};
static_assert(sizeof(StepSmem<8, true>) + 1024 <= 113 * 1024, "two CTAs per SM");
static_assert(sizeof(StepSmem<16, true>) + 1024 <= 227 * 1024, "one CTA per SM");
// The gate's part of the ring, at its end.
template <int NW, bool MULTI>
struct GateScratch {
    // Gate queries, from all CTAs: each channel in three bf16 parts (high, middle, low), which together are the fp32 number
    // exactly, two channels a word.  (Rows 64 bytes longer than the channels: neighbouring parts are in different banks.)
    __align__(16) uint32_t parts[MULTI ? kMaxQLen : 1][3][kMaxDGate / 2 + 16];
    __align__(16) int hist[kBins];                         // selection
};
// ... and of the selection, when queries and keys have been used.
struct Selected {
    unsigned taken[kStepMaxBlocks / 32];                   // a bit per candidate
    union {
        uint16_t list[kListed];                            // the taken ones, in order
        struct {                                           // on the way there, the short list:
            uint16_t tile[kStepMaxBlocks / kKeyTile];      // the tiles that may have a taken one
            uint16_t j[kFew];                              // their candidates that may be taken
            union {
                float tile_max[kStepMaxBlocks / kKeyTile]; // largest score of a key tile
                float score[kFew];
            };
        };
    };
};
template <int NW, bool MULTI>
struct GatePlace {                                         // offsets in the ring
    using Scratch = GateScratch<NW, MULTI>;
    static constexpr int kRing = Size<NW, MULTI>::kStages * kStageBytes;
    static constexpr int kScratch = kRing - (int)sizeof(Scratch);
    static constexpr int kSelected = kRing - (int)sizeof(Scratch::hist) - (int)sizeof(Selected);
    static_assert(offsetof(Scratch, hist) + sizeof(Scratch::hist) == sizeof(Scratch), "the histogram comes last");
    static_assert(kScratch % 16 == 0 && kSelected % 16 == 0 && kSelected >= 4 * kStepMaxBlocks, "behind the scores");
    static_assert(kScratch - 4 * kStepMaxBlocks - 64 >= 2 * kKeyTile * kMaxDGate, "room for a key tile whatever there is to score");
};
static_assert(kStepMaxBlocks <= 65536, "16 bits a block");

template <int NW>
__device__ __forceinline__ void tiles_listed_arrive() {
    __syncwarp();
    asm volatile("bar.arrive 3, %0;" ::"n"(32 * NW + 32) : "memory");
}
template <int NW>
__device__ __forceinline__ void tiles_listed_wait() {
    __syncwarp();
    asm volatile("bar.sync 3, %0;" ::"n"(32 * NW + 32) : "memory");
}

// ... and whether one of the worker threads says so
template <int NW>
__device__ __forceinline__ bool worker_any(bool x) {
    uint32_t any;
    __syncwarp();
    asm volatile(
        "{\n\t.reg .pred p, q;\n\t"
        "setp.ne.u32 p, %1, 0;\n\t"
        "bar.red.or.pred q, 1, %2, p;\n\t"
        "selp.u32 %0, 1, 0, q;\n\t}"
        : "=r"(any)
        : "r"((uint32_t)x), "n"(32 * NW)
        : "memory");
    return any != 0;
}

template <bool GATE>
struct GateArg { GateParams g; };
template <>
struct GateArg<false> {};

// The selection of the `need` best of the candidates [0, n_cand), 0 < need < n_cand, by a CTA's worker warps.  Comparisons
// only: the lower block number wins a tie, NaN is below every number.  A histogram over a monotone linear map of [min, max]
// leaves a few candidates in the boundary bin, which every warp ranks for itself; crowded bins and ranges that are not finite
// take radix passes over key - min instead.
// What bounds it: this code runs once per call, by two warps a scheduler, so that its time is the number of instructions
// on its longest path (some ten cycles each, mostly their fetch) and not the candidates; hence rolled loops, whose bodies stay
// in the instruction buffers.
template <int NW, typename Smem>
struct Selection {
    static constexpr int kThreads = 32 * NW, kPer = kBins / kThreads;
    Smem& sm;
    int* hist;
    const float* sc;
    int n_cand, need, warp, lane, tid;
    float smin, smax, scale;
    bool finite;
    // candidate j is taken if its key is above thr, or equal to it and j <= j_eq
    uint32_t thr = 0u;
    int j_eq = 0x7fffffff;

    __device__ __forceinline__ Selection(Smem& s, int* h, const float* scores, int n, int want, int w, int l)
        : sm(s), hist(h), sc(scores), n_cand(n), need(want), warp(w), lane(l), tid(32 * w + l) {
        smin = key_score(sm.pre_min);
        smax = key_score(sm.pre_max);
        const float range = smax - smin;
        scale = (kBins - 1.f) / range;
        // (every candidate's score is finite then; -0 and +0 have the same bin)
        finite = smin > -INFINITY && range > 0.f && range < INFINITY && scale < INFINITY;
    }
    __device__ __forceinline__ int bin_of(float s) const { return min(kBins - 1, (int)((s - smin) * scale)); }
    // the warps' totals before this one's
    __device__ __forceinline__ int before() const { return __reduce_add_sync(0xffffffffu, lane < warp ? sm.warp_tot[lane] : 0); }
    __device__ __forceinline__ int scan(int v) const {      // inclusive, over the warp
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int t = __shfl_up_sync(0xffffffffu, v, o);
            if (lane >= o) v += t;
        }
        return v;
    }
    // thread t owns kPer bins, from kBins-1-kPer*t downwards: finds the bin that straddles the rem-th best
    __device__ __forceinline__ void find_bin(int rem) {
        worker_sync<NW>();
        int c[kPer], mine = 0;
        if constexpr (kPer == 4) {
            const int4 v = *reinterpret_cast<const int4*>(hist + kBins - 4 * (tid + 1));
            c[0] = v.w; c[1] = v.z; c[2] = v.y; c[3] = v.x;
        } else {
            const int2 v = *reinterpret_cast<const int2*>(hist + kBins - 2 * (tid + 1));
            c[0] = v.y; c[1] = v.x;
        }
#pragma unroll
        for (int x = 0; x < kPer; ++x) mine += c[x];
        const int incl = scan(mine);
        if (lane == 31) sm.warp_tot[warp] = incl;
        worker_sync<NW>();
        int above = incl - mine + before();
        if (above < rem && rem <= above + mine) {
#pragma unroll
            for (int x = 0; x < kPer; ++x) {
                if (above < rem && rem <= above + c[x]) {
                    sm.prefix = (uint32_t)(kBins - 1 - kPer * tid - x);
                    sm.rem = rem - above;
                    sm.bin_cnt = c[x];
                }
                above += c[x];
            }
        }
        worker_sync<NW>();
    }
    __device__ __forceinline__ void clear_bins() {          // (a thread's own ones)
#pragma unroll
        for (int x = 0; x < kPer; ++x) hist[kBins - 1 - kPer * tid - x] = 0;
    }
    __device__ __forceinline__ void enlist(float v, int j) {
        const int slot = atomicAdd(&sm.list_n, 1) & 31;
        sm.list_key[slot] = score_key(v);
        sm.list_j[slot] = j;
    }
    // the `rem`-th best of the `cnt` <= 32 listed candidates, found by every warp for itself
    __device__ __forceinline__ void rank_list(int rem, int cnt) {
        const uint32_t key = lane < cnt ? sm.list_key[lane] : 0u;
        const int j = lane < cnt ? sm.list_j[lane] : 0x7fffffff;
        int rank = 0;
#pragma unroll 1
        for (int m = 0; m < cnt; ++m) {
            const uint32_t km = __shfl_sync(0xffffffffu, key, m);
            const int jm = __shfl_sync(0xffffffffu, j, m);
            rank += km > key || (km == key && jm < j);
        }
        const int src = __ffs(__ballot_sync(0xffffffffu, lane < cnt && rank == rem - 1)) - 1;
        thr = __shfl_sync(0xffffffffu, key, src);
        j_eq = __shfl_sync(0xffffffffu, j, src);
    }
    // Up to 4 * Q <= 16 candidates a thread: they stay in its registers from the histogram to take(e, j), for the e-th taken
    // one in block order.  False: the boundary bin is crowded.
    template <int Q, typename Take>
    __device__ __forceinline__ bool in_registers(Take&& take) {
        const int j0 = 4 * Q * tid, end = (n_cand + kKeyTile - 1) & ~(kKeyTile - 1);
        float v[4 * Q];
        int b[4 * Q];
#pragma unroll
        for (int x = 0; x < Q; ++x) {
            const float4 f = j0 + 4 * x < end ? *reinterpret_cast<const float4*>(sc + j0 + 4 * x)
                                              : make_float4(-INFINITY, -INFINITY, -INFINITY, -INFINITY);
            v[4 * x] = f.x; v[4 * x + 1] = f.y; v[4 * x + 2] = f.z; v[4 * x + 3] = f.w;
        }
        // (minus infinity, behind the last candidate, has a negative bin)
#pragma unroll
        for (int k = 0; k < 4 * Q; ++k) {
            b[k] = bin_of(v[k]);
            if (b[k] >= 0) atomicAdd(&hist[b[k]], 1);
        }
        find_bin(need);
        const int bin = (int)sm.prefix, rem = sm.rem, cnt = sm.bin_cnt;
        if (cnt > 32) return false;
#pragma unroll
        for (int k = 0; k < 4 * Q; ++k)
            if (b[k] == bin) enlist(v[k], j0 + k);
        worker_sync<NW>();
        rank_list(rem, cnt);
        const float last = key_score(thr);
        unsigned taken = 0u;
#pragma unroll
        for (int k = 0; k < 4 * Q; ++k) taken |= (unsigned)((v[k] > last) | ((v[k] == last) & (j0 + k <= j_eq))) << k;
        const int mine = __popc(taken), incl = scan(mine);
        if (lane == 31) sm.warp_tot[warp] = incl;
        worker_sync<NW>();
        int at = incl - mine + before();
#pragma unroll 1
        for (; taken; taken &= taken - 1) take(at++, j0 + __ffs(taken) - 1);
        return true;
    }
};

// The other cases: many candidates, crowded bins, scores that are not finite.  The taken ones' numbers in order, in sl.list.
// Neighbours are often taken together, so that a thread finds dozens: what is done per taken one is little more than its place
// in the list (with what an entry means to the tiles done by the thread that found it the lists of 625 of 15625
// blocks took 22 us, and now 13; those of 256 of 9375 up to 20, and now 8).  A function of its own: its loops' registers are not
// those of the short calls' path.
template <int NW, typename Smem>
__device__ __noinline__ void select_many(Smem* smem, int* hist, Selected* selected, const float* sc, int n_cand, int need) {
    __builtin_assume(__isShared(smem));
    __builtin_assume(__isShared(hist));
    __builtin_assume(__isShared(selected));
    __builtin_assume(__isShared(sc));
    constexpr int kThreads = 32 * NW;
    Smem& sm = *smem;
    Selected& sl = *selected;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    Selection<NW, Smem> sel(sm, hist, sc, n_cand, need, warp, lane);
    // the list, from the bits
    auto list_taken = [&]() {
        constexpr int kWords = kStepMaxBlocks / 32 / kThreads;
        worker_sync<NW>();                                 // (every bit is in place)
        unsigned words[kWords];
        int mine = 0;
#pragma unroll
        for (int x = 0; x < kWords; ++x) {
            words[x] = 32 * (kWords * tid + x) < n_cand ? sl.taken[kWords * tid + x] : 0u;
            mine += __popc(words[x]);
        }
        const int incl = sel.scan(mine);
        if (lane == 31) sm.warp_tot[warp] = incl;
        worker_sync<NW>();
        int at = incl - mine + sel.before();
#pragma unroll
        for (int x = 0; x < kWords; ++x)
#pragma unroll 1
            for (unsigned m = words[x]; m; m &= m - 1) sl.list[at++] = (uint16_t)(32 * (kWords * tid + x) + __ffs(m) - 1);
        worker_sync<NW>();
    };
    bool found = false;
    const bool many = sel.finite && n_cand > 16 * kThreads;
    // For one place in 32 or fewer a short list comes first: the need-th largest of the key tiles' maxima is a bound that at
    // least `need` candidates reach, and few others do.
    if (many && 32 * need <= n_cand) {
        const int n_tiles = (n_cand + kKeyTile - 1) / kKeyTile;
        for (int x = tid; x < kStepMaxBlocks / 32; x += kThreads) sl.taken[x] = 0u;
        // (places of the last tile behind the last candidate hold minus infinity)
#pragma unroll 1
        for (int t = tid; t < n_tiles; t += kThreads) {
            const float4* src = reinterpret_cast<const float4*>(sc + kKeyTile * t);
            float best = -INFINITY;
#pragma unroll
            for (int x = 0; x < 4; ++x) {                  // (neighbouring lanes begin at different banks)
                const float4 v = src[x ^ ((lane >> 1) & 3)];
                best = fmaxf(best, fmaxf(fmaxf(v.x, v.y), fmaxf(v.z, v.w)));
            }
            sl.tile_max[t] = best;
            atomicAdd(&hist[sel.bin_of(best)], 1);
        }
        sel.find_bin(need);
        const int bound = (int)sm.prefix;
        sel.clear_bins();
#pragma unroll 1
        for (int t = tid; t < n_tiles; t += kThreads)
            if (sel.bin_of(sl.tile_max[t]) >= bound) sl.tile[atomicAdd(&sm.tile_n, 1)] = (uint16_t)t;
        worker_sync<NW>();
        // bins of their own for the few, from about the bound's bin to the largest score
        const float lo = sel.smin + (float)bound / sel.scale, fine = (kBins - 1.f) / (sel.smax - lo);
        auto fine_of = [&](float s) -> int { return max(0, min(kBins - 1, (int)((s - lo) * fine))); };
        const int total = kKeyTile * sm.tile_n;
        if (fine > 0.f && fine < INFINITY) {
#pragma unroll 1
            for (int x = tid; x < total; x += kThreads) {
                const int j = kKeyTile * sl.tile[x / kKeyTile] + (x & (kKeyTile - 1));
                const float v = sc[j];
                if (sel.bin_of(v) >= bound) {
                    const int slot = atomicAdd(&sm.few_n, 1);
                    if (slot < kFew) { sl.score[slot] = v; sl.j[slot] = (uint16_t)j; }
                    atomicAdd(&hist[fine_of(v)], 1);
                }
            }
            sel.find_bin(need);
            const int few = sm.few_n, bin = (int)sm.prefix, rem = sm.rem, cnt = sm.bin_cnt;
            if (few <= kFew && cnt <= 32) {
#pragma unroll 1
                for (int e = tid; e < few; e += kThreads)
                    if (fine_of(sl.score[e]) == bin) sel.enlist(sl.score[e], sl.j[e]);
                worker_sync<NW>();
                sel.rank_list(rem, cnt);
#pragma unroll 1
                for (int e = tid; e < few; e += kThreads) {
                    const uint32_t key = score_key(sl.score[e]);
                    const int j = sl.j[e];
                    if (key > sel.thr || (key == sel.thr && j <= sel.j_eq)) atomicOr(&sl.taken[j >> 5], 1u << (j & 31));
                }
                list_taken();
                return;
            }
            sel.clear_bins();                              // (crowded, too: all candidates then)
        }
        worker_sync<NW>();
    }
    if (many) {
        // Neighbouring blocks have similar scores: the lanes of a warp take candidates that are far apart (lane l has
        // run l of an odd number of blocks: no bank conflicts); side by side, their additions would queue for a few bins.
        // (four at a time: their loads go out together)
        const int run = ((n_cand + 31) / 32) | 1;
        auto each_spread = [&](auto&& fn) {
            const int j0 = lane * run;
#pragma unroll 1
            for (int q = warp; q < run; q += 4 * NW) {
                float v[4];
#pragma unroll
                for (int x = 0; x < 4; ++x) v[x] = sc[min(j0 + q + x * NW, n_cand - 1)];
#pragma unroll
                for (int x = 0; x < 4; ++x)
                    if (q + x * NW < run && j0 + q + x * NW < n_cand) fn(v[x], j0 + q + x * NW);
            }
        };
        each_spread([&](float v, int) { atomicAdd(&hist[sel.bin_of(v)], 1); });
        sel.find_bin(need);
        const int bin = (int)sm.prefix, rem = sm.rem, cnt = sm.bin_cnt;
        if (cnt <= 32) {
            each_spread([&](float v, int j) { if (sel.bin_of(v) == bin) sel.enlist(v, j); });
            worker_sync<NW>();
            sel.rank_list(rem, cnt);
            found = true;
        }
    }
    // a warp has a run of blocks, a lane every 32nd of them
    const int words = (n_cand + 32 * NW - 1) / (32 * NW), w0 = warp * words, j0 = 32 * w0 + lane;
    if (!found) {
        const uint32_t kmin = sm.pre_min, kmax = sm.pre_max;
        auto each = [&](auto&& fn) {
#pragma unroll 1
            for (int e = 0; e < words; ++e) {
                const int j = j0 + 32 * e;
                fn(j < n_cand, score_key(sc[min(j, n_cand - 1)]), j);
            }
        };
        // radix passes of ten bits over key - kmin
        int bits_left = 32 - __clz(max(kmax - kmin, 1u)), rem = need;
        uint32_t prefix = 0u;
        while (bits_left > 0) {
            const int wbits = min(10, bits_left), shift = bits_left - wbits;
            sel.clear_bins();
            worker_sync<NW>();
            each([&](bool ok, uint32_t key, int) {
                const uint32_t rel = key - kmin;
                if (ok && (uint32_t)((unsigned long long)rel >> (shift + wbits)) == prefix)        // (shift + wbits can be 32)
                    atomicAdd(&hist[(rel >> shift) & ((1u << wbits) - 1u)], 1);
            });
            sel.find_bin(rem);
            prefix = (prefix << wbits) | sm.prefix;
            rem = sm.rem;
            bits_left = shift;
        }
        sel.thr = kmin + prefix;
        // the rem-th candidate whose key equals thr, in block order
        int n_eq = 0;
        each([&](bool ok, uint32_t key, int) { n_eq += __popc(__ballot_sync(0xffffffffu, ok && key == sel.thr)); });
        worker_sync<NW>();                                 // (everybody has read the last pass's totals)
        if (lane == 0) sm.warp_tot[warp] = n_eq;
        worker_sync<NW>();
        int eq_before = sel.before();
        if (eq_before < rem && rem <= eq_before + n_eq) {
            each([&](bool ok, uint32_t key, int j) {
                const bool eq = ok && key == sel.thr;
                const unsigned m = __ballot_sync(0xffffffffu, eq);
                if (eq && eq_before + __popc(m & ((1u << lane) - 1u)) == rem - 1) sm.last_eq = j;
                eq_before += __popc(m);
            });
        }
        worker_sync<NW>();
        sel.j_eq = sm.last_eq;
    }
#pragma unroll 1
    for (int e = 0; e < words; e += 4) {
        float v[4];
#pragma unroll
        for (int x = 0; x < 4; ++x) v[x] = sc[min(j0 + 32 * (e + x), n_cand - 1)];
#pragma unroll
        for (int x = 0; x < 4; ++x) {
            const uint32_t key = score_key(v[x]);
            const int j = j0 + 32 * (e + x);
            const unsigned m = __ballot_sync(0xffffffffu, (j < n_cand) & ((key > sel.thr) | ((key == sel.thr) & (j <= sel.j_eq))));
            if (lane == 0 && e + x < words) sl.taken[w0 + e + x] = m;
        }
    }
    list_taken();
}

// Cut off, not rounded: no finite number becomes infinite.
__device__ __forceinline__ uint32_t pack_bf16x2_toward_zero(float lo, float hi) {
    uint32_t d;
    asm("cvt.rz.bf16x2.f32 %0, %1, %2;" : "=r"(d) : "f"(hi), "f"(lo));
    return d;
}

// The compressed key of block j of the unit, which has just filled, in two parts.  The same sums in the same order as
// seer_kcomp.cu's append, so the same entry.  First the pooled features, by the producer warps of the cluster, which have
// nothing else to do while the gate is at work: 16 channels at a time, to every CTA of the cluster.
template <typename Smem>
__device__ __forceinline__ void append_pool(const GateParams& g, Smem& sm, int i, int h, int j, int rank, int S) {
    const int lane = threadIdx.x & 31, b = g.block_size;
    const __nv_bfloat16* src = g.k_nope + (size_t)i * g.k_stride_batch + (size_t)h * g.k_stride_head +
                               (g.k_rows_block_local ? 0 : (size_t)j * b) * g.k_stride_token;
    const int rg = lane >> 1;                              // lane: eight channels, rows lane / 2, lane / 2 + 16, ...
#pragma unroll 1
    for (int w0 = rank; w0 < 8; w0 += S) {
        const int c8 = 2 * w0 + (lane & 1);
        __nv_bfloat162 mx[4], mn[4];
        float sum[8];
#pragma unroll
        for (int c = 0; c < 4; ++c) { mx[c] = __float2bfloat162_rn(-INFINITY); mn[c] = __float2bfloat162_rn(INFINITY); }
#pragma unroll
        for (int c = 0; c < 8; ++c) sum[c] = 0.f;
#pragma unroll 4
        for (int r = rg; r < b; r += 16) {
            const uint4 v = *reinterpret_cast<const uint4*>(src + (size_t)r * g.k_stride_token + 8 * c8);
            const __nv_bfloat162* hh = reinterpret_cast<const __nv_bfloat162*>(&v);
#pragma unroll
            for (int c = 0; c < 4; ++c) {
                mx[c] = __hmax2(mx[c], hh[c]);
                mn[c] = __hmin2(mn[c], hh[c]);
                const float2 f = bf16x2_to_float2(hh[c]);
                sum[2 * c] += f.x;
                sum[2 * c + 1] += f.y;
            }
        }
#pragma unroll
        for (int off = 2; off < 32; off <<= 1) {
#pragma unroll
            for (int c = 0; c < 4; ++c) {
                const uint32_t a = __shfl_xor_sync(0xffffffffu, *reinterpret_cast<uint32_t*>(&mx[c]), off);
                const uint32_t d = __shfl_xor_sync(0xffffffffu, *reinterpret_cast<uint32_t*>(&mn[c]), off);
                mx[c] = __hmax2(mx[c], *reinterpret_cast<const __nv_bfloat162*>(&a));
                mn[c] = __hmin2(mn[c], *reinterpret_cast<const __nv_bfloat162*>(&d));
            }
        }
        // (row groups 2w and 2w + 1 first, then those pairs one after the other)
#pragma unroll
        for (int c = 0; c < 8; ++c) {
            const float pair = sum[c] + __shfl_xor_sync(0xffffffffu, sum[c], 2);
            float s = 0.f;
#pragma unroll
            for (int w = 0; w < 8; ++w) s += __shfl_sync(0xffffffffu, pair, 4 * w + (lane & 1));
            sum[c] = s / (float)b;
        }
        if (lane < 2) {
#pragma unroll
            for (int c = 0; c < 4; ++c) {
                const float2 a = bf16x2_to_float2(mx[c]), d = bf16x2_to_float2(mn[c]);
                *reinterpret_cast<float2*>(&sm.feat_own[0][8 * lane + 2 * c]) = a;
                *reinterpret_cast<float2*>(&sm.feat_own[1][8 * lane + 2 * c]) = d;
                *reinterpret_cast<float2*>(&sm.feat_own[2][8 * lane + 2 * c]) = make_float2(sum[2 * c], sum[2 * c + 1]);
            }
        }
        __syncwarp();
        if (lane < S) {                                    // lane r to CTA r of the cluster
            const uint32_t to = cluster_addr(sm.feat + 16 * w0, lane), bar = cluster_addr(&sm.got_feat, lane);
#pragma unroll 1
            for (int x = 0; x < 12; ++x)
                send_f32x4(to + (x >> 2) * (kHeadDim * 4) + (x & 3) * 16, *reinterpret_cast<const float4*>(&sm.feat_own[x >> 2][4 * (x & 3)]), bar);
        }
        __syncwarp();
    }
}

// Then the projection, by the worker warps of all CTAs, while their first tiles travel: two rotary pairs at a time.
template <int NW, typename Smem>
__device__ __forceinline__ void append_project(const GateParams& g, Smem& sm, int u, int h, int j, int rank, int S) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, half = g.d_gate / 2;
    const int ppc = half / S;                              // pairs of this CTA (an even number)
    if (2 * warp >= ppc) return;
    const float* feat = sm.feat;
    __nv_bfloat16* dst = const_cast<__nv_bfloat16*>(g.kcomp) + ((size_t)u * g.max_blocks + j) * g.d_gate;
    bool waited = false;
#pragma unroll 1
    for (int pair = rank * ppc + 2 * warp; pair < (rank + 1) * ppc; pair += 2 * NW) {
        uint4 wv[4][2];                                    // rows of W_k[h] of the rotary pairs `pair`, `pair` + 1
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const int r = pair + (k & 1) + (k >> 1) * half;
            const uint4* wrow = reinterpret_cast<const uint4*>(g.w_k + ((size_t)h * g.d_gate + r) * 3 * kHeadDim);
            wv[k][0] = __ldg(wrow + lane);
            wv[k][1] = lane < 16 ? __ldg(wrow + 32 + lane) : make_uint4(0u, 0u, 0u, 0u);
        }
        if (!waited) {                                     // (without the features nothing goes into the cache, which outlives the call)
            if (__any_sync(0xffffffffu, !wait_sent(&sm.got_feat, g.status))) return;
            waited = true;
        }
        float acc[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            acc[k] = 0.f;
#pragma unroll
            for (int x = 0; x < 2; ++x) {
                const int ch = lane + 32 * x;
                const __nv_bfloat162* hh = reinterpret_cast<const __nv_bfloat162*>(&wv[k][x]);
#pragma unroll
                for (int c = 0; c < 4; ++c) {
                    const float2 w = bf16x2_to_float2(hh[c]);
                    acc[k] = fmaf(w.x, ch < 48 ? feat[8 * ch + 2 * c] : 0.f, acc[k]);
                    acc[k] = fmaf(w.y, ch < 48 ? feat[8 * ch + 2 * c + 1] : 0.f, acc[k]);
                }
            }
        }
#pragma unroll
        for (int k = 0; k < 4; ++k)
#pragma unroll
            for (int off = 16; off > 0; off >>= 1) acc[k] += __shfl_xor_sync(0xffffffffu, acc[k], off);
        if (lane < 2) {
            const int c = pair + lane;
            const float a = lane ? acc[1] : acc[0], d = lane ? acc[3] : acc[2];
            float sn, cs;
            rope_sincos((double)j * (double)g.block_size, g.inv_freq[c], &sn, &cs);
            dst[c] = __float2bfloat16(a * cs - d * sn);
            dst[c + half] = __float2bfloat16(d * cs + a * sn);
        }
    }
}

// sin and cos like rope_sincos, with what the reduced angle loses when it is rounded to fp32 put back (first order): the
// gate query is made of MMAs' sums, whose accumulation cuts off, and gets back here what they lose.
__device__ __forceinline__ void rope_sincos_wide(double pos, double inv_freq, double* sn, double* cs) {
    double turns = pos * inv_freq * 0.15915494309189535;   // 1 / (2 pi)
    turns = 2. * (turns - rint(turns));
    const float x = (float)turns;
    float s, c;
    sincospif(x, &s, &c);
    const double rest = (turns - (double)x) * 3.14159265358979324;
    *sn = (double)s + (double)c * rest;
    *cs = (double)c - (double)s * rest;
}

// The score of one key by plain dot products (whole warp; the largest over the query tokens): for a key or gate query that
// is not finite, where the parts of the query (score_keys) would make NaN of what is an infinity.
__device__ __noinline__ float score_key_plain(const uint4* key, const uint32_t (*parts)[3][kMaxDGate / 2 + 16], int q_len, int d_gate, int lane) {
    const uint4 kv = lane < d_gate / 8 ? __ldcg(key + lane) : make_uint4(0u, 0u, 0u, 0u);
    float best = -INFINITY;
    for (int t = 0; t < q_len; ++t) {
        float a = 0.f;
        if (lane < d_gate / 8) {
            float q[8];
#pragma unroll
            for (int c = 0; c < 4; ++c) {
                const float2 hi = bf16x2_to_float2(parts[t][0][4 * lane + c]), mid = bf16x2_to_float2(parts[t][1][4 * lane + c]),
                             low = bf16x2_to_float2(parts[t][2][4 * lane + c]);
                q[2 * c] = hi.x + (mid.x + low.x);
                q[2 * c + 1] = hi.y + (mid.y + low.y);
            }
            a = dot8(kv, q);
        }
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) a += __shfl_xor_sync(0xffffffffu, a, off);
        best = q_len > 1 ? fmaxf(best, a) : a;
    }
    return best;
}

// The key tiles of a CTA (a run of the unit's keys) on their way through the ring: tile m comes in slot m mod `n` and slot s
// belongs to warp s mod NW.  A tile of 16 keys is two bulk copies, of its first and of its last eight keys; the second halves'
// memory begins 64 bytes off a bank line, so that lanes that read the same channels of a key of either half read different
// banks.  The producer warp asks for the slots' first tiles, a warp for its slots' others.  (What bounds the scores of many keys
// is how many are under way while the queries are made.  With a tile a warp, in its registers -- 64 of them for keys of 256
// channels, which spilled -- a step of batch 8 at 128k took 83.5 us and takes 82.7, with 64 blocks 40.3 and 38.6, of two
// sequences of 90k with 256 channels 32.2 and 24.0.  All other keys asked into L2 at the same time are too many for it where
// there are many units: of 200 units of 9375 keys, 480 MB, a step took 199 us and takes 142.)
struct KeySlots {
    unsigned char *a, *b;                                  // the halves of slot 0
    int n, shift;                                          // shift: log2 of a half's bytes

    __device__ __forceinline__ void place(unsigned char* ring, int n_tiles, int end, int d_gate) {
        const int first = (n_tiles * kKeyTile * 4 + 127) & ~127;
        shift = 34 - __clz(2 * d_gate);
        n = min((end - first - 64) >> (shift + 1), kKeySlots);
        a = ring + first;
        b = a + (n << shift) + 64;
    }
    __device__ __forceinline__ void request(int slot, uint64_t* full, const unsigned char* keys, int rows) const {      // rows: keys there are, from the tile's first one on
        const int na = min(rows, 8) << (shift - 3), nb = max(0, min(rows, 16) - 8) << (shift - 3);
        mbar_arrive_expect_tx(full, (uint32_t)(na + nb));
        bulk_load(a + (slot << shift), keys, (uint32_t)na, full);
        if (nb > 0) bulk_load(b + (slot << shift), keys + (1 << shift), (uint32_t)nb, full);
    }
};

// The sums of a key tile, by MMAs: row r of the first eight of the A operand is key (r & 1) * 8 + r / 2, row r + 8 the key
// four behind it.  A lane supplies the pieces lane % 4 + 4 * x of its rows' keys: `pieces` gives them.
// The B operand is the gate queries: columns 4t .. 4t + 3 are query token t's channels, the high part in the first two (one
// with the first and one with the last eight channels of an MMA, zero elsewhere: of sums half as long the MMA cuts off
// less), the middle and low parts in the others.  Both operands' contraction index is permuted alike: piece x of a lane is
// two MMAs' operand as it lies in memory.
// v0, v1: the sums of rows lane / 4 and lane / 4 + 8, the largest over the query tokens, the same in a row's four lanes; `odd0`, `odd1`:
// one of the row's sums is not finite.
template <int XS, bool MULTI, typename Pieces>
__device__ __forceinline__ void key_sums(Pieces&& pieces, const uint32_t (*parts)[3][kMaxDGate / 2 + 16], int q_len, int lane, float& v0, float& v1,
                                         bool& odd0, bool& odd1) {
    v0 = v1 = -INFINITY;
    odd0 = odd1 = false;
#pragma unroll 1
    for (int nt = 0; 2 * nt < q_len; ++nt) {
        // (each MMA begins at zero and its 16 products are added up outside: the MMA's own accumulation cuts off where the
        // addition rounds to nearest)
        float s[4] = {0.f, 0.f, 0.f, 0.f};
        const int col = (lane >> 2) & 3, t = 2 * nt + (lane >> 4);
        const uint32_t even = t < q_len && col != 1 ? 0xffffffffu : 0u, odd_w = t < q_len && col != 0 ? 0xffffffffu : 0u;
        const uint4* bq = reinterpret_cast<const uint4*>(parts[min(t, q_len - 1)][max(0, col - 1)]) + (lane & 3);
#pragma unroll
        for (int x = 0; x < XS; ++x) {
            const uint4 b = bq[4 * x];
            uint4 lo, hi;
            pieces(x, lo, hi);
            const uint32_t a0[4] = {lo.x, hi.x, lo.y, hi.y}, a1[4] = {lo.z, hi.z, lo.w, hi.w};
            float c0[4] = {0.f, 0.f, 0.f, 0.f}, c1[4] = {0.f, 0.f, 0.f, 0.f};
            mma_bf16_16816(c0, a0, b.x & even, b.y & odd_w);
            mma_bf16_16816(c1, a1, b.z & even, b.w & odd_w);
#pragma unroll
            for (int c = 0; c < 4; ++c) s[c] += c0[c] + c1[c];
        }
        // lanes 0 and 2 of a row's four have a token's high part, 1 and 3 its middle and low parts
        float r0 = s[0] + s[1], r1 = s[2] + s[3];
        r0 += __shfl_xor_sync(0xffffffffu, r0, 1);
        r1 += __shfl_xor_sync(0xffffffffu, r1, 1);
        odd0 |= !(fabsf(r0) < INFINITY);
        odd1 |= !(fabsf(r1) < INFINITY);
        if (2 * nt + ((lane >> 1) & 1) >= q_len) r0 = r1 = -INFINITY;
        v0 = fmaxf(v0, fmaxf(r0, __shfl_xor_sync(0xffffffffu, r0, 2)));
        v1 = fmaxf(v1, fmaxf(r1, __shfl_xor_sync(0xffffffffu, r1, 2)));
        if (!MULTI) break;
    }
}

// grid (S, units), cluster (S, 1, 1).  Short calls are bound by latency, and that by the number of instructions on the
// longest path: all of this runs once, by two warps a scheduler, at some ten cycles an instruction.  A step of 8 units x 64
// blocks (16.8 MB, 2.6 us at memory speed): by time stamps in the kernel (which make it a microsecond or two longer; medians
// over the CTAs, from the first read on) the gate query is there after 2.8 us, the scores after 4.4, the list after 6.9, the
// tiles from 8.4 to 10.1, the CTAs' parts after 11.7, the output after 13.  With a cluster barrier behind each of the first
// three, the selection by one CTA and its lists stored into the others, it was 2.9, 7.2, 10.6, 11.8 to 13.3, 15.3, 16.2.
// Longer calls by memory: of a step of 64 units x 205 blocks (430 MB) the tiles take 66 us, 6.5 TB/s, from the first CTA's
// first to the last one's last; CTAs that share a unit read neighbouring blocks at the same time.
// What it does: a step by the token budget; or one whose lists may be so long that it matters whether they are even (where they
// are not, the lists and the append are all that is done here, and the list kernel behind this launch does the rest); or the
// gate alone, by either method; or attention over given lists or all blocks.
enum Kind { STEP, SPREAD_STEP, GATE_ALONE, LISTS };
// SMALL: lists of blocks of 16 or 32 tokens, four or two to a tile.  (Told apart at run time both kinds' look-ups and copies took
// registers from one another, and spilled.)
// DG: channels of the gate, 0: known at run time (where the constant did not help the registers: several query tokens 35.4 ->
// 36.6 us, steps of 256 channels 10.6 -> 11.0)
template <int NW, Kind KIND, bool MULTI, bool SMALL, int DG>
__global__ void __launch_bounds__(Size<NW, MULTI>::kThreads, NW == 8 ? 2 : 1)
step_cluster_kernel(const __grid_constant__ CUtensorMap map_k, const __grid_constant__ CUtensorMap map_v,
                    const __grid_constant__ DecodeParams p, const __grid_constant__ GateArg<KIND != LISTS> ga) {
    constexpr bool GATE = KIND != LISTS, ALONE = KIND == GATE_ALONE;
    using Z = Size<NW, MULTI>;
    using Smem = StepSmem<NW, MULTI>;
    constexpr int kWorkers = Z::kWorkers, kStages = Z::kStages, kArrivals = Z::kArrivals, kRows = Z::kRows;
    using Place = GatePlace<NW, MULTI>;
    extern __shared__ unsigned char smem_raw[];
    // (aligned by an offset, not by a cast through an integer: the compiler then still knows the accesses for shared ones)
    Smem& sm = *reinterpret_cast<Smem*>(smem_raw + ((1024 - (smem_u32(smem_raw) & 1023)) & 1023));
    cg::cluster_group cluster = cg::this_cluster();
    const int S = (int)cluster.num_blocks(), rank = (int)cluster.block_rank(), s_shift = 31 - __clz(S);
    const int u = blockIdx.y, i = u / p.num_kv_heads, h = u - i * p.num_kv_heads;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const bool producer = warp == NW;
    const int q_len = MULTI ? p.q_len : 1;
    // The unit's rows (query token, head of the group) are cut into gridDim.z parts of p.rows; this cluster's: row0 ..
    const int row0 = MULTI ? blockIdx.z * p.rows : 0;
    const int rows = MULTI ? min(p.rows, q_len * p.group - row0) : p.group;
    // eight rows are an MMA's N side: `tiles_n` consumer groups share a K/V tile, `paces` such teams take alternate tiles
    const int tiles_n = MULTI ? (rows + 7) >> 3 : 1;
    const int paces = MULTI ? Z::kGroups / tiles_n : Z::kGroups;
    if (tid < 32) {
        if (GATE) mbar_init(&sm.key_full[tid], 1);
        if (tid < kArrivals) mbar_init(&sm.full[tid], 1);
        if (tid < kStages) mbar_init(&sm.empty[tid], 4 * tiles_n);
        if (tid == 0) {
            mbar_init(&sm.got_query, 1);
            mbar_init(&sm.got_scores, 1);
            mbar_init(&sm.got_feat, 1);
            mbar_init(&sm.got_parts, 1);
            sm.pre_min = 0xffffffffu;
            sm.pre_max = 0u;
            sm.list_n = sm.tile_n = sm.few_n = 0;
            sm.no_list = 0;
        }
        mbar_fence_init();
        if (tid == 0) {
            if constexpr (GATE) mbar_arrive_expect_tx(&sm.got_query, (uint32_t)(q_len * (DG ? DG : ga.g.d_gate) * 6));
            mbar_arrive_expect_tx(&sm.got_parts, (uint32_t)(rows * kHeadDim * 4 + S * rows * 8));
        }
    }
    // (another CTA's shared memory is written only after the barrier this opens: it is then known to be running, and its
    // mbarriers are initialised)
    cluster_arrive();
    if (producer && lane == 0 && !ALONE) {
        tma_prefetch_desc(&map_k);
        tma_prefetch_desc(&map_v);
    }

    int n_blocks = 0, L = 0;                               // listed blocks of the unit, cached tokens
    constexpr int kSubs = SMALL ? 4 : 1;                   // most blocks of a tile
    int entry[kSubs] = {};                                 // !GATE: the list's entries of this lane's first tile
    bool dead = false;                                     // a wait ran out: go through the motions, the results are invalid
    if constexpr (GATE) {
        const GateParams& g = ga.g;
        const int d_gate = DG ? DG : g.d_gate;
        const int n = g.group * kHeadDim, half = d_gate / 2;
        const unsigned char* kc = reinterpret_cast<const unsigned char*>(g.kcomp + (size_t)u * g.max_blocks * d_gate);
        // Gate query: a CTA makes the rotary pairs (c, c + d_gate/2) c_first .. c_first + ppc of all query tokens, by MMAs of 16
        // rows of W_q (eight pairs) by 8 tokens; the contraction, in units of 32 channels, is split over the warps that share
        // a row tile (`slices` of them), whose partial sums meet in shared memory.  A lane holds pieces of 16 bytes as they lie
        // in memory (channels 8 * (lane % 4) .. of a unit): the contraction index is permuted, in W_q and x alike.  What bounds
        // it is the way of the first bytes and, for several query tokens, was the arithmetic: with a warp per pair and token by
        // FMA the queries of four tokens were there after 7.2 us, now after 3.3.  (Each MMA begins at zero and
        // the rotation is in double: against 64 bits the scores are off by 7.4e-8 of their norm, by FMA 1.17e-7.)
        // How the units are dealt to warps depends on the cluster's size, and the scores shall not: a sequence's lists are the
        // same whatever the batch around it.  The units' sums are therefore added up in double, which is exact, in any order,
        // as long as none is 2^24 times another; beyond that the order is 2^-53 of the sum and all but never seen in fp32.
        const int ppc = half >> s_shift, c_first = rank * ppc;
        const int mt_shift = 31 - __clz(min((ppc + 7) >> 3, NW)), slices = NW >> mt_shift, slice = warp >> mt_shift;
        const int row8 = lane >> 2, units = n / 32;
        uint4 wa[4], wb[4], xx[4];
        auto load_w = [&](int m0, int u0) {
            const int pair = 8 * (m0 + (warp & ((1 << mt_shift) - 1))) + row8;
            const uint4* w = reinterpret_cast<const uint4*>(g.w_q + ((size_t)h * d_gate + c_first + min(pair, ppc - 1)) * n) + (lane & 3);
            const uint4* x = reinterpret_cast<const uint4*>(
                g.q_nope + (((size_t)i * q_len + min(row8, q_len - 1)) * g.num_q_heads + (size_t)h * g.group) * kHeadDim) + (lane & 3);
            const size_t step = (size_t)half * n / 8;
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                const int un = u0 + k * slices;
                if (un >= units) break;
                wa[k] = pair < ppc ? __ldg(w + 4 * un) : make_uint4(0u, 0u, 0u, 0u);
                wb[k] = pair < ppc ? __ldg(w + 4 * un + step) : make_uint4(0u, 0u, 0u, 0u);
                xx[k] = row8 < q_len ? __ldg(x + 4 * un) : make_uint4(0u, 0u, 0u, 0u);
            }
        };
        // (W_q into L2 only, which follows later writes: the kernel before this one may be the one that makes it)
        if (producer && lane < 2) prefetch_l2(g.w_q + ((size_t)h * d_gate + c_first + lane * half) * n, 2 * n * ppc);
        float* sc_all = reinterpret_cast<float*>(sm.ring);
        auto& gs = *reinterpret_cast<typename Place::Scratch*>(sm.ring + Place::kScratch);
        if (!producer) {
            for (int x = tid; x < kBins; x += kWorkers) gs.hist[x] = 0;
        }
        pdl_wait();                                        // queries, lengths and compressed keys are final
        if (ALONE && p.next_early) pdl_launch_dependents();     // (the gate alone has no work for which it wants the SMs)
        L = p.seq_lens[i];
        // (what the second round of loads reads of the queries, if there is one)
        if (producer && lane < q_len && units > 4 * slices)
            prefetch_l2(g.q_nope + (((size_t)i * q_len + lane) * g.num_q_heads + (size_t)h * g.group) * kHeadDim, 2 * n);
        if (!producer) load_w(0, slice);
        const int b_shift = 31 - __clz(g.block_size);
        const int n_i = L > 0 ? (L + g.block_size - 1) >> b_shift : 0;
        // the blocks that hold a query token's own position, j_f .. n_i - 1 (one, the last, for a single token), are always
        // taken; the candidates are those before them
        const int j_f = max(0, L - q_len) >> b_shift;
        int n_forced = min(n_i - j_f, g.max_sel);
        int n_cand = min(j_f, g.max_blocks);
        const bool appends = !ALONE && g.k_nope && blockIdx.z == 0 && L >= g.block_size && (L & (g.block_size - 1)) < q_len && (L >> b_shift) <= g.max_blocks;
        int need = 0;                                      // (threshold method: known once the scores are)
        if (n_i > 0 && !(ALONE && g.threshold_mode)) {
            const int k = min(max(g.token_budget >> b_shift, 1), min(n_i, g.max_sel));
            // (kListed: only a sequence longer than max_seq_len, which the host's rule went by, gets that far)
            need = max(0, min(min(k - n_forced, n_cand), kListed));
            n_blocks = need + n_forced;
        }
        // This CTA's key tiles: a run of those with a candidate.  The producer warp asks for as many as there are slots for, so
        // that they travel while the gate query is made.
        const int n_tiles = (n_cand + kKeyTile - 1) / kKeyTile, per_cta = (n_tiles + S - 1) >> s_shift;
        const int tile0 = min(rank * per_cta, n_tiles), my_tiles = min(per_cta, n_tiles - tile0);
        KeySlots slots;
        // (the queries' parts: those of the last q_len of kMaxQLen places, so that the keys have what is in front of them)
        const int t_skip = MULTI ? kMaxQLen - q_len : 0;
        uint32_t (*parts)[3][kMaxDGate / 2 + 16] = gs.parts + t_skip;
        slots.place(sm.ring, n_tiles, Place::kScratch + t_skip * (int)sizeof(gs.parts[0]), d_gate);
        const bool attends = KIND == SPREAD_STEP ? !step_uneven(p, S) : !ALONE;
        // who selects: every CTA that will read tiles, or (the gate alone) the first one
        const int n_sel = attends ? S : 1, sel_shift = attends ? s_shift : 0;
        const bool selects = rank < n_sel;
        if (producer) {
            // (the scores of the other CTAs' key tiles, and from every CTA their smallest and largest key)
            if (selects && lane == 0) mbar_arrive_expect_tx(&sm.got_scores, (uint32_t)((n_tiles - my_tiles) * kKeyTile * 4 + S * 8));
            if (appends && lane < 3) {
                if (lane == 0) mbar_arrive_expect_tx(&sm.got_feat, 3 * kHeadDim * 4);
                else prefetch_l2(g.w_k + ((size_t)h * d_gate + c_first + (lane - 1) * half) * 3 * kHeadDim, ppc * 3 * kHeadDim * 2);
            }
        }
        cluster_wait();                                    // every CTA of the cluster has started
        if (producer) {
            if (lane < min(my_tiles, slots.n)) {
                const int j = kKeyTile * (tile0 + lane);
                slots.request(lane, &sm.key_full[lane], kc + ((size_t)j << (slots.shift - 3)), g.max_blocks - j);
            }
        }
        // ---- gate query ------------------------------------------------------------------------------------------------
        if (!producer) {
            auto part = sm.sums;
            for (int m0 = 0; 8 * m0 < ppc; m0 += NW) {
                if (m0 > 0) {
                    worker_sync<NW>();                     // (the partial sums have been read)
                    load_w(m0, slice);
                }
                double acc[4] = {0., 0., 0., 0.};
#pragma unroll 1
                for (int u0 = slice;;) {
#pragma unroll
                    for (int k = 0; k < 4; ++k) {
                        if (u0 + k * slices >= units) break;
                        const uint32_t a0[4] = {wa[k].x, wb[k].x, wa[k].y, wb[k].y}, a1[4] = {wa[k].z, wb[k].z, wa[k].w, wb[k].w};
                        float c0[4] = {0.f, 0.f, 0.f, 0.f}, c1[4] = {0.f, 0.f, 0.f, 0.f};
                        mma_bf16_16816(c0, a0, xx[k].x, xx[k].y);
                        mma_bf16_16816(c1, a1, xx[k].z, xx[k].w);
#pragma unroll
                        for (int c = 0; c < 4; c += MULTI ? 1 : 2) acc[c] += (double)(c0[c] + c1[c]);      // (one token: column 0)
                    }
                    u0 += 4 * slices;
                    if (u0 >= units) break;
                    load_w(m0, u0);
                }
                if constexpr (MULTI) {
                    *reinterpret_cast<double2*>(&part[warp][row8][2 * (lane & 3)]) = make_double2(acc[0], acc[1]);
                    *reinterpret_cast<double2*>(&part[warp][row8 + 8][2 * (lane & 3)]) = make_double2(acc[2], acc[3]);
                } else if ((lane & 3) == 0) {
                    part[warp][row8][0] = acc[0];
                    part[warp][row8 + 8][0] = acc[2];
                }
                worker_sync<NW>();
                // a thread per pair, token and CTA that gets them
                const int np_shift = 31 - __clz(min(ppc, 8 << mt_shift));
#pragma unroll 1
                for (int x = tid; x < (q_len << (np_shift + s_shift)); x += kWorkers) {
                    const int to = x & (S - 1), pr = (x >> s_shift) & ((1 << np_shift) - 1), t = x >> (s_shift + np_shift);
                    const int c = c_first + 8 * m0 + pr;
                    double sn, cs;                         // query token t sits at position L - q_len + t
                    rope_sincos_wide((double)max(L - q_len + t, 0), g.inv_freq[c], &sn, &cs);
                    double a = 0., b = 0.;
#pragma unroll
                    for (int sl = 0; sl < NW; ++sl) {
                        if (sl >= slices) break;
                        a += part[(sl << mt_shift) + (pr >> 3)][pr & 7][t];
                        b += part[(sl << mt_shift) + (pr >> 3)][(pr & 7) + 8][t];
                    }
                    // A thread has channels c and c + d_gate/2, its neighbour S lanes on the ones next to them (c is even here and
                    // odd there, or the other way round): the even one sends the words of the lower two channels, the other
                    // one those of the upper two.
                    float f0 = (float)(a * cs - b * sn), f1 = (float)(b * cs + a * sn);
                    const bool upper = pr & 1;
                    const float got = __shfl_xor_sync(0xffffffffu, upper ? f0 : f1, S);
                    if (upper) f0 = got;
                    else f1 = got;
                    const uint32_t dst = cluster_addr(&parts[t][0][(c >> 1) + (upper ? half >> 1 : 0)], to), bar = cluster_addr(&sm.got_query, to);
#pragma unroll
                    for (int k = 0; k < 3; ++k) {
                        const uint32_t w = pack_bf16x2_toward_zero(f0, f1);
                        send_u32(dst + k * (uint32_t)sizeof(gs.parts[0][0]), w, bar);
                        const float2 r = bf16x2_to_float2(w);
                        // (each difference is exact: it has the bits behind the eight cut off, at most sixteen; what is not finite
                        // has no rest, and what is finite stays it)
                        f0 = fabsf(r.x) < INFINITY ? f0 - r.x : 0.f;
                        f1 = fabsf(r.y) < INFINITY ? f1 - r.y : 0.f;
                    }
                }
            }
        }
        // ---- scores, into the shared memory of the CTAs that select ------------------------------------------------
        // (keys through L2, not the read-only path: the entry that this launch appends, or the step before it did, is among them)
        uint32_t kmn = 0xffffffffu, kmx = 0u;              // smallest and largest key of this warp's scores
        auto scores = [&](auto xs_c) {
            constexpr int XS = decltype(xs_c)::value;
            const float inv = rsqrtf((float)d_gate);
            // this lane's first piece of its first key in slot 0; the second key is kOff bytes behind the first
            const int rr = lane >> 2, k_of = 8 * (rr & 1) + (rr >> 1) + 4 * (lane & 1);
            const unsigned char* at = ((rr & 1) ? slots.b : slots.a) + (rr >> 1) * (64 * XS) + 16 * (lane & 3);
            constexpr int kOff = 4 * (64 * XS);
            int slot = warp, use = 0;
            bool asked = false;
#pragma unroll 1
            for (int m = warp < slots.n ? warp : my_tiles;;) {
                const bool mine = m < my_tiles;
                const int j0 = kKeyTile * (tile0 + m), j = j0 + k_of;
                const unsigned char* here = at + (slot << slots.shift);
                auto in_slot = [&](int x, uint4& lo, uint4& hi) {
                    lo = *reinterpret_cast<const uint4*>(here + 64 * x);
                    hi = *reinterpret_cast<const uint4*>(here + kOff + 64 * x);
                };
                auto refill = [&]() {
                    __syncwarp();                          // (all lanes have read the slot)
                    if (lane == 0 && m + slots.n < my_tiles) {
                        const int jn = j0 + kKeyTile * slots.n;
                        fence_proxy_async_smem();
                        slots.request(slot, &sm.key_full[slot], kc + (size_t)jn * (64 * XS), g.max_blocks - jn);
                    }
                };
                uint4 held[2 * XS];                        // (not of 256 channels, which would be half of the thread's registers)
                if (mine) {
                    if (__any_sync(0xffffffffu, !mbar_wait(&sm.key_full[slot], use & 1, p.status))) {
                        dead = true;
                        break;
                    }
                    if constexpr (XS < 8) {
#pragma unroll
                        for (int x = 0; x < XS; ++x) in_slot(x, held[2 * x], held[2 * x + 1]);
                        refill();
                    }
                }
                if (!asked) {                              // (the first keys are there before the queries are)
                    asked = true;
                    if (!wait_sent(&sm.got_query, p.status)) dead = true;
                }
                if (!mine) break;
                float v0, v1;
                bool odd0, odd1;
                if constexpr (XS < 8) {
                    key_sums<XS, MULTI>([&](int x, uint4& lo, uint4& hi) { lo = held[2 * x]; hi = held[2 * x + 1]; }, parts, q_len, lane, v0, v1, odd0, odd1);
                } else {
                    key_sums<XS, MULTI>(in_slot, parts, q_len, lane, v0, v1, odd0, odd1);
                    refill();
                }
                // lane 4r has the score of row r, lane 4r + 1 (the others alike) that of row r + 8
                float v = (lane & 1) ? v1 : v0;
                // (only of keys that are candidates: behind them is whatever the cache or the slot holds, which has no part in this)
                const int j_lo = j0 + 8 * (rr & 1) + (rr >> 1);
                odd0 &= j_lo < n_cand;
                odd1 &= j_lo + 4 < n_cand;
                if (__any_sync(0xffffffffu, odd0 | odd1)) {
                    const unsigned odds0 = __ballot_sync(0xffffffffu, odd0), odds1 = __ballot_sync(0xffffffffu, odd1);
#pragma unroll 1
                    for (int k = 0; k < kKeyTile; ++k) {
                        if ((((k & 4) ? odds1 : odds0) >> (4 * (2 * (k & 3) + (k >> 3)))) & 15u) {
                            const float x = score_key_plain(reinterpret_cast<const uint4*>(kc + (size_t)(j0 + k) * (64 * XS)), parts, q_len, d_gate, lane);
                            if (k == k_of) v = x;
                        }
                    }
                }
                v *= inv;
                if ((lane & 2) == 0) {
                    const bool ok = j < n_cand;
                    sc_all[j] = ok ? v : -INFINITY;
                    if (ok) {
                        if (ALONE && g.scores_user) g.scores_user[(size_t)u * g.max_blocks + j] = v;
                        const uint32_t key = score_key(v);
                        kmn = min(kmn, key);
                        kmx = max(kmx, key);
                    }
                }
                slot += NW;
                m += NW;
                if (slot >= slots.n) {                     // (the tile behind the last slot's comes in slot 0)
                    m += slots.n + warp - slot;
                    slot = warp;
                    ++use;
                }
            }
        };
        if (!producer) {
            if (d_gate == 128) scores(std::integral_constant<int, 4>());
            else if (d_gate == 64) scores(std::integral_constant<int, 2>());
            else scores(std::integral_constant<int, 8>());
            kmn = __reduce_min_sync(0xffffffffu, kmn);
            kmx = __reduce_max_sync(0xffffffffu, kmx);
            if (lane == 0) { sm.warp_min[warp] = kmn; sm.warp_max[warp] = kmx; }
            worker_sync<NW>();
            // four scores at a time to the others (a lane each to sixteen CTAs, the scores of 8 units of 15625 keys took 5 us
            // longer to arrive)
            const int to = (tid >> 3) & (n_sel - 1);       // (eight lanes: a line of one CTA's)
            if (to != rank) {
                const uint32_t dst = cluster_addr(sc_all + kKeyTile * tile0, to), bar = cluster_addr(&sm.got_scores, to);
#pragma unroll 1
                for (int c = 8 * (tid >> (3 + sel_shift)) + (tid & 7); c < 4 * my_tiles; c += kWorkers >> sel_shift)
                    send_f32x4(dst + 16 * c, *reinterpret_cast<const float4*>(sc_all + kKeyTile * tile0 + 4 * c), bar);
            }
            if (warp == 0) {
                kmn = __reduce_min_sync(0xffffffffu, lane < NW ? sm.warp_min[lane] : 0xffffffffu);
                kmx = __reduce_max_sync(0xffffffffu, lane < NW ? sm.warp_max[lane] : 0u);
                if (lane < n_sel) {
                    const uint32_t bar = cluster_addr(&sm.got_scores, lane);
                    send_min(cluster_addr(&sm.pre_min, lane), kmn, bar);
                    send_max(cluster_addr(&sm.pre_max, lane), kmx, bar);
                }
            }
        }
        // ---- selection ---------------------------------------------------------------------------------------------
        if (selects && !producer) {
            int32_t* dst = g.block_idx + (size_t)u * g.max_sel;
            const bool lists = rank == 0 && blockIdx.z == 0;     // this CTA writes the caller's list, too
            // (a wait that has run out for one thread has for all: no list then, and the producer warp is told)
            dead = worker_any<NW>(!wait_sent(&sm.got_scores, p.status) || dead);
            if (dead) n_cand = need = n_forced = n_blocks = 0;
            if (dead && tid == 0) sm.no_list = 1;
            if (ALONE && g.threshold_mode) {
                // Threshold method (Sec. 3.1): softmax of the scores over the candidates; those above tau are the `above`
                // highest-scoring ones (equal scores have equal probabilities), so only the number differs
                auto sum_all = [&](float v) -> float {
#pragma unroll
                    for (int off = 16; off > 0; off >>= 1) v += __shfl_xor_sync(0xffffffffu, v, off);
                    worker_sync<NW>();                     // (the scratch may still be in use)
                    if (lane == 0) sm.warp_red[warp] = v;
                    worker_sync<NW>();
                    float r = 0.f;
#pragma unroll
                    for (int w2 = 0; w2 < NW; ++w2) r += sm.warp_red[w2];
                    return r;
                };
                const float mx = key_score(sm.pre_max);
                auto weight = [&](int j) { const float s = sc_all[j]; return s == s ? __expf(s - mx) : 0.f; };     // (NaN: as minus infinity)
                float z = 0.f, above = 0.f;
#pragma unroll 4
                for (int j = tid; j < n_cand; j += kWorkers) z += weight(j);
                z = sum_all(z);
#pragma unroll 4
                for (int j = tid; j < n_cand; j += kWorkers) above += weight(j) > g.threshold * z ? 1.f : 0.f;
                need = max(0, min(min((int)(sum_all(above) + 0.5f), g.max_sel - n_forced), min(n_cand, kListed)));
                n_blocks = n_i > 0 ? need + n_forced : 0;
            }
            // entry e of the list is block j: its tile(s) among this CTA's, if they are
            auto take = [&](int e, int j) {
                if (lists) dst[e] = j;
                if (!attends) return;
                if constexpr (!SMALL) {
                    for (int x = 0; x < p.tiles_per_block; ++x) {
                        const int t = (e << p.tpb_shift) + x;
                        if ((t & (S - 1)) == rank && (t >> s_shift) < kCodes) sm.codes[t >> s_shift] = (j << p.tpb_shift) + x;
                    }
                } else {
                    const int t = e >> p.bpt_shift, at = ((t >> s_shift) << p.bpt_shift) + (e & (p.blocks_per_tile - 1));
                    if ((t & (S - 1)) == rank && at < kCodes) sm.codes[at] = j;
                }
            };
            Selected& sl = *reinterpret_cast<Selected*>(sm.ring + Place::kSelected);
            int e0 = 0;                                    // entries that are in place
            if (need > 0 && need < n_cand) {
                Selection<NW, Smem> sel(sm, gs.hist, sc_all, n_cand, need, warp, lane);
                if (sel.finite && (n_cand <= 4 * kWorkers    ? sel.template in_registers<1>(take)
                                   : n_cand <= 8 * kWorkers  ? sel.template in_registers<2>(take)
                                   : n_cand <= 16 * kWorkers ? sel.template in_registers<4>(take)
                                                             : false))
                    e0 = need;
                else
                    select_many<NW>(&sm, gs.hist, &sl, sc_all, n_cand, need);
            }
            // the others: the list's, or every candidate; behind them the blocks taken without a score
#pragma unroll 1
            for (int e = e0 + tid; e < n_blocks; e += kWorkers)
                take(e, e >= need ? n_i - n_blocks + e : need < n_cand ? (int)sl.list[e] : e);
            if (lists) {
                if (tid == 0) g.block_cnt[u] = n_blocks;
                for (int e = n_blocks + tid; e < g.max_sel; e += kWorkers) dst[e] = -1;
            }
        }
        if (!attends) {                                  // the gate alone
            if (!ALONE && appends) {
                if (producer) append_pool(g, sm, i, h, (L >> b_shift) - 1, rank, S);
                else if (!dead) append_project<NW>(g, sm, u, h, (L >> b_shift) - 1, rank, S);
            }
            cluster_sync();                                // (as at the end)
            return;
        }
        fence_proxy_async_smem();                          // the ring's memory goes over to the copy engine
        if (producer) {
            // (nothing in this step reads the entry of the block that has just filled)
            if (appends) append_pool(g, sm, i, h, (L >> b_shift) - 1, rank, S);
            tiles_listed_wait<NW>();
            if (sm.no_list) n_blocks = 0;
        } else {
            tiles_listed_arrive<NW>();
            if (appends && !dead) append_project<NW>(g, sm, u, h, (L >> b_shift) - 1, rank, S);
        }
    } else {
        pdl_wait();
        // (the first entries are asked for beside the count that says how many there are, not behind it)
        if (producer && p.block_idx) {
            const int t = (lane << s_shift) + rank;
#pragma unroll
            for (int x = 0; x < kSubs; ++x) {
                const int e = SMALL ? (t << p.bpt_shift) + x : t >> p.tpb_shift;
                if (x < p.blocks_per_tile) entry[x] = p.block_idx[(size_t)u * p.max_sel + min(e, p.max_sel - 1)];
            }
        }
        L = p.seq_lens[i];
        if (p.block_idx) {
            const int cnt = p.block_cnt ? p.block_cnt[u] : p.max_sel;      // (not behind the test on L: both loads in flight)
            n_blocks = L > 0 ? max(0, min(cnt, p.max_sel)) : 0;
        }
        __syncthreads();                                   // barriers initialised
    }

    // ---- tiles ------------------------------------------------------------------------------------------------------
    const bool dense = !GATE && !p.block_idx;
    constexpr bool small = SMALL;
    const int T = dense ? (L > 0 ? min((L + kTileTokens - 1) / kTileTokens, p.max_blocks_cap) : 0)
                        : small ? (n_blocks + p.blocks_per_tile - 1) >> p.bpt_shift : n_blocks << p.tpb_shift;
    const int n_mine = (max(0, T - rank) + S - 1) >> s_shift;
    const int n_local = GATE ? min(n_mine, small ? kCodes >> p.bpt_shift : kCodes) : n_mine;     // (the host's rule keeps within kCodes)
    // output row of this cluster's row r: query token (row0 + r) / group, head (row0 + r) % group of the unit's
    auto out_row = [&](int r) -> size_t {
        const int tl = MULTI ? ((row0 + r) * p.group_magic) >> 16 : 0;
        return ((size_t)i * q_len + tl) * p.num_q_heads + (size_t)h * p.group + (row0 + r - tl * p.group);
    };
    const int qd = lane & 3, rw = lane >> 2;
    if (producer) {
        if (p.next_early) pdl_launch_dependents();
        if (GATE && n_local < n_mine && lane == 0) raise_status(p.status, DEV_BAD_INDEX);      // (a sequence longer than max_seq_len: tiles are left out)
        const int n_i = (L + p.block_size - 1) >> p.bs_shift;
        for (int base = 0; base < n_local; base += 32) {
            const int it = base + lane;
            int row[kSubs] = {}, outer[kSubs] = {}, nv_all = 0, n_sub = 0;
            if (it < n_local) {
                const int t = (it << s_shift) + rank;
                const int n_try = small ? p.blocks_per_tile : 1;
                const int span = small ? p.block_size : kTileTokens;
#pragma unroll
                for (int x = 0; x < kSubs; ++x) {
                    if (x < n_try) {
                        int tok0 = -1;
                        if (dense) {
                            tok0 = t * kTileTokens;
                        } else if (small) {
                            const int e = (t << p.bpt_shift) + x;
                            if (e < n_blocks) {
                                const int blk = GATE ? sm.codes[(it << p.bpt_shift) + x] : base == 0 ? entry[x] : p.block_idx[(size_t)u * p.max_sel + e];
                                if (!GATE && blk >= n_i) raise_status(p.status, DEV_BAD_INDEX);
                                if (blk >= 0 && blk < n_i) tok0 = blk << p.bs_shift;
                            }
                        } else if (GATE) {
                            tok0 = sm.codes[it] * kTileTokens;
                            if ((unsigned)tok0 >= (unsigned)(n_i << p.bs_shift)) {     // (never: the lists are this kernel's own)
                                raise_status(p.status, DEV_BAD_INDEX);
                                tok0 = -1;
                            }
                        } else {
                            const int blk = base == 0 ? entry[0] : p.block_idx[(size_t)u * p.max_sel + (t >> p.tpb_shift)];
                            if (blk >= n_i) raise_status(p.status, DEV_BAD_INDEX);
                            if (blk >= 0 && blk < n_i) tok0 = (blk << p.bs_shift) + (t & (p.tiles_per_block - 1)) * kTileTokens;
                        }
                        // (counted beyond the tile, so that earlier query tokens can be cut off)
                        int nv = tok0 >= 0 ? max(0, min(span + (MULTI ? kMaxQLen - 1 : 0), L - tok0)) : 0;
                        if (nv > 0) {
                            outer[x] = i;
                            row[x] = tok0;
                            if (p.page_table) {
                                const int pg = p.page_table[(size_t)i * p.page_table_stride + tok0 / p.page_size];
                                outer[x] = pg;
                                row[x] = tok0 % p.page_size;
                                if (pg < 0 || pg >= p.num_pages) { raise_status(p.status, DEV_BAD_INDEX); nv = 0; }
                            }
                        }
                        nv_all |= nv << (8 * x);
                        n_sub += nv > 0;
                    }
                }
            }
            __syncwarp();
            // Tile s of the batch, which lane s has looked up.  With up to sixteen copies a tile (blocks of 16 or 32 tokens) an
            // elected lane asks for them (see elect_one: 77 units, three query tokens, blocks of 16: 93.4 -> 82 us); with four
            // lane s itself, as handing over what it knows takes longer (one sequence of 32k 13.4, elected 13.65).
            const int m = min(32, n_local - base);
            for (int s = 0; s < m; ++s) {
                const int n = base + s, st = n % kStages;
                unsigned char* dst = sm.ring + st * kStageBytes;
                uint64_t* full = &sm.full[n % kArrivals];
                if constexpr (SMALL) {
                    const int nv = __shfl_sync(0xffffffffu, nv_all, s), subs = __shfl_sync(0xffffffffu, n_sub, s);
                    int r[4], o[4];
#pragma unroll
                    for (int x = 0; x < 4; ++x) {
                        r[x] = __shfl_sync(0xffffffffu, row[x], s);
                        o[x] = __shfl_sync(0xffffffffu, outer[x], s);
                    }
                    if (!dead && !mbar_wait(&sm.empty[st], ((n / kStages) & 1) ^ 1, p.status)) dead = true;
                    dead = __any_sync(0xffffffffu, dead);
                    if (elect_one()) {
                        sm.meta[n % kArrivals] = nv;       // (the tile kArrivals back has been read: the one kStages back has, which came after it)
                        if (dead || subs == 0) {
                            mbar_arrive(full);
                        } else {
                            const int sub_bytes = p.block_size * 128;      // one half (64 channels) of one block
                            mbar_arrive_expect_tx(full, (uint32_t)(subs * 4 * sub_bytes));
#pragma unroll
                            for (int x = 0; x < 4; ++x) {
                                if ((nv >> (8 * x)) & 0xff) {
                                    unsigned char* d2 = dst + x * sub_bytes;
                                    tma_load_4d(d2, &map_k, full, 0, r[x], h, o[x]);
                                    tma_load_4d(d2 + kHalfTileBytes, &map_k, full, 64, r[x], h, o[x]);
                                    tma_load_4d(d2 + kTileBytes, &map_v, full, 0, r[x], h, o[x]);
                                    tma_load_4d(d2 + kTileBytes + kHalfTileBytes, &map_v, full, 64, r[x], h, o[x]);
                                }
                            }
                        }
                    }
                } else if (lane == s) {
                    if (!dead && !mbar_wait(&sm.empty[st], ((n / kStages) & 1) ^ 1, p.status)) dead = true;
                    sm.meta[n % kArrivals] = nv_all;
                    if (dead || n_sub == 0) {
                        mbar_arrive(full);
                    } else {
                        mbar_arrive_expect_tx(full, kStageBytes);
                        tma_load_4d(dst, &map_k, full, 0, row[0], h, outer[0]);
                        tma_load_4d(dst + kHalfTileBytes, &map_k, full, 64, row[0], h, outer[0]);
                        tma_load_4d(dst + kTileBytes, &map_v, full, 0, row[0], h, outer[0]);
                        tma_load_4d(dst + kTileBytes + kHalfTileBytes, &map_v, full, 64, row[0], h, outer[0]);
                    }
                }
                __syncwarp();
            }
        }
        if (!GATE) cluster_wait();                         // (the barrier opened at the top)
        cluster_arrive_relaxed();
    } else {
        const int group = warp >> 2, my_n = MULTI ? group % tiles_n : 0, pace = MULTI ? group / tiles_n : group;
        // Q^T B-fragments: this thread supplies row 8 * my_n + rw of the unit's queries
        uint32_t bq[8][2];
        {
            const int r = 8 * my_n + rw;
            const uint32_t* qrow = reinterpret_cast<const uint32_t*>(p.q + out_row(r < rows ? r : 0) * kHeadDim);
#pragma unroll
            for (int ks = 0; ks < 8; ++ks) {
                bq[ks][0] = r < rows ? __ldg(qrow + 8 * ks + qd) : 0u;
                bq[ks][1] = r < rows ? __ldg(qrow + 8 * ks + 4 + qd) : 0u;
            }
        }
        // newest cached tokens that the query tokens of this thread's two rows (columns of S^T) may not see
        int back[2] = {0, 0};
        if (MULTI) {
#pragma unroll
            for (int c = 0; c < 2; ++c) {
                const int r = 8 * my_n + 2 * qd + c;
                if (r < rows) back[c] = q_len - 1 - (((row0 + r) * p.group_magic) >> 16);
            }
        }
        if (p.next_early) pdl_launch_dependents();
        const int w4 = warp & 3;                           // which 16 of a tile's tokens
        float o[8][4], m_run[2] = {-INFINITY, -INFINITY}, l_run[2] = {0.f, 0.f};
#pragma unroll
        for (int a = 0; a < 8; ++a) o[a][0] = o[a][1] = o[a][2] = o[a][3] = 0.f;
        // lane-constant parts of the ldmatrix addresses (swizzle: 16-B chunk ^= row & 7)
        const int k_row = 16 * w4 + ((lane >> 3) & 1) * 8 + (lane & 7), k_csel = lane >> 4;
        const int v_row = 16 * w4 + ((lane >> 4) & 1) * 8 + (lane & 7), v_csel = (lane >> 3) & 1;
        const int sw = lane & 7;
        // blocks of 16 or 32 tokens: which of the gathered blocks this warp's rows belong to, and where in it
        const int sub_w = !small ? 0 : p.block_size == 16 ? w4 : w4 >> 1;
        const int off_w = !small ? 16 * w4 : p.block_size == 16 ? 0 : (w4 & 1) * 16;
        for (int it = pace < paces ? pace : n_local; it < n_local; it += paces) {
            const int st = it % kStages;
            if (!dead && !mbar_wait(&sm.full[it % kArrivals], (it / kArrivals) & 1, p.status)) dead = true;
            const int nvw = (small ? (sm.meta[it % kArrivals] >> (8 * sub_w)) & 0xff : sm.meta[it % kArrivals]) - off_w;   // valid tokens from this warp's first row on
            if (nvw > 0 && !dead) {
                const uint32_t kbase = smem_u32(sm.ring + st * kStageBytes), vbase = kbase + kTileBytes;
                if (nvw < 16) {
                    // ragged tail: rows past the sequence end may hold anything; this warp's are cleared in V, so that
                    // a zero probability times garbage cannot produce NaN
                    unsigned char* vt = sm.ring + st * kStageBytes + kTileBytes;
                    for (int x = lane; x < (16 - nvw) * 16; x += 32) {
                        const int r = 16 * w4 + nvw + (x >> 4), part = x & 15;
                        *reinterpret_cast<uint4*>(vt + (part >> 3) * kHalfTileBytes + r * 128 + ((part & 7) << 4)) = make_uint4(0u, 0u, 0u, 0u);
                    }
                    fence_proxy_async_smem();
                    __syncwarp();
                }
                // ---- S^T = K . Q^T (four short accumulator chains) ----
                float sa[4][4];
#pragma unroll
                for (int x = 0; x < 4; ++x) sa[x][0] = sa[x][1] = sa[x][2] = sa[x][3] = 0.f;
#pragma unroll
                for (int ks = 0; ks < 8; ++ks) {
                    uint32_t a[4];
                    const int c8 = ((2 * ks) & 7) + k_csel;
                    ldmatrix_x4(a, kbase + (ks >> 2) * kHalfTileBytes + k_row * 128 + ((c8 ^ sw) << 4));
                    mma_bf16_16816(sa[ks & 3], a, bq[ks][0], bq[ks][1]);
                }
                float s[4];
#pragma unroll
                for (int x = 0; x < 4; ++x) s[x] = ((sa[0][x] + sa[1][x]) + (sa[2][x] + sa[3][x])) * p.scale_log2;
                const int lim0 = nvw - back[0], lim1 = nvw - back[1];      // tokens that a row sees of this warp's 16
                if (rw >= lim0) s[0] = -INFINITY;
                if (rw >= lim1) s[1] = -INFINITY;
                if (rw + 8 >= lim0) s[2] = -INFINITY;
                if (rw + 8 >= lim1) s[3] = -INFINITY;
                // ---- online softmax over this warp's 16 tokens, per row (column of S^T) ----
                float mx0 = fmaxf(s[0], s[2]), mx1 = fmaxf(s[1], s[3]);
#pragma unroll
                for (int off = 4; off < 32; off <<= 1) {
                    mx0 = fmaxf(mx0, __shfl_xor_sync(0xffffffffu, mx0, off));
                    mx1 = fmaxf(mx1, __shfl_xor_sync(0xffffffffu, mx1, off));
                }
                const float mn0 = fmaxf(m_run[0], mx0), mn1 = fmaxf(m_run[1], mx1);
                // a row that has seen nothing so far keeps max = -inf; exponents are then taken against 0
                const float mb0 = mn0 == -INFINITY ? 0.f : mn0, mb1 = mn1 == -INFINITY ? 0.f : mn1;
                const float al0 = fast_exp2(m_run[0] - mb0), al1 = fast_exp2(m_run[1] - mb1);
                const bool same_max = __all_sync(0xffffffffu, m_run[0] == mn0 && m_run[1] == mn1);
                m_run[0] = mn0;
                m_run[1] = mn1;
                const float p0 = fast_exp2(s[0] - mb0), p1 = fast_exp2(s[1] - mb1);
                const float p2 = fast_exp2(s[2] - mb0), p3 = fast_exp2(s[3] - mb1);
                l_run[0] = l_run[0] * al0 + (p0 + p2);
                l_run[1] = l_run[1] * al1 + (p1 + p3);
                if (!same_max) {
#pragma unroll
                    for (int a = 0; a < 8; ++a) { o[a][0] *= al0; o[a][1] *= al1; o[a][2] *= al0; o[a][3] *= al1; }
                }
                const uint32_t b0 = movmatrix_trans(pack_bf16x2(p0, p1));      // tokens 0-7 of the slice
                const uint32_t b1 = movmatrix_trans(pack_bf16x2(p2, p3));      // tokens 8-15
                // ---- O^T += V^T . P^T ----
#pragma unroll
                for (int a = 0; a < 8; ++a) {
                    uint32_t f[4];
                    const int c8 = ((2 * a) & 7) + v_csel;
                    ldmatrix_x4_trans(f, vbase + (a >> 2) * kHalfTileBytes + v_row * 128 + ((c8 ^ sw) << 4));
                    mma_bf16_16816(o[a], f, b0, b1);
                }
            }
            __syncwarp();
            if (lane == 0) mbar_arrive(&sm.empty[st]);
        }
        // ---- combine: warps, then CTAs ------------------------------------------------------------------------------
#pragma unroll
        for (int off = 4; off < 32; off <<= 1) {
            l_run[0] += __shfl_xor_sync(0xffffffffu, l_run[0], off);
            l_run[1] += __shfl_xor_sync(0xffffffffu, l_run[1], off);
        }
        worker_sync<NW>();                                     // every tile has been read: the ring is free
        float* part = reinterpret_cast<float*>(sm.ring) + warp * 8 * kMergeStride;
#pragma unroll
        for (int a = 0; a < 8; ++a) {
            const int d0 = 16 * a + rw;
            part[2 * qd * kMergeStride + d0] = o[a][0];
            part[(2 * qd + 1) * kMergeStride + d0] = o[a][1];
            part[2 * qd * kMergeStride + d0 + 8] = o[a][2];
            part[(2 * qd + 1) * kMergeStride + d0 + 8] = o[a][3];
        }
        if (rw == 0) {
            sm.warp_ml[warp][2 * qd] = make_float2(m_run[0], l_run[0]);
            sm.warp_ml[warp][2 * qd + 1] = make_float2(m_run[1], l_run[1]);
        }
        __syncwarp();
        if (!GATE) cluster_wait();                         // every CTA of the cluster has started (the barrier opened at the top)
        worker_sync<NW>();
        const int c_shift = 7 - s_shift;                   // log2 of the channels of a CTA's slice
        // a warp per row; lane: four channels
        for (int r = warp; r < rows; r += NW) {
            const int c = 4 * lane, n_part = 4 * paces;    // the warps that have a share of row r
            float M = -INFINITY, l = 0.f;
            float2 ml[NW];
            auto warp_of = [&](int x) { return MULTI ? ((x >> 2) * tiles_n + (r >> 3)) * 4 + (x & 3) : x; };
#pragma unroll
            for (int x = 0; x < NW; ++x) {
                ml[x] = x < n_part ? sm.warp_ml[warp_of(x)][r & 7] : make_float2(-INFINITY, 0.f);
                M = fmaxf(M, ml[x].x);
            }
            float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
            const float* src = reinterpret_cast<const float*>(sm.ring) + (r & 7) * kMergeStride + c;
#pragma unroll
            for (int x = 0; x < NW; ++x) {
                if (x < n_part) {
                    const float f = ml[x].x == -INFINITY ? 0.f : fast_exp2(ml[x].x - M);
                    const float4 v = *reinterpret_cast<const float4*>(src + warp_of(x) * 8 * kMergeStride);
                    l = fmaf(ml[x].y, f, l);
                    acc.x = fmaf(v.x, f, acc.x);
                    acc.y = fmaf(v.y, f, acc.y);
                    acc.z = fmaf(v.z, f, acc.z);
                    acc.w = fmaf(v.w, f, acc.w);
                }
            }
            const int to = c >> c_shift;
            send_f32x4(cluster_addr(sm.recv_o + (((rank * kRows + r) << c_shift) | (c & ((1 << c_shift) - 1))), to), acc, cluster_addr(&sm.got_parts, to));
            if (lane < S) send_f32x2(cluster_addr(&sm.recv_ml[rank][r], lane), make_float2(M, l), cluster_addr(&sm.got_parts, lane));
        }
    }
    if (!producer) {
        wait_sent(&sm.got_parts, p.status);
        cluster_arrive_relaxed();                          // (all that was sent to this CTA is here)
        const int c_shift = 7 - s_shift;
        const int pairs = rows << (c_shift - 1);           // channel pairs of this CTA's slice, all rows
#pragma unroll 1
        for (int x = tid; x < pairs; x += kWorkers) {
            const int r = x >> (c_shift - 1), c = 2 * (x & ((1 << (c_shift - 1)) - 1));
            float M = -INFINITY, l = 0.f, a0 = 0.f, a1 = 0.f;
            float2 ml[kMaxS];
#pragma unroll
            for (int s = 0; s < kMaxS; ++s) {
                ml[s] = s < S ? sm.recv_ml[s][r] : make_float2(-INFINITY, 0.f);
                M = fmaxf(M, ml[s].x);
            }
#pragma unroll
            for (int s = 0; s < kMaxS; ++s) {
                if (s < S) {
                    const float f = ml[s].x == -INFINITY ? 0.f : fast_exp2(ml[s].x - M);
                    const float2 v = *reinterpret_cast<const float2*>(&sm.recv_o[((s * kRows + r) << c_shift) + c]);
                    l = fmaf(ml[s].y, f, l);
                    a0 = fmaf(v.x, f, a0);
                    a1 = fmaf(v.y, f, a1);
                }
            }
            const float inv = l > 0.f ? 1.f / l : 0.f;
            const size_t row = out_row(r);
            *reinterpret_cast<uint32_t*>(p.out + row * kHeadDim + (rank << c_shift) + c) = pack_bf16x2(a0 * inv, a1 * inv);
            if (p.lse && rank == 0 && c == 0) p.lse[row] = l > 0.f ? (M + log2f(l)) * 0.6931471805599453f : -INFINITY;
        }
    }
    // No CTA leaves before every one has received all that was sent to it: neither the receiver's shared memory nor the
    // sender's place in the cluster may be gone while a store is under way.
    cluster_wait();
}

template <int NW, bool MULTI, typename Kernel>
cudaError_t configure(Kernel* kernel) {
    cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(StepSmem<NW, MULTI>) + 1024);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(kernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    return e;
}

template <int NW, bool MULTI>
cudaLaunchConfig_t config_of(int S, int units, int parts, cudaStream_t stream, cudaLaunchAttribute (&attr)[2]) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(S, units, parts);
    cfg.blockDim = dim3(Size<NW, MULTI>::kThreads);
    cfg.dynamicSmemBytes = sizeof(StepSmem<NW, MULTI>) + 1024;
    cfg.stream = stream;
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = S;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 2;
    return cfg;
}

constexpr int wide_gate(Kind kind) { return kind == GATE_ALONE ? 256 : 0; }

template <int NW, Kind KIND, bool MULTI, bool SMALL, int DG>
int resident_of(int k) {
    const auto kernel = step_cluster_kernel<NW, KIND, MULTI, SMALL, DG>;
    if (configure<NW, MULTI>(kernel) != cudaSuccess) return 0;
    cudaLaunchAttribute attr[2];
    cudaLaunchConfig_t cfg = config_of<NW, MULTI>(1 << k, 1, 1, nullptr, attr);
    cfg.numAttrs = 1;
    int n = 0;
    if (cudaOccupancyMaxActiveClusters(&n, kernel, &cfg) != cudaSuccess) n = 0;
    cudaGetLastError();                                    // (a refused size is no error of the caller's)
    return n;
}
template <int NW, Kind KIND, bool MULTI, bool SMALL>
int resident_of(int k) {
    if constexpr (KIND == LISTS || MULTI) return resident_of<NW, KIND, MULTI, SMALL, 0>(k);
    else return min(resident_of<NW, KIND, MULTI, SMALL, 64>(k), min(resident_of<NW, KIND, MULTI, SMALL, 128>(k), resident_of<NW, KIND, MULTI, SMALL, wide_gate(KIND)>(k)));
}
template <int NW, Kind KIND, bool MULTI>
int resident_of(int k) {
    return min(resident_of<NW, KIND, MULTI, false>(k), resident_of<NW, KIND, MULTI, true>(k));
}

// Clusters of 2^k CTAs that the device holds at once (`wide`: of the NW = 16 kernels), asked once per device; 0: the
// device or the driver does not take such clusters.
int resident_clusters(bool wide, int k) {
    static int cached[kMaxDevices][2][5];                  // (value + 1; 0: not asked yet.  A race asks twice and stores the same)
    int& c = cached[current_device_slot()][wide][k];
    if (c == 0) {
        c = wide ? min(resident_of<16, STEP, true>(k), resident_of<16, LISTS, true>(k)) + 1
                 : min(min(min(resident_of<8, STEP, false>(k), resident_of<8, SPREAD_STEP, false>(k)),
                           min(resident_of<8, STEP, true>(k), resident_of<8, LISTS, true>(k))),
                       min(resident_of<8, GATE_ALONE, false, false>(k), resident_of<8, GATE_ALONE, true, false>(k))) + 1;
    }
    return c - 1;
}

}  // namespace

// As many CTAs per unit as keep every cluster resident at once (a second wave would double the call) and still have
// something to do each.  Measured against the kernels of long calls, us a call (a step's append included):
//     step, 8 KV heads, budget 4096, 1 / 2 / 4 sequences     23.3 -> 16.9, 25.3 -> 19.8, 31.6 -> 28.8
//     step of batch 8 at 128k, 205 blocks (51 tiles a CTA)   98.4 -> 85.0
//     (as the step was when these were measured; its gate's parts have become shorter since)
//     four query tokens, 20 rows, 4 sequences, budget 4096   63.2 -> 38.6;  64 rows 92.3 -> 75.2;  8 rows, 1 sequence 27.2 -> 19.0
//     threshold gate alone in front of given lists, 4 sequences of 48k, blocks of 32: 42.5 -> 35.0 with both
// A cluster's CTAs go through their unit's tiles by themselves; the decode kernel's CTAs share all tiles.  The rule sees
// the longest list that there can be, not how uneven the lists are, and one long sequence among short ones leaves most
// clusters idle.  us a call, decode kernel -> clusters, 8 KV heads; one sequence's lists long / half of them / all, by the
// tiles a CTA of a long one:
//     lists, 16 sequences, 20 rows (S = 1)
//                                    16: 21.6 -> 18.8 / 27.6 -> 19.3 / 25.7 -> 20.1    32: 22.4 -> 30.7 / 39.7 -> 32.1 / 56.3 -> 33.5
//     steps, 16 sequences (S = 2)    64: 31.7 -> 46.8 / 72.3 -> 58.6 / 103 -> 93      128: 45.3 -> 82.7 / 108 -> 103 / 178 -> 173
//             8 sequences (S = 4)    64: 35.6 -> 47.4 / 69.6 -> 56.6 / 101 -> 91      128: 57.1 -> 80.6 / 105 -> 101 / 176 -> 172
// Given lists and dense calls of several query tokens, whose lengths follow the sequences', keep to where one long sequence
// does not lose much: 16 + 2 S tiles a CTA (a decode call pays for its parts whatever its size, and more the longer its
// longest unit is; lists of one query token are dealt: seer_lists.cu).  The lists of a step are all as long as the budget but for
// sequences shorter than that: one launch up to 64 tiles a CTA, where all but the most uneven batches gain.  So do 80 units in
// 160 CTAs, although twelve SMs have two of them; chain -> one launch, lists all long / spread evenly from an eighth on / half of the
// sequences' long, the others an eighth / a quarter long / one / one among nearly empty ones:
//     48 tiles a CTA    69.5 -> 53.8 / 62.8 -> 45.7 / 52.5 -> 42.4 / 40.4 -> 38.7 / 34.0 -> 37.4 / 27.6 -> 34.5
//     64                81.9 -> 65.6 / 69.8 -> 54.5 / 62.1 -> 50.7 / 46.5 -> 46.6 / 39.8 -> 46.0 / 33.1 -> 43.3
//     48, two tokens    72.8 -> 55.5 / 65.7 -> 47.7 / 54.5 -> 44.5 / 41.4 -> 40.3 / 36.2 -> 39.1 / 27.7 -> 36.0
// (The list kernel behind them as well, from 32 tiles a CTA on: 59.9 / 51.4 / 48.8 / 40.8 / 37.1 / 29.4 for 48, 71.8 / 60.1 / 60.2 / 48.3 /
// 43.1 / 32.7 for 64: six microseconds for all, for a gain in the last two.)  From there to 128 tiles (line_spread: one query
// token) it is the sequences' lengths that decide, in the kernels: even lists are done in the one launch, uneven ones by the list
// kernel behind it, which costs 5 us where it has nothing to do.  Chain -> two launches:
//     80, 8 sequences   124 -> 115 / 99.2 -> 88.0 / 88.2 -> 77.4 / 67.3 -> 59.3 / 53.3 -> 51.6 / 47.2 -> 41.1
//     96, 10 sequences  102 -> 96.7 / 86.4 -> 82.4 / 74.9 -> 73.2 / 54.3 -> 59.2 / 46.9 -> 49.1 / 38.2 -> 37.5
//     96, 16 sequences  146 -> 138 / 122 -> 111 / 98.9 -> 92.1 / 75.8 -> 75.6 / 55.7 -> 55.8 / 42.3 -> 39.4
// 149 to 296 units, a CTA each, gain like fewer: steps of 24 / 30 / 36 sequences, all long, 16 tiles a CTA 45.9 -> 33.8, 52.7 ->
// 39.1, 59.3 -> 43.1; 64 tiles 93.5 -> 82.1, 108 -> 96, 127 -> 109.
static StepPlan plan_of(bool wide, int units, int rows, long long max_tiles, long long max_codes, int max_keys, bool line_spread = false) {
    StepPlan plan = {0, 1, rows, wide, false, false};
    if (rows > 64) return plan;
    if (rows > 32) {
        plan.parts = (rows + 31) / 32;
        plan.rows = (rows + plan.parts - 1) / plan.parts;
    }
    units *= plan.parts;
    for (int k = 4; k >= 0; --k) {
        const int S = 1 << k;
        if (k > 0 && S > max_tiles && 128ll * S > max_keys) continue;      // a CTA would have nothing to do
        if (units > resident_clusters(wide, k)) continue;
        const long long line = (long long)S * (max_keys > 0 ? 64 : min(16 + 2 * S, 64));
        plan.spread = line_spread && max_tiles > line && max_tiles <= (long long)S * kListTiles;
        if ((max_tiles <= line || plan.spread) && max_codes <= (long long)S * kCodes) plan.S = S;
        // The next launch may start beside this one if both fit at once.  Otherwise its first clusters take places that the
        // last ones then lack: half the steps of 32 ragged units, in clusters of eight, had one to four clusters in a second
        // wave, 13 us late (mean 23.8 -> 22.6 us; threshold gate and lists 28.4 -> 27.8, batch 8 at 128k 82.7 -> 81.0).
        plan.next_early = 2 * units <= resident_clusters(wide, k);
        break;
    }
    return plan;
}

// Which of the two sizes.  Above 16 rows there is only the one of 16 warps.  One query token takes eight warps whatever the
// number of keys: two CTAs an SM make clusters twice as large, or twice as many units resident.  (With 16 warps above 8192
// keys a step of 8 units of 15625 keys and 625 blocks went to the kernels of long calls: 119 us, now 63; so did 200 units of
// 9375 keys, 233 and 142, and 192 units of short sequences in a cache of 16384 keys, 184 and 47; 16 units of 9375 took 50 and take
// 36, 96 took 153 and take 96.)  Several query tokens' parts leave the keys less room, which costs where the scores take most of
// it: 16 warps above 8192 keys where their clusters have eight CTAs or more (two tokens, 8 units of 15625: 36.3 -> 33.8; but 16
// units of 9375, in clusters of four, 36.6 -> 44.5).
StepPlan step_plan(int units, int rows, int q_len, long long max_tiles, long long max_codes, int max_keys) {
    if (rows <= 16) {
        if (q_len > 1 && max_keys > 8192) {
            const StepPlan plan = plan_of(true, units, rows, max_tiles, max_codes, max_keys);
            if (plan.S >= 8) return plan;
        }
        return plan_of(false, units, rows, max_tiles, max_codes, max_keys, q_len == 1 && max_keys > 0);
    }
    return plan_of(true, units, rows, max_tiles, max_codes, max_keys);
}

namespace {

template <int NW, bool MULTI, bool SMALL>
cudaError_t launch_of(const CUtensorMap& map_k, const CUtensorMap& map_v, const DecodeParams& p, const GateParams* g, const StepPlan& plan,
                      cudaStream_t stream) {
    cudaLaunchAttribute attr[2];
    const cudaLaunchConfig_t cfg = config_of<NW, MULTI>(plan.S, p.num_units, plan.parts, stream, attr);
    auto launch = [&](auto kind, auto multi, auto dg) {
        return cudaLaunchKernelEx(&cfg, step_cluster_kernel<NW, decltype(kind)::value, decltype(multi)::value, SMALL, decltype(dg)::value>, map_k, map_v, p,
                                  GateArg<true>{*g});
    };
    auto launch_gate = [&](auto kind, auto multi) {
        if constexpr (MULTI) return launch(kind, multi, std::integral_constant<int, 0>());
        else return g->d_gate == 64    ? launch(kind, multi, std::integral_constant<int, 64>())
                    : g->d_gate == 128 ? launch(kind, multi, std::integral_constant<int, 128>())
                                       : launch(kind, multi, std::integral_constant<int, wide_gate(decltype(kind)::value)>());
    };
    using Multi = std::integral_constant<bool, MULTI>;
    if (g) {
        if constexpr (NW == 8 && !SMALL)
            if (!p.q) return launch_gate(std::integral_constant<Kind, GATE_ALONE>(), Multi());
        if constexpr (!MULTI)
            if (plan.spread) return launch_gate(std::integral_constant<Kind, SPREAD_STEP>(), Multi());
        return launch_gate(std::integral_constant<Kind, STEP>(), Multi());
    }
    if constexpr (MULTI) return cudaLaunchKernelEx(&cfg, step_cluster_kernel<NW, LISTS, true, SMALL, 0>, map_k, map_v, p, GateArg<false>{});
    return cudaErrorInvalidValue;                          // (lists of one query token: seer_lists.cu)
}
template <int NW, bool MULTI>
cudaError_t launch_of(const CUtensorMap& map_k, const CUtensorMap& map_v, const DecodeParams& p, const GateParams* g, const StepPlan& plan,
                      cudaStream_t stream) {
    return p.block_idx && p.blocks_per_tile > 1 ? launch_of<NW, MULTI, true>(map_k, map_v, p, g, plan, stream)
                                                : launch_of<NW, MULTI, false>(map_k, map_v, p, g, plan, stream);
}

}  // namespace

cudaError_t launch_step_cluster(const CUtensorMap& map_k, const CUtensorMap& map_v, const DecodeParams& p, const GateParams* g,
                                const StepPlan& plan, cudaStream_t stream) {
    if (plan.wide) return launch_of<16, true>(map_k, map_v, p, g, plan, stream);
    return p.q_len == 1 ? launch_of<8, false>(map_k, map_v, p, g, plan, stream) : launch_of<8, true>(map_k, map_v, p, g, plan, stream);
}

bool launch_gate_cluster(const GateParams& p, cudaStream_t stream, cudaError_t* err) {
    if (p.scores_in || p.list_flags || !gate_one_kernel(p.max_blocks)) return false;
    const StepPlan plan = step_plan(p.batch * p.num_kv_heads, 1, 1, 0, 0, p.max_blocks);
    if (plan.S == 0) return false;
    CUtensorMap none;
    DecodeParams d;
    memset(&none, 0, sizeof none);
    memset(&d, 0, sizeof d);
    d.seq_lens = p.seq_lens;
    d.num_kv_heads = p.num_kv_heads;
    d.num_units = p.batch * p.num_kv_heads;
    d.group = p.group;
    d.q_len = p.q_len;
    d.rows = plan.rows;
    d.next_early = plan.next_early;
    d.status = p.status;
    *err = launch_step_cluster(none, none, d, &p, plan, stream);
    return true;
}

}  // namespace seer
