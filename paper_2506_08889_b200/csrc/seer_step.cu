// Short decode calls: one thread-block cluster per (sequence, KV head) unit does everything, in one launch.
//
// The chain of kernels that serves long calls (seer_gate.cu, seer_decode.cu) spends, on a short one, most of its
// time between its parts: lists through global memory, a schedule over all units, partial results published with
// a fence and a ticket and read back by the last CTA.  Here the S CTAs (S = 1 .. 16) of a unit's cluster share
// the unit from its first byte to its output:
//   1. gate (GATE): the unit's gate query, spread over the cluster's warps, into every CTA's shared memory; the
//      scores of the CTA's keys into the first CTA's; selection there; every listed tile's number into the
//      shared memory of the CTA that will read it (tile t belongs to CTA t mod S);
//      meanwhile other CTAs of the cluster compress the block that has just filled, if one has;
//      list (!GATE): the CTA reads its tiles' numbers from the caller's list, or counts them off (dense);
//   2. tiles: one producer warp keeps a ring of three 64-token K/V stages in flight; eight consumer warps, two
//      groups of four, take alternate tiles, a warp 16 tokens (the same tensor-core steps as decode_kernel);
//   3. combine: the warps' partials meet in shared memory, the CTA's go, a slice of the channels each, to the
//      cluster's CTAs, which write their slice of the output after one cluster barrier.
// Nothing between the steps leaves the SMs, and no CTA waits for another except at the cluster's hardware barrier.
#include <cooperative_groups.h>

#include "seer_gate_device.cuh"
#include "seer_internal.h"

namespace cg = cooperative_groups;

namespace seer {

namespace {

constexpr int kHalfTileBytes = kTileTokens * 128;          // 64 rows x 128 B (64 bf16 channels)
constexpr int kTileBytes = 2 * kHalfTileBytes;             // one K or V tile: 16 KiB
constexpr int kStageBytes = 2 * kTileBytes;                // K + V
constexpr int kMaxS = 16;
constexpr int kCodes = 256;                                // tile (or gathered block) numbers that a CTA holds
constexpr int kListed = kStageBytes / 4;                   // scored blocks that the first CTA's list holds
constexpr int kBins = 1024;                                // histogram of the selection
constexpr int kMergeStride = 132;                          // floats per row of a warp's partial (bank spread)
constexpr int kBatch = 8;                                  // 16-byte pieces of compressed keys per thread in flight
constexpr int kChunkKeys = 32;                             // keys are dealt to the cluster's CTAs in runs of 32
constexpr int kMaxQLen = 8;

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
    // K/V ring.  Before the first tile is asked for, the gate's: the scores of the unit (first CTA; up to
    // kStepMaxBlocks) in stages 0 and 1, the staged first batch of keys behind them, the list of the taken blocks in
    // its place later.  After the last tile: the warps' partials.
    unsigned char ring[Z::kStages][kStageBytes];
    // What the gate uses until the lists are out, and what arrives from the cluster's CTAs after their last tile.
    union {
        float qg[MULTI ? kMaxQLen : 1][kMaxDGate];         // gate queries
        __align__(16) float recv_o[Z::kRows * kHeadDim];   // [source CTA][row][this CTA's slice of the channels]
    };
    union {
        __align__(16) int hist[kBins + 4];                 // selection (first CTA); the one past the last is for nobody
        float2 recv_ml[kMaxS][Z::kRows];                   // [source CTA][row]: max, sum
    };
    float2 warp_ml[NW][8];
    // Tile n arrives in stage n % kStages and is announced on full[n % kArrivals].  The consumer groups that share a
    // tile's rows take all of one residue of the tile numbers, at their own pace, and every barrier belongs to one
    // residue, so its groups follow all of its phases.  (With a barrier per stage a group would miss the others' phases
    // and could take one that is two back for the one that it waits for.)
    uint64_t full[Z::kArrivals], empty[Z::kStages];
    int meta[Z::kArrivals];                                // tokens from the tile's first row on (blocks of 16 or 32 tokens: per block, 8 bits each)
    int codes[kCodes];                                     // GATE: this CTA's tiles: 64-token tile numbers, or the gathered blocks
    // selection (first CTA)
    int warp_tot[NW];
    float warp_red[NW];
    uint32_t list_key[32];
    int list_j[32];
    float feat[3 * kHeadDim];                              // pooled features of the block that has just filled
    uint32_t pre_min, pre_max;                             // smallest and largest key of a candidate
    uint32_t prefix;
    int rem, bin_cnt, list_n, last_eq;
};
static_assert(sizeof(StepSmem<8, true>) + 1024 <= 113 * 1024, "two CTAs per SM");
static_assert(sizeof(StepSmem<16, true>) + 1024 <= 227 * 1024, "one CTA per SM");
static_assert(kStepMaxBlocks * 4 <= 2 * kStageBytes && kBatch * 256 * 16 <= kStageBytes && kBatch * 512 * 16 <= 3 * kStageBytes, "the gate's use of the ring");
static_assert(kCodes * kMaxS <= kListed, "the list behind the scores");

template <int NW>
__device__ __forceinline__ void worker_sync() { asm volatile("bar.sync 1, %0;" ::"n"(32 * NW) : "memory"); }

template <bool GATE>
struct GateArg { GateParams g; };
template <>
struct GateArg<false> {};

// The selection of the token budget's `need` best of the candidates [0, n_cand), by the first CTA's worker warps.
// Leaves (thr, j_eq): candidate j is taken if its key is above thr, or equal to it and j <= j_eq.  Comparisons only:
// the lower block number wins a tie, NaN is below every number.  A histogram over a monotone linear map of
// [min, max] leaves a few candidates in the boundary bin, which every warp ranks for itself; crowded bins and ranges
// that are not finite take radix passes over key - min instead.
template <int NW, typename Smem>
__device__ __forceinline__ void select_threshold(Smem& sm, const float* sc, int n_cand, int need, int words, int warp, int lane,
                                                 uint32_t& thr, int& j_eq) {
    const int tid = 32 * warp + lane;
    if (need >= n_cand) { thr = 0u; j_eq = 0x7fffffff; return; }
    if (need <= 0) { thr = 0xffffffffu; j_eq = -1; return; }
    const uint32_t kmin = sm.pre_min, kmax = sm.pre_max;
    const float smin = key_score(kmin), smax = key_score(kmax);
    const float range = smax - smin, scale = (kBins - 1.f) / range;
    const int j0 = warp * words * 32 + lane;               // this lane's candidates: j0, j0 + 32, ...
    // (four at a time, without branches: their loads go out together)
    auto each = [&](auto&& fn) {
#pragma unroll 1
        for (int e = 0; e < words; e += 4) {
            float v[4];
#pragma unroll
            for (int x = 0; x < 4; ++x) v[x] = sc[min(j0 + 32 * (e + x), n_cand - 1)];
#pragma unroll
            for (int x = 0; x < 4; ++x) fn((e + x < words) & (j0 + 32 * (e + x) < n_cand), score_key(v[x]), j0 + 32 * (e + x));
        }
    };
    // The same for passes in any order, on the scores themselves: neighbouring blocks have similar scores, so the lanes of
    // a warp take candidates that are far apart (lane l has run l of `run` blocks, from its own place in it on: no bank
    // conflicts); side by side, their additions to the histogram would queue for a few bins.
    const int run = (n_cand + 31) / 32, rot = (run & 1) ? 0 : lane % run;
    auto each_spread = [&](auto&& fn) {
#pragma unroll 1
        for (int q = warp; q < run; q += 4 * NW) {
            float v[4];
            int jj[4];
#pragma unroll
            for (int x = 0; x < 4; ++x) {
                int at = q + x * NW + rot;
                at -= at >= run ? run : 0;
                jj[x] = q + x * NW < run ? min(lane * run + at, n_cand) : n_cand;      // (n_cand: none)
                v[x] = sc[min(jj[x], n_cand - 1)];
            }
            fn(v, jj);
        }
    };
    // thread t owns a few bins, from kBins-1-kPer*t downwards: finds the bin that straddles the rem-th best key
    constexpr int kPer = kBins / (32 * NW);
    auto find_bin = [&](int rem) {
        worker_sync<NW>();
        int c[kPer], mine = 0;
#pragma unroll
        for (int x = 0; x < kPer; ++x) { c[x] = sm.hist[kBins - 1 - kPer * tid - x]; mine += c[x]; }
        int incl = mine;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int t = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += t;
        }
        if (lane == 31) sm.warp_tot[warp] = incl;
        worker_sync<NW>();
        int above = incl - mine;
#pragma unroll
        for (int w2 = 0; w2 < NW; ++w2) above += w2 < warp ? sm.warp_tot[w2] : 0;
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
    };
    if (smin > -INFINITY && range > 0.f && range < INFINITY && scale < INFINITY) {
        // (every score is finite here; -0 and +0 have the same bin)
        auto bin_of = [&](float s, int j) -> int { return j < n_cand ? min(kBins - 1, (int)((s - smin) * scale)) : kBins; };
        each_spread([&](const float (&v)[4], const int (&j)[4]) {
#pragma unroll
            for (int x = 0; x < 4; ++x) atomicAdd(&sm.hist[bin_of(v[x], j[x])], 1);
        });
        find_bin(need);
        const int bin = (int)sm.prefix, rem = sm.rem, cnt = sm.bin_cnt;
        if (cnt <= 32) {
            each_spread([&](const float (&v)[4], const int (&j)[4]) {
                bool in[4], any = false;
#pragma unroll
                for (int x = 0; x < 4; ++x) any |= in[x] = bin_of(v[x], j[x]) == bin;
                if (any) {
#pragma unroll
                    for (int x = 0; x < 4; ++x) {
                        if (in[x]) {
                            const int slot = atomicAdd(&sm.list_n, 1);
                            sm.list_key[slot] = score_key(v[x]);
                            sm.list_j[slot] = j[x];
                        }
                    }
                }
            });
            worker_sync<NW>();
            const uint32_t key = lane < cnt ? sm.list_key[lane] : 0u;
            const int j = lane < cnt ? sm.list_j[lane] : 0x7fffffff;
            int rank = 0;
            for (int m = 0; m < cnt; ++m) {
                const uint32_t km = __shfl_sync(0xffffffffu, key, m);
                const int jm = __shfl_sync(0xffffffffu, j, m);
                rank += km > key || (km == key && jm < j);
            }
            const int src = __ffs(__ballot_sync(0xffffffffu, lane < cnt && rank == rem - 1)) - 1;
            thr = __shfl_sync(0xffffffffu, key, src);
            j_eq = __shfl_sync(0xffffffffu, j, src);
            return;
        }
    }
    // radix passes of ten bits over key - kmin
    int bits_left = 32 - __clz(max(kmax - kmin, 1u)), rem = need;
    uint32_t prefix = 0u;
    while (bits_left > 0) {
        const int wbits = min(10, bits_left), shift = bits_left - wbits;
#pragma unroll
        for (int x = 0; x < kPer; ++x) sm.hist[kPer * tid + x] = 0;
        worker_sync<NW>();
        each([&](bool ok, uint32_t key, int) {
            const uint32_t rel = key - kmin;
            if (ok && (uint32_t)((unsigned long long)rel >> (shift + wbits)) == prefix)        // (shift + wbits can be 32)
                atomicAdd(&sm.hist[(rel >> shift) & ((1u << wbits) - 1u)], 1);
        });
        find_bin(rem);
        prefix = (prefix << wbits) | sm.prefix;
        rem = sm.rem;
        bits_left = shift;
    }
    thr = kmin + prefix;
    // the rem-th candidate whose key equals thr, in block order (a warp's candidates are one run of blocks)
    int n_eq = 0;
    each([&](bool ok, uint32_t key, int) { n_eq += __popc(__ballot_sync(0xffffffffu, ok && key == thr)); });
    worker_sync<NW>();                                         // (everybody has read the last pass's totals)
    if (lane == 0) sm.warp_tot[warp] = n_eq;
    worker_sync<NW>();
    int before = 0;
#pragma unroll
    for (int w2 = 0; w2 < NW; ++w2) before += w2 < warp ? sm.warp_tot[w2] : 0;
    if (before < rem && rem <= before + n_eq) {
        each([&](bool ok, uint32_t key, int j) {
            const bool eq = ok && key == thr;
            const unsigned m = __ballot_sync(0xffffffffu, eq);
            if (eq && before + __popc(m & ((1u << lane) - 1u)) == rem - 1) sm.last_eq = j;
            before += __popc(m);
        });
    }
    worker_sync<NW>();
    j_eq = sm.last_eq;
}

// The compressed key of block j of the unit, which has just filled, by warps 0..7 of some of the cluster's CTAs: part
// `part` of `parts` of the rotary pairs.  The same sums in the same order as seer_kcomp.cu's append, so the same entry.
// (256 threads meet at barrier 2.)
__device__ __forceinline__ void append_block(const GateParams& g, float* feat, int u, int i, int h, int j, int part, int parts) {
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int b = g.block_size, half = g.d_gate / 2;
    uint4 wv[4][2];
    auto load_rows = [&](int pair) {                       // rows of W_k[h] of the rotary pairs `pair`, `pair` + 1
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const int r = min(pair + (k & 1), half - 1) + (k >> 1) * half;
            const uint4* wrow = reinterpret_cast<const uint4*>(g.w_k + ((size_t)h * g.d_gate + r) * 3 * kHeadDim);
            wv[k][0] = __ldg(wrow + lane);
            wv[k][1] = lane < 16 ? __ldg(wrow + 32 + lane) : make_uint4(0u, 0u, 0u, 0u);
        }
    };
    const int first = 2 * (part * 8 + warp), step = 2 * 8 * parts;
    if (first < half) load_rows(first);
    // warp: 16 channels; lane: eight of them, rows lane / 2, lane / 2 + 16, ...
    const int c8 = 2 * warp + (lane & 1), rg = lane >> 1;
    const __nv_bfloat16* src = g.k_nope + (size_t)i * g.k_stride_batch + (size_t)h * g.k_stride_head +
                               (g.k_rows_block_local ? 0 : (size_t)j * b) * g.k_stride_token + 8 * c8;
    __nv_bfloat162 mx[4], mn[4];
    float sum[8];
#pragma unroll
    for (int c = 0; c < 4; ++c) { mx[c] = __float2bfloat162_rn(-INFINITY); mn[c] = __float2bfloat162_rn(INFINITY); }
#pragma unroll
    for (int c = 0; c < 8; ++c) sum[c] = 0.f;
#pragma unroll 4
    for (int r = rg; r < b; r += 16) {
        const uint4 v = *reinterpret_cast<const uint4*>(src + (size_t)r * g.k_stride_token);
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
            feat[8 * c8 + 2 * c] = a.x;
            feat[8 * c8 + 2 * c + 1] = a.y;
            feat[kHeadDim + 8 * c8 + 2 * c] = d.x;
            feat[kHeadDim + 8 * c8 + 2 * c + 1] = d.y;
        }
#pragma unroll
        for (int c = 0; c < 8; ++c) feat[2 * kHeadDim + 8 * c8 + c] = sum[c];
    }
    asm volatile("bar.sync 2, 256;" ::: "memory");
    __nv_bfloat16* dst = const_cast<__nv_bfloat16*>(g.kcomp) + ((size_t)u * g.max_blocks + j) * g.d_gate;
    for (int pair = first; pair < half; pair += step) {
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
        if (pair + step < half) load_rows(pair + step);
#pragma unroll
        for (int k = 0; k < 4; ++k)
#pragma unroll
            for (int off = 16; off > 0; off >>= 1) acc[k] += __shfl_xor_sync(0xffffffffu, acc[k], off);
        if (lane < 2 && pair + lane < half) {
            const int c = pair + lane;
            const float a = lane ? acc[1] : acc[0], d = lane ? acc[3] : acc[2];
            float sn, cs;
            rope_sincos((double)j * (double)b, g.inv_freq[c], &sn, &cs);
            dst[c] = __float2bfloat16(a * cs - d * sn);
            dst[c + half] = __float2bfloat16(d * cs + a * sn);
        }
    }
}

// grid (S, units), cluster (S, 1, 1).  Short calls are bound by latency: a step of 8 units x 64 blocks (16.8 MB, 2.6 us at
// memory speed) takes 14.5 us.  Time stamps in the kernel (which make it a microsecond or two longer; medians over the CTAs,
// from the first read on) put 1.9 us on the gate query, 1.0 on the barrier behind it, 3.7 on the scores, 0.6 on the barrier,
// 1.5 on the selection, 2.1 on the lists and their barrier, 2.6 on the tiles, 1.0 on the warps' combine, 1.0 on the barrier,
// 0.9 on the output.  Longer ones by memory: of a step of 64 units x 205 blocks (430 MB; 83.5 us) the tiles take 66 us,
// 6.5 TB/s, from the first CTA's first to the last one's last; CTAs that share a unit read neighbouring blocks at the same time.
template <int NW, bool GATE, bool MULTI>
__global__ void __launch_bounds__(Size<NW, MULTI>::kThreads, NW == 8 ? 2 : 1)
step_cluster_kernel(const __grid_constant__ CUtensorMap map_k, const __grid_constant__ CUtensorMap map_v,
                    const __grid_constant__ DecodeParams p, const __grid_constant__ GateArg<GATE> ga) {
    using Z = Size<NW, MULTI>;
    using Smem = StepSmem<NW, MULTI>;
    constexpr int kWorkers = Z::kWorkers, kStages = Z::kStages, kArrivals = Z::kArrivals, kRows = Z::kRows;
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
    // (another CTA's shared memory is written only after the barrier this opens: it is then known to be running)
    cluster_arrive();
    if (tid < kArrivals) {
        mbar_init(&sm.full[tid], 1);
        if (tid < kStages) mbar_init(&sm.empty[tid], 4 * tiles_n);
        mbar_fence_init();
    }
    if (producer && lane == 0 && p.q) {
        tma_prefetch_desc(&map_k);
        tma_prefetch_desc(&map_v);
    }

    int n_blocks = 0, L = 0;                               // listed blocks of the unit, cached tokens
    if constexpr (GATE) {
        const GateParams& g = ga.g;
        const int n = g.group * kHeadDim, chunks = n / 8, half = g.d_gate / 2;
        const int nit = (chunks + 31) / 32;                // 16-byte pieces of a W_q row per lane (1..4)
        const int gw = rank * NW + warp, n_gw = S * NW;
        const int lpk_shift = g.d_gate == 64 ? 3 : g.d_gate == 128 ? 4 : 5, lpk = 1 << lpk_shift;   // lanes per key
        const int csub = tid & (lpk - 1);
        const uint4* kc = reinterpret_cast<const uint4*>(g.kcomp + (size_t)u * g.max_blocks * g.d_gate);
        // this CTA's key number lk (runs of kChunkKeys, dealt round robin) is block
        auto block_of = [&](int lk) { return (((lk / kChunkKeys) << s_shift) + rank) * kChunkKeys + (lk & (kChunkKeys - 1)); };
        // Rotary pairs (c, c + d_gate/2) of the gate query are dealt to the cluster's warps; with more warps than pairs
        // several of them take a pair, for every t_step-th query token each.
        const int c_step = min(n_gw, half), t_step = max(1, n_gw / half), t_first = gw / half, c_first = gw % half;
        uint4 wv[2][4];
        auto load_w = [&](int c) {
#pragma unroll
            for (int k = 0; k < 2; ++k) {
                const uint4* wrow = reinterpret_cast<const uint4*>(g.w_q + ((size_t)h * g.d_gate + c + k * half) * n);
#pragma unroll
                for (int it = 0; it < 4; ++it) {
                    const int ch = lane + 32 * it;
                    wv[k][it] = it < nit && ch < chunks ? __ldg(wrow + ch) : make_uint4(0u, 0u, 0u, 0u);
                }
            }
        };
        // (W_q into L2 only, which follows later writes: the kernel before this one may be the one that makes it)
        if (!producer && t_first < q_len && lane < 2) prefetch_l2(g.w_q + ((size_t)h * g.d_gate + c_first + lane * half) * n, 2 * n);
        if (rank == 0) {
            for (int x = tid; x < kBins; x += Z::kThreads) sm.hist[x] = 0;
            if (tid == 0) { sm.pre_min = 0xffffffffu; sm.pre_max = 0u; sm.list_n = 0; }
        }
        pdl_wait();                                        // queries, lengths and compressed keys are final
        if (!p.q) pdl_launch_dependents();                 // (the gate alone has no work for which it wants the SMs)
        L = p.seq_lens[i];
        uint4 xv[4];
        auto load_x = [&](int t) {
            const uint4* xsrc = reinterpret_cast<const uint4*>(
                g.q_nope + (((size_t)i * q_len + t) * g.num_q_heads + (size_t)h * g.group) * kHeadDim);
#pragma unroll
            for (int it = 0; it < 4; ++it) {
                const int ch = lane + 32 * it;
                xv[it] = it < nit && ch < chunks ? __ldg(xsrc + ch) : make_uint4(0u, 0u, 0u, 0u);
            }
        };
        const int all_chunks = (g.max_blocks + kChunkKeys - 1) / kChunkKeys;
        const int total_cap = ((max(0, all_chunks - rank) + S - 1) >> s_shift) << (lpk_shift + 5);    // pieces, block numbers past the cache among them
        uint4* staged = reinterpret_cast<uint4*>(sm.ring[2]);      // [kBatch * kWorkers]
        float* sc_all = reinterpret_cast<float*>(sm.ring[0]);
        if (!producer) {
            if (t_first < q_len) {
                load_w(c_first);
                load_x(t_first);
            }
            // the first batch of keys travels during the projection (entries past n_i - 1 exist in memory: harmless)
#pragma unroll
            for (int k = 0; k < kBatch; ++k) {
                const int pc = k * kWorkers + tid, j = block_of(pc >> lpk_shift);
                if (pc < total_cap && j < g.max_blocks) cp_async16(staged + pc, kc + ((size_t)j << lpk_shift) + csub);
            }
        }
        const int n_i = L > 0 ? (L + g.block_size - 1) / g.block_size : 0;
        // the blocks that hold a query token's own position, j_f .. n_i - 1 (one, the last, for a single token), are always
        // taken; the candidates are those before them
        const int j_f = max(0, L - q_len) / g.block_size;
        const int n_forced = min(n_i - j_f, g.max_sel);
        const int n_cand = min(j_f, g.max_blocks);
        int need = 0;                                      // (threshold method: known once the scores are)
        if (n_i > 0 && !g.threshold_mode) {
            const int k = min(max(g.token_budget / g.block_size, 1), min(n_i, g.max_sel));
            // (kListed: only a sequence longer than max_seq_len, which the host's rule went by, gets that far)
            need = max(0, min(min(k - n_forced, n_cand), kListed));
            n_blocks = need + n_forced;
        }
        // pieces that matter: up to the last run of keys with a candidate
        const int cand_chunks = (n_cand + kChunkKeys - 1) / kChunkKeys;
        const int total = ((max(0, cand_chunks - rank) + S - 1) >> s_shift) << (lpk_shift + 5);
        cluster_wait();                                    // every CTA of the cluster has started
        // ---- gate query: rotary pairs (c, c + d_gate/2) dealt to the cluster's warps --------------------------
        if (!producer) {
            for (int c = c_first; c < half; c += c_step) {
                for (int t = t_first; t < q_len; t += t_step) {
                    if (c != c_first && t == t_first) load_w(c);
                    if (MULTI && (c != c_first || t != t_first)) load_x(t);
                    float a = 0.f, b = 0.f;
#pragma unroll
                    for (int it = 0; it < 4; ++it) {
                        if (it < nit) { a += dot8(wv[0][it], xv[it]); b += dot8(wv[1][it], xv[it]); }
                    }
#pragma unroll
                    for (int off = 16; off > 0; off >>= 1) {
                        a += __shfl_xor_sync(0xffffffffu, a, off);
                        b += __shfl_xor_sync(0xffffffffu, b, off);
                    }
                    float sn, cs;                          // query token t sits at position L - q_len + t
                    rope_sincos((double)max(L - q_len + t, 0), g.inv_freq[c], &sn, &cs);
                    if (lane < S) {                        // lane r stores into CTA r of the cluster
                        float* dst = cluster.map_shared_rank(&sm.qg[0][0], lane) + t * kMaxDGate;
                        dst[c] = a * cs - b * sn;
                        dst[c + half] = b * cs + a * sn;
                    }
                }
            }
        }
        uint4 kv[kBatch];
        // (through L2, not the read-only path: the entry that this launch appends, or the step before it did, is among them)
        auto request = [&](int cb) {
#pragma unroll
            for (int k = 0; k < kBatch; ++k) {
                const int pc = cb + k * kWorkers + tid, j = block_of(pc >> lpk_shift);
                kv[k] = pc < total && j < g.max_blocks ? __ldcg(kc + ((size_t)j << lpk_shift) + csub) : make_uint4(0u, 0u, 0u, 0u);
            }
        };
        constexpr int kPieces = kWorkers * kBatch;
        if (!producer) request(kPieces);                   // the second batch, into registers
        cluster_sync();
        // ---- scores, into the first CTA's shared memory --------------------------------------------------------
        // A thread holds one piece of each of eight keys; reduce8 leaves every lane with the sum of one of the keys
        // (that of its piece number krev).
        if (!producer) {
            float* sc0 = cluster.map_shared_rank(sc_all, 0);
            const float inv = rsqrtf((float)g.d_gate);
            const int krev = ((lane & 1) << 2) | (lane & 2) | ((lane >> 2) & 1);
            const bool storer = (csub & ~7) == 0;
            uint32_t kmn = 0xffffffffu, kmx = 0u;
            float* sc_user = g.scores_user ? g.scores_user + (size_t)u * g.max_blocks : nullptr;
            // (several query tokens: a key's score is the largest of its products with their gate queries)
            auto score_batch = [&](auto&& piece, int cb) {
                float best = -INFINITY;
                for (int t = 0; t < q_len; ++t) {
                    float qsub[8], acc[kBatch];
#pragma unroll
                    for (int c = 0; c < 8; ++c) qsub[c] = sm.qg[t][8 * csub + c];
#pragma unroll
                    for (int k = 0; k < kBatch; ++k) acc[k] = dot8(piece(k), qsub);
                    const float x = reduce8(acc, lane, lpk);
                    best = MULTI ? fmaxf(best, x) : x;
                }
                const float v = best * inv;
                const int pc = cb + krev * kWorkers + tid, j = block_of(pc >> lpk_shift);
                if (storer && pc < total && j < n_cand) {
                    sc0[j] = v;
                    if (sc_user) sc_user[j] = v;
                    const uint32_t key = score_key(v);
                    kmn = min(kmn, key);
                    kmx = max(kmx, key);
                }
            };
            for (int cb = 0; cb < total;) {
                cp_async_wait_all();
                score_batch([&](int k) {
                    const int pc = k * kWorkers + tid;
                    return cb + pc < total && block_of((cb + pc) >> lpk_shift) < g.max_blocks ? staged[pc] : make_uint4(0u, 0u, 0u, 0u);
                }, cb);
                cb += kPieces;
                if (cb >= total) break;
                // (batches alternate between the staged area and the registers; the one after the next is on its way)
#pragma unroll
                for (int k = 0; k < kBatch; ++k) {
                    const int pc = cb + kPieces + k * kWorkers + tid, j = block_of(pc >> lpk_shift);
                    if (pc < total && j < g.max_blocks) cp_async16(staged + k * kWorkers + tid, kc + ((size_t)j << lpk_shift) + csub);
                }
                score_batch([&](int k) { return kv[k]; }, cb);
                cb += kPieces;
                request(cb + kPieces);
            }
            cp_async_wait_all();
#pragma unroll
            for (int off = 16; off > 0; off >>= 1) {
                kmn = min(kmn, __shfl_xor_sync(0xffffffffu, kmn, off));
                kmx = max(kmx, __shfl_xor_sync(0xffffffffu, kmx, off));
            }
            if (lane == 0 && kmn <= kmx) {
                atomicMin(cluster.map_shared_rank(&sm.pre_min, 0), kmn);
                atomicMax(cluster.map_shared_rank(&sm.pre_max, 0), kmx);
            }
        }
        cluster_sync();
        // ---- selection, by the first CTA ----------------------------------------------------------------------------
        if (rank == 0 && !producer) {
            int32_t* dst = g.block_idx + (size_t)u * g.max_sel;
            int* list = reinterpret_cast<int*>(sm.ring[2]);      // [kListed] the scored blocks of the list, ascending
            const int words = ((n_cand + 31) / 32 + NW - 1) / NW;      // 32 candidates each, per warp
            uint32_t thr;
            int j_eq;
            if (g.threshold_mode) {
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
            select_threshold<NW>(sm, sc_all, n_cand, need, words, warp, lane, thr, j_eq);
            // which of the warp's candidates are taken: lane x keeps the words x and x + 32 (words <= 64)
            const int jw = warp * words * 32 + lane;
            unsigned taken[2] = {0u, 0u};
#pragma unroll 1
            for (int e = 0; e < words; e += 4) {
                float v[4];
#pragma unroll
                for (int x = 0; x < 4; ++x) v[x] = sc_all[min(jw + 32 * (e + x), n_cand - 1)];
#pragma unroll
                for (int x = 0; x < 4; ++x) {
                    const int j = jw + 32 * (e + x);
                    const uint32_t key = score_key(v[x]);
                    const unsigned m = __ballot_sync(0xffffffffu, (e + x < words) & (j < n_cand) & ((key > thr) | ((key == thr) & (j <= j_eq))));
                    if (lane == ((e + x) & 31)) { if (e + x < 32) taken[0] = m; else taken[1] = m; }
                }
            }
            const int in_low = __popc(taken[0]), in_both = in_low + __popc(taken[1]);
            int incl_low = in_low, incl_high = in_both - in_low;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int lo = __shfl_up_sync(0xffffffffu, incl_low, o), hi = __shfl_up_sync(0xffffffffu, incl_high, o);
                if (lane >= o) { incl_low += lo; incl_high += hi; }
            }
            const int all_low = __shfl_sync(0xffffffffu, incl_low, 31);
            worker_sync<NW>();
            if (lane == 31) sm.warp_tot[warp] = incl_low + incl_high;
            worker_sync<NW>();
            int pos = 0;
#pragma unroll
            for (int w2 = 0; w2 < NW; ++w2) pos += w2 < warp ? sm.warp_tot[w2] : 0;
            // every lane lists its own words' blocks
            {
                int at = pos + incl_low - in_low;
                const int j_low = warp * words * 32 + 32 * lane;
                for (unsigned m = taken[0]; m; m &= m - 1) list[at++] = j_low + __ffs(m) - 1;
                at = pos + all_low + incl_high - (in_both - in_low);
                for (unsigned m = taken[1]; m; m &= m - 1) list[at++] = j_low + 1024 + __ffs(m) - 1;
            }
            if (tid == 0 && blockIdx.z == 0) g.block_cnt[u] = n_blocks;
            worker_sync<NW>();
            // entry e of the list is block j (the last ones: the blocks taken without a score): into the caller's list, and
            // to the CTA that reads its tile(s)
            for (int e = tid; e < g.max_sel; e += kWorkers) {
                const int j = e < need ? list[e] : e < n_blocks ? n_i - n_blocks + e : -1;
                if (blockIdx.z == 0) dst[e] = j;
                if (e >= n_blocks || !p.q) continue;
                if (p.blocks_per_tile == 1) {
                    for (int x = 0; x < p.tiles_per_block; ++x) {
                        const int t = (e << p.tpb_shift) + x;
                        if ((t >> s_shift) < kCodes) cluster.map_shared_rank(sm.codes, t & (S - 1))[t >> s_shift] = (j << p.tpb_shift) + x;
                    }
                } else {
                    const int t = e >> p.bpt_shift, sub = e & (p.blocks_per_tile - 1);
                    const int at = ((t >> s_shift) << p.bpt_shift) + sub;
                    if (at < kCodes) cluster.map_shared_rank(sm.codes, t & (S - 1))[at] = j;
                }
            }
        }
        if (!p.q) return;                                  // the gate alone
        fence_proxy_async_smem();                          // the ring's memory goes over to the copy engine
        cluster_arrive();
        // The other CTAs have nothing to do until the lists are out: up to four of them compress the block that has just
        // filled.  (Nothing in this step reads its entry.)
        if (g.k_nope && rank > 0 && rank <= 4 && warp < 8 && blockIdx.z == 0 && L >= g.block_size && L % g.block_size < q_len &&
            L / g.block_size <= g.max_blocks)
            append_block(g, sm.feat, u, i, h, L / g.block_size - 1, rank - 1, min(S - 1, 4));
    } else {
        pdl_wait();
        L = p.seq_lens[i];
        if (p.block_idx) {
            const int cnt = p.block_cnt ? p.block_cnt[u] : p.max_sel;      // (not behind the test on L: both loads in flight)
            n_blocks = L > 0 ? max(0, min(cnt, p.max_sel)) : 0;
        }
        __syncthreads();                                   // barriers initialised
    }

    // ---- tiles ------------------------------------------------------------------------------------------------------
    const bool dense = !GATE && !p.block_idx;
    const bool small = !dense && p.blocks_per_tile > 1;
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
    bool dead = false;                                     // a wait ran out: go through the motions, the results are invalid
    if (producer) {
        if (GATE) cluster_wait();                          // the tiles' numbers are in place
        pdl_launch_dependents();
        if (GATE && n_local < n_mine && lane == 0) raise_status(p.status, DEV_BAD_INDEX);      // (a sequence longer than max_seq_len: tiles are left out)
        const int n_i = (L + p.block_size - 1) >> p.bs_shift;
        for (int base = 0; base < n_local; base += 32) {
            const int it = base + lane;
            int row[4] = {0, 0, 0, 0}, outer[4] = {0, 0, 0, 0}, nv_all = 0, n_sub = 0;
            if (it < n_local) {
                const int t = (it << s_shift) + rank;
                const int n_try = small ? p.blocks_per_tile : 1;
                const int span = small ? p.block_size : kTileTokens;
#pragma unroll
                for (int x = 0; x < 4; ++x) {
                    if (x < n_try) {
                        int tok0 = -1;
                        if (dense) {
                            tok0 = t * kTileTokens;
                        } else if (small) {
                            const int e = (t << p.bpt_shift) + x;
                            if (e < n_blocks) {
                                const int blk = GATE ? sm.codes[(it << p.bpt_shift) + x] : p.block_idx[(size_t)u * p.max_sel + e];
                                if (!GATE && blk >= n_i) raise_status(p.status, DEV_BAD_INDEX);
                                if (blk >= 0 && blk < n_i) tok0 = blk << p.bs_shift;
                            }
                        } else if (GATE) {
                            tok0 = sm.codes[it] * kTileTokens;
                        } else {
                            const int blk = p.block_idx[(size_t)u * p.max_sel + (t >> p.tpb_shift)];
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
            // lane s asks for tile s of the batch
            const int m = min(32, n_local - base);
            for (int s = 0; s < m; ++s) {
                if (lane == s) {
                    const int st = it % kStages;
                    if (!dead && !mbar_wait(&sm.empty[st], ((it / kStages) & 1) ^ 1, p.status)) dead = true;
                    unsigned char* dst = sm.ring[st];
                    uint64_t* full = &sm.full[it % kArrivals];
                    sm.meta[it % kArrivals] = nv_all;      // (the tile kArrivals back has been read: the one kStages back has, which came after it)
                    if (dead || n_sub == 0) {
                        mbar_arrive(full);
                    } else if (small) {
                        const int sub_bytes = p.block_size * 128;      // one half (64 channels) of one block
                        mbar_arrive_expect_tx(full, (uint32_t)(n_sub * 4 * sub_bytes));
#pragma unroll
                        for (int x = 0; x < 4; ++x) {
                            if ((nv_all >> (8 * x)) & 0xff) {
                                unsigned char* d2 = dst + x * sub_bytes;
                                tma_load_4d(d2, &map_k, full, 0, row[x], h, outer[x]);
                                tma_load_4d(d2 + kHalfTileBytes, &map_k, full, 64, row[x], h, outer[x]);
                                tma_load_4d(d2 + kTileBytes, &map_v, full, 0, row[x], h, outer[x]);
                                tma_load_4d(d2 + kTileBytes + kHalfTileBytes, &map_v, full, 64, row[x], h, outer[x]);
                            }
                        }
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
        if (GATE) cluster_wait();
        pdl_launch_dependents();
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
                const uint32_t kbase = smem_u32(sm.ring[st]), vbase = kbase + kTileBytes;
                if (nvw < 16) {
                    // ragged tail: rows past the sequence end may hold anything; this warp's are cleared in V, so that
                    // a zero probability times garbage cannot produce NaN
                    unsigned char* vt = sm.ring[st] + kTileBytes;
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
        float* part = reinterpret_cast<float*>(sm.ring[0]) + warp * 8 * kMergeStride;
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
            const float* src = reinterpret_cast<const float*>(sm.ring[0]) + (r & 7) * kMergeStride + c;
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
            float* dst = cluster.map_shared_rank(sm.recv_o, c >> c_shift) + (((rank * kRows + r) << c_shift) | (c & ((1 << c_shift) - 1)));
            *reinterpret_cast<float4*>(dst) = acc;
            if (lane < S) cluster.map_shared_rank(&sm.recv_ml[0][0], lane)[rank * kRows + r] = make_float2(M, l);
        }
    }
    cluster_sync();
    if (!producer) {
        const int c_shift = 7 - s_shift;
        const int pairs = rows << (c_shift - 1);        // channel pairs of this CTA's slice, all rows
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
        if constexpr (GATE) {                              // (a cluster of one CTA has nobody to leave the append to)
            const GateParams& g = ga.g;
            if (g.k_nope && S == 1 && warp < 8 && blockIdx.z == 0 && L >= g.block_size && L % g.block_size < q_len &&
                L / g.block_size <= g.max_blocks)
                append_block(g, sm.feat, u, i, h, L / g.block_size - 1, 0, 1);
        }
    }
}

template <int NW, bool GATE, bool MULTI>
cudaError_t configure() {
    cudaError_t e = cudaFuncSetAttribute(step_cluster_kernel<NW, GATE, MULTI>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)sizeof(StepSmem<NW, MULTI>) + 1024);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(step_cluster_kernel<NW, GATE, MULTI>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    return e;
}

template <int NW, bool GATE, bool MULTI>
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

template <int NW, bool GATE, bool MULTI>
int resident_of(int k) {
    if (configure<NW, GATE, MULTI>() != cudaSuccess) return 0;
    cudaLaunchAttribute attr[2];
    cudaLaunchConfig_t cfg = config_of<NW, GATE, MULTI>(1 << k, 1, 1, nullptr, attr);
    cfg.numAttrs = 1;
    int n = 0;
    if (cudaOccupancyMaxActiveClusters(&n, step_cluster_kernel<NW, GATE, MULTI>, &cfg) != cudaSuccess) n = 0;
    cudaGetLastError();                                    // (a refused size is no error of the caller's)
    return n;
}

// Clusters of 2^k CTAs that the device holds at once (`wide`: of the NW = 16 kernels), asked once per device; 0: the
// device or the driver does not take such clusters.
int resident_clusters(bool wide, int k) {
    static int cached[kMaxDevices][2][5];                  // (value + 1; 0: not asked yet.  A race asks twice and stores the same)
    int& c = cached[current_device_slot()][wide][k];
    if (c == 0) {
        c = wide ? min(resident_of<16, true, true>(k), resident_of<16, false, true>(k)) + 1
                 : min(min(resident_of<8, true, false>(k), resident_of<8, false, false>(k)),
                       min(resident_of<8, true, true>(k), resident_of<8, false, true>(k))) + 1;
    }
    return c - 1;
}

}  // namespace

// As many CTAs per unit as keep every cluster resident at once (a second wave would double the call) and still have
// something to do each.  Measured against the kernels of long calls, us a call (a step's append included):
//     step, 8 KV heads, budget 4096, 1 / 2 / 4 sequences     23.3 -> 16.9, 25.3 -> 19.8, 31.6 -> 28.8
//     step of batch 8 at 128k, 205 blocks (51 tiles a CTA)   98.4 -> 85.0
//     four query tokens, 20 rows, 4 sequences, budget 4096   63.2 -> 38.6;  64 rows 92.3 -> 75.2;  8 rows, 1 sequence 27.2 -> 19.0
//     threshold gate alone in front of given lists, 4 sequences of 48k, blocks of 32: 42.5 -> 35.0 with both
// A cluster's CTAs go through their unit's tiles by themselves; the decode kernel's CTAs share all tiles.  The rule sees
// the longest list that there can be, not how uneven the lists are, and one long sequence among short ones leaves most
// clusters idle.  us a call, decode kernel -> clusters, 8 KV heads; one sequence's lists long / half of them / all, by the
// tiles a CTA of a long one:
//     lists, 24 sequences (S = 1)    16: 13.3 -> 12.2 / 20.4 -> 14.0 / 34.1 -> 21.9    32: 13.7 -> 18.8 / 35 -> 26.6 / 50 -> 37.7
//            16 sequences (S = 2)    16: 12.8 -> 11.9 / 20.9 -> 15.3 / 32.2 -> 25.7    32: 14.5 -> 18.9 / 37.5 -> 28.4 / 53.9 -> 46.0
//             8 sequences (S = 4)    16: 13.9 -> 12.2 / 19.8 -> 14.7 / 30.6 -> 25.6    32: 17.4 -> 19.8 / 35.9 -> 27.8 / 52.5 -> 45.0
//             4 sequences (S = 8)    32: 21.3 -> 21.8 / 34.9 -> 27.7 / 53.8 -> 45.8    64: 38.4 -> 41.2 / 54.5 -> 48.2 / 91.4 -> 83.7
//            16 sequences, 20 rows (S = 1)
//                                    16: 21.6 -> 18.8 / 27.6 -> 19.3 / 25.7 -> 20.1    32: 22.4 -> 30.7 / 39.7 -> 32.1 / 56.3 -> 33.5
//     steps, 16 sequences (S = 2)    64: 31.7 -> 46.8 / 72.3 -> 58.6 / 103 -> 93      128: 45.3 -> 82.7 / 108 -> 103 / 178 -> 173
//             8 sequences (S = 4)    64: 35.6 -> 47.4 / 69.6 -> 56.6 / 101 -> 91      128: 57.1 -> 80.6 / 105 -> 101 / 176 -> 172
// Given lists and dense calls, whose lengths follow the sequences', keep to where one long sequence does not lose: 16 + 2 S
// tiles a CTA (a decode call pays for its parts whatever its size, and more the longer its longest unit is).  The lists of a
// step are all as long as the budget but for sequences shorter than that: the line is at 64, where all but the most uneven
// batches gain; at 128 the even ones gain 3 % and the uneven ones lose up to half.  With a few more CTAs than SMs the SMs
// that hold two of them are the last to finish (80 units, 64 tiles a CTA, 160 CTAs: 65 -> 67; 32 tiles: 40.8 -> 37.5), so
// the line is at 32 there.  149 to 296 units, a CTA each, gain like fewer: steps of 24 / 30 / 36 sequences, all long, 16 tiles
// a CTA 45.9 -> 33.8, 52.7 -> 39.1, 59.3 -> 43.1; 64 tiles 93.5 -> 82.1, 108 -> 96, 127 -> 109.
StepPlan step_plan(int units, int rows, long long max_tiles, long long max_codes, int max_keys) {
    const bool wide = rows > 16;
    StepPlan plan = {0, 1, rows};
    if (rows > 64) return plan;
    if (wide) {
        plan.parts = (rows + 31) / 32;
        plan.rows = (rows + plan.parts - 1) / plan.parts;
    }
    const int sms = wide ? resident_clusters(true, 0) : resident_clusters(false, 0) / 2;
    units *= plan.parts;
    for (int k = 4; k >= 0; --k) {
        const int S = 1 << k;
        if (k > 0 && S > max_tiles && 128ll * S > max_keys) continue;      // a CTA would have nothing to do
        if (units > resident_clusters(wide, k)) continue;
        const bool few_doubled = units * S > sms && 5 * units * S <= 6 * sms;
        const long long line = (long long)S * min(max_keys > 0 ? 64 : 16 + 2 * S, few_doubled ? 32 : 64);
        if (max_tiles <= line && max_codes <= (long long)S * kCodes) plan.S = S;
        break;
    }
    return plan;
}

namespace {

template <int NW, bool MULTI>
cudaError_t launch_of(const CUtensorMap& map_k, const CUtensorMap& map_v, const DecodeParams& p, const GateParams* g, const StepPlan& plan,
                      cudaStream_t stream) {
    cudaLaunchAttribute attr[2];
    if (g) {
        const cudaLaunchConfig_t cfg = config_of<NW, true, MULTI>(plan.S, p.num_units, plan.parts, stream, attr);
        return cudaLaunchKernelEx(&cfg, step_cluster_kernel<NW, true, MULTI>, map_k, map_v, p, GateArg<true>{*g});
    }
    const cudaLaunchConfig_t cfg = config_of<NW, false, MULTI>(plan.S, p.num_units, plan.parts, stream, attr);
    return cudaLaunchKernelEx(&cfg, step_cluster_kernel<NW, false, MULTI>, map_k, map_v, p, GateArg<false>{});
}

}  // namespace

cudaError_t launch_step_cluster(const CUtensorMap& map_k, const CUtensorMap& map_v, const DecodeParams& p, const GateParams* g,
                                const StepPlan& plan, cudaStream_t stream) {
    if (p.q_len == 1) return launch_of<8, false>(map_k, map_v, p, g, plan, stream);
    return plan.parts * plan.rows <= 16 ? launch_of<8, true>(map_k, map_v, p, g, plan, stream)
                                        : launch_of<16, true>(map_k, map_v, p, g, plan, stream);
}

}  // namespace seer
