// Sparse decode over given lists, and dense decode, of one query token (up to eight heads per KV head): one launch of
// thread-block clusters.
//
// Every (sequence, KV head) unit has S CTAs (two per SM) that meet in shared memory, as in the one-launch step: a producer
// warp keeps a ring of three 64-token K/V stages in flight, eight consumer warps in two groups take alternate tiles, the
// warps' partials and then the CTAs' (a slice of the channels each, by stores that count their bytes down on the
// receiver's mbarrier) are merged without a trip through global memory.  How the work is dealt is decided in the kernel,
// which alone knows the lists' lengths:
//   even lists     cluster c takes unit c from end to end;
//   uneven ones    every cluster takes its unit's first tiles, up to a line; what is left of the long units, laid end to end,
//                  is dealt to the clusters whose own lists end well before it.  A cluster goes through its share piece by
//                  piece, each a run of tiles of one unit; a unit of several pieces is put together from their partial
//                  results, in global memory, by the CTAs that deliver the last one (rank r of the clusters has slice r of the
//                  channels, so each slice is a matter of its own, with its own counter).  Where units are few and long there are
//                  clusters without a unit of their own for it, as many as there is room for.
// Every CTA comes to the same decision from the same numbers, so that nothing is waited for across clusters.  A warp of its own
// decides while a unit's first tiles, which are never dealt, travel and are consumed.
//
// What bounds it: memory, from the first tiles (2.8 us after the kernel may read its inputs) to the last; 128 ragged lists of 13 to
// 102 tiles (247 MB) take 44.5 us, 52.7 by the decode kernel, whose CTAs make a schedule first and publish their partial
// results with a fence and a ticket each; 64 lists of 103 tiles (216 MB) 37.0 and 47.1.  A CTA by itself is bound by its three
// stages, of which the consumers hold one or two: 0.46 us a tile.  Short uneven lists: the chain of two pieces.  24 sequences, one of
// 32 tiles a CTA among ones of 4, by time stamps: deal seen 4.5 us, first pieces over 5 (long ones 9.4), their output 6.8,
// second pieces over 9.7 to 10.5, their partials written 11 to 11.8, counted 12.1, put together 14.2.
#include <cooperative_groups.h>

#include <type_traits>

#include "seer_cluster.cuh"

namespace cg = cooperative_groups;

namespace seer {

namespace {

constexpr int kNW = 8;                                     // consumer warps; with the producer warp two CTAs per SM
template <bool SPREAD>
constexpr int kThreads = 32 * (kNW + (SPREAD ? 2 : 1));    // uneven lists are dealt by a warp of its own
constexpr int kStages = 3, kGroups = kNW / 4, kArrivals = kStages * kGroups;
constexpr int kRows = kMaxGroup;
// A unit's first tiles, by the CTA, that are never dealt: a helper ends a piece's cost and half of it again below the line.
constexpr int kOwnTiles = kPieceTiles + kPieceTiles / 2;

struct __align__(1024) ListSmem {
    unsigned char ring[kStages * kStageBytes];
    // what the cluster's CTAs send after a piece's last tile, by turns: a CTA that sends its part of piece k + 2 has received all
    // of piece k + 1, whose senders had read piece k's
    __align__(16) float recv_o[2][kRows * kHeadDim];       // [source CTA][row][this CTA's slice of the channels]
    float2 recv_ml[2][kMaxS][kRows];                       // [source CTA][row]: max, sum
    float2 warp_ml[kNW][kRows];
    // Tile n arrives in stage (n + pieces before) % kStages (behind a piece is a stage without a tile) and is announced on
    // full[n % kArrivals]: a barrier belongs to one residue of the tile numbers and so to one consumer group, which follows all
    // of its phases.
    uint64_t full[kArrivals], empty[kStages];
    // A stage, behind a piece, to put its partials together: given[piece % kStages].  (Pieces may be without a tile for a CTA; that
    // of three before has been put together when a stage is given.)
    uint64_t got_parts[2], given[kStages];
    int meta[kArrivals];                                   // tokens from the tile's first row on (blocks of 16 or 32 tokens: per block, 8 bits each)
    // uneven lists: how the tiles are dealt
    int rest[kListUnits + 1];                              // tiles above the line of the units before
    int room[kListUnits + 1];                              // tiles that the helpers before take (on the way there: the units' tiles)
    int line, helpers, helper, is_last;                    // helper: number of this cluster among the helpers, or -1
    int share[2], pieces[2];                               // the helper's share of the rest; first and last helper with a piece of a unit
};
static_assert(sizeof(ListSmem) + 1024 <= 113 * 1024, "two CTAs per SM");

__device__ __forceinline__ void consumers_sync() { worker_sync<kNW>(); }
// The deal is made: the dealing warp arrives for the consumer groups (barriers 2 and 3) and the producer (4), which wait for it.
// (Barriers of the hardware, not mbarriers: the dealing warp waits for nothing, and a wait that could run out would leave its warp
// with another idea of its pieces than the others.)
__device__ __forceinline__ void deal_made() {
    __syncwarp();
    asm volatile("bar.arrive 2, 160;\n\tbar.arrive 3, 160;\n\tbar.arrive 4, 64;" ::: "memory");
}
__device__ __forceinline__ void await_deal(int group) {    // (group 2: the producer)
    __syncwarp();
    asm volatile("bar.sync %0, %1;" ::"r"(2 + group), "r"(group < kGroups ? 160 : 64) : "memory");
}
static_assert(kNW == 8 && kGroups == 2, "five warps at each of barriers 2 and 3");
__device__ __forceinline__ void mbar_arrive_n(uint64_t* bar, uint32_t n) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)), "r"(n) : "memory");
}

// A consumer warp's step over a staged K/V tile (as in the one-launch step, whose registers do not allow a copy of it that both
// kernels share: 0.2 us of 14), for the unit's up to eight heads: the 16 tokens `w4` of the tile,
// online softmax with running maximum m_run, sum l_run and output o of its own.  S^T = K . Q^T and O^T += V^T . P^T by mma.sync,
// tokens (channels) on M, rows on N.
// stage: K and V of the tile; bq: the Q^T fragments; nvw: valid tokens from this warp's first one on (at least one).
__device__ __forceinline__ void tile_step(float (&o)[8][4], float (&m_run)[2], float (&l_run)[2], unsigned char* stage,
                                          const uint32_t (&bq)[8][2], int nvw, float scale_log2, int lane, int w4) {
    const int rw = lane >> 2;
    // lane-constant parts of the ldmatrix addresses (swizzle: 16-B chunk ^= row & 7)
    const int k_row = 16 * w4 + ((lane >> 3) & 1) * 8 + (lane & 7), k_csel = lane >> 4;
    const int v_row = 16 * w4 + ((lane >> 4) & 1) * 8 + (lane & 7), v_csel = (lane >> 3) & 1;
    const int sw = lane & 7;
    const uint32_t kbase = smem_u32(stage), vbase = kbase + kTileBytes;
    if (nvw < 16) {
        // ragged tail: rows past the sequence end may hold anything; this warp's are cleared in V, so that
        // a zero probability times garbage cannot produce NaN
        unsigned char* vt = stage + kTileBytes;
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
    for (int x = 0; x < 4; ++x) s[x] = ((sa[0][x] + sa[1][x]) + (sa[2][x] + sa[3][x])) * scale_log2;
    if (rw >= nvw) s[0] = s[1] = -INFINITY;
    if (rw + 8 >= nvw) s[2] = s[3] = -INFINITY;
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

// A cluster's piece of a unit: its tiles a .. b.  `x`, `end`: what is left of the cluster's share of the rest.
struct Piece {
    int u, a, b, n;                                        // n: tiles of the unit
    int x, end;
};

// The place of x in the ascending v[0 .. n]: the last i < n with v[i] <= x.
__device__ __forceinline__ int place_of(const int* v, int n, int x) {
    int lo = 0, hi = n;
    while (hi - lo > 1) {
        const int mid = (lo + hi) >> 1;
        if (v[mid] <= x) lo = mid; else hi = mid;
    }
    return lo;
}

// Where helper k's share of the rest begins.  Where that is a little before or behind a unit's end it is there: a helper with parts of
// two units pays for two pieces.  Each unit's end takes the nearest share's only, so that no share becomes empty but the last.
__device__ __forceinline__ int share_begin(const ListSmem& sm, int clusters, int k, int cost) {
    const int x = sm.room[k];
    if (k == 0 || k == sm.helpers || x >= sm.rest[clusters]) return x;
    const int prev = sm.room[k - 1], next = sm.room[k + 1], u = place_of(sm.rest, clusters, x), r0 = sm.rest[u], r1 = sm.rest[u + 1];
    const int back = r0 > prev && x - r0 <= r0 - prev ? x - r0 : cost, ahead = r1 < next && r1 - x < next - r1 ? r1 - x : cost;
    return min(back, ahead) >= cost ? x : back <= ahead ? r0 : r1;
}

// The deal, by one warp, from the units' tiles in sm.room: the lowest line at which the helpers have room below it for what is
// above it.  (Few tiles are not worth a piece: a unit that ends a little above the line keeps what is its, a cluster with little
// room is no helper.)  A lane has the tiles of `per` clusters that follow one another, so that one scan over the lanes is enough: with
// every 32nd, and shares' ends moved for all helpers, the deal of 192 units was seen at 6.4 us instead of 4.5.
template <int COUNTS>
__device__ __forceinline__ void deal(ListSmem& sm, int clusters, int s_shift, int cluster_id, int total, int most) {
    const int lane = threadIdx.x & 31, per = (clusters + 31) >> 5, v0 = lane * per, cost = kPieceTiles << s_shift, few = cost / 2;
    auto above = [&](int line, int t) { return t - line >= few ? t - line : 0; };
    auto below = [&](int line, int t) { return line - cost - t >= few ? line - cost - t : 0; };
    int n[COUNTS];
#pragma unroll
    for (int k = 0; k < COUNTS; ++k) n[k] = k < per && v0 + k < clusters ? sm.room[v0 + k] : 0;
    __syncwarp();
    const int S1 = (1 << s_shift) - 1;
    int lo = max((total / clusters + S1) >> s_shift, kOwnTiles), hi = max(lo, (most + S1) >> s_shift);      // (tiles a CTA; line `hi`: nothing is above it)
#pragma unroll 1
    while (lo < hi) {
        const int mid = (lo + hi) >> 1, line = mid << s_shift;
        int free = 0;
#pragma unroll
        for (int k = 0; k < COUNTS; ++k) {
            if (k >= per) break;
            if (v0 + k < clusters) free += below(line, n[k]) - above(line, n[k]);
        }
        if (__reduce_add_sync(0xffffffffu, free) >= 0) hi = mid;
        else lo = mid + 1;
    }
    const int line = lo << s_shift;
    int rest = 0, room = 0, helpers = 0;                   // this lane's, then all lanes' up to it
#pragma unroll
    for (int k = 0; k < COUNTS; ++k) {
        if (k >= per) break;
        if (v0 + k >= clusters) break;
        const int mine = below(line, n[k]);
        rest += above(line, n[k]);
        room += mine;
        helpers += mine > 0;
    }
    int a = rest, b = room, c = helpers;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int ta = __shfl_up_sync(0xffffffffu, a, o), tb = __shfl_up_sync(0xffffffffu, b, o), tc = __shfl_up_sync(0xffffffffu, c, o);
        if (lane >= o) { a += ta; b += tb; c += tc; }
    }
    int at = a - rest, to = b - room, helper = c - helpers;
    rest = __shfl_sync(0xffffffffu, a, 31);
    room = __shfl_sync(0xffffffffu, b, 31);
    helpers = __shfl_sync(0xffffffffu, c, 31);
#pragma unroll
    for (int k = 0; k < COUNTS; ++k) {
        if (k >= per) break;
        const int v = v0 + k, mine = below(line, n[k]);
        if (v >= clusters) break;
        sm.rest[v] = at;
        at += above(line, n[k]);
        if (mine > 0) {
            sm.room[helper] = to;
            if (v == cluster_id) sm.helper = helper;
            to += mine;
            ++helper;
        }
    }
    if (lane == 0) {
        sm.rest[clusters] = rest;
        sm.room[helpers] = room;
        sm.helpers = helpers;
        sm.line = line;
    }
    __syncwarp();
    helper = sm.helper;
    if (helper >= 0 && lane < 2) sm.share[lane] = min(share_begin(sm, clusters, helper + lane, cost), rest);
    __syncwarp();
}

// grid (S, clusters), cluster (S, 1, 1).  SPREAD: the lists may be so long that it matters whether they are even.
template <bool SPREAD>
__device__ __forceinline__ void list_body(const CUtensorMap& map_k, const CUtensorMap& map_v, const DecodeParams& p) {
    extern __shared__ unsigned char smem_raw[];
    // (aligned by an offset, not by a cast through an integer: the compiler then still knows the accesses for shared ones)
    ListSmem& sm = *reinterpret_cast<ListSmem*>(smem_raw + ((1024 - (smem_u32(smem_raw) & 1023)) & 1023));
    cg::cluster_group cluster = cg::this_cluster();
    const int S = (int)cluster.num_blocks(), rank = (int)cluster.block_rank(), s_shift = 31 - __clz(S);
    const int c_shift = 7 - s_shift;                       // log2 of the channels of a CTA's slice
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const bool producer = warp == kNW;
    const int rows = p.group, cluster_id = blockIdx.y;
    const uint32_t part_bytes = (uint32_t)(rows * kHeadDim * 4 + S * rows * 8);      // what a CTA receives per piece
    if (tid < 32) {
        if (tid < kArrivals) mbar_init(&sm.full[tid], 1);
        if (tid < kStages) {
            mbar_init(&sm.empty[tid], kNW);
            mbar_init(&sm.given[tid], 1);
        }
        if (tid < 2) mbar_init(&sm.got_parts[tid], 1);
        if (tid == 0) {
            sm.line = 0x7fffffff;                          // (even lists)
            sm.helper = -1;
        }
        mbar_fence_init();
        if (tid < 2) mbar_arrive_expect_tx(&sm.got_parts[tid], part_bytes);
    }
    // (another CTA's shared memory is written only after the barrier this opens: it is then known to be running, and its
    // mbarriers are initialised)
    cluster_arrive();
    if (producer && lane == 0) {
        tma_prefetch_desc(&map_k);
        tma_prefetch_desc(&map_v);
    }
    const bool dense = !p.block_idx;
    const bool small = !dense && p.blocks_per_tile > 1;
    auto sequence_of = [&](int u) { return p.kvh_magic ? (int)__umulhi((unsigned)u, p.kvh_magic) : u; };
    // a unit's listed blocks, and its tiles
    auto listed = [&](int count, int L) -> int { return L > 0 ? max(0, min(count, p.max_sel)) : 0; };
    auto blocks_of = [&](int u, int L) -> int {
        if (dense) return 0;
        return listed(p.block_cnt ? p.block_cnt[u] : p.max_sel, L);        // (not behind a test on L: both loads in flight)
    };
    auto tiles_of = [&](int n_blocks, int L) -> int {
        if (dense) return L > 0 ? min((L + kTileTokens - 1) / kTileTokens, p.max_blocks_cap) : 0;
        return small ? (n_blocks + p.blocks_per_tile - 1) >> p.bpt_shift : n_blocks << p.tpb_shift;
    };
    pdl_wait();
    if (SPREAD && p.sel_from_lens > 0 && !step_uneven(p, S)) {     // (a step whose attention is done)
        pdl_launch_dependents();
        cluster_wait();
        return;
    }
    // (the first entries are asked for beside the count that says how many there are, not behind it)
    int entry[4] = {-1, -1, -1, -1}, entry2[4] = {-1, -1, -1, -1};      // the list's entries of this lane's first tile, and of the second piece's
    const bool owner = cluster_id < p.num_units;           // (the others have no unit of their own)
    if (producer && !dense && owner) {
        const int t = (lane << s_shift) + rank;
#pragma unroll
        for (int x = 0; x < 4; ++x) {
            const int e = small ? (t << p.bpt_shift) + x : t >> p.tpb_shift;
            if (x < p.blocks_per_tile) entry[x] = p.block_idx[(size_t)cluster_id * p.max_sel + min(e, p.max_sel - 1)];
        }
    }
    Piece pc;
    int L = owner ? p.seq_lens[sequence_of(cluster_id)] : 0, n_blocks = owner ? blocks_of(cluster_id, L) : 0;
    pc.u = cluster_id;
    pc.a = 0;
    pc.b = pc.n = tiles_of(n_blocks, L);
    pc.x = pc.end = 0;
    __syncthreads();                                       // barriers initialised
    // what the deal makes of this cluster's own unit, and its share of the rest
    auto take_share = [&]() {
        if (sm.line < 0x7fffffff && sm.rest[cluster_id + 1] > sm.rest[cluster_id]) pc.b = sm.line;
        if (sm.helper >= 0) {
            pc.x = sm.share[0];
            pc.end = sm.share[1];
        }
    };
    // on to the next piece; false: that was the last
    auto next_piece = [&]() -> bool {
        if (pc.x >= pc.end) return false;
        pc.u = place_of(sm.rest, p.clusters, pc.x);        // (the last one that begins there: the others have nothing above the line)
        const int r0 = sm.rest[pc.u], r1 = sm.rest[pc.u + 1], line = sm.line;
        pc.a = line + pc.x - r0;
        pc.x = min(r1, pc.end);
        pc.b = line + pc.x - r0;
        pc.n = line + r1 - r0;
        return true;
    };
    auto mine_of = [&]() -> int { return max(0, pc.b - pc.a - rank + S - 1) >> s_shift; };      // this CTA's tiles of the piece
    bool dead = false;                                     // a wait ran out: go through the motions, the results are invalid
    int tiles_before = 0, pieces_before = 0;               // this CTA's tiles, and the cluster's pieces, before the current one
    // (What is done for a piece is written once and compiled twice: for the cluster's own unit, which mostly is all there is, the
    // numbers before it are known to be zero.)
    using First = std::true_type;
    using Later = std::false_type;
    if (producer) {
        if (p.next_early) pdl_launch_dependents();
        // a helper's first piece is looked up as soon as the deal is made
        int L2 = 0, count2 = 0;
        auto see_deal = [&]() {
            await_deal(kGroups);
            take_share();
            if (pc.x < pc.end) {
                const int u = place_of(sm.rest, p.clusters, pc.x), t = sm.line + pc.x - sm.rest[u] + (lane << s_shift) + rank;
                L2 = p.seq_lens[sequence_of(u)];
                if (!dense) count2 = p.block_cnt ? p.block_cnt[u] : p.max_sel;
                if (!dense) {
#pragma unroll
                    for (int x = 0; x < 4; ++x) {
                        const int e = small ? (t << p.bpt_shift) + x : t >> p.tpb_shift;
                        if (x < p.blocks_per_tile) entry2[x] = p.block_idx[(size_t)u * p.max_sel + min(e, p.max_sel - 1)];
                    }
                }
            }
        };
        int tile0 = 0, piece = 0;
        do {
            if (SPREAD && piece > 0) {
                const bool first = piece == 1;
                L = first ? L2 : p.seq_lens[sequence_of(pc.u)];
                n_blocks = first ? listed(count2, L) : blocks_of(pc.u, L);
#pragma unroll
                for (int x = 0; x < 4; ++x) entry[x] = entry2[x];
            }
            const int i = sequence_of(pc.u), h = pc.u - i * p.num_kv_heads;
            int n_local = mine_of();
            if (SPREAD && piece == 0 && n_local == 0) see_deal();
            const int n_i = (L + p.block_size - 1) >> p.bs_shift;
            const int32_t* list = p.block_idx + (size_t)pc.u * p.max_sel;
            // (a CTA's first tiles do not depend on the deal)
            const bool own = SPREAD && piece == 0;
            for (int base = 0, count; base < n_local; base += count) {
                count = !own || base > kOwnTiles ? 32 : base == 0 ? kOwnTiles : 32 - kOwnTiles;
                const int it = base + lane;
                int row[4] = {0, 0, 0, 0}, outer[4] = {0, 0, 0, 0}, nv_all = 0, n_sub = 0;
                if (it < n_local) {
                    const int t = pc.a + (it << s_shift) + rank;
                    const int n_try = small ? p.blocks_per_tile : 1;
                    const int span = small ? p.block_size : kTileTokens;
                    const bool have = it < 32 && (!SPREAD || piece <= 1);
#pragma unroll
                    for (int x = 0; x < 4; ++x) {
                        if (x < n_try) {
                            int tok0 = -1;
                            if (dense) {
                                tok0 = t * kTileTokens;
                            } else if (small) {
                                const int e = (t << p.bpt_shift) + x;
                                if (e < n_blocks) {
                                    const int blk = have ? entry[x] : list[e];
                                    if (blk >= n_i) raise_status(p.status, DEV_BAD_INDEX);
                                    if (blk >= 0 && blk < n_i) tok0 = blk << p.bs_shift;
                                }
                            } else {
                                const int blk = have ? entry[0] : list[t >> p.tpb_shift];
                                if (blk >= n_i) raise_status(p.status, DEV_BAD_INDEX);
                                if (blk >= 0 && blk < n_i) tok0 = (blk << p.bs_shift) + (t & (p.tiles_per_block - 1)) * kTileTokens;
                            }
                            int nv = tok0 >= 0 ? max(0, min(span, L - tok0)) : 0;
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
                // tile s of the batch, which lane s has looked up, is asked for by an elected lane
                const int m = min(count, n_local - base);
                for (int s = 0; s < m; ++s) {
                    const int n = tile0 + base + s, slot = n + piece, st = slot % kStages;
                    const int nv = __shfl_sync(0xffffffffu, nv_all, s), subs = __shfl_sync(0xffffffffu, n_sub, s);
                    int r[4], o[4];
                    r[0] = __shfl_sync(0xffffffffu, row[0], s);
                    o[0] = __shfl_sync(0xffffffffu, outer[0], s);
                    if (small) {
#pragma unroll
                        for (int x = 1; x < 4; ++x) {
                            r[x] = __shfl_sync(0xffffffffu, row[x], s);
                            o[x] = __shfl_sync(0xffffffffu, outer[x], s);
                        }
                    }
                    if (!dead && !mbar_wait(&sm.empty[st], ((slot / kStages) & 1) ^ 1, p.status)) dead = true;
                    dead = __any_sync(0xffffffffu, dead);
                    if (elect_one()) {
                        unsigned char* dst = sm.ring + st * kStageBytes;
                        uint64_t* full = &sm.full[n % kArrivals];
                        sm.meta[n % kArrivals] = nv;       // (the tile kArrivals back has been read: a later one of its group had this stage or a later one)
                        if (dead || subs == 0) {
                            mbar_arrive(full);
                        } else if (small) {
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
                        } else {
                            mbar_arrive_expect_tx(full, kStageBytes);
                            tma_load_4d(dst, &map_k, full, 0, r[0], h, o[0]);
                            tma_load_4d(dst + kHalfTileBytes, &map_k, full, 64, r[0], h, o[0]);
                            tma_load_4d(dst + kTileBytes, &map_v, full, 0, r[0], h, o[0]);
                            tma_load_4d(dst + kTileBytes + kHalfTileBytes, &map_v, full, 64, r[0], h, o[0]);
                        }
                    }
                    __syncwarp();
                }
                dead = __any_sync(0xffffffffu, dead);
                if (own && base == 0) {
                    see_deal();
                    n_local = mine_of();
#pragma unroll
                    for (int x = 0; x < 4; ++x) entry[x] = __shfl_down_sync(0xffffffffu, entry[x], kOwnTiles);
                }
            }
            if (!SPREAD) break;
            // The slot behind a piece's last tile is the consumers': its stage is where they put their partials together.  They
            // take it when the producer gives it, which it does, as with a tile, when the stage is free: every phase of its
            // barrier is thus seen before the next one can end.  (Behind the last piece nobody asks for the stage again.)
            tile0 += n_local;
            if (pc.x < pc.end) {
                const int slot = tile0 + piece;
                if (!dead && !mbar_wait(&sm.empty[slot % kStages], ((slot / kStages) & 1) ^ 1, p.status)) dead = true;
                dead = __any_sync(0xffffffffu, dead);
                if (lane == 0) mbar_arrive(&sm.given[piece % kStages]);
            }
            ++piece;
        } while (next_piece());
        cluster_wait();                                    // (the barrier opened at the top)
        cluster_arrive_relaxed();
    } else if (SPREAD && warp > kNW) {
        // The deal, while the first tiles travel.  The units' tiles (read by neighbouring lanes from neighbouring places: the lanes'
        // own runs of them cost even lists 0.4 us):
        constexpr int kCounts = (kListUnits + 31) / 32;
        int n[kCounts], len[kCounts], total = 0, most = 0;
#pragma unroll
        for (int k = 0; k < kCounts; ++k) {                // (all loads on their way before the first is looked at)
            if (32 * k >= p.clusters) break;
            const int v = min(lane + 32 * k, p.num_units - 1);
            len[k] = p.seq_lens[sequence_of(v)];
            n[k] = p.block_cnt ? p.block_cnt[v] : p.max_sel;
        }
#pragma unroll
        for (int k = 0; k < kCounts; ++k) {
            const int v = lane + 32 * k;
            if (32 * k >= p.clusters) break;
            n[k] = v < p.num_units ? tiles_of(listed(n[k], len[k]), len[k]) : 0;
            total += n[k];
            most = max(most, n[k]);
            if (v < p.clusters) sm.room[v] = n[k];
        }
        __syncwarp();
        total = __reduce_add_sync(0xffffffffu, total);
        most = __reduce_max_sync(0xffffffffu, most);
        if (list_uneven(total, most, p.clusters, S)) deal<kCounts>(sm, p.clusters, s_shift, cluster_id, total, most);
        deal_made();
        cluster_wait();                                    // (the barrier opened at the top)
        cluster_arrive_relaxed();
    } else {
        const int group = warp >> 2, w4 = warp & 3, qd = lane & 3, rw = lane >> 2;
        // Q^T B-fragments: this thread supplies row rw of the unit's queries
        uint32_t bq[8][2];
        auto load_q = [&](int u) {
            const int i = sequence_of(u), h = u - i * p.num_kv_heads;
            const uint32_t* qrow = reinterpret_cast<const uint32_t*>(
                p.q + ((size_t)i * p.num_q_heads + (size_t)h * p.group + (rw < rows ? rw : 0)) * kHeadDim);
#pragma unroll
            for (int ks = 0; ks < 8; ++ks) {
                bq[ks][0] = rw < rows ? __ldg(qrow + 8 * ks + qd) : 0u;
                bq[ks][1] = rw < rows ? __ldg(qrow + 8 * ks + 4 + qd) : 0u;
            }
        };
        load_q(min(pc.u, p.num_units - 1));
        if (p.next_early) pdl_launch_dependents();
        // blocks of 16 or 32 tokens: which of the gathered blocks this warp's rows belong to, and where in it
        const int sub_w = !small ? 0 : p.block_size == 16 ? w4 : w4 >> 1;
        const int off_w = !small ? 16 * w4 : p.block_size == 16 ? 0 : (w4 & 1) * 16;
        // false: that was the last piece
        auto consume = [&](auto first_c) -> bool {
            constexpr bool FIRST = decltype(first_c)::value;
            const int tile0 = FIRST ? 0 : tiles_before, piece = FIRST ? 0 : pieces_before;
            int n_end = tile0 + mine_of();
float o[8][4], m_run[2] = {-INFINITY, -INFINITY}, l_run[2] = {0.f, 0.f};
#pragma unroll
            for (int a = 0; a < 8; ++a) o[a][0] = o[a][1] = o[a][2] = o[a][3] = 0.f;
            bool dealt = !(SPREAD && FIRST);               // (a CTA's first tiles do not depend on the deal)
            int stop = dealt ? n_end : min(n_end, kOwnTiles);
            for (int n = FIRST ? group : tile0 + ((tile0 ^ group) & 1);; n += kGroups) {
                if (n >= stop) {
                    if (dealt) break;
                    await_deal(group);
                    take_share();
                    stop = n_end = mine_of();
                    dealt = true;
                    if (n >= stop) break;
                }
                const int st = (n + piece) % kStages;
                if (!dead && !mbar_wait(&sm.full[n % kArrivals], (n / kArrivals) & 1, p.status)) dead = true;
                const int nvw = (small ? (sm.meta[n % kArrivals] >> (8 * sub_w)) & 0xff : sm.meta[n % kArrivals]) - off_w;   // valid tokens from this warp's first row on
                if (nvw > 0 && !dead) tile_step(o, m_run, l_run, sm.ring + st * kStageBytes, bq, nvw, p.scale_log2, lane, w4);
                __syncwarp();
                if (lane == 0) mbar_arrive_n(&sm.empty[st], kNW / 4);
            }
            const bool more = SPREAD && pc.x < pc.end;
            // ---- the warps' partials, then the CTAs' -----------------------------------------------------------------
#pragma unroll
            for (int off = 4; off < 32; off <<= 1) {
                l_run[0] += __shfl_xor_sync(0xffffffffu, l_run[0], off);
                l_run[1] += __shfl_xor_sync(0xffffffffu, l_run[1], off);
            }
            const int st = (n_end + piece) % kStages, turn = piece & 1;
            // [warp][row][channel]; the channel's place is swizzled by the row, so that a warp's stores meet different banks
            float* parts = reinterpret_cast<float*>(sm.ring + st * kStageBytes);
            if (more && !dead && !mbar_wait(&sm.given[piece % kStages], (piece / kStages) & 1, p.status)) dead = true;
            consumers_sync();                              // every tile of the piece has been read: the slot's stage is free
            float* part = parts + warp * (kRows * kHeadDim);
            const int sw = qd << 3;
#pragma unroll
            for (int a = 0; a < 8; ++a) {
                const int d0 = (16 * a + rw) ^ sw, d1 = (16 * a + rw + 8) ^ sw;
                part[2 * qd * kHeadDim + d0] = o[a][0];
                part[(2 * qd + 1) * kHeadDim + d0] = o[a][1];
                part[2 * qd * kHeadDim + d1] = o[a][2];
                part[(2 * qd + 1) * kHeadDim + d1] = o[a][3];
            }
            if (rw == 0) {
                sm.warp_ml[warp][2 * qd] = make_float2(m_run[0], l_run[0]);
                sm.warp_ml[warp][2 * qd + 1] = make_float2(m_run[1], l_run[1]);
            }
            __syncwarp();
            if (FIRST) cluster_wait();                // every CTA of the cluster has started (the barrier opened at the top)
            consumers_sync();
            // a warp per row; lane: four channels
            if (warp < rows) {
                const int c = 4 * lane;
                float M = -INFINITY, l = 0.f;
                float2 ml[kNW];
#pragma unroll
                for (int x = 0; x < kNW; ++x) {
                    ml[x] = sm.warp_ml[x][warp];
                    M = fmaxf(M, ml[x].x);
                }
                float4 sum = make_float4(0.f, 0.f, 0.f, 0.f);
                const float* src = parts + warp * kHeadDim + (c ^ ((warp >> 1) << 3));
#pragma unroll
                for (int x = 0; x < kNW; ++x) {
                    const float f = ml[x].x == -INFINITY ? 0.f : fast_exp2(ml[x].x - M);
                    const float4 v = *reinterpret_cast<const float4*>(src + x * (kRows * kHeadDim));
                    l = fmaf(ml[x].y, f, l);
                    sum.x = fmaf(v.x, f, sum.x);
                    sum.y = fmaf(v.y, f, sum.y);
                    sum.z = fmaf(v.z, f, sum.z);
                    sum.w = fmaf(v.w, f, sum.w);
                }
                const int to = c >> c_shift;
                send_f32x4(cluster_addr(sm.recv_o[turn] + (((rank * kRows + warp) << c_shift) | (c & ((1 << c_shift) - 1))), to), sum,
                           cluster_addr(&sm.got_parts[turn], to));
                if (lane < S) send_f32x2(cluster_addr(&sm.recv_ml[turn][rank][warp], lane), make_float2(M, l), cluster_addr(&sm.got_parts[turn], lane));
            }
            const Piece done = pc;
            if (more) {
                next_piece();
                load_q(pc.u);                              // (on their way under what follows)
                fence_proxy_async_smem();                  // the stage goes over to the copy engine
                __syncwarp();
                if (lane == 0) mbar_arrive(&sm.empty[st]);
            }
            wait_sent(&sm.got_parts[turn], p.status, (piece >> 1) & 1);
            if (!more) cluster_arrive_relaxed();           // (all that was sent to this CTA is here)
            else if (tid == 0) mbar_arrive_expect_tx(&sm.got_parts[turn], part_bytes);       // (for the piece after the next)
            // ---- this CTA's slice of the channels: the output, or the piece's part of it --------------------------------
            const int pairs = rows << (c_shift - 1);       // channel pairs of the slice, all rows
            const bool whole = !SPREAD || done.b - done.a == done.n;
            const int i = sequence_of(done.u), h = done.u - i * p.num_kv_heads;
            // partial results in global memory: of the owner's piece and the helpers' (helper k's of unit u: k + u grows from one
            // piece to the next), by rank: max and sum of the rows, then the sums
            const int slice = 1 << c_shift, part_stride = 2 * kRows + (kRows << c_shift);
            auto part_of = [&](int slot) { return p.part_o + (size_t)(slot * S + rank) * part_stride; };
            auto write_out = [&](int r, int c, float M, float l, float a0, float a1) {
                const float inv = l > 0.f ? 1.f / l : 0.f;
                const size_t row = (size_t)i * p.num_q_heads + (size_t)h * p.group + r;
                *reinterpret_cast<uint32_t*>(p.out + row * kHeadDim + (rank << c_shift) + c) = pack_bf16x2(a0 * inv, a1 * inv);
                if (p.lse && rank == 0 && c == 0) p.lse[row] = l > 0.f ? (M + log2f(l)) * 0.6931471805599453f : -INFINITY;
            };
#pragma unroll 1
            for (int x = tid; x < pairs; x += 32 * kNW) {
                const int r = x >> (c_shift - 1), c = 2 * (x & ((slice >> 1) - 1));
                float M = -INFINITY, l = 0.f, a0 = 0.f, a1 = 0.f;
                float2 ml[kMaxS];
#pragma unroll
                for (int s = 0; s < kMaxS; ++s) {
                    ml[s] = s < S ? sm.recv_ml[turn][s][r] : make_float2(-INFINITY, 0.f);
                    M = fmaxf(M, ml[s].x);
                }
#pragma unroll
                for (int s = 0; s < kMaxS; ++s) {
                    if (s < S) {
                        const float f = ml[s].x == -INFINITY ? 0.f : fast_exp2(ml[s].x - M);
                        const float2 v = *reinterpret_cast<const float2*>(&sm.recv_o[turn][((s * kRows + r) << c_shift) + c]);
                        l = fmaf(ml[s].y, f, l);
                        a0 = fmaf(v.x, f, a0);
                        a1 = fmaf(v.y, f, a1);
                    }
                }
                if (whole) {
                    if (!SPREAD || done.u < p.num_units) write_out(r, c, M, l, a0, a1);
                } else {
                    float* dst = part_of(done.a == 0 ? done.u : p.num_units + sm.helper + done.u);
                    if (c == 0) *reinterpret_cast<float2*>(dst + 2 * r) = make_float2(M, l);
                    *reinterpret_cast<float2*>(dst + 2 * kRows + (r << c_shift) + c) = make_float2(a0, a1);
                }
            }
            if (!whole) {
                // whoever counts the unit's last tiles puts its pieces together, in order
                int* count = reinterpret_cast<int*>(p.tickets) + done.u * kMaxS + rank;
                consumers_sync();
                if (tid == 32) {                           // (behind the barrier: its release and acquire are all threads')
                    int before;
                    asm volatile("atom.add.acq_rel.gpu.global.s32 %0, [%1], %2;" : "=r"(before) : "l"(count), "r"(done.b - done.a) : "memory");
                    sm.is_last = before + done.b - done.a == done.n;
                } else if (warp == 0) {                    // the helpers that have a piece of the unit
                    const int r0 = sm.rest[done.u], r1 = sm.rest[done.u + 1], at = place_of(sm.room, sm.helpers, lane == 0 ? r0 : r1 - 1);
                    const int begin = share_begin(sm, p.clusters, lane == 0 ? at + 1 : at, kPieceTiles << s_shift);
                    if (lane < 2) sm.pieces[lane] = lane == 0 ? at + (begin <= r0) : at - (begin >= r1);
                }
                consumers_sync();
                if (sm.is_last) {
                    if (tid == 0) *count = 0;              // (as every launch finds it)
                    const int k_lo = sm.pieces[0], count_k = sm.pieces[1] - k_lo + 1;
#pragma unroll 1
                    for (int x = tid; x < pairs; x += 32 * kNW) {
                        const int r = x >> (c_shift - 1), c = 2 * (x & ((slice >> 1) - 1));
                        float M = -INFINITY, l = 0.f, a0 = 0.f, a1 = 0.f;
                        // piece -1: the owner's
                        const float* const first = part_of(done.u);
                        const float* const others = part_of(p.num_units + k_lo + done.u);
                        const int at_ml = 2 * r, at_v = 2 * kRows + (r << c_shift) + c, step = S * part_stride;
#pragma unroll 1
                        for (int k0 = -1; k0 < count_k; k0 += 4) {
                            float2 ml[4], v[4];        // (so many pieces' numbers on their way at a time)
#pragma unroll
                            for (int e = 0; e < 4; ++e) {
                                const float* src = k0 + e < 0 ? first : others + min(k0 + e, count_k - 1) * step;
                                ml[e] = __ldcg(reinterpret_cast<const float2*>(src + at_ml));
                                v[e] = __ldcg(reinterpret_cast<const float2*>(src + at_v));
                            }
                            float m = M;
#pragma unroll
                            for (int e = 0; e < 4; ++e) {
                                if (k0 + e >= count_k) ml[e].x = -INFINITY;
                                m = fmaxf(m, ml[e].x);
                            }
                            const float mb = m == -INFINITY ? 0.f : m, f = fast_exp2(M - mb);
                            M = m;
                            l *= f;
                            a0 *= f;
                            a1 *= f;
#pragma unroll
                            for (int e = 0; e < 4; ++e) {
                                const float g = fast_exp2(ml[e].x - mb);
                                l = fmaf(ml[e].y, g, l);
                                a0 = fmaf(v[e].x, g, a0);
                                a1 = fmaf(v[e].y, g, a1);
                            }
                        }
                        write_out(r, c, M, l, a0, a1);
                    }
                }
            }
            tiles_before = n_end;
            pieces_before = piece + 1;
            return more;
        };
        bool more = consume(First());
        if constexpr (SPREAD) {
#pragma unroll 1
            while (more) more = consume(Later());
        }
    }
    // No CTA leaves before every one has received all that was sent to it: neither the receiver's shared memory nor the
    // sender's place in the cluster may be gone while a store is under way.
    cluster_wait();
}

__global__ void __launch_bounds__(kThreads<false>, 2)
list_step_cluster_kernel(const __grid_constant__ CUtensorMap map_k, const __grid_constant__ CUtensorMap map_v,
                         const __grid_constant__ DecodeParams p) {
    list_body<false>(map_k, map_v, p);
}
__global__ void __launch_bounds__(kThreads<true>, 2)
dealt_decode_kernel(const __grid_constant__ CUtensorMap map_k, const __grid_constant__ CUtensorMap map_v,
                    const __grid_constant__ DecodeParams p) {
    list_body<true>(map_k, map_v, p);
}

cudaLaunchConfig_t config_of(bool spread, int S, int units, cudaStream_t stream, cudaLaunchAttribute (&attr)[2]) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(S, units);
    cfg.blockDim = dim3(spread ? kThreads<true> : kThreads<false>);
    cfg.dynamicSmemBytes = sizeof(ListSmem) + 1024;
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

template <typename Kernel>
int resident_of(Kernel* kernel, bool spread, int k) {
    int n = 0;
    cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(ListSmem) + 1024);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(kernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    if (e == cudaSuccess) {
        cudaLaunchAttribute attr[2];
        cudaLaunchConfig_t cfg = config_of(spread, 1 << k, 1, nullptr, attr);
        cfg.numAttrs = 1;
        if (cudaOccupancyMaxActiveClusters(&n, kernel, &cfg) != cudaSuccess) n = 0;
    }
    cudaGetLastError();                                    // (a refused size is no error of the caller's)
    return n;
}

// Clusters of 2^k CTAs that the device holds at once, asked once per device; 0: it does not take such clusters.
int resident_lists(int k) {
    static int cached[kMaxDevices][5];                     // (value + 1; 0: not asked yet.  A race asks twice and stores the same)
    int& c = cached[current_device_slot()][k];
    if (c == 0) c = min(resident_of(list_step_cluster_kernel, false, k), resident_of(dealt_decode_kernel, true, k)) + 1;
    return c - 1;
}

}  // namespace

// As many CTAs per unit as keep every cluster resident at once and still have something to do each.  Above 128 tiles a CTA the
// decode kernel, whose CTAs share all tiles throughout, is ahead where lists are ragged.  us a call, decode kernel -> clusters, 8
// KV heads; all lists equally long / lengths spread evenly from an eighth on / one sequence's lists eight times the others':
//     32 tiles a CTA      16 sequences (S = 2)  56.2 -> 45.8 / 39.8 -> 30.9 / 18.7 -> 15.5      24 (S = 1)  51.6 -> 35.8 / 39.1 -> 27.1 / 13.8 -> 15.1
//                          8 sequences (S = 4)  54.4 -> 45.1 / 38.8 -> 30.5 / 24.4 -> 19.1      10 (S = 2)  40.9 -> 31.3 / 30.5 -> 24.6 / 14.9 -> 13.8
//     48                  16 sequences          74.5 -> 64.0 / 50.1 -> 43.0 / 25.9 -> 21.3       8, dense   70.8 -> 62.5 / 47.7 -> 41.7 / 31.1 -> 22.9
//     96, dense           10 sequences (S = 2)  85.3 -> 77.1 / 55.9 -> 58.0 / 32.1 -> 26.6       4 (S = 8)  90.9 -> 83.0 / 59.1 -> 52.4 / 43.8 -> 34.8
//     128, dense           8 sequences           164 -> 155 / 101 -> 101 / 51.5 -> 46.0
//     192, dense           8 sequences           241 -> 228 / 147 -> 151
//     256, dense           8 sequences           313 -> 305 / 193 -> 201
// One long sequence among nearly empty ones: 32 tiles a CTA 16.3 -> 14.6 (24 sequences), 15.7 -> 13.9 (16), 16.8 -> 14.4 (8); 48
// 15.5 -> 15.9 (16); 64 15.3 -> 16.3 (24).  What still loses is one long list of 32 tiles a CTA among ones of 4, a CTA each (24 sequences
// 13.8 -> 15.1, dense 12.6 -> 14.7; 20 13.3 -> 14.2): the decode kernel has four tiles a CTA there, the clusters nine and a second piece.
// (A deal of 8 us, that all of a CTA's tiles but three waited for, lost up to 30 %.)
// Where half of the clusters that fit would do, and a list may have more than 32 tiles a CTA, all that fit are launched, and the long
// units dealt to those without one (a CTA by itself is far from what the memory gives): dense, one KV head of 128k 54.9 (decode
// kernel) -> 24.4, two of 55k and 156k 48.9 -> 29.6, lists of 615 tiles 21.5 -> 15.8; with 25 tiles a CTA or less nothing is gained.
ListPlan list_plan(int units, long long max_tiles) {
    ListPlan plan = {0, units, false, false};
    if (units > kListUnits || units * max_tiles >= (1ll << 30)) return plan;
    for (int k = 4; k >= 0; --k) {
        const int S = 1 << k;
        if (k > 0 && S > max_tiles) continue;              // a CTA would have nothing to do
        if (units > resident_lists(k)) continue;
        plan.spread = max_tiles > (long long)S * max(16 + 2 * S, kUndealtTiles);       // (shorter lists gain nothing by a deal)
        if (2 * units <= resident_lists(k) && max_tiles > 32ll * S) {
            plan.clusters = resident_lists(k);
            plan.spread = true;
        }
        if (max_tiles * units <= (long long)kListTiles * S * plan.clusters) plan.S = S;
        plan.next_early = 2 * plan.clusters <= resident_lists(k);
        break;
    }
    return plan;
}

size_t list_part_bytes(int units, int clusters, int S) {
    return (size_t)(2 * units + clusters) * S * (2 * kRows + (size_t)kRows * kHeadDim / S) * sizeof(float);
}

cudaError_t launch_lists(const CUtensorMap& map_k, const CUtensorMap& map_v, const DecodeParams& p, int S, cudaStream_t stream) {
    cudaLaunchAttribute attr[2];
    const cudaLaunchConfig_t cfg = config_of(p.spread, S, p.clusters, stream, attr);
    return cudaLaunchKernelEx(&cfg, p.spread ? dealt_decode_kernel : list_step_cluster_kernel, map_k, map_v, p);
}

}  // namespace seer
