// Parts shared by the kernels that give a unit (one sequence's KV head) a thread-block cluster: stores that count their bytes
// down on the receiver's mbarrier, the layout of a staged K/V tile.
#pragma once

#include "seer_gate_device.cuh"
#include "seer_internal.h"

namespace seer {

constexpr int kHalfTileBytes = kTileTokens * 128;          // 64 rows x 128 B (64 bf16 channels)
constexpr int kTileBytes = 2 * kHalfTileBytes;             // one K or V tile: 16 KiB
constexpr int kStageBytes = 2 * kTileBytes;                // K + V
constexpr int kMaxS = 16;                                  // CTAs of a cluster

// Barriers among the worker warps, and between them and the producer.  The aligned forms are for a warp whose lanes are
// together; behind a loop or branch of some lanes they need not be, so they are brought together here.
template <int NW>
__device__ __forceinline__ void worker_sync() {
    __syncwarp();
    asm volatile("bar.sync 1, %0;" ::"n"(32 * NW) : "memory");
}

// ---- stores into a CTA of the cluster (addr, bar: of its shared memory, cluster_addr), counted on its mbarrier ----------
__device__ __forceinline__ uint32_t cluster_addr(const void* mine, int rank) {
    uint32_t a;
    asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(a) : "r"(smem_u32(mine)), "r"(rank));
    return a;
}
__device__ __forceinline__ void send_u32(uint32_t addr, uint32_t v, uint32_t bar) {
    asm volatile("st.async.shared::cluster.mbarrier::complete_tx::bytes.u32 [%0], %1, [%2];" ::"r"(addr), "r"(v), "r"(bar) : "memory");
}
__device__ __forceinline__ void send_f32x2(uint32_t addr, float2 v, uint32_t bar) {
    asm volatile("st.async.shared::cluster.mbarrier::complete_tx::bytes.v2.f32 [%0], {%1, %2}, [%3];" ::"r"(addr), "f"(v.x), "f"(v.y), "r"(bar)
                 : "memory");
}
__device__ __forceinline__ void send_f32x4(uint32_t addr, float4 v, uint32_t bar) {
    asm volatile("st.async.shared::cluster.mbarrier::complete_tx::bytes.v4.f32 [%0], {%1, %2, %3, %4}, [%5];" ::"r"(addr), "f"(v.x), "f"(v.y),
                 "f"(v.z), "f"(v.w), "r"(bar)
                 : "memory");
}
__device__ __forceinline__ void send_min(uint32_t addr, uint32_t v, uint32_t bar) {
    asm volatile("red.async.relaxed.cluster.shared::cluster.mbarrier::complete_tx::bytes.min.u32 [%0], %1, [%2];" ::"r"(addr), "r"(v), "r"(bar)
                 : "memory");
}
__device__ __forceinline__ void send_max(uint32_t addr, uint32_t v, uint32_t bar) {
    asm volatile("red.async.relaxed.cluster.shared::cluster.mbarrier::complete_tx::bytes.max.u32 [%0], %1, [%2];" ::"r"(addr), "r"(v), "r"(bar)
                 : "memory");
}
// Bounded wait for what the cluster's CTAs have sent (by default the first phase of `bar`).
__device__ __forceinline__ bool wait_sent(uint64_t* bar, unsigned int* status, uint32_t parity = 0) {
    uint32_t ok = 0;
    for (uint32_t it = 0; it < (1u << 24) && !ok; ++it) {
        asm volatile(
            "{\n\t.reg .pred p;\n\t"
            "mbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\n\t"
            "selp.u32 %0, 1, 0, p;\n\t}"
            : "=r"(ok)
            : "r"(smem_u32(bar)), "r"(parity)
            : "memory");
        if (!ok && it > 64) __nanosleep(64);
    }
    if (!ok) raise_status(status, DEV_TIMEOUT);
    __syncwarp();                                          // (the lanes need not have left the loop together)
    return ok != 0;
}

// Whether the lists are dealt.  In hundredths of a microsecond: a CTA that has the memory to itself gets through a tile in 0.46
// us (three stages, of which one or two are being read); all CTAs together through one in 0.0047 us, taken as 0.004 because
// the last ones are alone with their tiles; a deal costs 5 us: the pieces' way through global memory and the helpers' second start.
// Dealt lists take as long as twelve tiles a CTA at least, nine that are never dealt and a piece's three (24 sequences, one of 20 tiles a
// CTA, the others of 2: not dealt 13.0, dealt, without this bound, 14.0).
// (24 sequences, a quarter of them with 32 tiles a CTA, the others with 4: dealt 20.3 us, not dealt, as by a line of 8 us, 24.2; 10
// sequences, lengths spread evenly up to 48 tiles a CTA: not dealt 34.1, dealt, as by a line of 3 us, 43.2.)
// A step's lists are dealt by a kernel behind it: 8 us (10 sequences, half of them with 72 tiles a CTA, the others with 9: not dealt
// 62.2, dealt, as by a line of 5 us, 68.6; 8, a quarter with 80: dealt 59.3, not dealt, as by one of 11 us, 70.6).
constexpr int kTileTime = 46, kDealTime = 500, kStepDealTime = 800;
constexpr int kPieceTiles = 6;                             // a piece costs a helper as much as so many tiles a CTA (by 8, lists of 17 us 18)
// Lists of so many tiles a CTA are even to list_uneven: the kernel that does not ask (24 sequences, one of 20 tiles a CTA, the others of 2,
// 13.1 -> 11.4 us; half of them of 20 19.5 -> 18.8).
constexpr int kUndealtTiles = 2 * kPieceTiles + kDealTime / kTileTime;
__device__ __forceinline__ bool list_uneven(int total, int most, int units, int S, int deal = kDealTime) {
    // (most * kTileTime / S > max(0.4 * total, total * kTileTime / (units * S), 12 * kTileTime) + deal, without its divisions)
    return 5ll * kTileTime * most * units >
           max(max(2ll * total * S * units, 5ll * kTileTime * total), 5ll * kTileTime * (2 * kPieceTiles) * S * units) + 5ll * deal * S * units;
}
// The same of a step's lists, as the sequences' lengths give them (whole warp).
__device__ __forceinline__ bool step_uneven(const DecodeParams& p, int S) {
    int total = 0, most = 0;
    for (int i = threadIdx.x & 31; i < p.batch; i += 32) {
        const int L = p.seq_lens[i], n = L > 0 ? min((L + p.block_size - 1) >> p.bs_shift, p.sel_from_lens) : 0;
        const int tiles = p.blocks_per_tile > 1 ? (n + p.blocks_per_tile - 1) >> p.bpt_shift : n << p.tpb_shift;
        total += tiles;
        most = max(most, tiles);
    }
    return list_uneven(__reduce_add_sync(0xffffffffu, total) * p.num_kv_heads, __reduce_max_sync(0xffffffffu, most), p.num_units, S, kStepDealTime);
}

}  // namespace seer
