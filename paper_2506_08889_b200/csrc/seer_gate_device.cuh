// Device-side parts of the gate that its kernels share with the one-kernel decode step: dot products of
// bf16 pieces, the reduction over a key's lanes, the order-preserving key of a score, the cluster barrier.
#pragma once

#include "seer_device.cuh"

namespace seer {

__device__ __forceinline__ float dot8(const uint4& a, const float* x) {
    const __nv_bfloat162* h = reinterpret_cast<const __nv_bfloat162*>(&a);
    float acc = 0.f;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        float2 f = bf16x2_to_float2(h[k]);
        acc = fmaf(f.x, x[2 * k], acc);
        acc = fmaf(f.y, x[2 * k + 1], acc);
    }
    return acc;
}
__device__ __forceinline__ float dot8(const uint4& a, const uint4& b) {
    const __nv_bfloat162* h = reinterpret_cast<const __nv_bfloat162*>(&a);
    const __nv_bfloat162* g = reinterpret_cast<const __nv_bfloat162*>(&b);
    float acc = 0.f;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        const float2 f = bf16x2_to_float2(h[k]), e = bf16x2_to_float2(g[k]);
        acc = fmaf(f.x, e.x, acc);
        acc = fmaf(f.y, e.y, acc);
    }
    return acc;
}

// v[k], k = 0..7, summed over a group of `group` = 8, 16 or 32 neighbouring lanes, eight sums for
// 8 + (log2(group) - 3) shuffles: lanes exchange half of what they carry and go on with the other half,
// so a lane ends with the group's sum of v[r], r = its low three lane bits in reverse order.
__device__ __forceinline__ float reduce8(const float (&v)[8], int lane, int group) {
    const bool b0 = lane & 1, b1 = lane & 2, b2 = lane & 4;
    float w4[4], w2[2];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const float keep = b0 ? v[i + 4] : v[i], send = b0 ? v[i] : v[i + 4];
        w4[i] = keep + __shfl_xor_sync(0xffffffffu, send, 1);
    }
#pragma unroll
    for (int i = 0; i < 2; ++i) {
        const float keep = b1 ? w4[i + 2] : w4[i], send = b1 ? w4[i] : w4[i + 2];
        w2[i] = keep + __shfl_xor_sync(0xffffffffu, send, 2);
    }
    const float keep = b2 ? w2[1] : w2[0], send = b2 ? w2[0] : w2[1];
    float x = keep + __shfl_xor_sync(0xffffffffu, send, 4);
    for (int off = 8; off < group; off <<= 1) x += __shfl_xor_sync(0xffffffffu, x, off);
    return x;
}

// Order-preserving key: larger score <-> larger key; -0 == +0; NaN below everything.
__device__ __forceinline__ uint32_t score_key(float s) {
    if (s != s) return 0u;
    uint32_t b = __float_as_uint(s);
    if (b == 0x80000000u) b = 0u;
    return (b & 0x80000000u) ? ~b : (b | 0x80000000u);
}

// Inverse of score_key (NaN came out as key 0 and goes back as -inf).
__device__ __forceinline__ float key_score(uint32_t key) {
    if (key == 0u) return -INFINITY;
    return __uint_as_float((key & 0x80000000u) ? (key ^ 0x80000000u) : ~key);
}

// Split cluster barrier (all threads of all CTAs of the cluster execute both halves).  The aligned forms are for a warp
// whose lanes are together; behind a branch that only some lanes take they need not be, so they are brought together here.
#define SEER_CLUSTER_ARRIVE(sem) do { __syncwarp(); asm volatile("barrier.cluster.arrive" sem ".aligned;" ::: "memory"); } while (0)
__device__ __forceinline__ void cluster_arrive() { SEER_CLUSTER_ARRIVE(".release"); }
// ... where nothing that this thread has written is handed over with it: it does not wait for its stores.
__device__ __forceinline__ void cluster_arrive_relaxed() { SEER_CLUSTER_ARRIVE(".relaxed"); }
__device__ __forceinline__ void cluster_wait() {
    __syncwarp();
    asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}
__device__ __forceinline__ void cluster_sync() {
    cluster_arrive();
    cluster_wait();
}

}  // namespace seer
