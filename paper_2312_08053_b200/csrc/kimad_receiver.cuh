// Receiving side of a message and the model step (Algorithm 1, server lines):
//   k_apply_packed  u^_m += C_m(.)  scatter-add of the packed (index, value) entries of every worker
//   k_aggregate     x <- x - gamma * sum_m w_m u^_m, a dense stream over W + 1 arrays
#pragma once
#include "kimad_kernels.cuh"

namespace kimad {

// One CTA row per worker (blockIdx.y); entries are visited with a grid-stride loop because their number is only known on the
// device (offs[L]).  A warp takes 128 consecutive entries, four per lane: one bisection in offs for the first of them (the
// layers of the others follow it), then four indices and values and four estimator entries per lane in flight.  Bound by
// the scattered 32-byte sectors it reads and writes back.  One entry per thread with a bisection each took
// 816 us for 33 M bf16 entries of each of four workers, this form 714; 3.1 M entries of each (150 us) are bound by the sectors.
template <bool BF16>
__global__ void __launch_bounds__(kThreads)
k_apply_packed(const uint32_t* __restrict__ idx, const void* __restrict__ val, const uint64_t* __restrict__ offs,
               const LayerDesc* __restrict__ layers, uint32_t L, uint64_t cap, uint64_t stride,
               float* __restrict__ est) {
    pdl_wait();
    constexpr int PER = 4;
    const uint32_t w = blockIdx.y, lane = threadIdx.x & 31;
    const uint64_t* of = offs + (size_t)w * (L + 1);
    const uint64_t total = min(of[L], cap);
    const uint32_t* ix = idx + (size_t)w * cap;
    float* e = est + (size_t)w * stride;
    const uint64_t step = (uint64_t)gridDim.x * (kThreads * PER);
    for (uint64_t p0 = ((uint64_t)blockIdx.x * (kThreads / 32) + (threadIdx.x >> 5)) * (32 * PER); p0 < total; p0 += step) {
        uint32_t i[PER];
        float v[PER];
#pragma unroll
        for (int u = 0; u < PER; ++u) {
            const uint64_t p = p0 + lane + 32u * u;
            i[u] = 0xffffffffu;
            v[u] = 0.f;
            if (p < total) {
                i[u] = __ldcs(ix + p);
                v[u] = BF16 ? __bfloat162float(reinterpret_cast<const __nv_bfloat16*>(val)[(size_t)w * cap + p])
                            : __ldcs(reinterpret_cast<const float*>(val) + (size_t)w * cap + p);
            }
        }
        uint32_t lo = 0, hi = L; // invariant: of[lo] <= p0 < of[hi]
        while (hi - lo > 1) {
            const uint32_t mid = (lo + hi) >> 1;
            if (of[mid] <= p0) lo = mid; else hi = mid;
        }
        float* dst[PER];
        float was[PER];
        uint64_t end = of[lo + 1];
        LayerDesc ld = layers[lo];
#pragma unroll
        for (int u = 0; u < PER; ++u) {
            const uint64_t p = p0 + lane + 32u * u;
            dst[u] = nullptr;
            was[u] = 0.f;
            if (p < total) {
                if (p >= end) {
                    do end = of[++lo + 1]; while (p >= end);
                    ld = layers[lo];
                }
                if ((uint64_t)i[u] < ld.n) { // every index occurs once per message: no two threads share an element
                    dst[u] = e + ld.begin + i[u];
                    was[u] = *dst[u];
                }
            }
        }
#pragma unroll
        for (int u = 0; u < PER; ++u)
            if (dst[u]) *dst[u] = __fadd_rn(was[u], v[u]);
    }
}

struct AggWeights { float w[KIMAD_MAX_AGG_WORKERS]; };

template <bool VEC>
__global__ void __launch_bounds__(kThreads)
k_aggregate(float* __restrict__ x, const float* __restrict__ est, uint64_t stride, uint32_t W, uint64_t n,
            AggWeights wt, float gamma) {
    pdl_wait();
    const uint64_t step = (uint64_t)gridDim.x * kThreads;
    if (VEC) {
        const uint64_t nq = n / 4;
        for (uint64_t q = (uint64_t)blockIdx.x * kThreads + threadIdx.x; q < nq; q += step) {
            float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
            for (uint32_t m = 0; m < W; ++m) {
                const float4 e = __ldcs(reinterpret_cast<const float4*>(est + (size_t)m * stride) + q);
                const float wm = wt.w[m];
                acc.x = __fadd_rn(acc.x, __fmul_rn(wm, e.x)); acc.y = __fadd_rn(acc.y, __fmul_rn(wm, e.y));
                acc.z = __fadd_rn(acc.z, __fmul_rn(wm, e.z)); acc.w = __fadd_rn(acc.w, __fmul_rn(wm, e.w));
            }
            float4 v = reinterpret_cast<float4*>(x)[q];
            v.x = __fsub_rn(v.x, __fmul_rn(gamma, acc.x)); v.y = __fsub_rn(v.y, __fmul_rn(gamma, acc.y));
            v.z = __fsub_rn(v.z, __fmul_rn(gamma, acc.z)); v.w = __fsub_rn(v.w, __fmul_rn(gamma, acc.w));
            reinterpret_cast<float4*>(x)[q] = v;
        }
    }
    const uint64_t tail0 = VEC ? (n / 4) * 4 : 0;
    for (uint64_t i = tail0 + (uint64_t)blockIdx.x * kThreads + threadIdx.x; i < n; i += step) {
        float acc = 0.f;
        for (uint32_t m = 0; m < W; ++m) acc = __fadd_rn(acc, __fmul_rn(wt.w[m], est[(size_t)m * stride + i]));
        x[i] = __fsub_rn(x[i], __fmul_rn(gamma, acc));
    }
}

} // namespace kimad
