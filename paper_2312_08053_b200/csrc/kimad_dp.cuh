// Stage (c): the knapsack dynamic program over the budget axis (Eq. 2, Eq. 3, Section 3.2, Algorithm 3), one CTA per
// worker, and what every way of choosing the candidates ends with (offsets, statistics, the select records).
//
// The recursion cur[b] = min_j fl(prev[b - u_j] + e_j) is serial in the layers and its binary32 sums must be taken left
// to right (the value decides ties), so the only parallelism is over the cells of a row.
//
//   * The row is cut to the cells that can matter.  Every layer takes at least its smallest candidate's cells, so the
//     row is kept relative to the sum of those: width = D - sum_l u_{l,0} + 1, candidates shifted by u_{l,0}.
//   * Where all candidates of a layer take the same number of cells (small tensors under a coarse cell) the shifted
//     layer reads its own cell only: such layers are applied in registers.  Between other layers the row is exchanged
//     through shared memory.
//   * A candidate only reads cells at or below its own, so an exchange needs no barrier: a warp owns consecutive cells and
//     waits for the warps below it only, by a progress counter per warp; rows live in a ring of a few slots, so lower
//     warps run ahead and the latencies of the warps' chains overlap.
//   * The recursion carries values only, and of several candidates with the same cells only the smallest error.  The
//     exchanged rows go to the workspace, and the winning candidates -- the first that attains the minimum -- are found on
//     the chosen path alone, last layer first, by repeating the one cell's sums.
//
// With many layers a second kernel (k_dp_windows) looks at the few cells of every row that the chosen path can visit
// (kimad_dp_window.cuh), at the same time: whole rows start as soon as the windows have, on another SM.  Both come to the same answer; the
// first to have it gives it (a worker's flags), and the other one stops when it next looks there.  Windows are up to six times as fast where they
// decide, but whether they will is known only at their end.  Where they do not, the whole rows now take 1 to 5 % longer than alone, and 4 us:
// 148 layers, 16 candidates, D = 8191, errors of a few distinct values 516 us alone, 521 (one after the other: 569); 1000 such layers
// 2780, 2865 (3480); 40 layers, 5 candidates, D = 2000 43, 46 (62).
//
// Whole rows: bound by instruction issue and shared-memory reads of one SM on wide axes (a record's uniform 128-bit reads cost about as
// much as the cells they address), by the chain of latencies per exchange on short ones, and by the cold start of the
// records and of the backtracking's rows.  Against one CTA with a barrier per layer, every candidate's index carried along
// and back-pointers for every cell: GPT-2 small's 148 layers, 16 candidates, D = 1000: 163 -> 69 us; 1995 blocks of it,
// D = 3990: 12.4 -> 1.76 ms; ResNet-18's 62 layers, 7 candidates: 60 -> 32 us.
//
// Waits are on warps of the same CTA and are bounded: a wait that runs out marks the worker's result KIMAD_ERR_TIMEOUT and
// the remaining waits are skipped.
#pragma once
#include <type_traits>

#include "kimad_kernels.cuh"

namespace kimad {

constexpr int kDpMaxThreads = 1024;
constexpr int kDpMaxRing = 8;                  // rows in flight at most
constexpr uint32_t kDpMaxChunkLayers = 256;    // layers whose records are staged at a time (two buffers)
constexpr long long kDpWaitClocks = 1ll << 31; // limit of a wait unless set otherwise: about a second (an exchange takes about a microsecond)
constexpr uint32_t kDpTimedOut = 1u, kDpStopped = 2u; // why a search over whole rows ends early: a wait ran out, the answer is there already
constexpr uint32_t kDpMostLooks = 1u << 22; // of a thread that looks whether the answer is there: about a second
constexpr uint32_t kDpSameBit = 0x10000u;      // head: all usable candidates of the layer take the same number of cells

// Plan of a launch (host).  A layer has two records of rw = 2 kr + 4 words (kr = K rounded up to 8): {byte offsets of the
// cells read, i.e. -4 (u_j - u_0), [kr] | errors [kr] | head}.  The first holds the distinct cells with their smallest
// error (head: their number | kDpSameBit, smallest error of all), the second all usable candidates (head: their number,
// the smallest error, the largest u_j - u_0); entries that cannot be used repeat candidate 0.
// Shared memory: work_bytes (two chunks of first records | ring of rows; the backtracking's rows and records lie over
// them), then a value, the exchange's layer and the choice per layer (7 bytes).
struct DpPlan {
    uint32_t kr, rw;
    uint32_t chunk_layers;
    uint32_t work_bytes;
    uint32_t smem; // dynamic shared memory in all
    uint32_t window; // bytes of work_bytes behind the records for the search over windows (kimad_dp_window.cuh); 0: whole rows only
    uint32_t window_mem; // ... and of the workspace, per worker
    uint32_t in_turn;    // whole rows only after the windows
    long long wait_clocks; // limit of a wait
};

__device__ __forceinline__ void cp_async_16(uint32_t dst, const void* src) { asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(src) : "memory"); }
__device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_all;" ::: "memory"); }
template <int OFF>
__device__ __forceinline__ float lds_f32(uint32_t addr) { float x; asm volatile("ld.shared.f32 %0, [%1+%2];" : "=f"(x) : "r"(addr), "n"(OFF)); return x; }
// x[q][k] = word 32 q of the row at addr, q < CPT
template <int CPT, int N, int Q = 0>
__device__ __forceinline__ void lds_cells(float (&x)[CPT][N], int k, uint32_t addr) {
    if constexpr (Q < CPT) {
        x[Q][k] = lds_f32<128 * Q>(addr);
        lds_cells<CPT, N, Q + 1>(x, k, addr);
    }
}
__device__ __forceinline__ float min3(float a, float b, float c) { float m; asm("min.f32 %0, %1, %2, %3;" : "=f"(m) : "f"(a), "f"(b), "f"(c)); return m; }
// A warp's progress: published by one lane after __syncwarp, which orders the warp's accesses before it, and waited for
// (bounded) by a warp until every lane's counter has reached the lane's target.  Release and acquire on the counters themselves:
// with a fence before and after plain accesses the 1995 blocks took 1.87 instead of 1.76 ms.
__device__ __forceinline__ void progress_set(uint32_t* counter, uint32_t x) { asm volatile("st.release.cta.shared.u32 [%0], %1;" ::"r"(smem_u32(counter)), "r"(x) : "memory"); }
__device__ __forceinline__ int progress_get(uint32_t counter) { int x; asm volatile("ld.acquire.cta.shared.u32 %0, [%1];" : "=r"(x) : "r"(counter) : "memory"); return x; }
// A worker's flags: non-finite values were met; the search over windows runs, and what the kernels before it wrote can be read; one of the
// searches has the answer; one of them is done (the other one clears the word for the next step).
constexpr uint32_t kFlagNonfinite = 1u, kFlagReady = 2u, kFlagChosen = 4u, kFlagDone = 8u;
// (acquire: what the one who set a flag has seen is seen; in a loop it would empty the SM's cache each time)
__device__ __forceinline__ uint32_t flags_now(const uint32_t* flags) { uint32_t x; asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(x) : "l"(flags) : "memory"); return x; }
__device__ __forceinline__ uint32_t flags_look(const uint32_t* flags) { uint32_t x; asm volatile("ld.relaxed.gpu.global.u32 %0, [%1];" : "=r"(x) : "l"(flags) : "memory"); return x; }

// A look at a worker's flags that nobody waits for: the sixteen bytes they lie in are copied to shared memory now and then, and read
// there.  (A load to a register makes its warp wait at the next branch: 10 to 35 % of the rows' time.)
struct FlagsCopy {
    const uint32_t* from;
    uint32_t to, at; // in shared memory
    __device__ __forceinline__ FlagsCopy(const uint32_t* flags, const uint32_t* copy /* [4], on a 16-byte boundary */)
        : from(reinterpret_cast<const uint32_t*>(reinterpret_cast<uintptr_t>(flags) & ~(uintptr_t)15u)), to(smem_u32(copy)),
          at(smem_u32(copy) + (uint32_t)(reinterpret_cast<uintptr_t>(flags) & 15u)) {}
    __device__ __forceinline__ void ask() const { cp_async_16(to, from); }
    __device__ __forceinline__ uint32_t chosen() const { uint32_t x; asm volatile("ld.volatile.shared.u32 %0, [%1];" : "=r"(x) : "r"(at) : "memory"); return x & kFlagChosen; }
};

// CAN_STOP: false when the warp has to wait and the search is over.  (The warps of a search that is timed out skip their waits.)
template <bool CAN_STOP>
__device__ __forceinline__ bool progress_wait(const uint32_t* counter, int target, volatile uint32_t* failed, long long limit) {
    const uint32_t at = smem_u32(counter);
    if (!__all_sync(0xffffffffu, progress_get(at) >= target)) {
        const long long start = clock64();
        while (!__all_sync(0xffffffffu, progress_get(at) >= target)) {
            if (clock64() - start > limit) *failed = kDpTimedOut;
            if (__any_sync(0xffffffffu, *failed != 0u)) {
                if (CAN_STOP) return false;
                break;
            }
        }
    }
    __syncwarp();
    return true;
}

} // namespace kimad
#include "kimad_dp_window.cuh"
namespace kimad {

// ------------------------------------------------------------------------------------------------
// What follows the choice of a candidate per layer, by one CTA: totals, capacity check, output offsets, statistics and
// the records of the select stage.
// ------------------------------------------------------------------------------------------------
struct DpBudgets { uint64_t c[kDpWorkersPerLaunch]; };

struct ChooseArgs {
    uint32_t W, L, K, D, bpe, check_finite, cost_model;
    uint64_t full_bytes, cap;
    const LayerDesc* layers;
    KTab ktab;
    const float* err;          // [W][L][K]
    const uint32_t *tau, *keep_eq, *shift; // shift: log2 of the interval's width | (code of its keys | kSelMany) << 8
    uint32_t* flags;
    Sel* sel;
    uint32_t *out_k, *out_j;
    uint64_t* out_offs;
    kimad_stats* out_stats;
    uint32_t* out_dense;       // may be null
    FbList* lists;
    uint32_t when; // 0: always; 1: only if no layer is listed for refinement or the exact path; 2: only if one is
};

// a layer listed for refinement may move on to the exact path's list while a launch with when = 1 runs, but then the
// refinement's list alone decides
__device__ __forceinline__ bool choose_applies(const ChooseArgs& a) {
    return a.when == 0u || ((a.lists->rf_layers != 0u || a.lists->n_layers != 0u) == (a.when == 2u));
}

// s_j[L]: the chosen candidates (read when status >= 0); s_k[L], s_e[L]: scratch.  `fitted`: the candidates come from the
// ratio sized to the budget, feasibility is decided here.  The total error is added left to right in binary32, over the
// layers in order, unless the caller already has that sum (`total`: the knapsack's own value of the chosen cell).  CLEAR: the worker's
// flags have served.
template <bool CLEAR = true, typename J>
__device__ __forceinline__ void choose_finish(const ChooseArgs& a, uint32_t w, uint64_t c, int status, bool fitted,
                                              const float* total, const J* s_j, uint32_t* s_k, float* s_e) {
    __shared__ unsigned long long s_nsel, s_used, s_part[kDpMaxThreads / 32];
    __shared__ int s_final;
    const uint32_t L = a.L, K = a.K, lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = blockDim.x >> 5;
    const float* e_w = a.err + (size_t)w * L * K;
    if (threadIdx.x == 0) { s_nsel = 0; s_used = 0; }
    __syncthreads();
    auto record = [&](uint32_t l) { // everything of the select record that does not depend on the totals
        const size_t o = ((size_t)w * L + l) * K + s_j[l];
        Sel s;
        s.tau = a.tau[o];
        s.keep_eq = a.keep_eq[o];
        s.shift = a.shift[o];
        s.tau_low = 0;
        s.code = s.shift >> 8; // (kept beside the interval's width)
        s.shift &= 255u;
        s.k = 0;
        s.base = 0;
        return s;
    };
    if (status >= 0) {
        unsigned long long my_n = 0, my_b = 0;
        for (uint32_t l = threadIdx.x; l < L; l += blockDim.x) {
            const uint64_t n = a.layers[l].n, k = a.ktab.at(w, (size_t)l * K + s_j[l]);
            bool dense;
            my_b += candidate_bytes(n, k, a.bpe, a.cost_model, &dense);
            const uint32_t k_eff = (uint32_t)(dense ? n : k);
            my_n += k_eff;
            s_k[l] = k_eff;
            if (!total) s_e[l] = dense ? 0.f : e_w[(size_t)l * K + s_j[l]];
            if (a.out_dense) a.out_dense[(size_t)w * L + l] = dense ? 1u : 0u;
        }
#pragma unroll
        for (int o = 16; o; o >>= 1) {
            my_n += __shfl_xor_sync(0xffffffffu, my_n, o);
            my_b += __shfl_xor_sync(0xffffffffu, my_b, o);
        }
        if (lane == 0) { atomicAdd(&s_nsel, my_n); atomicAdd(&s_used, my_b); }
    } else if (a.out_dense) {
        for (uint32_t l = threadIdx.x; l < L; l += blockDim.x) a.out_dense[(size_t)w * L + l] = 0u;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        const uint64_t nsel = s_nsel;
        float tot = 0.f;
        if (status >= 0) {
            if (total) tot = *total;
            else
                for (uint32_t l = 0; l < L; ++l) tot = __fadd_rn(tot, s_e[l]);
        }
        if (status == KIMAD_OK && fitted && s_used > c) status = KIMAD_STATUS_INFEASIBLE; // not even one entry per layer fits
        if (status >= 0 && nsel > a.cap) status = KIMAD_ERR_CAPACITY;
        kimad_stats s;
        s.budget_bytes = c;
        s.n_selected = status >= 0 ? nsel : 0;
        s.used_bytes = status >= 0 ? s_used : 0;
        s.total_err = status >= 0 ? tot : 0.f;
        s.status = status;
        a.out_stats[w] = s;
        s_final = status;
        if (CLEAR) a.flags[w] = 0;
    }
    __syncthreads();
    status = s_final;
    unsigned long long run = 0; // entries kept in the layers before this pass
    for (uint32_t l0 = 0; l0 < L; l0 += blockDim.x) {
        const uint32_t l = l0 + threadIdx.x;
        const unsigned long long k = l < L && status >= 0 ? s_k[l] : 0u;
        unsigned long long incl = k;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const unsigned long long y = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= (uint32_t)o) incl += y;
        }
        __syncthreads(); // s_part may still be read from the previous pass
        if (lane == 31) s_part[wid] = incl;
        __syncthreads();
        unsigned long long before = run, all = 0;
        for (uint32_t i = 0; i < nw; ++i) {
            const unsigned long long t = s_part[i];
            if (i < wid) before += t;
            all += t;
        }
        if (l < L) {
            const size_t wl = (size_t)w * L + l;
            const unsigned long long base = before + incl - k;
            a.out_offs[(size_t)w * (L + 1) + l] = base;
            Sel s{};
            uint32_t j = 0;
            if (status >= 0) {
                j = s_j[l];
                s = record(l);
                s.k = (uint32_t)k;
                s.base = base;
            }
            a.out_k[wl] = s.k;
            a.out_j[wl] = j;
            a.sel[wl] = s;
        }
        run += all;
    }
    if (threadIdx.x == 0) a.out_offs[(size_t)w * (L + 1) + L] = run;
}

// ------------------------------------------------------------------------------------------------
// The search over whole rows; a thread owns CPT cells of a row (32 apart: a warp owns 32 CPT consecutive cells).  Returns the
// status, or kRowsStopped.  The chosen candidates are left in shared memory, the total in *total where there was a search.
// ------------------------------------------------------------------------------------------------
constexpr int kRowsStopped = 1 << 30;
struct RowsArgs {
    uint32_t L, K, D;
    uint64_t c;            // budget in bytes
    const double* cost;    // [L][K] and the worker's errors
    const float* err;
    uint32_t* tab;         // [L][2][rw]
    float* hist;           // [exchanges][hist_row], on a 16-byte boundary
    uint32_t hist_row;
    const uint32_t* flags; // of the worker
};

// RACE: beside the search over windows, until that has the answer.
enum Race { kAlone, kWarpLooks, kFirstWarpLooks }; // no other search; a warp without cells looks for its answer; all have cells, the first looks
template <int CPT, Race RACE>
__device__ __forceinline__ int rows_search(const RowsArgs& a, const DpPlan& plan, int status, float* total) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ uint32_t s_prog[32], s_failed, s_reach, s_cell, s_left, s_signed, s_rows;
    __shared__ unsigned long long s_sum;
    __shared__ float s_redv[kDpMaxThreads / 32];
    __shared__ uint32_t s_redb[kDpMaxThreads / 32];
    __shared__ __align__(16) uint32_t s_seen[4];
    __shared__ const uint32_t* s_w_flags;

    const uint32_t L = a.L, K = a.K, D = a.D, T = blockDim.x, hist_row = a.hist_row;
    const uint32_t t = threadIdx.x, lane = t & 31, wid = t >> 5;
    const uint64_t c = a.c;
    const double* __restrict__ cost = a.cost;
    const float* __restrict__ err = a.err;
    const float kInf = __int_as_float(0x7f800000);
    const uint32_t kr = plan.kr, rw = plan.rw, rec16 = rw / 4u, CL = plan.chunk_layers, work_bytes = plan.work_bytes;
    const long long wait_clocks = plan.wait_clocks;
    uint32_t* s_tab = reinterpret_cast<uint32_t*>(smem_raw);           // [2][CL * rw]
    float* ring = reinterpret_cast<float*>(s_tab + 2u * CL * rw);
    float* s_p = reinterpret_cast<float*>(smem_raw + work_bytes);      // [L] smallest error, later the value before the layer
    uint16_t* s_ex = reinterpret_cast<uint16_t*>(s_p + L);             // [L] layer of every exchange
    uint8_t* s_j = reinterpret_cast<uint8_t*>(s_ex + L);               // [L]
    uint32_t* tab = a.tab;
    float* hist = a.hist;
    if (t == 0) { s_failed = 0; s_sum = 0; s_reach = 0; s_signed = 0; }
    if (RACE && t < 4u) s_seen[t] = 0;
    if (RACE && t == 0) { s_rows = 0; s_w_flags = a.flags; }
    const uint32_t* const volatile* w_flags = &s_w_flags; // (in shared memory: the recursion has no registers to spare)
    volatile uint32_t* failed = &s_failed;
    auto look_while = [&](auto busy) -> bool {
        for (uint32_t n = 0; n < kDpMostLooks && busy(); ++n) {
            if (flags_look(*w_flags) & kFlagChosen) {
                *failed = kDpStopped;
                return true;
            }
            __nanosleep(200);
        }
        return false;
    };
    __syncthreads();

    // ---- the layers' records; 8, 16 or 32 lanes per layer, the loads of the next layers ahead of the current ones' work
    const uint32_t G = kr <= 8u ? 8u : (kr <= 16u ? 16u : 32u), per = 32u / G; // lanes per layer, layers per warp
    const uint32_t sub = lane / G, jj = lane % G, stride = (T >> 5) * per;
    if (status == KIMAD_OK) {
        const uint32_t gmask = G == 32u ? 0xffffffffu : (((1u << G) - 1u) << (sub * G));
        constexpr int AHEAD = 4; // layers per group of lanes whose inputs are requested together (they come from DRAM on most steps)
        const uint32_t rounds = (kr + G - 1u) / G; // above 1: more than 32 candidates
        unsigned long long sum = 0;
        uint32_t reach = 0;
        bool negative = false;
        const CellsOf cells_of(c, D);
        for (uint32_t l4 = wid * per; l4 < L; l4 += AHEAD * stride) {
            double x_[AHEAD];
            float e_[AHEAD];
            auto fetch = [&](uint32_t l, uint32_t j, double& x, float& e) {
                x = 0.0; e = 0.f;
                if (l < L && j < K) { x = cost[(size_t)l * K + j]; e = err[(size_t)l * K + j]; }
            };
#pragma unroll
            for (int i = 0; i < AHEAD; ++i) fetch(l4 + i * stride + sub, jj, x_[i], e_[i]);
#pragma unroll
            for (int i = 0; i < AHEAD; ++i) {
                if (l4 + i * stride >= L) break;
                const uint32_t l = l4 + i * stride + sub;
                const bool have = l < L;
                uint32_t* rec = tab + (size_t)l * 2u * rw; // (written where `have`)
                uint32_t u0 = 0, nu = 0, nd = 0, far = 0;
                float e0 = 0.f, emin = kInf;
                bool same = true;
                for (uint32_t r = 0; r < rounds; ++r) {
                    const uint32_t j = r * G + jj;
                    if (r) fetch(l, j, x_[i], e_[i]);
                    const uint32_t u = cells_of(x_[i]);
                    const bool in = have && j < K, ok = in && u <= D; // sizes ascend with j: the usable candidates come first
                    const float e = x_[i] < 0.0 ? 0.f : e_[i];        // a layer sent densely (negative cost) loses nothing
                    if (r == 0) { u0 = __shfl_sync(0xffffffffu, u, sub * G); e0 = __shfl_sync(0xffffffffu, e, sub * G); }
                    const uint32_t du = min(u - u0, D - L + 1u); // (a row has at most D - L + 1 cells: that far is out of it from anywhere)
                    const uint32_t oks = __ballot_sync(0xffffffffu, ok) & gmask;
                    same &= (__ballot_sync(0xffffffffu, ok && u != u0) & gmask) == 0u;
                    if (oks) far = __shfl_sync(gmask, du, 31 - __clz(oks));
                    nu += __popc(oks);
                    emin = fminf(emin, ok ? e : kInf);
                    negative |= ok && e < 0.f;
                    // of two neighbours with the same cells the first is left out unless its error is the smaller one
                    const float e_right = __shfl_down_sync(0xffffffffu, e, 1);
                    const uint32_t u_right = __shfl_down_sync(0xffffffffu, u, 1);
                    const bool keep = ok && !(jj + 1u < G && ((oks >> lane) & 2u) && u_right == u && e_right <= e);
                    const uint32_t kept = __ballot_sync(0xffffffffu, keep) & gmask;
                    if (keep) {
                        const uint32_t at = nd + __popc(kept & ((1u << lane) - 1u));
                        rec[at] = 0u - 4u * du;
                        rec[kr + at] = __float_as_uint(e);
                    }
                    nd += __popc(kept);
                    if (have && j < kr) {
                        rec[rw + j] = ok ? 0u - 4u * (u - u0) : 0u;
                        rec[rw + kr + j] = __float_as_uint(ok ? e : e0);
                    }
                }
                for (uint32_t o = G >> 1; o; o >>= 1) emin = fminf(emin, __shfl_xor_sync(0xffffffffu, emin, o));
                if (have) {
                    for (uint32_t x = nd + jj; x < ((nd + 7u) & ~7u); x += G) { // the last batch repeats candidate 0
                        rec[x] = 0u;
                        rec[kr + x] = __float_as_uint(e0);
                    }
                    if (jj == 0) {
                        *reinterpret_cast<uint4*>(rec + 2u * kr) = make_uint4(nd | (same ? kDpSameBit : 0u), __float_as_uint(emin), far, 0u);
                        *reinterpret_cast<uint4*>(rec + rw + 2u * kr) = make_uint4(nu, __float_as_uint(emin), far, 0u);
                        sum += nu ? u0 : D + 1u; // not even the smallest candidate fits
                        reach = max(reach, far);
                    }
                }
            }
        }
        if (negative) s_signed = 1u;
        if (jj == 0 && sum) { atomicAdd(&s_sum, sum); atomicMax(&s_reach, reach); }
    }
    __syncthreads();
    const uint64_t least = s_sum;
    if (status == KIMAD_OK && least > D) status = KIMAD_STATUS_INFEASIBLE;
    if (status != KIMAD_OK) { // nothing to search
        for (uint32_t l = t; l < L; l += T) s_j[l] = (uint8_t)(status == KIMAD_STATUS_PLATEAU ? K - 1 : 0u);
        __syncthreads();
        return status;
    }
    const uint32_t width = D - (uint32_t)least + 1u; // cells 0 .. width - 1 above the smallest total
    const uint32_t reach = s_reach;                  // cells that a candidate reads below its own at most
    // a row has +inf in front of it, for the cells below its start
    const uint32_t margin = (reach + 3u) & ~3u, slot_words = margin + ((width + 3u) & ~3u);
    const uint32_t n_ring = min((uint32_t)kDpMaxRing, (work_bytes - 8u * CL * rw) / (4u * slot_words)); // (at least 2)
    if (t == 0) (void)KIMAD_CHECK(n_ring >= 2u && 8u * CL * rw + 4u * n_ring * slot_words <= work_bytes, 4);
    for (uint32_t i = t; i < n_ring * margin; i += T) ring[(i / margin) * slot_words + i % margin] = kInf;


    // ---- the recursion
    const uint32_t wcell = wid * (32u * CPT), cell0 = wcell + lane; // the thread's cells: cell0 + 32 q
    const bool busy = wcell < width;
    // Progress: a warp publishes s + 1 when its part of row s is written; it is then done with reading row s - 1.
    if (t < 32u) s_prog[t] = t < T / 32u && t * (32u * CPT) < width ? 0u : 0x7fffffffu; // no work: never holds anybody up
    uint32_t* prog = s_prog;
    const uint32_t n_chunks = (L + CL - 1) / CL;
    auto stage_tab = [&](uint32_t ch) { // the first records of a chunk of layers
        const uint32_t l0 = ch * CL, n16 = min(CL, L - l0) * rec16;
        const uint4* src = reinterpret_cast<const uint4*>(tab + (size_t)l0 * 2u * rw);
        const uint32_t dst = smem_u32(s_tab + (ch & 1u) * CL * rw);
        for (uint32_t i = t; i < n16; i += T) cp_async_16(dst + 16u * i, src + (i / rec16) * 2u * rec16 + i % rec16);
    };
    float v[CPT];
#pragma unroll
    for (int q = 0; q < CPT; ++q) v[q] = cell0 + 32u * q == 0u ? 0.f : kInf;
    __syncthreads(); // the records are final
    stage_tab(0);
    uint32_t seq = 0, slot = 0; // exchanges so far; slot of the next one
    float* hist_at = hist + cell0;
    // A thread of a warp without cells looks whether the other search has the answer, until the first warp is through with the chunk, and
    // then holds up the others by the counter of a warp without cells: those that work never look.  (A look at shared memory by every
    // warp and row took 3 to 5 % of the rows' time.)  Where all warps have cells the first one looks, every four
    // rows where these are short (at every row: 10 %).
    volatile uint32_t* rows_of = &s_rows;
    for (uint32_t ch = 0; ch < n_chunks; ++ch) {
        cp_async_wait();
        // this chunk's records are there, nobody reads the other buffer any more
        if (RACE) {
            if (__syncthreads_or(*failed == kDpStopped)) break; // (for all threads or none)
        } else {
            __syncthreads();
        }
        if (ch + 1 < n_chunks) stage_tab(ch + 1);
        if (!busy) {
            if (RACE == kWarpLooks && t == T - 32u && look_while([&]() { return *rows_of <= ch; })) progress_set(prog + 31, 0x80000000u); // everybody has to wait
            continue;
        }
        const uint32_t* rec = s_tab + (ch & 1u) * CL * rw;
        const uint32_t l0 = ch * CL, nl = min(CL, L - l0);
        uint2 head = *reinterpret_cast<const uint2*>(rec + 2u * kr);
        for (uint32_t i = 0; i < nl; ++i, rec += rw) {
            const uint2 h = head;
            if (i + 1 < nl) head = *reinterpret_cast<const uint2*>(rec + rw + 2u * kr);
            if (h.x & kDpSameBit) { // own cell only: the smallest error decides the value
#pragma unroll
                for (int q = 0; q < CPT; ++q) v[q] = __fadd_rn(v[q], __uint_as_float(h.y));
                if (t == 0) s_p[l0 + i] = __uint_as_float(h.y);
                continue;
            }
            const uint32_t nd = h.x;
            float* row = ring + slot * slot_words + margin;
#pragma unroll
            for (int q = 0; q < CPT; ++q)
                if (cell0 + 32u * q < width) row[cell0 + 32u * q] = v[q];
            if (t == 0 && KIMAD_CHECK(seq < L && l0 + i < L, 4)) s_ex[seq] = (uint16_t)(l0 + i);
            __syncwarp();
            if (lane == 0) progress_set(prog + wid, seq + 1u);
            const uint32_t* er = rec + kr;
            uint4 u4 = *reinterpret_cast<const uint4*>(rec), e4 = *reinterpret_cast<const uint4*>(er);
            // Two cells per thread (short rows: bound by the chain of latencies per layer): up to sixteen candidates' records
            // are read ahead of the wait and all their cells requested together.
            const bool wide = CPT == 2 && nd <= 16u;
            uint32_t u[16];
            float e[16];
            if (wide) {
                auto take = [&](int i, uint4 a, uint4 b) {
                    u[i] = a.x; u[i + 1] = a.y; u[i + 2] = a.z; u[i + 3] = a.w;
                    e[i] = __uint_as_float(b.x); e[i + 1] = __uint_as_float(b.y); e[i + 2] = __uint_as_float(b.z); e[i + 3] = __uint_as_float(b.w);
                };
                take(0, u4, e4);
                take(4, *reinterpret_cast<const uint4*>(rec + 4), *reinterpret_cast<const uint4*>(er + 4));
                if (nd > 8u) {
                    take(8, *reinterpret_cast<const uint4*>(rec + 8), *reinterpret_cast<const uint4*>(er + 8));
                    take(12, *reinterpret_cast<const uint4*>(rec + 12), *reinterpret_cast<const uint4*>(er + 12));
                }
            }
            // the warps below have written their part of this row; the others are done with the slot of the next one
            if (RACE == kFirstWarpLooks && wid == 0) { // asks at one row, looks at the next
                const FlagsCopy copy(*w_flags, s_seen);
                if ((kr > 16u || (seq & 3u) == 1u) && __any_sync(0xffffffffu, copy.chosen())) {
                    *failed = kDpStopped;
                    break;
                }
                if ((kr > 16u || (seq & 3u) == 0u) && lane == 0) copy.ask();
            }
            if (!progress_wait<RACE != kAlone>(prog + lane, lane < wid ? (int)seq + 1 : (lane == wid ? 0 : (int)seq + 3 - (int)n_ring), failed, wait_clocks)) break;
            const uint32_t addr = smem_u32(row + cell0);
            // a candidate's cells: no further below the row's start than its margin (the last warp's, past the row's end, stay in the CTA's memory)
            auto at = [&](uint32_t off) {
                return addr + (KIMAD_CHECK((int)cell0 + ((int)off >> 2) >= -(int)margin && row + cell0 + 32u * (CPT - 1) < reinterpret_cast<float*>(smem_raw + plan.smem), 5) ? off : 0u);
            };
            const int top = -4 * (int)(wcell + 32u * CPT - 1u); // offset from the warp's last cell to the row's start
#pragma unroll
            for (int q = 0; q < CPT; ++q) {
                if (cell0 + 32u * q < width) hist_at[32u * q] = v[q];
                v[q] = kInf;
            }
            hist_at += hist_row;
            auto gather = [&](auto count) { // the first `count` candidates
                constexpr int N = decltype(count)::value;
                float x[CPT][N];
#pragma unroll
                for (int k = 0; k < N; ++k) lds_cells<CPT, N>(x, k, at(u[k]));
#pragma unroll
                for (int q = 0; q < CPT; ++q) {
#pragma unroll
                    for (int k = 0; k < N; ++k) x[q][k] = __fadd_rn(x[q][k], e[k]);
#pragma unroll
                    for (int k = 0; k < N; k += 4) v[q] = min3(min3(x[q][k], x[q][k + 1], x[q][k + 2]), x[q][k + 3], v[q]);
                }
            };
            if (wide) {
                if (nd <= 8u || (int)u[8] < top) gather(std::integral_constant<int, 8>{}); // (the rest: out of reach for the warp's cells)
                else gather(std::integral_constant<int, 16>{});
            } else
            for (uint32_t j0 = 4;; j0 += 4u) { // the offsets' sizes ascend with the entry
                const uint32_t u[4] = {u4.x, u4.y, u4.z, u4.w};
                const float e[4] = {__uint_as_float(e4.x), __uint_as_float(e4.y), __uint_as_float(e4.z), __uint_as_float(e4.w)};
                float x[CPT][4]; // cells beyond the row (last warp) read what lies behind it and are never stored
#pragma unroll
                for (int k = 0; k < 4; ++k) lds_cells<CPT, 4>(x, k, at(u[k]));
                bool more = j0 < nd;
                if (more) {
                    u4 = *reinterpret_cast<const uint4*>(rec + j0);
                    e4 = *reinterpret_cast<const uint4*>(er + j0);
                    more = (int)u4.x >= top; // else out of reach for all of the warp's cells, and so are the rest
                }
#pragma unroll
                for (int q = 0; q < CPT; ++q)
                    v[q] = min3(min3(__fadd_rn(x[q][0], e[0]), __fadd_rn(x[q][1], e[1]), __fadd_rn(x[q][2], e[2])), __fadd_rn(x[q][3], e[3]), v[q]);
                if (!more) break;
            }
            ++seq;
            if (++slot == n_ring) slot = 0;
        }
        if (RACE && t == 0) *rows_of = ch + 1u;
    }

    // ---- lowest cell attaining the minimum: lexicographic (value, cell)
    float bv = kInf;
    uint32_t bb = 0xffffffffu;
#pragma unroll
    for (int q = 0; q < CPT; ++q) {
        const uint32_t b = cell0 + 32u * q;
        if (b < width && v[q] < bv) { bv = v[q]; bb = b; } // q ascending: cells ascend
    }
    auto lower = [](float ov, uint32_t ob, float v, uint32_t b) { return ov < v || (ov == v && ob < b); };
#pragma unroll
    for (int o = 16; o; o >>= 1) {
        const float ov = __shfl_xor_sync(0xffffffffu, bv, o);
        const uint32_t ob = __shfl_xor_sync(0xffffffffu, bb, o);
        if (lower(ov, ob, bv, bb)) { bv = ov; bb = ob; }
    }
    if (lane == 0) { s_redv[wid] = bv; s_redb[wid] = bb; }
    if (t == 0) s_left = seq; // (warp 0 owns the lowest cells: always busy)
    __syncthreads();          // the recursion is over for all warps, its rows are in the workspace
    if (RACE && *failed == kDpStopped) return kRowsStopped;
    const uint32_t n_ex = s_left;
    bv = s_redv[0]; bb = s_redb[0];
    for (uint32_t i = 1; i < T / 32; ++i)
        if (lower(s_redv[i], s_redb[i], bv, bb)) { bv = s_redv[i]; bb = s_redb[i]; }
    if (*failed) {
        status = KIMAD_ERR_TIMEOUT;
    } else if (!(bv < kInf)) {
        status = KIMAD_STATUS_INFEASIBLE;
        for (uint32_t l = t; l < L; l += T) s_j[l] = 0;
    } else {
        // Backtracking over the exchanged rows, last to first.  The whole CTA stages the rows of some exchanges (a window of
        // cells below the current one) and their layers' second records, then one warp walks them, a lane per candidate:
        // the first candidate that attains the minimum, and the cell it came from.
        __syncthreads(); // everybody has read the number of exchanges
        if (t == 0) s_cell = bb;
        const volatile uint32_t* walked = &s_left; // exchanges left: less once the first warp is through with the staged ones
        // Errors that the curve stage computes are not negative, and neither are their sums: they order as their bits do.
        const bool any_sign = s_signed != 0u;
        auto warp_min = [](float x, auto any) {
            if constexpr (decltype(any)::value) {
#pragma unroll
                for (int o = 16; o; o >>= 1) x = fminf(x, __shfl_xor_sync(0xffffffffu, x, o));
                return x;
            } else {
                return __uint_as_float(__reduce_min_sync(0xffffffffu, __float_as_uint(x)));
            }
        };
        __syncthreads();
        for (uint32_t left = n_ex; left;) {
            const uint32_t b0 = s_cell, lo = (b0 - min(b0, reach + 256u)) & ~3u;
            const uint32_t row16 = (b0 - lo) / 4u + 1u, per16 = rec16 + row16;
            const uint32_t nx = min(left, work_bytes / (16u * per16));
            uint4* buf = reinterpret_cast<uint4*>(smem_raw);
            for (uint32_t i = wid; i < nx; i += T / 32) { // a warp per exchange
                const uint4* r16 = reinterpret_cast<const uint4*>(tab + (size_t)s_ex[left - 1u - i] * 2u * rw + rw);
                const uint4* h16 = reinterpret_cast<const uint4*>(hist + (size_t)(left - 1u - i) * hist_row + lo);
                const uint32_t dst = smem_u32(buf + i * per16);
                for (uint32_t x = lane; x < per16; x += 32u) cp_async_16(dst + 16u * x, x < rec16 ? r16 + x : h16 + (x - rec16));
            }
            cp_async_wait();
            __syncthreads();
            // (while the first warp walks, which does not look: a test per exchange took 7 % of the search's time with 50 candidates)
            if (RACE && t == 32u) (void)look_while([&]() { return *walked == left; });
            if (wid == 0) {
                uint32_t b = b0, i = 0;
                const uint32_t* rec = reinterpret_cast<const uint32_t*>(buf);
                if (kr <= 32u) { // the next exchange's record is read ahead; lane i mod 32 keeps the result of exchange i
                    const float* row = reinterpret_cast<const float*>(rec + rw) - lo;
                    uint32_t my_j = 0;
                    float my_best = 0.f;
                    auto keep = [&](uint32_t n, uint32_t upto) { // results of the n exchanges before `upto`
                        if (lane < n) {
                            const uint32_t l = s_ex[left - 1u - (upto - n + lane)];
                            s_j[l] = (uint8_t)my_j;
                            s_p[l] = my_best;
                        }
                    };
                    const uint32_t lane_j = min(lane, kr - 1u);
                    uint32_t nu = rec[2u * kr], far = rec[2u * kr + 2u], off = (0u - rec[lane_j]) >> 2;
                    float e = __uint_as_float(rec[kr + lane_j]);
                    auto walk = [&](auto any) {
                        while (i < nx) {
                            if (lo && b - lo < far) break; // left the window: staged anew from here (never on the first exchange)
                            const bool fits = lane < nu && off <= b && KIMAD_CHECK(b - off >= lo && b <= b0, 5);
                            const float sum = fits ? __fadd_rn(row[b - off], e) : kInf;
                            const uint32_t mine = lane << 16 | off;
                            row += 4u * per16; rec += 4u * per16; // (the last ones read lie inside the buffer: work_bytes is below its end)
                            nu = rec[2u * kr]; far = rec[2u * kr + 2u]; off = (0u - rec[lane_j]) >> 2;
                            e = __uint_as_float(rec[kr + lane_j]);
                            const float best = warp_min(sum, any);
                            const uint32_t win = __reduce_min_sync(0xffffffffu, fits && sum == best ? mine : 0xffffffffu); // the first of them
                            if (lane == (i & 31u)) { my_j = win >> 16; my_best = best; }
                            b -= KIMAD_CHECK(win != 0xffffffffu, 5) ? win & 0xffffu : 0u;
                            if ((++i & 31u) == 0) keep(32u, i);
                        }
                    };
                    if (any_sign) walk(std::true_type{}); // (not a test per exchange: that took 1.6 us on 148 layers, 10 on 1995)
                    else walk(std::false_type{});
                    keep(i & 31u, i);
                } else {
                    for (; i < nx; ++i, rec += 4u * per16) {
                        const float* row = reinterpret_cast<const float*>(rec + rw) - lo;
                        const uint32_t nu = rec[2u * kr], far = rec[2u * kr + 2u];
                        if (lo && b - lo < far) break;
                        uint32_t off[4], step = 0, j = 0;
                        float sum[4], best = kInf;
#pragma unroll
                        for (int h = 0; h < 4; ++h) {
                            const uint32_t x = 32u * h + lane;
                            off[h] = 0;
                            sum[h] = kInf;
                            if (x < nu) {
                                off[h] = (0u - rec[x]) >> 2;
                                if (off[h] <= b && KIMAD_CHECK(b - off[h] >= lo && b <= b0, 5)) sum[h] = __fadd_rn(row[b - off[h]], __uint_as_float(rec[kr + x]));
                            }
                            best = fminf(best, sum[h]);
                        }
                        best = any_sign ? warp_min(best, std::true_type{}) : warp_min(best, std::false_type{});
#pragma unroll
                        for (int h = 3; h >= 0; --h) {
                            const uint32_t eq = __ballot_sync(0xffffffffu, sum[h] == best);
                            const uint32_t from = __shfl_sync(0xffffffffu, off[h], eq ? __ffs(eq) - 1 : 0);
                            if (eq) { j = 32u * h + __ffs(eq) - 1u; step = from; }
                        }
                        if (lane == 0) {
                            const uint32_t l = s_ex[left - 1u - i];
                            s_j[l] = (uint8_t)j;
                            s_p[l] = best;
                        }
                        b -= step;
                    }
                }
                if (lane == 0) { s_cell = b; s_left = left - i; }
            }
            __syncthreads();
            if (RACE && *failed) return kRowsStopped;
            left = s_left;
        }
        // The layers in between: the value before each of them (a thread per run of such layers), then the first candidate
        // that attains the layer's smallest sum.
        for (uint32_t x = t; x <= n_ex; x += T) { // run x follows exchange x - 1
            const uint32_t l0 = x ? s_ex[x - 1] + 1u : 0u, l1 = x < n_ex ? s_ex[x] : L;
            float p = x ? s_p[l0 - 1] : 0.f;
            for (uint32_t l = l0; l < l1; ++l) {
                const float q = __fadd_rn(p, s_p[l]);
                s_p[l] = p;
                s_j[l] = 0xffu;
                p = q;
            }
        }
        __syncthreads();
        for (uint32_t l = t; l < L; l += T) {
            if (s_j[l] != 0xffu) continue;
            const uint32_t* rec = tab + (size_t)l * 2u * rw + rw;
            const uint4 head = __ldcg(reinterpret_cast<const uint4*>(rec + 2u * kr));
            const float p = s_p[l], least_sum = __fadd_rn(p, __uint_as_float(head.y));
            uint32_t j = 0;
            for (uint32_t j0 = (head.x - 1u) & ~7u;; j0 -= 8u) {
                const float4 ea = __ldcg(reinterpret_cast<const float4*>(rec + kr + j0)), eb = __ldcg(reinterpret_cast<const float4*>(rec + kr + j0 + 4));
                const float e[8] = {ea.x, ea.y, ea.z, ea.w, eb.x, eb.y, eb.z, eb.w};
#pragma unroll
                for (int i = 7; i >= 0; --i) j = __fadd_rn(p, e[i]) == least_sum ? j0 + i : j;
                if (j0 == 0) break;
            }
            s_j[l] = (uint8_t)j;
        }
    }
    *total = bv;
    __syncthreads();
    return status;
}

// ------------------------------------------------------------------------------------------------
// k_dp, k_dp_windows: a CTA per worker
// ------------------------------------------------------------------------------------------------
__device__ __forceinline__ int choose_status(const ChooseArgs& a, uint64_t c, uint32_t flags) {
    if (a.check_finite && (flags & kFlagNonfinite)) return KIMAD_ERR_NONFINITE;
    return c >= a.full_bytes ? KIMAD_STATUS_PLATEAU : (c == 0 ? KIMAD_STATUS_INFEASIBLE : KIMAD_OK);
}
// Of two searches: gives the answer left in shared memory, unless the other one has given it.
__device__ __forceinline__ void choose_first(const ChooseArgs& a, const DpPlan& plan, uint32_t w, uint64_t c, int status, float total) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ uint32_t s_flags;
    __shared__ float s_total;
    if (threadIdx.x == 0) {
        s_flags = atomicOr(&a.flags[w], kFlagChosen);
        s_total = total;
    }
    __syncthreads();
    if (s_flags & kFlagChosen) return;
    uint32_t* s_k = reinterpret_cast<uint32_t*>(smem_raw); // [L], [L]: scratch (work_bytes >= 8 L)
    choose_finish<false>(a, w, c, status, false, status == KIMAD_OK ? &s_total : nullptr, smem_raw + plan.work_bytes + 6u * a.L, s_k, reinterpret_cast<float*>(s_k + a.L));
}
__device__ __forceinline__ void choose_done(const ChooseArgs& a, uint32_t w) { // (both searches get here, once)
    if (threadIdx.x == 0 && (atomicOr(&a.flags[w], kFlagDone) & kFlagDone)) a.flags[w] = 0;
}

// RACE: beside k_dp_windows, which precedes it on the stream.
template <int CPT, Race RACE>
__global__ void __launch_bounds__(CPT == 2 ? 512 : (CPT == 4 ? (RACE ? 544 : 512) : kDpMaxThreads), 1)
k_dp(DpBudgets budgets, uint32_t w_base, ChooseArgs a, DpPlan plan, const double* __restrict__ cost /* [L][K], see kimad_common.h */,
     uint32_t* __restrict__ tab_all /* [W] at tab_stride words, [L][2][rw] each */, size_t tab_stride,
     float* __restrict__ hist_all /* [W] at hist_stride words, [exchanges][hist_row] each */, size_t hist_stride, uint32_t hist_row) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ uint32_t s_flags;
    __shared__ float s_total;
    const uint32_t w = w_base + blockIdx.x, L = a.L, K = a.K, D = a.D, t = threadIdx.x;
    const float* err = a.err + (size_t)w * L * K;
    uint32_t flags = 0;
    if (RACE) {
        // Started while the windows' kernel runs, once that has started: it says when what the kernels before it wrote can be read (or it
        // has ended, if it does not).  Its end is waited for at the end here: the kernels that follow wait for this one.
        if (t == 0) s_flags = flags_now(a.flags + w);
        __syncthreads();
        if (plan.in_turn || !(s_flags & kFlagReady)) {
            __syncthreads();
            pdl_wait();
            if (t == 0) s_flags = flags_now(a.flags + w);
            __syncthreads();
        } else {
            pdl_launch();
        }
        flags = s_flags;
        if (!choose_applies(a)) return;
    } else {
        pdl_wait();
        if (!choose_applies(a)) return;
        if (a.check_finite) flags = a.flags[w];
    }
    const uint64_t c = budgets.c[blockIdx.x];
    const int known = choose_status(a, c, flags);
    if (!RACE || !(flags & kFlagChosen)) {
        float* hist = reinterpret_cast<float*>((reinterpret_cast<uintptr_t>(hist_all + w * hist_stride) + 15u) & ~(uintptr_t)15u);
        // the records and the rows fit where they are put
        if (t == 0) (void)KIMAD_CHECK((size_t)L * 2u * plan.rw <= tab_stride && (size_t)L * hist_row + (hist - (hist_all + w * hist_stride)) <= hist_stride &&
                                      D - L + 1u <= hist_row, 4);
        const RowsArgs ra{L, K, D, c, cost, err, tab_all + w * tab_stride, hist, hist_row, a.flags + w};
        float value = 0.f;
        const int status = rows_search<CPT, RACE>(ra, plan, known, &value); // (the flags are read before the end of the choice resets them)
        if constexpr (RACE) {
            if (status != kRowsStopped) choose_first(a, plan, w, c, status, value);
        } else {
            if (t == 0) s_total = value;
            __syncthreads();
            uint32_t* s_k = reinterpret_cast<uint32_t*>(smem_raw); // [L], [L]: scratch (work_bytes >= 8 L)
            choose_finish(a, w, c, status, false, status == KIMAD_OK ? &s_total : nullptr, smem_raw + plan.work_bytes + 6u * L, s_k, reinterpret_cast<float*>(s_k + L));
        }
    }
    if (RACE) {
        choose_done(a, w);
        pdl_wait();
    }
}

// ONE: all layers' records are staged at once.
template <bool ONE>
__global__ void __launch_bounds__(kWindowThreads, 1)
k_dp_windows(DpBudgets budgets, uint32_t w_base, ChooseArgs a, DpPlan plan, const double* __restrict__ cost,
             unsigned char* __restrict__ mem_all /* [W] at mem_stride bytes, mem_room each */, size_t mem_stride, size_t mem_room) {
    pdl_wait_only();
    const uint32_t w = w_base + blockIdx.x, L = a.L, t = threadIdx.x;
    if (!choose_applies(a)) return;
    if (t == 0) { // (release: what this kernel waited for is there for those who see it)
        asm volatile("red.release.gpu.global.or.b32 [%0], %1;" ::"l"(a.flags + w), "r"(kFlagReady) : "memory");
        pdl_launch();
    }
    const uint64_t c = budgets.c[blockIdx.x];
    const int status = choose_status(a, c, a.check_finite ? flags_now(a.flags + w) : 0u); // (the word is cleared when both searches are done)
    if (status == KIMAD_OK) { // (else whole rows have nothing to search either)
        unsigned char* mem = reinterpret_cast<unsigned char*>((reinterpret_cast<uintptr_t>(mem_all + w * mem_stride) + 15u) & ~(uintptr_t)15u);
        const uint32_t at_p = plan.work_bytes, at_x = at_p + 4u * L, at_j = at_x + 2u * L; // the tail of the shared memory
        const WindowArgs wa{L, a.K, a.D, plan.kr, plan.rw, c, cost, a.err + (size_t)w * L * a.K, plan.chunk_layers, 8u * plan.chunk_layers * plan.rw, plan.window,
                            mem, mem_all ? mem_room - (size_t)(mem - (mem_all + w * mem_stride)) : 0u, a.flags + w, at_p, at_x, at_j};
        float value;
        const uint32_t how = window_search<ONE>(wa, &value);
        if (t == 0 && how != kWindowStopped) atomicAdd(&a.lists->windows[how], 1u);
        if (how == kWindowFirst || how == kWindowSecond) choose_first(a, plan, w, c, KIMAD_OK, value);
    }
    choose_done(a, w);
}

// ------------------------------------------------------------------------------------------------
// k_pick: the other ways to choose a candidate per layer, one CTA per worker.
// mode 1: candidates given (j_in); mode 2: one candidate index for all layers, the largest whose total size fits the
// budget (Kimad on the grid, Section 3.1); mode 3: Algorithm 3 read with the discretised error as the axis and the size
// as the value; mode 4: the table holds, per worker, the single candidate of the ratio fitted to the budget
// (k_fit_ratio): nothing to search.
// Shared memory (the host computes the same sizes): two rows of (D + 2) "none" followed by D + 1 values | j[L] | mode 3:
// cells[L Kp], sizes[L Kp], Kp = K rounded up to 4 | back-pointers, where they fit.  The margin in front of each row lets
// prev[b - u] be read without a bounds test.  Back-pointers: a nibble when K <= 16, else a byte.
// ------------------------------------------------------------------------------------------------
constexpr int kPickThreads = 512;
constexpr int kPickCells = 2; // budget cells per thread (mode 3)
struct PickPlan {
    uint32_t pd_in_smem; // else in the caller's workspace
    uint32_t pd_nibble;
    uint32_t pd_row_bytes;
};

__global__ void __launch_bounds__(kPickThreads)
k_pick(DpBudgets budgets, uint32_t w_base, ChooseArgs a, int mode, PickPlan plan, const uint32_t* __restrict__ j_in,
       uint8_t* __restrict__ pd_global) {
    pdl_wait();
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const uint32_t w = w_base + blockIdx.x, L = a.L, K = a.K, D = a.D;
    if (!choose_applies(a)) return;
    const uint64_t c = budgets.c[blockIdx.x];
    const uint32_t row = D + 1, pad = D + 2, rowp = row + pad, Kp = (K + 3) & ~3u;
    uint32_t* prow = reinterpret_cast<uint32_t*>(smem_raw);
    uint32_t* s_j = prow + 2 * rowp; // [L]
    __shared__ int s_status;
    const LayerDesc* layers = a.layers;
    const KTab ktab = a.ktab;

    int status = KIMAD_OK;
    if (a.check_finite && (a.flags[w] & kFlagNonfinite)) status = KIMAD_ERR_NONFINITE;
    __syncthreads(); // the flags are read before the end of the choice resets them
    if (status == KIMAD_OK) {
        if (mode == 1) {
            for (uint32_t l = threadIdx.x; l < L; l += blockDim.x) s_j[l] = min(j_in[(size_t)w * L + l], K - 1);
        } else if (c >= a.full_bytes) {
            status = KIMAD_STATUS_PLATEAU;
            for (uint32_t l = threadIdx.x; l < L; l += blockDim.x) s_j[l] = K - 1;
        } else if (c == 0) {
            status = KIMAD_STATUS_INFEASIBLE;
            for (uint32_t l = threadIdx.x; l < L; l += blockDim.x) s_j[l] = 0;
        } else if (mode == 2) {
            // total size of candidate j over the layers; sizes ascend with j.  A warp per j, layers dealt out to its lanes
            __shared__ uint32_t s_fit; // number of candidates that fit
            if (threadIdx.x == 0) s_fit = 0;
            __syncthreads();
            for (uint32_t j = threadIdx.x >> 5; j < K; j += blockDim.x >> 5) {
                unsigned long long bytes = 0;
                for (uint32_t l = threadIdx.x & 31u; l < L; l += 32u)
                    bytes += candidate_bytes(layers[l].n, ktab.at(w, (size_t)l * K + j), a.bpe, a.cost_model, nullptr);
#pragma unroll
                for (int o = 16; o; o >>= 1) bytes += __shfl_xor_sync(0xffffffffu, bytes, o);
                if ((threadIdx.x & 31u) == 0 && bytes <= c) atomicMax(&s_fit, j + 1);
            }
            __syncthreads();
            const uint32_t fit = s_fit;
            if (fit == 0) status = KIMAD_STATUS_INFEASIBLE;
            for (uint32_t l = threadIdx.x; l < L; l += blockDim.x) s_j[l] = fit ? fit - 1 : 0;
        } else if (mode == 4) {
            for (uint32_t l = threadIdx.x; l < L; l += blockDim.x) s_j[l] = 0; // feasibility is decided on the totals
        } else {
            // Error axis: E_max = sum_l err_{l,0} (binary64, layers in order), cells e_{l,j} = floor(err D / E_max),
            // value = fewest kept entries for a total of exactly e cells; answer = lowest e whose value fits c.
            __shared__ double s_emax;
            __shared__ uint32_t s_best;
            uint32_t* pv = prow + pad;
            uint32_t* cu = prow + rowp + pad;
            const float* e_w = a.err + (size_t)w * L * K;
            uint32_t* s_units = s_j + L;       // [L * Kp]
            uint32_t* s_kk = s_units + L * Kp; // [L * Kp]
            uint8_t* pd = plan.pd_in_smem ? reinterpret_cast<uint8_t*>(s_kk + L * Kp) : pd_global + (size_t)w * L * plan.pd_row_bytes;
            const uint32_t kNone = 0xffffffffu;
            if (threadIdx.x == 0) {
                double e = 0.0;
                for (uint32_t l = 0; l < L; ++l) e = __dadd_rn(e, (double)e_w[(size_t)l * K]);
                s_emax = e;
                s_best = kNone;
            }
            __syncthreads();
            const double emax = s_emax;
            for (uint32_t i = threadIdx.x; i < L * Kp; i += blockDim.x) {
                const uint32_t l = i / Kp, j = i % Kp;
                uint32_t u = D + 1, kk = 0; // padding reads the margin
                if (j < K) {
                    const double q = emax > 0.0 ? floor(__ddiv_rn(__dmul_rn((double)e_w[(size_t)l * K + j], (double)D), emax)) : 0.0;
                    u = q > (double)D ? D : (uint32_t)q;
                    kk = (uint32_t)ktab.at(w, (size_t)l * K + j);
                }
                s_units[i] = u;
                s_kk[i] = kk;
            }
            for (uint32_t i = threadIdx.x; i < 2 * rowp; i += blockDim.x) prow[i] = kNone;
            __syncthreads();
            if (threadIdx.x == 0) pv[0] = 0;
            for (uint32_t l = 0; l < L; ++l) {
                __syncthreads();
                const uint32_t* un = s_units + l * Kp;
                const uint32_t* kk = s_kk + l * Kp;
                uint8_t* pdl = pd + (size_t)l * plan.pd_row_bytes;
                for (uint32_t bb = 0; bb < row; bb += kPickCells * blockDim.x) {
#pragma unroll
                    for (int q = 0; q < kPickCells; ++q) {
                        const uint32_t b = bb + threadIdx.x + q * blockDim.x;
                        const uint32_t bc = min(b, row - 1);
                        uint32_t best = kNone, bj = 0;
                        for (uint32_t j = 0; j < K; ++j) {
                            const uint32_t p = pv[(int)bc - (int)un[j]];
                            const uint32_t t = p > kNone - kk[j] ? kNone : p + kk[j];
                            if (t < best) { best = t; bj = j; }
                        }
                        if (b < row) cu[b] = best;
                        if (plan.pd_nibble) {
                            const uint32_t nb = __shfl_down_sync(0xffffffffu, bj, 1);
                            if (!(threadIdx.x & 1) && b < row) pdl[b >> 1] = (uint8_t)(bj | (nb << 4));
                        } else if (b < row) {
                            pdl[b] = (uint8_t)bj;
                        }
                    }
                }
                uint32_t* sw = pv; pv = cu; cu = sw;
            }
            __syncthreads();
            const uint64_t cap_k = c / a.bpe;
            for (uint32_t b = threadIdx.x; b < row; b += blockDim.x)
                if (pv[b] != kNone && (uint64_t)pv[b] <= cap_k) atomicMin(&s_best, b);
            __syncthreads();
            if (threadIdx.x == 0) {
                if (s_best == kNone) {
                    s_status = KIMAD_STATUS_INFEASIBLE;
                } else {
                    s_status = KIMAD_OK;
                    uint32_t b = s_best;
                    for (uint32_t l = L; l-- > 0;) {
                        const uint8_t* pdl = pd + (size_t)l * plan.pd_row_bytes;
                        const uint32_t j = plan.pd_nibble ? ((pdl[b >> 1] >> (4 * (b & 1))) & 15u) : pdl[b];
                        s_j[l] = j;
                        b -= s_units[l * Kp + j];
                    }
                }
            }
            __syncthreads();
            status = s_status;
            if (status == KIMAD_STATUS_INFEASIBLE)
                for (uint32_t l = threadIdx.x; l < L; l += blockDim.x) s_j[l] = 0;
        }
    }
    __syncthreads();
    // (the rows are free now; L <= D < the rows' size)
    choose_finish(a, w, c, status, mode == 4, nullptr, s_j, prow, reinterpret_cast<float*>(prow) + rowp);
}

// The ratio of Section 3.1 sized to the budget: r = q / 2^32 with the largest q whose entries
// sum_l min(n_l, max(1, floor(q n_l / 2^32))) fit floor(c / (4 + vb)); the worker's table row gets those k_l.
// One CTA per worker; the sums are order-free integers.  The interval of q is cut into 33 at a time, a warp per cut: seven
// rounds instead of the 33 of a bisection (ResNet-18's 62 layers: 24 -> 8 us, ahead of everything else of the step).
constexpr int kFitThreads = 1024;
__global__ void __launch_bounds__(kFitThreads)
k_fit_ratio(DpBudgets budgets, uint32_t w_base, uint32_t W, uint32_t L, uint32_t bpe, uint64_t N,
            const LayerDesc* __restrict__ layers, uint64_t* __restrict__ ktab_w /* [W][L] */) {
    pdl_wait();
    constexpr uint32_t kCuts = kFitThreads / 32;
    constexpr int kNear = 1024; // layer sizes kept in shared memory (the others are read where they are)
    __shared__ uint32_t s_n[kNear], s_fits;
    const uint32_t w = w_base + blockIdx.x, lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const uint64_t entries = budgets.c[blockIdx.x] / bpe;
    auto k_of = [&](uint64_t q, uint64_t n) {
        uint64_t k = q >= 4294967296ull ? n : (q * n) >> 32;
        k = k < 1 ? 1 : k;
        return k > n ? n : k;
    };
    for (uint32_t l = threadIdx.x; l < min(L, (uint32_t)kNear); l += kFitThreads) s_n[l] = (uint32_t)layers[l].n;
    auto size = [&](uint32_t l) -> uint64_t { return l < (uint32_t)kNear ? s_n[l] : layers[l].n; };
    if (threadIdx.x == 0) s_fits = 0;
    __syncthreads();
    uint64_t q;
    if (entries < (uint64_t)L) q = 0;
    else if (entries >= N) q = 4294967296ull;
    else {
        uint64_t lo = 0, hi = 4294967296ull; // sum(lo) <= entries < sum(hi)
        while (hi - lo > 1) {
            const uint64_t at = lo + ((hi - lo) * (wid + 1)) / (kCuts + 1); // ascending with the warp; may repeat once hi - lo is small
            unsigned long long sum = 0;
            for (uint32_t l = lane; l < L; l += 32) sum += k_of(at, size(l));
#pragma unroll
            for (int o = 16; o; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
            if (lane == 0 && sum <= entries) atomicMax(&s_fits, wid + 1); // sums ascend with q
            __syncthreads();
            const uint32_t fits = s_fits;
            __syncthreads();
            if (threadIdx.x == 0) s_fits = 0;
            const uint64_t span = hi - lo, base = lo;
            if (fits) lo = base + (span * fits) / (kCuts + 1);
            if (fits < kCuts) hi = base + (span * (fits + 1)) / (kCuts + 1);
            __syncthreads();
        }
        q = lo;
    }
    if (w < W)
        for (uint32_t l = threadIdx.x; l < L; l += kFitThreads) ktab_w[(size_t)w * L + l] = k_of(q, size(l));
}

} // namespace kimad
