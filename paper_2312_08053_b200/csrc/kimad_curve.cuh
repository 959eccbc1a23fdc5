// Stage (a)+(b), fast path: EF21 difference fused with a banded histogram that yields the error curve of
// every candidate in ONE sweep over the gradients.
//
//   k_sample     per (worker, layer): histogram of a stratified sample of |d| over 16-bit key prefixes
//                ("cells"); for every candidate k_j the cells that can contain the k_j-th largest key
//                (sample rank +- 6 sigma) form a band.  Band cells are cut into fine bins of 2^shift
//                keys, everything else into coarse "gap" bins.  Every region (a gap, or a group of bands with
//                one bin width) maps a key to its bin as base + (key >> shift); which region a key lies in is
//                read from a table over the window of cells between the lowest and the highest band.
//                A mass of exact zeros in the sample (a sparse gradient) is counted apart: such a layer's zeros
//                stay out of the sweep's histogram, candidates whose rank lies among them need no band, and
//                sigma grows by what the spread of the zeros over the sampled units says about their clustering.
//   k_pass_a     the sweep: d = grad - g (one code byte per element goes to scratch), bin = base + (key >> shift)
//                with (base, shift) = table(cell(key)), two u32 shared-memory atomics per element: the count, and
//                the exact integer sum of squares in a u32 word whose (rare) carries go straight to the 64-bit sum
//                in global memory.  CTAs own static runs of chunks of equal cost.
//   k_resolve_a  per (worker, layer): totals of every group of 32 bins, a scan over the groups, then a warp per
//                candidate finds the group and the bin that hold its threshold (zeros left out by the sweep = the
//                layer's size minus the counted entries) and the squares below it.  The candidate's error is certified to 5e-6 relative from the bin's width.  A
//                threshold in a gap bin (the sample mispredicted) sends the layer to the exact radix path; a bound
//                that is too loose sends the candidate to the refinement.
//   k_refine     loose candidates: the entries of the threshold's bin, found by their code byte, are counted in
//                1024 pieces of the bin; error and interval from the pieces (still loose: exact path).
//   k_tiny_exact layers of at most kTinyMax elements are sorted in shared memory instead.
//   k_fb1, k_fb23 exact three-digit radix select over the chunks of the layers handed over (rare).
#pragma once
#include "kimad_kernels.cuh"
#include <type_traits>

namespace kimad {

constexpr int kTinyMax = 4096;
#ifndef KIMAD_FINE_BINS
#define KIMAD_FINE_BINS 12288
#endif
constexpr int kFineBins = KIMAD_FINE_BINS;          // fine bins per (worker, layer)
constexpr int kMaxGaps = KIMAD_MAX_RATIOS + 2;      // gap regions: below / between / above the band groups, + non-finite keys
constexpr int kBaseWords = kMaxGaps + 2;            // first bin of every gap and of the keys that are not finite; the number of bins
constexpr int kMaxBins = kFineBins + kL1Bins + 2 * kMaxGaps; // fine bins + gap regions cut at every 11-bit prefix
static_assert(kBaseWords > KIMAD_MAX_RATIOS + 1 + 2, "a group of bands per candidate and one above them");
constexpr int kMaxShift = 15;                       // a fine bin is 2^shift keys wide, at most a whole cell
constexpr int kBigThreads = 1024;
static_assert(kSampleRound == 8 * (kBigThreads / kSampleUnit), "eight units per warp and round");
constexpr uint32_t kGapBit = 1u;                    // bin_lo entries carry this bit when the bin is a gap bin


struct WarpLanes {
    uint32_t lane = threadIdx.x & 31u, lanes = 32;
    __device__ __forceinline__ uint32_t sum(uint32_t x) const { return __reduce_add_sync(0xffffffffu, x); }
    __device__ __forceinline__ void sync() const { __syncwarp(); }
};

__device__ __forceinline__ uint32_t select(uint32_t c, uint32_t x, uint32_t y) { // c != 0 ? x : y, without a branch
    uint32_t r;
    asm("{.reg .pred p; setp.ne.u32 p, %1, 0; selp.b32 %0, %2, %3, p;}" : "=r"(r) : "r"(c), "r"(x), "r"(y));
    return r;
}
__device__ __forceinline__ uint32_t hash_u32(uint32_t x) {
    x ^= x >> 16; x *= 0x7feb352du; x ^= x >> 15; x *= 0x846ca68bu; x ^= x >> 16;
    return x;
}

// A cluster's CTAs meet; what one of them wrote before is seen by all of them after.
__device__ __forceinline__ void cluster_arrive() { asm volatile("barrier.cluster.arrive.release;" ::: "memory"); }
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait.acquire;" ::: "memory"); }
// The word at `addr` (shared memory of this CTA) in the shared memory of the cluster's CTA `rank`.
__device__ __forceinline__ uint32_t cluster_word(uint32_t addr, uint32_t rank) {
    uint32_t at, x;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(at) : "r"(addr), "r"(rank));
    asm volatile("ld.shared::cluster.u32 %0, [%1];" : "=r"(x) : "r"(at) : "memory");
    return x;
}

// ------------------------------------------------------------------------------------------------
// k_sample: one CTA per (regular layer, worker), or a cluster of up to kSampleClusterMost that read the layer's sample together.  A CTA's
// 64 units per warp take 20 us of its 35 at the latency of DRAM, whatever the other SMs do: where the layers are large enough and the
// clusters of all of them resident at once (sample_cluster; a CTA fills an SM but for a CTA of the tiny layers' kernel), the others count
// their part of the units and the first one adds the cells that hold anything to its own.
// ------------------------------------------------------------------------------------------------
// (48 registers: a CTA of the tiny layers' kernel, which runs beside this one, then fits on the same SM)
__global__ void __maxnreg__(48)
k_sample(const float* __restrict__ grads, const float* __restrict__ state, uint64_t stride,
         const LayerDesc* __restrict__ layers, const uint32_t* __restrict__ reg_layers, uint32_t R,
         const KTab ktab, uint32_t K, uint32_t force_exact, uint32_t* __restrict__ cell_tab,
         int4* __restrict__ cell_win, uint32_t* __restrict__ bin_lo, BandMeta* __restrict__ meta) {
    pdl_wait();
    extern __shared__ __align__(16) uint32_t sh[];
    float* s_sq = reinterpret_cast<float*>(sh);   // [1024] squares (cell midpoints) below each thread segment
    float* s_wd = s_sq + 1024;                    // [32]
    uint32_t* h32 = sh + 1024 + 32;               // [32768] two u16 cell counters per word
    uint32_t* s_pre = h32 + 32768;                // [1024] inclusive sample count of the thread segments, from the top
    uint32_t* s_base = s_pre + 1024;              // [2 kBaseWords] first bin id of every gap region, of every group
    uint32_t* s_w = s_base + 2 * kBaseWords;      // [32]
    uint32_t* s_cb = s_w + 32;                    // [128] per candidate, then per merged group: lowest cell,
    uint32_t* s_ct = s_cb + 128;                  // [128] highest cell,
    uint32_t* s_cs = s_ct + 128;                  // [128] shift
    __shared__ uint32_t s_flag, s_ng, s_cg, s_z, s_clip, s_top, s_fine;
    __shared__ unsigned long long s_zz;
    __shared__ float s_nd[128]; // bins per cell needed, per candidate, then per merged group
    const uint32_t r = blockIdx.x, w = blockIdx.y;
    const uint32_t l = reg_layers[r];
    const size_t wr = (size_t)w * R + r;
    BandMeta* mt = meta + wr;
    const uint32_t rank = blockIdx.z, ranks = gridDim.z; // in the layer's cluster
    if (force_exact) {
        if (threadIdx.x == 0 && rank == 0) *mt = BandMeta{0, 0, 1, 0};
        return;
    }
    const LayerDesc ld = layers[l];
    const uint32_t n = (uint32_t)ld.n;
    for (int i = threadIdx.x; i < 32768 / 4; i += kBigThreads) reinterpret_cast<uint4*>(h32)[i] = make_uint4(0u, 0u, 0u, 0u);
    if (threadIdx.x == 0) { s_flag = 0; s_ng = 0; s_cg = 0; s_z = 0; s_zz = 0ull; s_clip = 0; s_top = 0; s_fine = 0; }
    __syncthreads();

    // ---- stratified sample of |grad - g|.  Exact zeros (the untouched rows of a sparse gradient) are counted apart:
    // they sit below every other key, add nothing to any error, and the sweep leaves them out of its histogram.
    const float* gr = grads + (size_t)w * stride + ld.begin;
    const float* st = state + (size_t)w * stride + ld.begin;
    const uint32_t n_units = n / kSampleUnit + ((n % kSampleUnit) != 0); // n may be as large as 2^32 - 1
    const uint32_t m_units = sample_units(n_units);
    const bool whole = m_units == n_units;
    const uint32_t sq_ = n / m_units, sr_ = n % m_units; // used when sampled
    const uint32_t m = whole ? n : kSampleUnit * m_units; // sample size (a stratum is no shorter than a unit), exact zeros included
    uint32_t top_key = 0;                                  // largest finite key
    // a warp reads one unit (128 bytes); eight units per thread are in flight before their keys are counted (this phase runs at
    // the DRAM's random-access rate on large layers; four and four, counted alternately, took a fifth longer)
    for (uint32_t ib = rank * kSampleRound + threadIdx.x / kSampleUnit; ib < m_units; ib += ranks * kSampleRound) {
        float a[8], b[8];
        bool ok[8];
        // where the round's eight units start is the same for all lanes: lane u (mod 8) works out unit u's start
        // and the others fetch it with a shuffle
        uint32_t my_start;
        {
            const uint32_t i = ib + (threadIdx.x & 7u) * (kBigThreads / kSampleUnit);
            my_start = kSampleUnit * i;
            if (!whole && i < m_units) { // unit i somewhere inside stratum i = [i q + i r / m, (i+1) q + (i+1) r / m)
                const uint32_t s0 = i * sq_ + (i * sr_) / m_units;
                const uint32_t s1 = (i + 1) * sq_ + ((i + 1) * sr_) / m_units;
                const uint32_t room = s1 > s0 + kSampleUnit ? s1 - s0 - kSampleUnit : 0;
                my_start = s0 + __umulhi(hash_u32(i * 0x9e3779b9u + l * 0x85ebca6bu + 1u), room + 1);
            }
        }
#pragma unroll
        for (int u = 0; u < 8; ++u) {
            const uint32_t i = ib + u * (kBigThreads / kSampleUnit);
            const uint32_t p = __shfl_sync(0xffffffffu, my_start, u) + (threadIdx.x % kSampleUnit);
            ok[u] = i < m_units && p < n;
            a[u] = ok[u] ? gr[p] : 0.f;
            b[u] = ok[u] ? st[p] : 0.f;
        }
#pragma unroll
        for (int u = 0; u < 8; ++u) {
            const uint32_t key = ok[u] ? key_of(__fsub_rn(a[u], b[u])) : 1u;
            if ((u & 3) == 0) { // every fourth unit: its exact zeros, for the spread of the zeros over the units
                const uint32_t zu = __popc(__ballot_sync(0xffffffffu, key == 0u));
                if (zu && (threadIdx.x & 31) == 0) { atomicAdd(&s_z, zu); atomicAdd(&s_zz, (unsigned long long)(zu * zu)); }
            }
            if (ok[u]) {
                if (key) atomicAdd(&h32[key >> 16], 1u << (16 * ((key >> 15) & 1)));
                top_key = max(top_key, key < 0x7f800000u ? key : 0u);
            }
        }
    }
    top_key = __reduce_max_sync(0xffffffffu, top_key);
    if ((threadIdx.x & 31) == 0) atomicMax(&s_top, top_key);
    __syncthreads();
    if (ranks > 1u) {
        const uint32_t ln = threadIdx.x & 31u, wd = threadIdx.x >> 5;
        // segments of 64 cells (32 words) that hold anything, a bit each: bit w of word i stands for segment 32 i + w, so that the segments of a
        // distribution, which lie side by side, fall to different warps below
        if (rank) {
            for (uint32_t i = 0; i < 32u; ++i) {
                const uint32_t any = __reduce_or_sync(0xffffffffu, h32[32u * (32u * i + wd) + ln]);
                if (ln == i) s_sq[32u * wd + i] = __uint_as_float(any ? 1u : 0u);
            }
            __syncthreads();
            const uint32_t bits = __ballot_sync(0xffffffffu, __float_as_uint(s_sq[32u * ln + wd]) != 0u); // word wd: warp ln's segment
            if (ln == 0) s_pre[wd] = bits;
        }
        cluster_arrive();
        cluster_wait();
        if (rank == 0) {
            uint32_t all = 0; // lane i: the segments 32 i ... of the others
            for (uint32_t r2 = 1; r2 < ranks; ++r2) all |= cluster_word(smem_u32(s_pre + ln), r2);
            for (uint32_t todo = __ballot_sync(0xffffffffu, (all >> wd) & 1u); todo; todo &= todo - 1u) {
                const uint32_t at = 32u * (32u * (__ffs(todo) - 1u) + wd) + ln;
                uint32_t x[kSampleClusterMost];
#pragma unroll
                for (uint32_t r2 = 1; r2 < kSampleClusterMost; ++r2) x[r2] = r2 < ranks ? cluster_word(smem_u32(h32 + at), r2) : 0u;
                uint32_t sum = h32[at];
#pragma unroll
                for (uint32_t r2 = 1; r2 < kSampleClusterMost; ++r2) sum += x[r2]; // (two counters a word: of 65504 entries at most in all)
                h32[at] = sum;
            }
            if (threadIdx.x >= 1u && threadIdx.x < ranks) {
                atomicMax(&s_top, cluster_word(smem_u32(&s_top), threadIdx.x));
                atomicAdd(&s_z, cluster_word(smem_u32(&s_z), threadIdx.x));
                const uint32_t lo = cluster_word(smem_u32(&s_zz), threadIdx.x), hi = cluster_word(smem_u32(&s_zz) + 4u, threadIdx.x);
                atomicAdd(&s_zz, (unsigned long long)hi << 32 | lo);
            }
        }
        cluster_arrive(); // the others' memory has been read
        cluster_wait();
        if (rank) return;
    }
    auto cell_count = [&](uint32_t cell) { return (h32[cell >> 1] >> (16 * (cell & 1))) & 0xffffu; };
    // Square of the cell's middle value, in units that put the sample's largest value into [2^40, 2^41): sums of squares over the
    // layer stay finite, and squares of values down to 2^-113 of the largest one are there.  Only ratios of sums are used.
    const float unit = __uint_as_float(min(254u, 294u - max(s_top >> 23, 1u)) << 23);
    auto cell_sq = [&](uint32_t cell) {
        const float v = __uint_as_float((cell << 15) | 0x4000u) * unit;
        return v * v;
    };

    // ---- per segment t (cells 65535 - 64 t - (0..63)): sample count and squares.  Eight lanes take a segment, four words (two
    // cells each) per lane; the few segments that hold anything lie side by side, so fours of them are dealt out over the warps.
    uint32_t mz; // sample entries in the histogram: all but the exact zeros
    {
        const uint32_t ln = threadIdx.x & 31u, wd = threadIdx.x >> 5;
        for (uint32_t four = wd; four < (uint32_t)kBigThreads / 4; four += kBigThreads / 32) {
            const uint32_t seg = 4u * four + (ln >> 3), word = 32736u - 32u * seg + 4u * (ln & 7u);
            const uint4 x4 = *reinterpret_cast<const uint4*>(h32 + word);
            uint32_t sum = 0;
            float sq = 0.f;
            if (__any_sync(0xffffffffu, (x4.x | x4.y | x4.z | x4.w) != 0u)) {
                const uint32_t x[4] = {x4.x, x4.y, x4.z, x4.w};
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    const uint32_t c0 = x[i] & 0xffffu, c1 = x[i] >> 16;
                    sum += c0 + c1;
                    if (c0) sq += (float)c0 * cell_sq(2u * (word + i));
                    if (c1) sq += (float)c1 * cell_sq(2u * (word + i) + 1u);
                }
#pragma unroll
                for (int o = 4; o; o >>= 1) {
                    sum += __shfl_xor_sync(0xffffffffu, sum, o);
                    sq += __shfl_xor_sync(0xffffffffu, sq, o);
                }
            }
            if ((ln & 7u) == 0) { s_pre[seg] = sum; s_sq[seg] = sq; }
        }
        __syncthreads();
        const uint32_t sum = s_pre[threadIdx.x];
        const float sq = s_sq[kBigThreads - 1 - threadIdx.x]; // squares are added up from the bottom: no cancellation
        const uint32_t ex = block_excl_scan<uint32_t, kBigThreads>(sum, s_w, &mz);
        const float exd = block_excl_scan<float, kBigThreads>(sq, s_wd, nullptr);
        s_pre[threadIdx.x] = ex + sum;
        s_sq[kBigThreads - 1 - threadIdx.x] = exd; // squares in the segments below this one (higher index)
    }
    __syncthreads();
    const uint32_t z = m - mz; // the sample's exact zeros
    // Variance of the sample's zero count, from the spread of the zero counts of the units looked at (the units i with
    // i mod 128 < 32): zeros that come in runs (whole rows) make the sample's share of zeros, and with it the sample
    // rank of every threshold among the other keys, far less certain than independent draws would.
    float var_z = 0.f;
    if (z && !whole) {
        const float ns = (float)((m_units / 128u) * 32u + min(m_units % 128u, 32u)), zs = (float)s_z;
        var_z = fmaxf(0.f, ((float)s_zz - zs * zs / ns) / ns) * (float)m_units;
    }
    // cell holding sample rank rk (1-based, from the top); the whole warp takes part
    const uint32_t lane = threadIdx.x & 31;
    auto cell_of_rank = [&](uint32_t rk) {
        // the first segment that reaches the rank: 32 segments' ends, then the segments of one of those 32 (as a bisection, ten rounds)
        static_assert(kBigThreads == 1024, "two rounds of 32");
        const uint32_t ends = __ballot_sync(0xffffffffu, s_pre[32u * lane + 31u] >= rk);
        const uint32_t part = ends ? __ffs(ends) - 1u : 31u;
        const uint32_t here = __ballot_sync(0xffffffffu, s_pre[32u * part + lane] >= rk);
        const int lo = 32 * (int)part + (here ? __ffs(here) - 1 : 31);
        const uint32_t before = lo ? s_pre[lo - 1] : 0u;
        const uint32_t top = 65535u - 64u * lo;
        // lanes take cells top - 2 lane and top - 2 lane - 1; inclusive counts along the lanes
        const uint32_t c0 = cell_count(top - 2 * lane), c1 = cell_count(top - 2 * lane - 1);
        uint32_t incl = c0 + c1;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t y = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= (uint32_t)o) incl += y;
        }
        const uint32_t upto0 = before + incl - c1; // entries in the cells top .. top - 2 lane
        const uint32_t hit0 = __ballot_sync(0xffffffffu, upto0 >= rk);
        const uint32_t hit1 = __ballot_sync(0xffffffffu, before + incl >= rk);
        if (!hit1) return top - 63u;
        const uint32_t l1 = __ffs(hit1) - 1;
        return (hit0 >> l1) & 1u ? top - 2 * l1 : top - 2 * l1 - 1;
    };

    // ---- bands: the cells that can hold the k_j-th largest key, and how finely to cut them (one warp per candidate)
    for (uint32_t j = threadIdx.x >> 5; j < K; j += kBigThreads / 32) {
        const uint64_t k = ktab.at(w, (size_t)l * K + j);
        uint32_t o_cb = 1, o_ct = 0, o_cs = 15; // k == n keeps everything: no threshold, no band
        float o_nd = 1.f;                        // bins per cell it needs
        if (k < n) {
            uint32_t r_lo, r_hi;
            if (whole) {
                r_lo = r_hi = (uint32_t)k;
            } else {
                const float p = (float)((double)k / (double)n);
                const float rho = p * (float)m, rel = mz ? rho / (float)mz : 0.f;
                const float left_out = fmaxf(0.f, 1.f - (float)m / (float)n); // drawn without replacement
                const float sg = sqrtf((float)m * p * (1.f - p) * left_out + rel * rel * var_z);
                const float a = floorf(rho - 6.f * sg - 2.f), b = ceilf(rho + 6.f * sg + 2.f);
                r_lo = a < 1.f ? 0u : (uint32_t)a;
                r_hi = b > (float)m ? 0u : (uint32_t)b;
            }
            // a rank window wholly among the zeros: the threshold is 0 unless the sample misleads, no band (the curve
            // stage knows the exact number of zeros); a window that reaches into the zeros ends at the lowest cell
            // the sample saw, a quarter octave further down
            const bool zero_cand = z && (mz == 0 || r_lo > mz);
            const bool clip_bot = z && !zero_cand && (r_hi == 0 || r_hi > mz);
            if (zero_cand) {
                if (lane == 0) { s_cb[j] = o_cb; s_ct[j] = o_ct; s_cs[j] = o_cs; }
                continue;
            }
            // rank window clipped at the top: the threshold may lie above the largest sample, so the band goes a
            // quarter octave further up; clipped at the bottom: no bound from the sample, exact path
            // bands stay among the finite keys (a sample with non-finite values is reported by the curve stage)
            uint32_t c_top = min(cell_of_rank(max(r_lo, 1u)), 65279u);
            if (r_lo == 0) {
                c_top = min(c_top + 64u, 65279u);
                if (lane == 0) s_clip = 1;
            }
            if (r_hi == 0 && !z && lane == 0) s_flag = 1;
            uint32_t c_bot = cell_of_rank(clip_bot ? mz : max(r_hi, 1u));
            if (clip_bot) c_bot = c_bot > 64u ? c_bot - 64u : 0u;
            c_bot = min(c_bot, c_top);
            const uint32_t ncell = c_top - c_bot + 1;
            if (ncell > (uint32_t)kFineBins) {
                if (lane == 0) s_flag = 2;
            } else {
                // sample entries in each quarter of the band (a tail band is much denser at its bottom)
                const uint32_t nq = (ncell + 3) / 4;
                uint32_t inq[4] = {0, 0, 0, 0};
                for (uint32_t c = c_bot + lane; c <= c_top; c += 32) {
                    const uint32_t cc = cell_count(c), qi = (c - c_bot) / nq;
#pragma unroll
                    for (int i = 0; i < 4; ++i) inq[i] += qi == (uint32_t)i ? cc : 0u;
                }
                // estimate of this candidate's error: squares of everything below the band
                const uint32_t seg = (65535u - c_bot) >> 6;
                float below = 0.f;
                for (uint32_t c = 65535u - 64u * seg - 63u + lane; c < c_bot; c += 32) {
                    const uint32_t cc = cell_count(c);
                    if (cc) below += (float)cc * cell_sq(c);
                }
#pragma unroll
                for (int o = 16; o; o >>= 1) {
#pragma unroll
                    for (int i = 0; i < 4; ++i) inq[i] += __shfl_xor_sync(0xffffffffu, inq[i], o);
                    below += __shfl_xor_sync(0xffffffffu, below, o);
                }
                below += s_sq[seg];
                const float scale = (float)n / (float)m;
                // entries per cell and v^2 are taken quarter by quarter
                float dens = 0.f, load = 0.f;
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    const uint32_t qtop = min(c_top, c_bot + (uint32_t)(i + 1) * nq - 1);
                    const float per_cell = (float)(inq[i] + 1) / (float)nq * scale; // + 1: never plan on an empty sample
                    dens = per_cell > dens ? per_cell : dens;
                    const float ld = per_cell * cell_sq(qtop);
                    load = ld > load ? ld : load;
                }
                const float bins = bins_needed(dens, load, below * scale); // (about 2048 entries of a bin are listed by the select stage)
                uint32_t sh_j = kCellShift;
                while (sh_j > kMinShift && (float)(1u << (kCellShift - sh_j)) < bins) --sh_j;
                o_cb = c_bot; o_ct = c_top; o_cs = sh_j;
                o_nd = bins;
            }
        }
        if (lane == 0) { s_cb[j] = o_cb; s_ct[j] = o_ct; s_cs[j] = o_cs; s_nd[j] = o_nd; }
    }
    __syncthreads();
    // merge overlapping / adjacent bands (they descend in key with j) into groups; groups end up in s_c*[0..ng)
    // (by a warp that holds the candidates, 32 at a time: one thread that read them from shared memory took 1.9 us)
    if (threadIdx.x < 32 && !s_flag) {
        // The sweep reads a key's region from a table over the cells between the lowest and the highest band.  If
        // that window has more cells than the table has entries, an entry stands for 2^cg cells and the bands
        // are widened to whole entries (more fine bins; the common case is cg = 0).
        uint32_t lo_all = 0xffffffffu, hi_all = 0, cg = 0;
        for (uint32_t j = lane; j < K; j += 32u)
            if (s_cb[j] <= s_ct[j]) { lo_all = min(lo_all, s_cb[j]); hi_all = max(hi_all, s_ct[j]); }
        lo_all = __reduce_min_sync(0xffffffffu, lo_all);
        hi_all = __reduce_max_sync(0xffffffffu, hi_all);
        if (lo_all <= hi_all)
            while ((hi_all >> cg) - (lo_all >> cg) + 3 > (uint32_t)kCellTab) ++cg;
        const uint32_t cmask = (1u << cg) - 1u;
        // The group that is open goes to slot ng, again with every band that joins it (ng <= j: slots already consumed).
        uint32_t ng = 0, open = 0;
        uint32_t gb = 1, gt = 0, gs = 15;
        float gn = 0.f;
        for (uint32_t j0 = 0; j0 < K; j0 += 32u) {
            const uint32_t jl = min(j0 + lane, K - 1u);
            const uint32_t my_cb = s_cb[jl], my_ct = s_ct[jl], my_cs = s_cs[jl], upto = min(32u, K - j0);
            const float my_nd = s_nd[jl];
            __syncwarp();
#pragma unroll 4
            for (uint32_t i = 0; i < upto; ++i) {
                uint32_t cb = __shfl_sync(0xffffffffu, my_cb, i), ct = __shfl_sync(0xffffffffu, my_ct, i);
                const uint32_t cs = __shfl_sync(0xffffffffu, my_cs, i);
                const float cn = __shfl_sync(0xffffffffu, my_nd, i);
                const uint32_t valid = cb <= ct;
                cb &= ~cmask; ct |= cmask; // stays below the non-finite cells: 65279 ends a block of 32
                const uint32_t join = open & (uint32_t)(ct + 1 >= gb);
                ng += valid & open & (join ^ 1u);
                // joined, first of a group, left out: written out as selections (branches took as long as one thread that walked the list)
                gb = select(valid, select(join, min(gb, cb), cb), gb);
                gt = select(valid, select(join, max(gt, ct), ct), gt);
                gs = select(valid, select(join, min(gs, cs), cs), gs);
                gn = __uint_as_float(select(valid, select(join, __float_as_uint(fmaxf(gn, cn)), __float_as_uint(cn)), __float_as_uint(gn)));
                open |= valid;
                if (lane == 0) { s_cb[ng] = gb; s_ct[ng] = gt; s_cs[ng] = gs; s_nd[ng] = gn; }
            }
            __syncwarp();
        }
        ng += open;
        uint32_t fine = 0, cells = 0;
        for (uint32_t g = lane; g < ng; g += 32u) {
            const uint32_t c = s_ct[g] - s_cb[g] + 1;
            fine += c << (15 - s_cs[g]);
            cells += c;
        }
        fine = __reduce_add_sync(0xffffffffu, fine);
        cells = __reduce_add_sync(0xffffffffu, cells);
        if (lane == 0) {
            s_cg = cg;
            if (cells > (uint32_t)kFineBins) s_flag = 3;
            s_fine = fine; // (below 2^24 unless flagged)
            s_ng = ng;
        }
    }
    uint32_t left = 0; // fine bins not given away
    if (threadIdx.x < 32) {
        __syncwarp();
        if (!s_flag) {
            const bool fit = coarsen_groups(WarpLanes{}, s_cb, s_ct, s_cs, s_nd, s_ng, s_fine, (uint32_t)kFineBins, &left);
            __syncwarp();
            if (!fit && threadIdx.x == 0) s_flag = 3;
        }
        __syncwarp();
    }
    if (threadIdx.x == 0 && !s_flag) {
        uint32_t ng = s_ng;
        const uint32_t cg = s_cg, cmask = (1u << cg) - 1u;
        // Where the rank window of the highest band reached beyond the largest sample, up to four more octaves above the band
        // get one bin per cell, as far as bins and table entries are left.  A sample without an entry as large as the smallest
        // candidate's threshold is not rare where large entries lie together (a few rows of a gradient, seven samples
        // expected), and the exact path costs far more than these bins (1.1 B Llama shape, gradients moved across
        // the tensors' borders: 4.5 layers of 402 per step on the exact path without them, 1 with one octave).
        if (s_clip && ng) {
            const uint32_t window = (s_ct[0] >> cg) - (s_cb[ng - 1] >> cg) + 3u;
            uint32_t ext = min(min(1024u, left), window < (uint32_t)kCellTab ? ((uint32_t)kCellTab - window) << cg : 0u) & ~cmask;
            ext = min(ext, 65279u - s_ct[0]);
            if (ext) {
                for (uint32_t g = ng; g; --g) { s_cb[g] = s_cb[g - 1]; s_ct[g] = s_ct[g - 1]; s_cs[g] = s_cs[g - 1]; }
                s_cb[0] = s_ct[1] + 1u; s_ct[0] = s_ct[1] + ext; s_cs[0] = 15;
                ++ng;
            }
        }
        s_ng = ng;
    }
    __syncthreads();
    const uint32_t ng = s_ng, cg = s_cg;
    // ---- bin ids in ascending key order: gap_0, fine bins of the lowest group, gap_1, ..., gap_ng, non-finite keys.
    // A gap region is cut at every 11-bit prefix (one bin per piece: keeps the shared-memory atomics of the sweep
    // spread over many words); keys with exponent 255 take the eight pieces that follow gap_ng's, so that one
    // formula serves everything above the highest band.  Groups are stored with descending keys; a = ng - 1 - g
    // is the ascending index.  s_base[a] = first id of gap_a, s_glo[a] = lowest cell of gap_a.
    // Every region -- a gap or a group of fine bins -- maps a key to its bin as base + (key >> shift) with one
    // (base, shift) pair: shift 20 for the gap pieces, the group's bin width for the fine bins.
    uint32_t* s_glo = s_pre; // [kMaxGaps] reuse: the rank prefix is no longer needed
    if (threadIdx.x < 32 && !s_flag) {
        uint32_t id = 0;
        for (uint32_t a0 = 0; a0 <= ng; a0 += 32u) { // a lane per gap and the group above it
            const uint32_t a = a0 + lane;
            uint32_t gap = 0, bins = 0;
            if (a <= ng) {
                const uint32_t lo = a == 0 ? 0u : s_ct[ng - a] + 1;          // lowest cell of the gap
                const uint32_t hi = a == ng ? 65279u : s_cb[ng - 1 - a] - 1;  // highest cell (may be lo - 1: empty)
                s_glo[a] = lo;
                if (hi + 1 > lo) gap = (hi >> 5) - (lo >> 5) + 1;
                if (a < ng) {
                    const uint32_t g = ng - 1 - a;
                    bins = (s_ct[g] - s_cb[g] + 1) << (15 - s_cs[g]);
                }
            }
            uint32_t incl = gap + bins;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const uint32_t y = __shfl_up_sync(0xffffffffu, incl, o);
                if (lane >= (uint32_t)o) incl += y;
            }
            if (a <= ng) {
                s_base[a] = id + incl - gap - bins;
                if (a < ng) s_base[kBaseWords + a] = id + incl - bins; // first fine bin of group a
            }
            id += __shfl_sync(0xffffffffu, incl, 31);
        }
        if (lane == 0) {
            s_base[ng + 1] = id;     // keys with exponent 255: the pieces 2040..2047
            s_base[ng + 2] = id + 8; // number of bins
        }
    }
    __syncthreads();
    const uint32_t tot_bins = s_flag ? 0u : s_base[ng + 2];
    // window of the cell table: the cells from the lowest to the highest band cell and one entry on either side
    // (everything below lies in gap_0, everything above in gap_ng or among the non-finite keys)
    // (in table entries of 2^cg cells each)
    const uint32_t wlo = (ng ? s_cb[ng - 1] : 1u) >> cg, whi = (ng ? s_ct[0] : 1u) >> cg;
    const uint32_t used = whi - wlo + 3;
    const bool bad = s_flag || tot_bins > (uint32_t)kMaxBins || used > (uint32_t)kCellTab;
    if (bad) {
        if (threadIdx.x == 0) *mt = BandMeta{tot_bins, used, 2, s_flag};
        return;
    }
    uint32_t* tab = cell_tab + wr * kCellTab;
    uint32_t* blo = bin_lo + wr * (kMaxBins + 1);
    // entry i serves the cells (wlo - 1 + i) << cg ...; the first one everything below the window, the last one
    // everything above it
    // (base, shift) of a region, as base << 5 | shift (base may be negative)
    auto group_entry = [&](uint32_t a) {
        const uint32_t g = ng - 1 - a, cs = s_cs[g];
        return (uint32_t)(((int)s_base[kBaseWords + a] - (int)(s_cb[g] << (15 - cs))) * 32) | cs;
    };
    auto gap_entry = [&](uint32_t a) { return (uint32_t)(((int)s_base[a] - (int)(s_glo[a] >> 5)) * 32) | 20u; };
    // The tables are filled region by region (gap a, the group above it), the CTA's warps dealt out to the regions, several to each where
    // there are few: a region's entries are all the same, its bins' keys equally spaced.
    const uint32_t regions = 2u * ng + 2u, wid = threadIdx.x >> 5, sub = max(1u, (uint32_t)(kBigThreads / 32) / regions);
    const uint32_t from = 32u * (wid % sub) + lane, step = 32u * sub;
    if (threadIdx.x == 0) {
        tab[0] = wlo == 0 && ng && s_cb[ng - 1] == 0u ? group_entry(0) : gap_entry(0);
        tab[used - 1u] = gap_entry(ng);
        if (ng == 0) tab[1] = gap_entry(0); // (no band: one gap)
    }
    for (uint32_t r = wid / sub; r < regions; r += (uint32_t)(kBigThreads / 32) / sub) {
        const uint32_t a = r >> 1;
        if (r == regions - 1u) {
            if (from < 8u) blo[s_base[ng + 1] + from] = ((2040u + from) << 20) | kGapBit;
        } else if (r & 1u) {
            const uint32_t g = ng - 1 - a, cs = s_cs[g], bins = (s_ct[g] - s_cb[g] + 1) << (15 - cs), key = s_cb[g] << 15, e = group_entry(a);
            for (uint32_t i = (s_cb[g] >> cg) - wlo + 1u + from; i <= (s_ct[g] >> cg) - wlo + 1u; i += step) tab[i] = e;
            uint32_t* to = blo + s_base[kBaseWords + a];
#pragma unroll 4
            for (uint32_t i = from; i < bins; i += step) to[i] = key + (i << cs);
        } else {
            const uint32_t lo = s_glo[a], bins = s_base[a < ng ? kBaseWords + a : ng + 1] - s_base[a], e = gap_entry(a);
            if (a != 0u && a < ng)
                for (uint32_t i = (lo >> cg) - wlo + 1u + from; i < (s_cb[ng - 1 - a] >> cg) - wlo + 1u; i += step) tab[i] = e;
            uint32_t* to = blo + s_base[a];
#pragma unroll 4
            for (uint32_t i = from; i < bins; i += step) to[i] = (max(lo, ((lo >> 5) + i) << 5) << 15) | kGapBit;
        }
    }
    if (threadIdx.x == 0) {
        blo[tot_bins] = 0x80000000u;
        uint32_t ls = 0; // bins per code of the byte plane: the codes stay below 128
        while (((tot_bins - 1) >> ls) > 127u) ++ls;
        cell_win[wr] = make_int4((int)wlo - 1, (int)whi + 1, (int)(15 + cg), (int)(ls | (z ? 256u : 0u))); // bit 8: zeros are left out
        *mt = BandMeta{tot_bins, used, 0, ng + 2};
    }
}

// ------------------------------------------------------------------------------------------------
// k_pass_a: every CTA owns one static run of consecutive chunks of one worker (runs balanced by cost, a few
// per SM); histogram words and the cell table of the current layer live in shared memory
// ------------------------------------------------------------------------------------------------
struct SweepRun { uint32_t w, c0, c1; }; // chunks [c0, c1) of worker w
constexpr int kRunDesc = 64;             // chunk descriptors staged in shared memory at a time

template <bool VEC>
__global__ void __launch_bounds__(kBigThreads, 1)
k_pass_a(const float* __restrict__ grads, const float* __restrict__ state, uint8_t* __restrict__ d_code,
         const Chunk* __restrict__ chunks, const SweepRun* __restrict__ runs, uint64_t stride, uint64_t dstride, const Phase phases,
         const uint32_t* __restrict__ reg_index /* [L], 0xffffffff: tiny layer */, uint32_t R,
         const uint32_t* __restrict__ cell_tab, const int4* __restrict__ cell_win, const BandMeta* __restrict__ meta,
         uint32_t* __restrict__ bh_cnt, unsigned long long* __restrict__ bh_sum) {
    extern __shared__ __align__(16) uint32_t sh[];
    __shared__ Chunk s_desc[kRunDesc];
    uint32_t* h_cnt = sh;
    uint32_t* h_lo = sh + kMaxBins;
    uint32_t* tab = sh + 2 * kMaxBins; // [kCellTab]
    // the run, its first chunk descriptors and the clean histogram do not depend on the kernels before this one
    const SweepRun run = runs[blockIdx.x];
    auto chunk_at = [&](uint32_t c) { // in positions counted from the worker's 128-bit boundary
        Chunk ch = chunks[c];
        const uint32_t phase = VEC ? phases.at(run.w) : 0u;
        ch.begin += phase;
        ch.end += phase;
        return ch;
    };
    for (int i = threadIdx.x; i < 2 * kMaxBins; i += kBigThreads) sh[i] = 0;
    for (uint32_t i = threadIdx.x; i < min(run.c1 - run.c0, (uint32_t)kRunDesc); i += kBigThreads) s_desc[i] = chunk_at(run.c0 + i);
    pdl_wait();
    __syncthreads();
    const float* gr0 = grads + (size_t)run.w * stride - (VEC ? phases.at(run.w) : 0u);
    const float* st0 = state + (size_t)run.w * stride - (VEC ? phases.at(run.w) : 0u);
    uint8_t* dc0 = d_code + (size_t)run.w * dstride;
    int cur_layer = -1;
    // slot of the current layer's histogram; 0xffffffff: none (tiny or handed-over layer); bit 30 (kSkipZeros): the
    // layer's exact zeros are left out of the histogram
    constexpr uint32_t kSkipZeros = 0x40000000u;
    uint32_t wr = 0xffffffffu;
    __shared__ uint32_t s_bins; // of the current layer's histogram
    bool dirty = false;
    int wlo_m1 = 0, whi_p1 = 0;  // cells of the table's first and last entry, in units of 2^(cshift - 15) cells
    uint32_t cshift = 15, lshift = 0; // keys per table entry, bins per code (log2)

    auto flush = [&]() {
        __syncthreads();
        const uint32_t slot = wr & ~kSkipZeros;
        const uint32_t n_bins = s_bins;
        uint32_t* gc = bh_cnt + (size_t)slot * kMaxBins;
        unsigned long long* gs = bh_sum + (size_t)slot * kMaxBins;
        for (uint32_t i0 = threadIdx.x; i0 < n_bins; i0 += 4 * kBigThreads) { // four bins at a time
            uint32_t c[4], lo[4];
#pragma unroll
            for (uint32_t q = 0; q < 4; ++q) {
                const uint32_t i = min(i0 + q * kBigThreads, (uint32_t)kMaxBins - 1u);
                c[q] = i0 + q * kBigThreads < n_bins ? h_cnt[i] : 0u;
                lo[q] = h_lo[i];
            }
#pragma unroll
            for (uint32_t q = 0; q < 4; ++q) {
                const uint32_t i = i0 + q * kBigThreads;
                if (c[q]) {
                    atomicAdd(&gc[i], c[q]);
                    atomicAdd(&gs[i], (unsigned long long)lo[q]);
                    h_cnt[i] = 0; h_lo[i] = 0;
                }
            }
        }
        __syncthreads();
        dirty = false;
    };
    // (base, shift) of the region a key lies in: one table read; the clamp sends everything outside the window to
    // the table's first or last entry
    auto look = [&](uint32_t key) -> uint32_t { return tab[min(max((int)(key >> cshift), wlo_m1), whi_p1) - wlo_m1]; };
    auto bin_of = [&](uint32_t key, uint32_t e) -> uint32_t { return (uint32_t)(((int)e >> 5) + (int)(key >> (e & 31u))); };
    auto add = [&](uint32_t id, uint32_t key) {
        // 24 significant bits of the square (truncation < 2^-22 relative) summed exactly: the word wraps, the
        // returned old value tells when, and a wrap adds 2^32 to the layer's 64-bit sum in global memory
        const uint32_t sq = (uint32_t)(sq_fixed(key) >> 8);
#ifdef KIMAD_CHECKED
        if (!KIMAD_CHECK(id < meta[wr & ~kSkipZeros].n_bins, 0)) return;
#endif
        atomicAdd(&h_cnt[id], 1u);
        const uint32_t old = atomicAdd(&h_lo[id], sq);
        if (old + sq < old) atomicAdd(bh_sum + (size_t)(wr & ~kSkipZeros) * kMaxBins + id, 1ull << 32); // rare
    };
    // one element: its bin's count and sum; returns its code
    auto acc = [&](uint32_t key) -> uint32_t {
        const uint32_t id = bin_of(key, look(key));
        if (key || !(wr & kSkipZeros)) add(id, key);
        return id >> lshift;
    };
    // The four elements of a quad go through the stages together (all table reads, then the bin ids, then the
    // atomics): four independent chains of dependent shared-memory accesses instead of one after the other.
    // Returns the quad's four codes.
    // Where the sample found a mass of exact zeros (the untouched rows of a sparse gradient), zeros are left out:
    // they add nothing to any sum, they would all hit one word, and the curve stage takes their number from the
    // layer's size.
    auto acc4 = [&](const uint32_t (&k)[4], auto skip) -> uint32_t {
        uint32_t e[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) e[i] = look(k[i]);
#pragma unroll
        for (int i = 0; i < 4; ++i) e[i] = bin_of(k[i], e[i]);
        if (decltype(skip)::value) {
#pragma unroll
            for (int i = 0; i < 4; ++i) if (k[i]) add(e[i], k[i]);
        } else {
#pragma unroll
            for (int i = 0; i < 4; ++i) add(e[i], k[i]);
        }
        return pack_low_bytes(e[0] >> lshift, e[1] >> lshift, e[2] >> lshift, e[3] >> lshift);
    };

    for (uint32_t c = run.c0; c < run.c1; ++c) {
        const uint32_t di = (c - run.c0) % (uint32_t)kRunDesc;
        if (di == 0 && c != run.c0) { // next window of descriptors
            __syncthreads();
            for (uint32_t i = threadIdx.x; i < min(run.c1 - c, (uint32_t)kRunDesc); i += kBigThreads) s_desc[i] = chunk_at(c + i);
            __syncthreads();
        }
        Chunk ch = s_desc[di];
        // the chunks of one layer follow each other without a gap: those among the staged descriptors are swept as
        // one span, so that the load pipeline below is filled once per span and not once per chunk
        while (c + 1 < run.c1 && (c + 1 - run.c0) % (uint32_t)kRunDesc != 0) {
            const Chunk& nx = s_desc[(c + 1 - run.c0) % (uint32_t)kRunDesc];
            if (nx.layer != ch.layer || nx.begin != ch.end) break;
            ch.end = nx.end;
            ++c;
        }
        if ((int)ch.layer != cur_layer) {
            if (dirty) flush();
            cur_layer = (int)ch.layer;
            const uint32_t r = reg_index[ch.layer];
            wr = 0xffffffffu;
            __syncthreads(); // the table is no longer read
            if (r != 0xffffffffu && !meta[run.w * R + r].flagged) {
                wr = run.w * R + r;
                const int4 win = cell_win[wr];
                const uint32_t used = meta[wr].n_cells;
                wlo_m1 = win.x; whi_p1 = win.y; cshift = (uint32_t)win.z; lshift = (uint32_t)win.w & 31u;
                if (threadIdx.x == 0) s_bins = meta[wr].n_bins;
                static_assert(kCellTab == 4 * kBigThreads && 2 * kMaxBins % 4 == 0, "the table in one round of 128-bit loads");
                if (4 * threadIdx.x < used) reinterpret_cast<uint4*>(tab)[threadIdx.x] = reinterpret_cast<const uint4*>(cell_tab + (size_t)wr * kCellTab)[threadIdx.x];
                if ((uint32_t)win.w & 256u) wr |= kSkipZeros;
            }
            __syncthreads();
        }
        const bool active = wr != 0xffffffffu;
        const ChunkView cv(ch, 0);
        uint8_t* dc = dc0 + cv.a0;
        {
            const uint32_t q_lo = (cv.first + 3) >> 2, q_hi = cv.len >> 2; // whole quads [q_lo, q_hi)
            // One quad per thread and round; the loads of the round three rounds ahead are issued before the current
            // round is processed (four register sets, taken in turn), so that a round's memory latency lies behind
            // the work of the rounds before it.  VEC: both inputs are 16-byte aligned at every worker's start and a
            // quad is one 128-bit load per input; otherwise four 32-bit loads, served from L1 after the first.
            const float4* gr4 = reinterpret_cast<const float4*>(gr0 + cv.a0); // (only dereferenced as float4 when VEC)
            const float4* st4 = reinterpret_cast<const float4*>(st0 + cv.a0);
            auto fetch = [&](float4& a, float4& b, uint32_t q) {
                if (q < q_hi) {
                    if (VEC) {
                        a = __ldcg(gr4 + q);
                        b = __ldcg(st4 + q);
                    } else {
                        const float* g = reinterpret_cast<const float*>(gr4 + q);
                        const float* t = reinterpret_cast<const float*>(st4 + q);
                        a = make_float4(__ldg(g), __ldg(g + 1), __ldg(g + 2), __ldg(g + 3));
                        b = make_float4(__ldg(t), __ldg(t + 1), __ldg(t + 2), __ldg(t + 3));
                    }
                }
            };
            auto work = [&](const float4& a, const float4& b, uint32_t q, auto skip) {
                const uint32_t k[4] = {key_of(__fsub_rn(a.x, b.x)), key_of(__fsub_rn(a.y, b.y)),
                                       key_of(__fsub_rn(a.z, b.z)), key_of(__fsub_rn(a.w, b.w))};
                reinterpret_cast<uint32_t*>(dc)[q] = active ? acc4(k, skip) : pack_key_codes(k[0], k[1], k[2], k[3]);
            };
            float4 a0, b0, a1, b1, a2, b2, a3, b3;
            uint32_t qb = q_lo + threadIdx.x;
            constexpr uint32_t S = kBigThreads;
            fetch(a0, b0, qb); fetch(a1, b1, qb + S); fetch(a2, b2, qb + 2 * S);
            // four rounds; false when the span ends inside them.  Two forms (with and without the exact zeros), chosen
            // once per four rounds
            auto rounds = [&](auto skip) -> bool {
                fetch(a3, b3, qb + 3 * S); work(a0, b0, qb, skip); qb += S; if (qb >= q_hi) return false;
                fetch(a0, b0, qb + 3 * S); work(a1, b1, qb, skip); qb += S; if (qb >= q_hi) return false;
                fetch(a1, b1, qb + 3 * S); work(a2, b2, qb, skip); qb += S; if (qb >= q_hi) return false;
                fetch(a2, b2, qb + 3 * S); work(a3, b3, qb, skip); qb += S;
                return true;
            };
            const bool zs = active && (wr & kSkipZeros);
            while (qb < q_hi)
                if (!(zs ? rounds(std::true_type{}) : rounds(std::false_type{}))) break;
            if (threadIdx.x < 8) { // ragged edges: [first, min(4 q_lo, len)) and [max(4 q_hi, 4 q_lo), len)
                uint32_t e;
                if (threadIdx.x < 4) { e = cv.first + threadIdx.x; if (e >= min(4 * q_lo, cv.len)) e = 0xffffffffu; }
                else { e = max(4 * q_hi, 4 * q_lo) + (threadIdx.x - 4); if (e >= cv.len) e = 0xffffffffu; }
                if (e != 0xffffffffu) {
                    const uint32_t key = key_of(__fsub_rn(gr0[cv.a0 + e], st0[cv.a0 + e]));
                    dc[e] = (uint8_t)(active ? acc(key) : code_of_key(key));
                }
            }
        }
        if (active) dirty = true;
    }
    if (dirty) flush();
}

// ------------------------------------------------------------------------------------------------
// The slow paths of a layer: refinement of loose candidates, exact radix select.  Both go over the layer's chunks and
// end with a step that needs all of them.  Layers of large contexts are listed with their chunks (k_refine, k_fb1, k_fb23), which
// costs every step four launches, a second launch of the DP and two event waits although the lists are usually empty.  Where no
// layer has more than kInlineChunks chunks the curve kernel takes them itself (layer_by_itself): 62 tensors of up to
// 147 K elements 116.5 -> 112 us a step, a small model through a built-in workspace 98 -> 86 us.  With one layer of thirty
// candidates on the exact path a step takes 190 us with two chunks, 242 with four, 268 with five and about 340 with eight by one CTA,
// 234 over lists with nine; hence the bound for contexts that take it always.  Beyond four chunks a cluster of two or four CTAs
// takes a layer (227 us with five chunks, 209 with eight).  The clusters of all layers have to be resident at once (a CTA fills
// an SM), though those whose layer needs nothing only wait; where they are not, one CTA takes layers of up to six chunks (293 us: the
// lists would cost every step without such a layer 4 to 5 us) and the lists take more.
// ------------------------------------------------------------------------------------------------
constexpr uint32_t kInlineChunks = 8, kInlineChunksAlone = 6; // with clusters, with a CTA per layer where those are too many
constexpr uint32_t kInlineChunksExact = 2;                     // ... where every layer takes the exact path
constexpr uint32_t kInlineCtas = 128;                          // of a launch of clusters
KIMAD_HD uint32_t inline_cluster(uint32_t most_chunks) { return most_chunks <= 4 ? 1u : (most_chunks <= 6 ? 2u : 4u); }
struct ListArgs {
    DSource src;
    const LayerDesc* layers;
    const Chunk* chunks;
    uint32_t L, K;
    KTab ktab;
    FbList* fb;
    RefineCand* rf;     // [W][L][K]
    uint32_t* h1_cnt;   // [W][R][kL1Bins]
    unsigned long long* h1_ss;
    uint32_t* h23_cnt;  // [W][R][K][kL23Bins]
    unsigned long long* h23_ss;
    Cand* cands;        // [W][L][K]
    SlotTab* slots;     // [W][L]
    uint32_t* flags;
    float* err;         // [W][L][K], and the three below
    uint32_t *tau, *keep_eq, *shift;
    CodeSpace codes;
    uint32_t* arrived;  // [W][L] finished chunks of a listed layer; zero in between
};

// ------------------------------------------------------------------------------------------------
// Refinement of loose candidates: the bin that holds such a candidate's threshold is cut into up to 1024 pieces, and
// the entries of the bin -- found by their code byte, completed from the inputs -- are counted and their squares
// summed per piece (the level-2/3 arrays of the exact path serve as storage: a layer is never on both paths at once).
// Costs one pass over the layer's code bytes instead of the exact path's three passes over its inputs.
// ------------------------------------------------------------------------------------------------
template <int NT>
__device__ __forceinline__ void refine_chunk(const ListArgs& a, uint32_t w, const Chunk& ch, size_t wl, size_t wr) {
    __shared__ uint32_t s_klo[KIMAD_MAX_RATIOS], s_shift[KIMAD_MAX_RATIOS], s_j[KIMAD_MAX_RATIOS];
    __shared__ uint32_t s_mask[4]; // the 7-bit codes of the loose candidates' bins
    __shared__ uint32_t s_n;
    __syncthreads();
    if (threadIdx.x < 4) s_mask[threadIdx.x] = 0;
    if (threadIdx.x == 0) s_n = 0;
    __syncthreads();
    if (threadIdx.x < 32) { // the layer's loose candidates in order of j, every bin once (under its lowest j); a lane each
        const uint32_t lane = threadIdx.x;
        uint32_t p = 0, last = 0; // bins so far, the last one's lower key
        for (uint32_t j0 = 0; j0 < a.K; j0 += 32u) {
            const uint32_t j = j0 + lane;
            RefineCand r{0, kNoRefine, 0, 0, 0.0};
            if (j < a.K) r = a.rf[wl * a.K + j];
            const bool loose = r.shift != kNoRefine;
            const uint32_t m = __ballot_sync(0xffffffffu, loose), before = m & ((1u << lane) - 1u);
            const uint32_t left = __shfl_sync(0xffffffffu, r.klo, before ? 31 - __clz(before) : 0);
            const bool first = loose && (before ? left != r.klo : (p == 0 || last != r.klo)); // thresholds descend with j
            const uint32_t f = __ballot_sync(0xffffffffu, first);
            if (first) {
                const uint32_t at = p + __popc(f & ((1u << lane) - 1u));
                s_klo[at] = r.klo; s_shift[at] = r.shift; s_j[at] = j;
                const uint32_t code = a.codes.code(w, ch.layer, r.klo) & 127u;
                atomicOr(&s_mask[code >> 5], 1u << (code & 31u));
            }
            if (m) last = __shfl_sync(0xffffffffu, r.klo, 31 - __clz(m));
            p += __popc(f);
        }
        if (lane == 0) s_n = p;
    }
    __syncthreads();
    const uint32_t nc = s_n;
    const uint32_t m0 = s_mask[0], m1 = s_mask[1], m2 = s_mask[2], m3 = s_mask[3];
    const ChunkView cv(ch, a.src.phase.at(w));
    const DView dd(a.src, w, cv.a0);
    const bool vec = ((reinterpret_cast<uintptr_t>(dd.gr) | reinterpret_cast<uintptr_t>(dd.st)) & 15u) == 0;
    auto wanted = [&](uint32_t code) -> bool {
        const uint32_t word = code < 64u ? (code < 32u ? m0 : m1) : (code < 96u ? m2 : m3);
        return (word >> (code & 31u)) & 1u;
    };
    auto place = [&](uint32_t key) { // the entry's piece, if it lies in one of the loose bins
        for (uint32_t p = 0; p < nc; ++p) {
            const uint32_t d1 = key - s_klo[p], sh = s_shift[p];
            if (d1 < (1u << sh)) {
                const size_t at = (wr * a.K + s_j[p]) * kL23Bins + (d1 >> (sh > 10u ? sh - 10u : 0u));
                atomicAdd(&a.h23_cnt[at], 1u);
                atomicAdd(&a.h23_ss[at], (unsigned long long)sq_fixed(key));
                break; // bins are disjoint; candidates that share a bin share a piece histogram (see refine_resolve_layer)
            }
        }
    };
    const uint32_t units = (cv.len + 15u) >> 4;
    for (uint32_t u = threadIdx.x; u < units; u += NT) {
        const uint32_t e0 = 16u * u;
        uint32_t hit = 0; // the unit's elements whose code is one of the loose bins'
        if (e0 + 16u > cv.first) { // (a unit at the chunk's edge holds codes of the neighbouring chunk, too)
            const uint4 c4 = __ldcs(reinterpret_cast<const uint4*>(dd.code) + u);
            const uint32_t x[4] = {c4.x, c4.y, c4.z, c4.w};
#pragma unroll
            for (int i = 0; i < 4; ++i)
#pragma unroll
                for (int b = 0; b < 4; ++b)
                    if (wanted((x[i] >> (8 * b)) & 127u)) hit |= 1u << (4 * i + b);
            if (e0 < cv.first) hit &= ~0u << (cv.first - e0);
            if (e0 + 16u > cv.len) hit &= ~(~0u << (cv.len - e0));
        }
        if (!hit) continue;
        // the unit's entries are completed from the inputs with independent loads: eight at a time
        if (vec && e0 >= cv.first && e0 + 16u <= cv.len) {
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                if (!((hit >> (8 * h)) & 255u)) continue;
                const float4* g4 = reinterpret_cast<const float4*>(dd.gr + e0 + 8 * h);
                const float4* t4 = reinterpret_cast<const float4*>(dd.st + e0 + 8 * h);
                const float4 ga = __ldg(g4), gb = __ldg(g4 + 1), ta = __ldg(t4), tb = __ldg(t4 + 1);
                const float v[8] = {__fsub_rn(ga.x, ta.x), __fsub_rn(ga.y, ta.y), __fsub_rn(ga.z, ta.z), __fsub_rn(ga.w, ta.w),
                                    __fsub_rn(gb.x, tb.x), __fsub_rn(gb.y, tb.y), __fsub_rn(gb.z, tb.z), __fsub_rn(gb.w, tb.w)};
#pragma unroll
                for (int i = 0; i < 8; ++i)
                    if ((hit >> (8 * h + i)) & 1u) place(key_of(v[i]));
            }
        } else {
            for (; hit; hit &= hit - 1u) place(key_of(dd.at(e0 + (uint32_t)__ffs(hit) - 1u)));
        }
    }
}

// The pieces of a layer's loose bins resolved, a warp per candidate and a lane per 32 consecutive pieces (ascending keys).  Candidates
// that share a bin were counted into the histogram of the first of them (the lowest j): the later ones read it there.  True where a
// bound is still too loose (a bin with very many entries): the layer needs the exact path after all.
template <int NT>
__device__ __forceinline__ bool refine_resolve_layer(const ListArgs& a, uint32_t l, uint32_t w, size_t wl, size_t wr) {
    __shared__ int s_bad;
    const uint32_t lane = threadIdx.x & 31;
    __syncthreads();
    if (threadIdx.x == 0) s_bad = 0;
    __syncthreads();
    for (uint32_t j = threadIdx.x >> 5; j < a.K; j += NT / 32) {
        const RefineCand rc = a.rf[wl * a.K + j];
        if (rc.shift == kNoRefine) continue;
        uint32_t owner = j; // the first loose candidate with this bin holds the pieces
        for (uint32_t i0 = 0; i0 < j && owner == j; i0 += 32u) {
            bool same = false;
            if (i0 + lane < j) {
                const RefineCand o = a.rf[wl * a.K + i0 + lane];
                same = o.shift != kNoRefine && o.klo == rc.klo;
            }
            const uint32_t m = __ballot_sync(0xffffffffu, same);
            if (m) owner = i0 + __ffs(m) - 1u;
        }
        const uint32_t sub = rc.shift > 10u ? rc.shift - 10u : 0u, b0 = 32u * lane;
        const uint32_t* gc = a.h23_cnt + (wr * a.K + owner) * kL23Bins; // (pieces beyond 2^(shift - sub) are zero)
        const unsigned long long* gs = a.h23_ss + (wr * a.K + owner) * kL23Bins;
        const double scale = sq_scale(rc.klo >> 23);
        uint32_t c[32], csum = 0;
        load_counts(c, gc, b0);
        const double qsum = add_squares(0.0, gs, b0, 32u, scale);
#pragma unroll
        for (int i = 0; i < 32; ++i) csum += c[i];
        uint32_t upto = csum; // entries in the lane's pieces and those of the lanes below
        double below = qsum;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t yc = __shfl_up_sync(0xffffffffu, upto, o);
            const double ys = __shfl_up_sync(0xffffffffu, below, o);
            if (lane >= (uint32_t)o) { upto += yc; below += ys; }
        }
        below = __shfl_up_sync(0xffffffffu, below, 1); // exclusive value from the left neighbour: no cancellation
        if (lane == 0) below = 0.0;
        const uint32_t tot = __shfl_sync(0xffffffffu, upto, 31);
        if (!KIMAD_CHECK(tot == rc.cb, 7)) s_bad = 1;
        const size_t o = wl * a.K + j;
        if (upto - csum <= rc.drop && rc.drop < upto) { // one lane: the piece that holds the threshold is one of its own
            uint32_t i = 0, before = upto - csum, ci = 0;
            bool open = true;
#pragma unroll
            for (int x = 0; x < 32; ++x) {
                if (open && rc.drop - before < c[x]) { open = false; i = x; ci = c[x]; }
                if (open) before += c[x];
            }
            const uint32_t b = b0 + i, klo = rc.klo + (b << sub), d2 = rc.drop - before;
            const double vlo = (double)__uint_as_float(klo), qi = (double)__ldcg(gs + b) * scale;
            const double upper = qi * ((double)d2 / (double)ci), lower = (double)d2 * vlo * vlo;
            double part = 0.5 * (upper + lower), slack = 0.5 * (upper - lower);
            if (d2 == 0 || sub == 0) { part = lower; slack = 0.0; }
            const double e = rc.below + add_squares(below, gs, b0, i, scale) + part;
            if (slack > e * 5e-6) {
                s_bad = 1;
            } else {
                a.err[o] = (float)e; a.tau[o] = klo; a.keep_eq[o] = ci - d2;
                a.shift[o] = sub | (a.codes.code(w, l, klo) | (sub && ci > kListCap ? kSelMany : 0u)) << 8;
            }
        }
    }
    __syncthreads(); // the pieces have been read
    // clean the pieces, close the candidates
    for (uint32_t j = 0; j < a.K; ++j) {
        if (a.rf[wl * a.K + j].shift == kNoRefine) continue;
        for (uint32_t b = threadIdx.x; b < (uint32_t)kL23Bins; b += NT) {
            a.h23_cnt[(wr * a.K + j) * kL23Bins + b] = 0;
            a.h23_ss[(wr * a.K + j) * kL23Bins + b] = 0ull;
        }
    }
    __syncthreads();
    for (uint32_t j = threadIdx.x; j < a.K; j += NT) a.rf[wl * a.K + j].shift = kNoRefine;
    return s_bad != 0;
}

// ------------------------------------------------------------------------------------------------
// exact radix path over the handed-over chunks.  The list is usually empty, but a handed-over layer may be large and
// may hold one key millions of times (the exact zeros of a sparse gradient): every thread therefore adds up the run
// of consecutive elements of its own that fall into one bin and issues its atomics when the bin changes, and keeps
// eight elements' loads in flight (every layer of GPT-2 small on this path: 2254 us a step, with four 2319).
// ------------------------------------------------------------------------------------------------
constexpr int kFbAhead = 8; // elements per thread whose loads are issued together

// s_cnt, s_below [kL1Bins]; s_below holds the two words of the chunk's sums
template <int NT>
__device__ __forceinline__ void fb1_chunk(const ListArgs& a, uint32_t w, const Chunk& ch, size_t wr, uint32_t* s_cnt, double* s_below) {
    uint32_t *s_hi = reinterpret_cast<uint32_t*>(s_below), *s_lo = s_hi + kL1Bins;
    __syncthreads(); // (the arrays may still be read from the chunk or layer before)
    const ChunkView cv(ch, a.src.phase.at(w));
    const DView dd(a.src, w, cv.a0);
    for (int b = threadIdx.x; b < kL1Bins; b += NT) { s_cnt[b] = 0; s_hi[b] = 0; s_lo[b] = 0; }
    __syncthreads();
    // a thread sees at most kChunkElems / NT elements of a chunk: its two partial sums stay below 2^32
    uint32_t cur = 0, cn = 0, chi = 0, clo = 0;
    bool nonfinite = false;
    auto flush = [&]() {
        if (cn) { atomicAdd(&s_cnt[cur], cn); atomicAdd(&s_hi[cur], chi); atomicAdd(&s_lo[cur], clo); }
    };
    for (uint32_t x0 = cv.first + threadIdx.x; x0 < cv.len; x0 += kFbAhead * NT) {
        float v[kFbAhead];
#pragma unroll
        for (int u = 0; u < kFbAhead; ++u) v[u] = x0 + u * NT < cv.len ? dd.at(x0 + u * NT) : 0.f;
#pragma unroll
        for (int u = 0; u < kFbAhead; ++u) {
            if (x0 + u * NT >= cv.len) break;
            const uint32_t key = key_of(v[u]);
            const uint32_t sq = (uint32_t)sq_fixed(key);
            if ((key >> 20) != cur) { flush(); cur = key >> 20; cn = 0; chi = 0; clo = 0; }
            ++cn; chi += sq >> 16; clo += sq & 0xffffu;
            nonfinite |= key >= 0x7f800000u;
        }
    }
    flush();
    if (nonfinite) atomicOr(&a.flags[w], 1u);
    __syncthreads();
    uint32_t* gc = a.h1_cnt + wr * kL1Bins;
    unsigned long long* gs = a.h1_ss + wr * kL1Bins;
    for (int b = threadIdx.x; b < kL1Bins; b += NT)
        if (s_cnt[b]) {
            atomicAdd(&gc[b], s_cnt[b]);
            atomicAdd(&gs[b], ((unsigned long long)s_hi[b] << 16) + s_lo[b]);
        }
}

template <int LEVEL, int NT>
__device__ __forceinline__ void fb23_chunk(const ListArgs& a, uint32_t w, const Chunk& ch, size_t wl, size_t wr) {
    __shared__ uint8_t s_first[kL1Bins]; // level-1 bin -> first slot whose prefix starts with it (0xff: none)
    __shared__ uint8_t s_num[kL1Bins];   // ... and how many consecutive slots share that bin (level 3)
    __shared__ uint32_t s_prefix[KIMAD_MAX_RATIOS];
    __syncthreads(); // (they may still be read from the chunk before)
    const SlotTab& stab = a.slots[wl];
    const uint32_t ns = stab.n;
    for (int b = threadIdx.x; b < kL1Bins; b += NT) { s_first[b] = 0xff; s_num[b] = 0; }
    for (uint32_t s = threadIdx.x; s < ns; s += NT) s_prefix[s] = stab.prefix[s];
    __syncthreads();
    auto bin1 = [&](uint32_t s) { return LEVEL == 2 ? s_prefix[s] : s_prefix[s] >> 10; };
    for (uint32_t s = threadIdx.x; s < ns; s += NT) { // slots that share a level-1 bin follow each other
        const uint32_t b1 = bin1(s);
        if (s && bin1(s - 1u) == b1) continue;
        uint32_t n = 1;
        while (s + n < ns && bin1(s + n) == b1) ++n;
        s_first[b1] = (uint8_t)s;
        s_num[b1] = (uint8_t)n;
    }
    __syncthreads();
    const ChunkView cv(ch, a.src.phase.at(w));
    const DView dd(a.src, w, cv.a0);
    uint32_t* gc = a.h23_cnt + wr * a.K * kL23Bins;
    unsigned long long* gs = a.h23_ss + wr * a.K * kL23Bins;
    uint32_t cur = 0xffffffffu, cn = 0; // (slot, bin) of the thread's current run, its entries and squares
    unsigned long long csq = 0;
    auto flush = [&]() {
        if (cn) {
            atomicAdd(&gc[cur], cn);
            if (LEVEL == 2) atomicAdd(&gs[cur], csq);
        }
    };
    for (uint32_t x0 = cv.first + threadIdx.x; x0 < cv.len; x0 += kFbAhead * NT) {
        float v[kFbAhead];
#pragma unroll
        for (int u = 0; u < kFbAhead; ++u) v[u] = x0 + u * NT < cv.len ? dd.at(x0 + u * NT) : 0.f;
#pragma unroll
        for (int u = 0; u < kFbAhead; ++u) {
            if (x0 + u * NT >= cv.len) break;
            const uint32_t key = key_of(v[u]);
            const uint32_t f = s_first[key >> 20];
            if (f == 0xff) continue;
            uint32_t at = 0xffffffffu;
            if (LEVEL == 2) {
                at = f * (uint32_t)kL23Bins + ((key >> 10) & 1023u);
            } else {
                const uint32_t nn = s_num[key >> 20], p21 = key >> 10;
                for (uint32_t s = f; s < f + nn; ++s)
                    if (s_prefix[s] == p21) { at = s * (uint32_t)kL23Bins + (key & 1023u); break; }
                if (at == 0xffffffffu) continue;
            }
            if (at != cur) { flush(); cur = at; cn = 0; csq = 0; }
            ++cn;
            if (LEVEL == 2) csq += (unsigned long long)sq_fixed(key);
        }
    }
    flush();
}

template <int LEVEL, int NT>
__device__ __forceinline__ void fb23_resolve(const ListArgs& a, uint32_t l, uint32_t w, size_t wl, size_t wr) {
    fb_resolve23_layer<LEVEL, NT>(l, w, wl, wr, a.K, a.h23_cnt, a.h23_ss, a.cands, a.slots, a.err, a.tau, a.keep_eq, a.shift, a.codes);
}

// All of it for one layer, by a cluster of n CTAs of kBigThreads threads: the chunks are dealt out to them, the steps that need all
// chunks are the first one's.  exact: the exact path at once, else the refinement first.  word: the cluster's verdict, zero afterwards.
__device__ __noinline__ void layer_by_itself(const ListArgs& a, uint32_t l, uint32_t w, bool exact, uint32_t rank, uint32_t n, uint32_t* word) {
    constexpr int NT = kBigThreads;
    __shared__ __align__(16) uint32_t s_cnt[kL1Bins];
    __shared__ __align__(16) double s_below[kL1Bins];
    __shared__ uint32_t s_w32[NT / 32];
    __shared__ double s_w64[NT / 32];
    const LayerDesc ld = a.layers[l];
    const size_t wl = (size_t)w * a.L + l, wr = a.codes.slot(w, l);
    auto meet = [&]() {
        __threadfence();
        __syncthreads();
        if (n > 1u) {
            cluster_arrive();
            cluster_wait();
        }
    };
    auto each_chunk = [&](auto f) {
        for (uint32_t i = rank; i < ld.n_chunks; i += n) f(a.chunks[ld.first_chunk + i]);
        meet();
    };
    if (!exact) {
        each_chunk([&](const Chunk& ch) { refine_chunk<NT>(a, w, ch, wl, wr); });
        bool loose = false;
        if (rank == 0) {
            loose = refine_resolve_layer<NT>(a, l, w, wl, wr);
            if (threadIdx.x == 0) {
                if (n > 1u) *word = loose ? 1u : 0u;
                if (loose) { atomicAdd(&a.fb->total_layers, 1u); atomicAdd(&a.fb->why[3], 1u); }
            }
        }
        meet();
        if (rank) loose = __ldcg(word) != 0u;
        if (!loose) return;
    }
    each_chunk([&](const Chunk& ch) { fb1_chunk<NT>(a, w, ch, wr, s_cnt, s_below); });
    if (rank == 0) fb_resolve1_layer<NT>(l, w, wl, wr, a.K, a.h1_cnt, a.h1_ss, a.ktab, a.cands, a.slots, s_cnt, s_below, s_w32, s_w64);
    meet();
    each_chunk([&](const Chunk& ch) { fb23_chunk<2, NT>(a, w, ch, wl, wr); });
    if (rank == 0) fb23_resolve<2, NT>(a, l, w, wl, wr);
    meet();
    each_chunk([&](const Chunk& ch) { fb23_chunk<3, NT>(a, w, ch, wl, wr); });
    if (rank) return;
    fb23_resolve<3, NT>(a, l, w, wl, wr);
    if (n > 1u && threadIdx.x == 0) *word = 0; // (read by all of the cluster before the last meeting)
}

// A CTA's share of a list: consecutive entries, which are mostly of one layer (a layer's chunks follow each other), so that a layer's
// counter and the fence before it are touched once per CTA and not per chunk.  work(w, chunk, wl, wr) per entry, finish(w, layer, wl, wr)
// in the CTA that finishes a layer.
template <typename Work, typename Finish>
__device__ __forceinline__ void over_list(const ListArgs& a, const uint2* __restrict__ list, uint32_t n, Work work, Finish finish) {
    const uint32_t per = (n + gridDim.x - 1u) / gridDim.x, end = min(n, (blockIdx.x + 1u) * per);
    uint32_t done = 0;
    for (uint32_t it = blockIdx.x * per; it < end; ++it) {
        const uint2 e = list[it];
        const Chunk ch = a.chunks[e.y];
        const size_t wl = (size_t)e.x * a.L + ch.layer, wr = a.codes.slot(e.x, ch.layer);
        work(e.x, ch, wl, wr);
        ++done;
        if (it + 1u < end) {
            const uint2 next = list[it + 1u];
            if (next.x == e.x && a.chunks[next.y].layer == ch.layer) continue;
        }
        if (last_of_layer(a.arrived + wl, done, a.layers[ch.layer].n_chunks)) finish(e.x, ch.layer, wl, wr);
        done = 0;
    }
}

__global__ void __launch_bounds__(kThreads, 5)
k_refine(const ListArgs a, const uint2* __restrict__ rf_chunks, uint2* __restrict__ fb_chunks, uint32_t list_cap) {
    pdl_wait();
    __shared__ uint32_t s_at;
    over_list(a, rf_chunks, a.fb->rf_chunks,
        [&](uint32_t w, const Chunk& ch, size_t wl, size_t wr) { refine_chunk<kThreads>(a, w, ch, wl, wr); },
        [&](uint32_t w, uint32_t l, size_t wl, size_t wr) {
            if (!refine_resolve_layer<kThreads>(a, l, w, wl, wr)) return;
            const LayerDesc ld = a.layers[l]; // to the exact path after all
            if (threadIdx.x == 0) {
                s_at = atomicAdd(&a.fb->n_chunks, ld.n_chunks);
                atomicAdd(&a.fb->n_layers, 1u);
                atomicAdd(&a.fb->total_layers, 1u);
                atomicAdd(&a.fb->why[3], 1u);
            }
            __syncthreads();
            for (uint32_t i = threadIdx.x; i < ld.n_chunks; i += kThreads)
                if (KIMAD_CHECK(s_at + i < list_cap, 2)) fb_chunks[s_at + i] = make_uint2(w, ld.first_chunk + i);
            __syncthreads(); // s_at may be written again
        });
}

// (four CTAs per SM: the step that follows a layer's last chunk would take twice the registers)
__global__ void __launch_bounds__(kThreads, 4)
k_fb1(const ListArgs a, const uint2* __restrict__ fb_chunks) {
    pdl_wait();
    __shared__ __align__(16) uint32_t s_cnt[kL1Bins];
    __shared__ __align__(16) double s_below[kL1Bins];
    __shared__ uint32_t s_w32[8];
    __shared__ double s_w64[8];
    over_list(a, fb_chunks, a.fb->n_chunks,
        [&](uint32_t w, const Chunk& ch, size_t, size_t wr) { fb1_chunk<kThreads>(a, w, ch, wr, s_cnt, s_below); },
        [&](uint32_t w, uint32_t l, size_t wl, size_t wr) {
            fb_resolve1_layer<kThreads>(l, w, wl, wr, a.K, a.h1_cnt, a.h1_ss, a.ktab, a.cands, a.slots, s_cnt, s_below, s_w32, s_w64);
        });
}

template <int LEVEL>
__global__ void __launch_bounds__(kThreads, 4)
k_fb23(const ListArgs a, const uint2* __restrict__ fb_chunks) {
    pdl_wait();
    over_list(a, fb_chunks, a.fb->n_chunks,
        [&](uint32_t w, const Chunk& ch, size_t wl, size_t wr) { fb23_chunk<LEVEL, kThreads>(a, w, ch, wl, wr); },
        [&](uint32_t w, uint32_t l, size_t wl, size_t wr) { fb23_resolve<LEVEL, kThreads>(a, l, w, wl, wr); });
}

// ------------------------------------------------------------------------------------------------
// k_resolve_a: one CTA per (regular layer, worker)
// ------------------------------------------------------------------------------------------------
template <bool LISTS> // false: no layer has more than kInlineChunks chunks; the slow paths are taken here, by the clusters along z
__global__ void __launch_bounds__(kBigThreads)
k_resolve_a(const LayerDesc* __restrict__ layers, const uint32_t* __restrict__ reg_layers, uint32_t R, uint32_t L,
            const KTab ktab, uint32_t K, const BandMeta* __restrict__ meta, const int4* __restrict__ cell_win,
            const uint32_t* __restrict__ bin_lo, uint32_t* __restrict__ bh_cnt, unsigned long long* __restrict__ bh_sum,
            float* __restrict__ err_out, uint32_t* __restrict__ tau_out, uint32_t* __restrict__ rank_out,
            uint32_t* __restrict__ shift_out, uint32_t* __restrict__ flags, FbList* __restrict__ fb,
            uint2* __restrict__ fb_chunks, RefineCand* __restrict__ rf, uint2* __restrict__ rf_chunks, uint32_t list_cap, uint32_t w_base,
            const __grid_constant__ ListArgs la) {
    pdl_wait();
    __shared__ uint32_t s_drop[KIMAD_MAX_RATIOS]; // entries not kept by candidate j: n - k_j
    __shared__ int s_loose;
    constexpr int kGroups32 = (kMaxBins + 31) / 32;
    __shared__ uint32_t s_gc[kGroups32]; // per group of 32 bins: entries, then the entries of the groups below it
    __shared__ double s_gs[kGroups32];   // ... and their squares
    __shared__ uint32_t s_w32[32];
    __shared__ double s_w64[32];
    __shared__ int s_bad;
    const uint32_t r = blockIdx.x, w = w_base + blockIdx.y;
    const uint32_t l = reg_layers[r];
    const size_t wr = (size_t)w * R + r, wl = (size_t)w * L + l;
    if constexpr (!LISTS) {
        if (blockIdx.z) { // the first CTA of the cluster decides
            cluster_arrive();
            cluster_wait();
            uint32_t* word = la.arrived + wl;
            const uint32_t verdict = __ldcg(word);
            if (verdict) layer_by_itself(la, l, w, verdict == 2u, blockIdx.z, gridDim.z, word);
            return;
        }
    }
    const BandMeta mt = meta[wr];
    const LayerDesc ld = layers[l];
    if (threadIdx.x == 0) { s_bad = mt.flagged; s_loose = 0; }
    if (threadIdx.x < K) {
        const uint64_t k = ktab.at(w, (size_t)l * K + threadIdx.x);
        s_drop[threadIdx.x] = (uint32_t)(ld.n - k);
    }
    __syncthreads();
    if (!mt.flagged) {
        const uint32_t nb = mt.n_bins, ngrp = (nb + 31u) >> 5; // groups of 32 consecutive bins (ascending keys)
        const uint32_t* blo = bin_lo + wr * (kMaxBins + 1);
        const uint32_t ls = (uint32_t)cell_win[wr].w & 31u;
        uint32_t* gc = bh_cnt + wr * kMaxBins;
        unsigned long long* gs = bh_sum + wr * kMaxBins;
        const uint32_t lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
        auto bin_sq = [&](uint32_t b) { // the sweep summed squares in units of 2^8 sq_fixed
            return (double)gs[b] * (256.0 * sq_scale(blo[b] >> 23));
        };
        // (1) entries and squares of every group; (2) exclusive prefixes over the groups; (3) a warp per candidate:
        // the group where the running count passes n - k_j by bisection over the prefixes, then the bin inside it
        bool nonfinite = false;
        constexpr uint32_t AHEAD = 4; // groups per warp whose bins are requested together
        for (uint32_t g0 = wid; g0 < ngrp; g0 += AHEAD * (kBigThreads / 32)) {
            uint32_t c[AHEAD], key[AHEAD];
            unsigned long long sq[AHEAD];
#pragma unroll
            for (uint32_t q = 0; q < AHEAD; ++q) {
                const uint32_t bb = 32u * (g0 + q * (kBigThreads / 32)) + lane;
                c[q] = key[q] = 0;
                sq[q] = 0ull;
                if (bb < nb) { c[q] = gc[bb]; sq[q] = gs[bb]; key[q] = blo[bb]; }
            }
#pragma unroll
            for (uint32_t q = 0; q < AHEAD; ++q) {
                const uint32_t g = g0 + q * (kBigThreads / 32);
                double sv = (double)sq[q] * (256.0 * sq_scale(key[q] >> 23)); // (as bin_sq; nothing where nothing was counted)
                nonfinite |= c[q] && key[q] >= 0x7f800000u;
#pragma unroll
                for (int o = 16; o; o >>= 1) {
                    c[q] += __shfl_xor_sync(0xffffffffu, c[q], o);
                    sv += __shfl_xor_sync(0xffffffffu, sv, o);
                }
                if (lane == 0 && g < ngrp) { s_gc[g] = c[q]; s_gs[g] = sv; }
            }
        }
        if (nonfinite) atomicOr(&flags[w], 1u);
        __syncthreads();
        uint32_t counted;
        {
            const uint32_t c = threadIdx.x < ngrp ? s_gc[threadIdx.x] : 0u;
            const double sv = threadIdx.x < ngrp ? s_gs[threadIdx.x] : 0.0;
            const uint32_t ec = block_excl_scan<uint32_t, kBigThreads>(c, s_w32, &counted);
            const double es = block_excl_scan<double, kBigThreads>(sv, s_w64, nullptr);
            __syncthreads();
            if (threadIdx.x < ngrp) { s_gc[threadIdx.x] = ec; s_gs[threadIdx.x] = es; }
        }
        __syncthreads();
        const uint32_t zeros = (uint32_t)ld.n - counted; // the sweep leaves exact zeros out of its histogram
        for (uint32_t j = wid; j < K; j += kBigThreads / 32) {
            const size_t o = wl * K + j;
            const uint32_t dj = s_drop[j];
            if (lane == 0) rf[o].shift = kNoRefine;
            if (dj == 0 || dj < zeros) { // everything kept; or the threshold is 0 and nothing but zeros is dropped
                if (lane == 0) { err_out[o] = 0.f; tau_out[o] = 0; rank_out[o] = dj ? zeros - dj : 0u; shift_out[o] = 0; }
                continue;
            }
            const uint32_t target = dj - zeros; // entries of the histogram that are dropped, counted from the bottom
            uint32_t lo = 0, hi = ngrp - 1;     // the last group whose prefix does not exceed the target
            while (lo < hi) { const uint32_t mid = (lo + hi + 1) >> 1; if (s_gc[mid] <= target) lo = mid; else hi = mid - 1; }
            const uint32_t bin = 32u * lo + lane;
            uint32_t c = 0;
            double sv = 0.0;
            if (bin < nb) { c = gc[bin]; if (c) sv = bin_sq(bin); }
            uint32_t ic = c;
            double is = sv;
#pragma unroll
            for (int q = 1; q < 32; q <<= 1) {
                const uint32_t yc = __shfl_up_sync(0xffffffffu, ic, q);
                const double ys = __shfl_up_sync(0xffffffffu, is, q);
                if (lane >= (uint32_t)q) { ic += yc; is += ys; }
            }
            const uint32_t before = s_gc[lo] + ic - c;
            double ex_s = __shfl_up_sync(0xffffffffu, is, 1); // exclusive value from the left neighbour: no cancellation
            if (lane == 0) ex_s = 0.0;
            const double below = s_gs[lo] + ex_s;
            const bool mine = c && target >= before && target - before < c; // this bin holds the threshold
            if (!__ballot_sync(0xffffffffu, mine)) { if (lane == 0) atomicMax(&s_bad, 3); continue; }
            if (!mine) continue;
            if (blo[bin] & kGapBit) { atomicMax(&s_bad, 3); continue; } // outside its band
            const uint32_t klo = blo[bin], width = (blo[bin + 1] & ~kGapBit) - klo;
            const uint32_t cb = c, drop = target - before; // entries of the bin that are not kept, < cb
            const double vlo = (double)__uint_as_float(klo);
            // the dropped entries are the `drop` smallest of the bin: their squares sum to something in
            // [drop * vlo^2, drop * mean]; take the midpoint and certify the half-width
            const double upper = sv * ((double)drop / (double)cb);
            const double lower = (double)drop * vlo * vlo;
            double part = 0.5 * (upper + lower), slack = 0.5 * (upper - lower);
            if (drop == 0 || width == 1) { part = lower; slack = 0.0; }
            const double e = below + part;
            if (slack > e * 5e-6) { // acceptance bound on the curve is 1e-5: this candidate's bin is looked at once more
                if (klo == 0u && zeros) { atomicMax(&s_bad, 4); continue; } // (not a bin whose zeros were left out)
                s_loose = 1;
                atomicAdd(&fb->loose_j[j], 1u);
                rf[o] = RefineCand{klo, (uint32_t)(31 - __clz(width)), cb, drop, below};
                continue;
            }
            err_out[o] = (float)e;
            tau_out[o] = klo;
            rank_out[o] = cb - drop;
            // with the code of the bin's entries (zeros that the sweep left out lie in the bin of key 0)
            const bool many = cb > kListCap || (klo == 0u && zeros);
            shift_out[o] = (31 - __clz(width)) | ((bin >> ls) | (many ? kSelMany : 0u)) << 8;
        }
    }
    __syncthreads();
    const int bad = s_bad;
    const uint32_t verdict = bad ? 2u : (s_loose ? 1u : 0u);
    if constexpr (!LISTS) { // the cluster's other CTAs need not wait for what follows
        if (gridDim.z > 1u) {
            if (verdict && threadIdx.x == 0) la.arrived[wl] = verdict;
            cluster_arrive();
        }
    }
    if (!mt.flagged) { // clean for the next step
        uint32_t* gc = bh_cnt + wr * kMaxBins;
        unsigned long long* gs = bh_sum + wr * kMaxBins;
        for (uint32_t bb = threadIdx.x; bb < mt.n_bins; bb += kBigThreads) { gc[bb] = 0; gs[bb] = 0ull; } // (without a look at what is there)
    }
    __shared__ uint32_t s_at;
    if constexpr (!LISTS) {
        if (gridDim.z > 1u) cluster_wait();
        if (!verdict) return;
        if (threadIdx.x == 0) {
            if (bad) { atomicAdd(&fb->total_layers, 1u); atomicAdd(&fb->why[bad - 1], 1u); }
            else atomicAdd(&fb->refined, 1u);
        }
        layer_by_itself(la, l, w, bad != 0, 0u, gridDim.z, la.arrived + wl);
        return;
    }
    if (bad) { // hand the layer and its chunks to the exact path
        if (threadIdx.x == 0) {
            s_at = atomicAdd(&fb->n_chunks, ld.n_chunks);
            atomicAdd(&fb->n_layers, 1u);
            atomicAdd(&fb->total_layers, 1u);
            atomicAdd(&fb->why[bad - 1], 1u);
        }
        __syncthreads();
        for (uint32_t i = threadIdx.x; i < ld.n_chunks; i += kBigThreads)
            if (KIMAD_CHECK(s_at + i < list_cap, 2)) fb_chunks[s_at + i] = make_uint2(w, ld.first_chunk + i);
    } else if (verdict) { // only loose bounds: refine those candidates
        if (threadIdx.x == 0) {
            s_at = atomicAdd(&fb->rf_chunks, ld.n_chunks);
            atomicAdd(&fb->rf_layers, 1u);
            atomicAdd(&fb->refined, 1u);
        }
        __syncthreads();
        for (uint32_t i = threadIdx.x; i < ld.n_chunks; i += kBigThreads)
            if (KIMAD_CHECK(s_at + i < list_cap, 2)) rf_chunks[s_at + i] = make_uint2(w, ld.first_chunk + i);
    }
}

// ------------------------------------------------------------------------------------------------
// Bitonic sort (descending) of kThreads E keys in shared memory with E consecutive keys per thread
// held in registers: compare-exchanges at distances below E stay inside a thread, those of E .. 16 E are a
// shuffle with the thread 1 .. 16 lanes away, and only larger distances go through shared memory.  The stages are a chain of
// latencies, so every thread of the CTA takes part (E = 2 .. 16) and all of them are written out: as loops they took 150 to 200
// cycles each, most of it branches.
// ------------------------------------------------------------------------------------------------
template <int E, int STRIDE>
__device__ __forceinline__ void tiny_ce_inside(uint32_t (&v)[E], bool desc) {
    if constexpr (STRIDE > 0) {
#pragma unroll
        for (int e = 0; e < E; ++e)
            if (!(e & STRIDE)) {
                const uint32_t hi = max(v[e], v[e | STRIDE]), lo = min(v[e], v[e | STRIDE]);
                v[e] = desc ? hi : lo;
                v[e | STRIDE] = desc ? lo : hi;
            }
        tiny_ce_inside<E, STRIDE / 2>(v, desc);
    }
}
// the stages of the sizes 2 .. E / 2: direction by the key's position inside the thread
template <int E, int SIZE>
__device__ __forceinline__ void tiny_sort_inside(uint32_t (&v)[E]) {
    if constexpr (SIZE < E) {
#pragma unroll
        for (int str = SIZE / 2; str > 0; str >>= 1)
#pragma unroll
            for (int e = 0; e < E; ++e)
                if (!(e & str)) {
                    const uint32_t hi = max(v[e], v[e | str]), lo = min(v[e], v[e | str]);
                    const bool desc = (e & SIZE) == 0;
                    v[e] = desc ? hi : lo;
                    v[e | str] = desc ? lo : hi;
                }
        tiny_sort_inside<E, SIZE * 2>(v);
    }
}
template <int E>
__device__ __forceinline__ void tiny_store(uint32_t* at, const uint32_t (&v)[E]) {
    if constexpr (E == 2) {
        *reinterpret_cast<uint2*>(at) = make_uint2(v[0], v[1]);
    } else {
#pragma unroll
        for (int q = 0; q < E / 4; ++q) reinterpret_cast<uint4*>(at)[q] = make_uint4(v[4 * q], v[4 * q + 1], v[4 * q + 2], v[4 * q + 3]);
    }
}
template <int E>
__device__ __forceinline__ void tiny_load(uint32_t (&v)[E], const uint32_t* at) {
    if constexpr (E == 2) {
        const uint2 x = *reinterpret_cast<const uint2*>(at);
        v[0] = x.x; v[1] = x.y;
    } else {
#pragma unroll
        for (int q = 0; q < E / 4; ++q) {
            const uint4 x = reinterpret_cast<const uint4*>(at)[q];
            v[4 * q] = x.x; v[4 * q + 1] = x.y; v[4 * q + 2] = x.z; v[4 * q + 3] = x.w;
        }
    }
}
template <int E>
__device__ __forceinline__ void tiny_sort_blocked(uint32_t* s_key) {
    const uint32_t t = threadIdx.x;
    uint32_t v[E];
    tiny_load<E>(v, s_key + E * t);
    tiny_sort_inside<E, 2>(v);
#pragma unroll
    for (int size = E; size <= E * kThreads; size <<= 1) { // from here on the direction depends on the thread
        const bool desc = ((E * t) & (uint32_t)size) == 0;
#pragma unroll
        for (int str = size >> 1; str >= E; str >>= 1) {
            const int dt = str / E;                                  // the partner thread is t ^ dt
            const bool keep_max = ((t & (uint32_t)dt) == 0) == desc; // the lower position keeps the larger key when descending
            uint32_t pv[E];
            if (dt >= 32) { // another warp: through shared memory
                __syncthreads(); // s_key is no longer read
                tiny_store<E>(s_key + E * t, v);
                __syncthreads();
                tiny_load<E>(pv, s_key + E * (t ^ (uint32_t)dt));
            } else { // a lane of the same warp
#pragma unroll
                for (int e = 0; e < E; ++e) pv[e] = __shfl_xor_sync(0xffffffffu, v[e], dt);
            }
#pragma unroll
            for (int e = 0; e < E; ++e) v[e] = keep_max ? max(v[e], pv[e]) : min(v[e], pv[e]);
        }
        tiny_ce_inside<E, E / 2>(v, desc);
    }
    __syncthreads();
    tiny_store<E>(s_key + E * t, v);
    __syncthreads();
}

// ------------------------------------------------------------------------------------------------
// k_tiny_exact: layers of at most kTinyMax elements, sorted in shared memory (one CTA each)
// ------------------------------------------------------------------------------------------------
__global__ void __launch_bounds__(kThreads)
k_tiny_exact(const float* __restrict__ grads, const float* __restrict__ state, uint64_t stride,
             const LayerDesc* __restrict__ layers,
             const uint32_t* __restrict__ tiny_layers, uint32_t L, const KTab ktab, uint32_t K,
             float* __restrict__ err_out, uint32_t* __restrict__ tau_out, uint32_t* __restrict__ rank_out,
             uint32_t* __restrict__ shift_out, uint32_t* __restrict__ flags) {
    pdl_wait();
    extern __shared__ __align__(16) unsigned char tiny_smem[];
    double* s_suf = reinterpret_cast<double*>(tiny_smem);                // [kTinyMax] squares of the entries ranked >= i
    uint32_t* s_key = reinterpret_cast<uint32_t*>(s_suf + kTinyMax);     // [kTinyMax]
    __shared__ double s_w64[8];
    const uint32_t l = tiny_layers[blockIdx.x], w = blockIdx.y;
    const LayerDesc ld = layers[l];
    const uint32_t n = (uint32_t)ld.n;
    // d is recomputed here (the same single subtraction as in the sweep), so that this kernel depends on the
    // step's inputs only and can run beside the sample and sweep kernels
    const float* gr = grads + (size_t)w * stride + ld.begin;
    const float* st = state + (size_t)w * stride + ld.begin;
    uint32_t np = 1;
    while (np < n) np <<= 1;
    bool nonfinite = false;
    for (uint32_t i = threadIdx.x; i < np; i += kThreads) {
        const uint32_t key = i < n ? key_of(__fsub_rn(gr[i], st[i])) : 0u;
        nonfinite |= key >= 0x7f800000u;
        s_key[i] = key;
    }
    if (nonfinite) atomicOr(&flags[w], 1u);
    __syncthreads();
    // Keys per thread by the padded size; layers that a thread per key covers are ranked by counting (256 keys sorted with a
    // barrier per stage: 12000 to 17000 cycles).
    if (np > 2048u) tiny_sort_blocked<16>(s_key);
    else if (np > 1024u) tiny_sort_blocked<8>(s_key);
    else if (np > 512u) tiny_sort_blocked<4>(s_key);
    else if (np > (uint32_t)kThreads) tiny_sort_blocked<2>(s_key);
    else {
        uint32_t rank = 0; // keys ahead of this thread's: larger ones, and equal ones with a lower index
        const uint32_t mine = threadIdx.x < np ? s_key[threadIdx.x] : 0u;
        uint32_t i = 0;
        for (; i + 4u <= np; i += 4u) {
            const uint4 x = *reinterpret_cast<const uint4*>(s_key + i);
            rank += (uint32_t)(x.x > mine) + (uint32_t)(x.y > mine) + (uint32_t)(x.z > mine) + (uint32_t)(x.w > mine);
            rank += (uint32_t)((x.x == mine) & (i < threadIdx.x)) + (uint32_t)((x.y == mine) & (i + 1u < threadIdx.x)) +
                    (uint32_t)((x.z == mine) & (i + 2u < threadIdx.x)) + (uint32_t)((x.w == mine) & (i + 3u < threadIdx.x));
        }
        for (; i < np; ++i) {
            const uint32_t x = s_key[i];
            rank += (uint32_t)(x > mine) + (uint32_t)((x == mine) & (i < threadIdx.x));
        }
        __syncthreads();
        if (threadIdx.x < np) s_key[rank] = mine;
        __syncthreads();
    }
    // suffix sums of squares, smallest magnitudes first: position q = n-1-i runs over ascending magnitude
    constexpr int PER = kTinyMax / kThreads;
    double loc[PER];
    double sum = 0.0;
#pragma unroll
    for (int i = 0; i < PER; ++i) {
        const uint32_t q = threadIdx.x * PER + i; // q-th smallest
        double v = 0.0;
        if (q < n) v = (double)__uint_as_float(s_key[n - 1 - q]);
        loc[i] = v * v;
        sum += loc[i];
    }
    double run = block_excl_scan<double>(sum, s_w64, nullptr);
#pragma unroll
    for (int i = 0; i < PER; ++i) {
        const uint32_t q = threadIdx.x * PER + i;
        run += loc[i];
        if (q < n) s_suf[n - 1 - q] = run; // squares of the ranks >= n-1-q
    }
    __syncthreads();
    const size_t wl = (size_t)w * L + l;
    for (uint32_t j = threadIdx.x; j < K; j += kThreads) {
        const uint32_t k = (uint32_t)ktab.at(w, (size_t)l * K + j);
        const size_t o = wl * K + j;
        const uint32_t t = s_key[k - 1];
        uint32_t lo = 0; // first rank whose key equals t: larger ones are counted
#pragma unroll
        for (uint32_t b = kTinyMax / 2; b; b >>= 1) lo += select((uint32_t)(lo + b < k) & (uint32_t)(s_key[min(lo + b, k) - 1u] > t), b, 0u);
        err_out[o] = k < n ? (float)s_suf[k] : 0.f;
        tau_out[o] = t;
        rank_out[o] = k - lo;
        shift_out[o] = code_of_key(t) << 8;
    }
}

} // namespace kimad
