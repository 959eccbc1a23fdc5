// Device code of the Kimad+ compression pass for sm_100a: helpers shared by all stages, the exact radix
// resolve kernels.
//
// Stage map of one step (letters as in include/kimad.h; file in brackets):
//   k_sample        (a)+(b) per (worker, layer): stratified sample of |grad - g| -> for every candidate k_j the
//                   band of 16-bit key prefixes that can hold its threshold -> bins and the cell table [kimad_curve.cuh]
//   k_pass_a        (a)+(b) the sweep: d = grad - g (Section 3 footnote, Eq. 6), bin = table(key(d)), count and
//                   exact integer sum of squares per bin in shared memory; one byte per element (a monotone code
//                   of its bin) goes to scratch, d itself is never stored                         [kimad_curve.cuh]
//   k_resolve_a     (b) Eq. 4 / the "Errors" matrix of Algorithm 3: err_l(k_j) from the bins, certified to the
//                   curve tolerance; layers that fail the certificate are handed to the exact path [kimad_curve.cuh]
//   k_tiny_exact    (b) layers of at most 4096 elements, sorted in shared memory                 [kimad_curve.cuh]
//   k_refine
//                   (b) candidates whose certified bound is too loose: one more look at their bin (usually none)
//   k_fb1, k_fb23<2|3>
//                   (b) exact 11+10+10-bit radix select over the handed-over layers (usually none)
//                                                                          [kimad_curve.cuh, this file]
//   k_dp            (c) Algorithm 3 on the budget axis (Eq. 2, Eq. 3, Section 3.2), one CTA per worker [kimad_dp.cuh]
//   k_pick          (c) the uniform-ratio policies and the error-axis reading                     [kimad_dp.cuh]
//   k_sel_count, k_sel_offsets, k_sel_recount
//                   (d) exact threshold and per-slice output offsets at the chosen k             [kimad_select.cuh]
//   k_sel_write     (e)+(f) ordered (index, value) pack and g += C(d) (Algorithm 1, Eq. 6)       [kimad_select.cuh]
//   k_apply_packed, k_aggregate   receiving side and model step (Algorithm 1, server lines)      [kimad_receiver.cuh]
//
// Nothing here is a dense contraction, so there is no tensor-core path.  The sweep runs at 83-90 % of the measured HBM
// copy rate on its 9 bytes per element (one shared-memory table read and two shared-memory atomics per element keep it
// from the rest); the counting and write sweeps are bound by HBM on large layers and by load latency on small ones.
// After the sample kernel the workers go through the stages as two groups on streams of their own (kimad_api.cu).
#pragma once
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include "kimad_common.h"

namespace kimad {

constexpr int kThreads = 256;
constexpr int kL1Bins = 2048;  // 8 exponent bits + 3 mantissa bits
constexpr int kL23Bins = 1024; // 10 bits each

__device__ __forceinline__ uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }
__device__ __forceinline__ uint32_t key_of(float d) { return __float_as_uint(d) & 0x7fffffffu; }

// Kernels launched with programmatic stream serialisation may be scheduled before their predecessor in the
// stream has finished (which hides their launch latency); they wait here, before touching anything it wrote.
// A no-op for an ordinary launch.  From then on the next kernel in the stream may be scheduled as SMs come free: its CTAs
// start and wait here in their turn, which takes most of a launch off every link of the chain.
__device__ __forceinline__ void pdl_wait_only() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void pdl_launch() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void pdl_wait() {
    pdl_wait_only();
    pdl_launch();
}

// Aligned view of a chunk for 128-bit loads of the inputs (quads of elements) and of the code plane (sixteen
// codes): units start at a0 = begin & ~15; only the first and the last ones can be partial.  All offsets are
// 32-bit and relative to a0.
// Where a worker's vectors start at an odd element (unpadded strides, an offset base), both inputs are `phase` elements past a
// 128-bit boundary.  Positions counted from that boundary (element + phase) are aligned as the memory is; the code plane is laid
// out in them, and chunks are cut into quads and units of sixteen there.
struct Phase {
    uint32_t first, step; // elements past the boundary of worker 0; what the stride adds per worker (0, 0: inputs that are
                          // not equally far past one, which are read element by element)
    __device__ __forceinline__ uint32_t at(uint32_t w) const { return (first + w * step) & 3u; }
};
struct ChunkView {
    uint64_t a0;         // aligned start: element + phase
    uint32_t first, len; // valid element offsets are [first, len)
    __device__ __forceinline__ ChunkView(const Chunk& ch, uint32_t phase)
        : a0((ch.begin + phase) & ~15ull), first((uint32_t)(ch.begin + phase - a0)), len((uint32_t)(ch.end + phase - a0)) {}
};

// The difference vector d = grad - g is never stored.  The sweep leaves one BYTE per element (u8 [W][dstride]): a
// 7-bit code that never decreases with the magnitude key inside a layer -- the element's histogram bin divided by
// a power of two for layers swept with a histogram, the upper seven bits of the key otherwise (code_of_key).  The
// counting sweep of the select stage classifies an entry as above or below the threshold by its code and needs the
// exact value only for the entries whose code equals the threshold's; whoever needs an exact d recomputes the one
// subtraction from the inputs (the estimator is not written before the write sweep, and there every element is
// read before it is updated).
struct DSource {
    uint8_t* code;
    const float* grads;
    const float* state;
    uint64_t stride;  // elements between workers in grads / state
    uint64_t dstride; // ... in the code plane
    Phase phase;
};
struct DView { // one worker's data at a chunk's aligned start
    const uint8_t* code;
    const float* gr;
    const float* st;
    __device__ __forceinline__ DView(const DSource& p, uint32_t w, uint64_t a0)
        : code(p.code + (size_t)w * p.dstride + a0), gr(p.grads + (size_t)w * p.stride + a0 - p.phase.at(w)),
          st(p.state + (size_t)w * p.stride + a0 - p.phase.at(w)) {}
    __device__ __forceinline__ float at(uint32_t e) const { return __fsub_rn(gr[e], st[e]); }
};
// code of layers without a histogram: the upper seven bits of the 31-bit key
__device__ __forceinline__ uint32_t code_of_key(uint32_t key) { return key >> 24; }
// the lowest bytes of four words as one word (element 0 in the lowest byte)
__device__ __forceinline__ uint32_t pack_low_bytes(uint32_t a, uint32_t b, uint32_t c, uint32_t d) {
    return __byte_perm(__byte_perm(a, b, 0x0040), __byte_perm(c, d, 0x0040), 0x5410);
}
// the codes of a quad of keys of a layer without a histogram (the highest byte of every key)
__device__ __forceinline__ uint32_t pack_key_codes(uint32_t k0, uint32_t k1, uint32_t k2, uint32_t k3) {
    return __byte_perm(__byte_perm(k0, k1, 0x0073), __byte_perm(k2, k3, 0x0073), 0x5410);
}

// ------------------------------------------------------------------------------------------------
// block-wide exclusive scans (NT threads), result valid in every thread; `total` optional
// ------------------------------------------------------------------------------------------------
template <typename T, int NT = kThreads>
__device__ __forceinline__ T block_excl_scan(T v, T* s_warp /* [NT / 32] */, T* total) {
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    T x = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        T y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += y;
    }
    __syncthreads(); // s_warp may still be read from a previous call
    if (lane == 31) s_warp[wid] = x;
    __syncthreads();
    T base = 0, tot = 0;
    if (NT <= 256) {
#pragma unroll
        for (int i = 0; i < NT / 32; ++i) {
            const T t = s_warp[i];
            if (i < wid) base += t;
            tot += t;
        }
    } else { // every warp scans the warps' totals
        T t = lane < NT / 32 ? s_warp[lane] : T(0);
#pragma unroll
        for (int o = 1; o < NT / 32; o <<= 1) {
            const T y = __shfl_up_sync(0xffffffffu, t, o);
            if (lane >= o) t += y;
        }
        base = wid ? __shfl_sync(0xffffffffu, t, wid - 1) : T(0);
        tot = __shfl_sync(0xffffffffu, t, NT / 32 - 1);
    }
    if (total) *total = tot;
    // the lane's exclusive value is taken from its left neighbour, not as inclusive - own: a subtraction would
    // cancel the small terms of a floating-point scan whose values span many orders of magnitude
    T ex = __shfl_up_sync(0xffffffffu, x, 1);
    if (lane == 0) ex = 0;
    return base + ex;
}

// ------------------------------------------------------------------------------------------------
// (a) difference + level-1 histogram
// ------------------------------------------------------------------------------------------------
// Squares are accumulated as exact integers.  Every histogram bin holds keys of one exponent e, so
// value^2 = M^2 * 4^(max(e,1)-150) with M the 24-bit significand (no hidden bit for subnormals);
// bins sum (M^2 >> 16), a 32-bit quantity (truncation <= 2^-30 relative).  Integer adds commute, so
// the sums -- and with them the error curve -- do not depend on the order the atomics land in.
__device__ __forceinline__ uint64_t sq_fixed(uint32_t key) {
    const uint32_t e = key >> 23, mant = key & 0x7fffffu;
    const uint32_t M = e ? (mant | 0x800000u) : mant;
    return ((uint64_t)M * (uint64_t)M) >> 16;
}
// scale that turns a bin's integer sum back into a sum of squared values; e = exponent field of the bin
__device__ __forceinline__ double sq_scale(uint32_t e) { // 2^(2 (max(e,1) - 150) + 16), always a normal double
    const int x = 2 * ((int)(e ? e : 1u) - 150) + 16;
    return __longlong_as_double((long long)(x + 1023) << 52);
}

// ------------------------------------------------------------------------------------------------
// (b) resolve: candidates -> bins.  One CTA per (worker, layer).
// ------------------------------------------------------------------------------------------------
// In-place: on return s_incl[p] (p = position counted from the TOP bin, p = NB-1-bin) holds the
// inclusive count of keys in bins >= that bin; s_below[bin] holds the sum of ss over bins < bin.
template <int NB, int NT>
__device__ __forceinline__ void scan_bins(uint32_t* s_incl /* in: counts by position */, double* s_below /* in: ss by bin */,
                                          uint32_t* s_w32, double* s_w64) {
    constexpr int PER = NB / NT;
    static_assert(PER % 2 == 0, "8-byte shared-memory accesses");
    uint32_t loc[PER];
    uint32_t sum = 0;
    uint2* v2 = reinterpret_cast<uint2*>(s_incl + threadIdx.x * PER);
#pragma unroll
    for (int i = 0; i < PER / 2; ++i) { const uint2 t = v2[i]; loc[2 * i] = t.x; loc[2 * i + 1] = t.y; }
#pragma unroll
    for (int i = 0; i < PER; ++i) sum += loc[i];
    uint32_t ex = block_excl_scan<uint32_t, NT>(sum, s_w32, nullptr);
#pragma unroll
    for (int i = 0; i < PER; ++i) { ex += loc[i]; loc[i] = ex; }
#pragma unroll
    for (int i = 0; i < PER / 2; ++i) v2[i] = make_uint2(loc[2 * i], loc[2 * i + 1]);
    if (s_below) {
        double dl[PER];
        double ds = 0.0;
        double2* d2 = reinterpret_cast<double2*>(s_below + threadIdx.x * PER);
#pragma unroll
        for (int i = 0; i < PER / 2; ++i) { const double2 t = d2[i]; dl[2 * i] = t.x; dl[2 * i + 1] = t.y; }
#pragma unroll
        for (int i = 0; i < PER; ++i) ds += dl[i];
        double de = block_excl_scan<double, NT>(ds, s_w64, nullptr);
#pragma unroll
        for (int i = 0; i < PER; ++i) { const double t = dl[i]; dl[i] = de; de += t; }
#pragma unroll
        for (int i = 0; i < PER / 2; ++i) d2[i] = make_double2(dl[2 * i], dl[2 * i + 1]);
    }
    __syncthreads();
}

// first position p (0 = top bin) whose inclusive count reaches `rank` (1-based)
template <int NB>
__device__ __forceinline__ int find_pos(const uint32_t* s_incl, uint32_t rank) {
    int lo = 0, hi = NB - 1;
    while (lo < hi) {
        const int mid = (lo + hi) >> 1;
        if (s_incl[mid] >= rank) hi = mid; else lo = mid + 1;
    }
    return lo;
}

// The exact radix kernels below run over the list of layers handed over in this step (usually empty).
struct FbList { // layers handed to the exact radix path in this step, and their chunks
    uint32_t n_chunks;
    uint32_t n_layers;
    uint32_t total_layers; // never reset: how many layers were handed over since the workspace was attached
    uint32_t why[5];       // never reset: ... because 0: forced, 1: bands too wide for the tables, 2: threshold
                           // outside its band, 3: error bound too loose
    uint32_t loose_j[KIMAD_MAX_RATIOS + 1]; // never reset: which candidate's bound was too loose
    // layers whose only defect is a loose bound are refined instead: one more look at the entries of the bins that
    // hold the loose candidates' thresholds (k_refine)
    uint32_t rf_chunks;
    uint32_t rf_layers;
    uint32_t refined; // never reset: layers that took the refinement
    uint32_t windows[3]; // never reset: searches over windows that did not decide, that did in the first windows, in the second
};
// A candidate of a refined layer: its threshold lies in the bin [klo, klo + 2^shift), which holds cb entries of which
// the `drop` smallest are not kept; `below` = the squares of everything below the bin.  shift = kNoRefine: this
// candidate's curve entry is final.
struct RefineCand {
    uint32_t klo, shift, cb, drop;
    double below;
};
constexpr uint32_t kNoRefine = 0xffffffffu;

// ------------------------------------------------------------------------------------------------
// What the sample kernel leaves per (worker, regular layer) for the sweep (details in kimad_curve.cuh)
// ------------------------------------------------------------------------------------------------
constexpr int kCellTab = 4096; // entries of the cell table: the window of cells from the lowest to the highest band
                               // and one entry on either side
struct BandMeta {
    uint32_t n_bins;
    uint32_t n_cells; // entries of the cell table in use
    uint32_t flagged; // != 0: this layer takes the exact radix path in this step (and is swept without a histogram)
    uint32_t n_gaps;  // gap regions (when flagged: detail of the misfit)
};
// entry of the cell table: base << 5 | shift (base signed): the bin of a key is base + (key >> shift).
// window of a layer: {cell of the first entry, cell of the last entry, log2 of the keys per entry, log2 of the bins
// per code of the byte plane (bits 0..4) | 256 when the sweep leaves the layer's exact zeros out of its histogram}
struct CodeSpace { // how the sweep coded the elements of one (worker, layer)
    const uint32_t* reg_index; // [L], 0xffffffff: tiny layer
    const BandMeta* meta;      // [W][R]
    const uint32_t* cell_tab;  // [W][R][kCellTab]
    const int4* cell_win;      // [W][R]
    uint32_t R;
    // index of a (worker, regular layer) in the per-layer arrays of the curve stage
    __device__ __forceinline__ size_t slot(uint32_t w, uint32_t l) const { return (size_t)w * R + reg_index[l]; }
    // code of a key of layer l of worker w, as the sweep wrote it for every element of that layer
    __device__ __forceinline__ uint32_t code(uint32_t w, uint32_t l, uint32_t key) const {
        const uint32_t r = reg_index[l];
        if (r == 0xffffffffu) return key >> 24;
        const size_t wr = (size_t)w * R + r;
        if (meta[wr].flagged) return key >> 24;
        const int4 win = cell_win[wr];
        const uint32_t e = cell_tab[wr * kCellTab + (size_t)(min(max((int)(key >> win.z), win.x), win.y) - win.x)];
        return (uint32_t)(((int)e >> 5) + (int)(key >> (e & 31u))) >> (win.w & 31);
    }
};

// Work over chunks of listed layers ends, per layer, with a step that needs all of them: the CTA that finishes the layer's
// last chunk takes that step.  True (for the whole CTA) in that CTA, which then sees what the others wrote; the counter is
// back at zero.  Every thread of the CTA calls it after its last write for the `done` chunks.
__device__ __forceinline__ bool last_of_layer(uint32_t* counter, uint32_t done, uint32_t n_chunks) {
    __shared__ uint32_t s_last;
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) {
        s_last = atomicAdd(counter, done) + done == n_chunks;
        if (s_last) *counter = 0;
    }
    __syncthreads();
    const bool last = s_last != 0;
    if (last) __threadfence();
    return last;
}

// The 32 counts from b0 on (a lane's share of a histogram of kL23Bins), requested together.
__device__ __forceinline__ void load_counts(uint32_t (&c)[32], const uint32_t* gc, uint32_t b0) {
#pragma unroll
    for (int q = 0; q < 8; ++q) {
        const uint4 x = __ldcg(reinterpret_cast<const uint4*>(gc + b0) + q);
        c[4 * q] = x.x; c[4 * q + 1] = x.y; c[4 * q + 2] = x.z; c[4 * q + 3] = x.w;
    }
}
// `from` and the first `upto` of the 32 sums of squares from b0 on, added in order.
__device__ __forceinline__ double add_squares(double from, const unsigned long long* gs, uint32_t b0, uint32_t upto, double scale) {
#pragma unroll 8
    for (uint32_t q = 0; q < 16; ++q) {
        if (2u * q >= upto) break;
        const ulonglong2 x = __ldcg(reinterpret_cast<const ulonglong2*>(gs + b0) + q);
        from += (double)x.x * scale;
        if (2u * q + 1u < upto) from += (double)x.y * scale;
    }
    return from;
}
// Slots of a layer's candidates: one per distinct prefix, in candidate order (prefixes do not increase with the candidate).  By a warp.
__device__ __forceinline__ void assign_slots(Cand* cd, SlotTab& stab, uint32_t K) {
    const uint32_t lane = threadIdx.x & 31;
    uint32_t n = 0, last = 0;
    for (uint32_t j0 = 0; j0 < K; j0 += 32u) {
        const uint32_t j = j0 + lane, pfx = j < K ? cd[j].prefix : 0u;
        const uint32_t left = __shfl_up_sync(0xffffffffu, pfx, 1);
        const bool first = j < K && (lane ? left != pfx : (n == 0u || last != pfx));
        const uint32_t m = __ballot_sync(0xffffffffu, first), slot = n + __popc(m & (0xffffffffu >> (31u - lane))) - 1u;
        if (first) stab.prefix[slot] = pfx;
        if (j < K) cd[j].slot = slot;
        last = __shfl_sync(0xffffffffu, pfx, min(K - 1u - j0, 31u));
        n += __popc(m);
    }
    if (lane == 0) stab.n = n;
}

// Level 1 of the exact radix select of one (worker, layer): candidates -> level-1 bins.  By a whole CTA; s_incl and s_below are
// [kL1Bins].  Leaves the histogram clean.
template <int NT>
__device__ __forceinline__ void fb_resolve1_layer(uint32_t l, uint32_t w, size_t wl, size_t wr, uint32_t K, uint32_t* __restrict__ g_cnt,
                                                  unsigned long long* __restrict__ g_ss, const KTab& ktab, Cand* __restrict__ cands,
                                                  SlotTab* __restrict__ slots, uint32_t* s_incl, double* s_below, uint32_t* s_w32,
                                                  double* s_w64) {
    uint32_t* gc = g_cnt + wr * kL1Bins;
    unsigned long long* gs = g_ss + wr * kL1Bins;
    for (int b = threadIdx.x; b < kL1Bins; b += NT) {
        s_incl[kL1Bins - 1 - b] = __ldcg(gc + b);
        s_below[b] = (double)__ldcg(gs + b) * sq_scale((uint32_t)b >> 3);
        gc[b] = 0;
        gs[b] = 0ull;
    }
    __syncthreads();
    scan_bins<kL1Bins, NT>(s_incl, s_below, s_w32, s_w64);
    Cand* cd = cands + wl * K;
    for (uint32_t j = threadIdx.x; j < K; j += NT) {
        const uint32_t k = (uint32_t)ktab.at(w, (size_t)l * K + j);
        const int p = find_pos<kL1Bins>(s_incl, k);
        const uint32_t above = p ? s_incl[p - 1] : 0u;
        Cand c;
        c.prefix = (uint32_t)(kL1Bins - 1 - p);
        c.rank = k - above;
        c.gt = above;
        c.err_low = s_below[kL1Bins - 1 - p];
        c.slot = 0;
        cd[j] = c;
    }
    __syncthreads();
    if (threadIdx.x < 32) assign_slots(cd, slots[wl], K);
    __syncthreads();
}

// LEVEL 2: refine inside a level-1 bin; LEVEL 3: inside a (level-1, level-2) bin.  By a whole CTA, a warp per slot: a lane takes
// 32 consecutive bins, whose counts it keeps.  Leaves the histograms clean.  Bound by the latency of a few rounds of loads per slot;
// with bins read one at a time, again for every candidate, it was the longest part of a layer's exact path.
template <int LEVEL, int NT>
__device__ __forceinline__ void fb_resolve23_layer(uint32_t l, uint32_t w, size_t wl, size_t wr, uint32_t K, uint32_t* __restrict__ g_cnt,
                                                   unsigned long long* __restrict__ g_ss, Cand* __restrict__ cands,
                                                   SlotTab* __restrict__ slots, float* __restrict__ err_out, uint32_t* __restrict__ tau_out,
                                                   uint32_t* __restrict__ keep_eq_out, uint32_t* __restrict__ shift_out,
                                                   const CodeSpace& codes) {
    const uint32_t lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    SlotTab& stab = slots[wl];
    Cand* cd = cands + wl * K;
    const uint32_t ns = stab.n;
    for (uint32_t s = wid; s < ns; s += NT / 32) {
        uint32_t* gc = g_cnt + (wr * K + s) * kL23Bins;
        unsigned long long* gs = g_ss + (wr * K + s) * kL23Bins;
        const uint32_t prefix = stab.prefix[s], b0 = 32u * lane;
        const double scale = LEVEL == 2 ? sq_scale(prefix >> 3) : 0.0; // LEVEL 2: prefix = level-1 bin (8 exponent + 3 mantissa bits)
        auto value = [&](uint32_t b) { return (double)__uint_as_float((prefix << 10) | b); };
        uint32_t c[32], cnt = 0;
        load_counts(c, gc, b0);
        double sq = 0.0;
        if (LEVEL == 2) {
            sq = add_squares(sq, gs, b0, 32u, scale);
#pragma unroll
            for (int i = 0; i < 32; ++i) cnt += c[i];
        } else { // all 31 bits known, the sum of squares is count * value^2
#pragma unroll
            for (int i = 0; i < 32; ++i) { const double v = value(b0 + i); cnt += c[i]; sq += (double)c[i] * v * v; }
        }
        uint32_t upto = cnt; // entries in the lane's bins and those of the lanes above
        double below = sq;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t yc = __shfl_down_sync(0xffffffffu, upto, o);
            const double ys = __shfl_up_sync(0xffffffffu, below, o);
            if (lane + o < 32u) upto += yc;
            if (lane >= (uint32_t)o) below += ys;
        }
        const uint32_t above = upto - cnt;
        below = __shfl_up_sync(0xffffffffu, below, 1); // exclusive value from the left neighbour: no cancellation
        if (lane == 0) below = 0.0;
        for (uint32_t j0 = 0; j0 < K; j0 += 32u) { // the slot's candidates, asked for by a lane each
            const bool in = j0 + lane < K;
            const uint32_t my_rank = in ? cd[j0 + lane].rank : 0u;
            uint32_t here = __ballot_sync(0xffffffffu, in && cd[j0 + lane].slot == s);
            for (; here; here &= here - 1u) {
                const uint32_t j = j0 + __ffs(here) - 1u, rank = __shfl_sync(0xffffffffu, my_rank, j - j0);
                if (above < rank && rank <= upto) { // one lane
                    uint32_t i = 0, gt = above, found_c = 0; // its bin that holds the rank, counted from the top
                    bool open = true;
#pragma unroll
                    for (int x = 31; x >= 0; --x) {
                        if (open && gt + c[x] >= rank) { open = false; i = x; found_c = c[x]; }
                        if (open) gt += c[x];
                    }
                    double e = below;
                    if (LEVEL == 2) {
                        e = add_squares(e, gs, b0, i, scale);
                    } else {
#pragma unroll
                        for (int x = 0; x < 31; ++x)
                            if ((uint32_t)x < i) { const double v = value(b0 + x); e += (double)c[x] * v * v; }
                    }
                    e += cd[j].err_low;
                    const uint32_t found = (prefix << 10) | (b0 + i);
                    if (LEVEL == 2) {
                        cd[j].prefix = found;
                        cd[j].gt += gt;
                        cd[j].err_low = e;
                        cd[j].rank = rank - gt;
                    } else {
                        const uint32_t keep = rank - gt; // 1 <= keep <= found_c
                        const double v = (double)__uint_as_float(found);
                        err_out[wl * K + j] = (float)(e + (double)(found_c - keep) * v * v);
                        tau_out[wl * K + j] = found;
                        keep_eq_out[wl * K + j] = keep;
                        shift_out[wl * K + j] = codes.code(w, l, found) << 8;
                    }
                }
                __syncwarp();
            }
        }
        __syncwarp();
        for (uint32_t b = lane; b < (uint32_t)kL23Bins / 4; b += 32u) reinterpret_cast<uint4*>(gc)[b] = make_uint4(0u, 0u, 0u, 0u);
        if (LEVEL == 2)
            for (uint32_t b = lane; b < (uint32_t)kL23Bins / 2; b += 32u) reinterpret_cast<ulonglong2*>(gs)[b] = make_ulonglong2(0ull, 0ull);
    }
    __syncthreads();
    if (LEVEL == 2 && threadIdx.x < 32) assign_slots(cd, stab, K); // new slots = distinct 21-bit prefixes
    __syncthreads();
}

} // namespace kimad
