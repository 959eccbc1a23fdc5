// Stages (d)-(f): Top-K selection at the chosen k, ordered sparse pack, EF21 update.
//
// After the DP every (worker, layer) knows a key interval [lo, lo + 2^shift) that contains its
// threshold and the rank of the threshold inside that interval (shift = 0 when the curve stage already
// resolved all 31 bits).  k_sel_count, one sweep over the byte codes the curve stage left, counts, per 2048-element
// slice, the entries above the interval, lists the few entries inside it per layer and marks the 16-element groups that
// can hold a kept entry; k_sel_offsets (a CTA per layer) takes the exact threshold from the listed entries and leaves one
// job record per chunk with the chunk's output offset; k_sel_write compacts in index order and updates the estimator,
// reading only the marked groups of sparse slices.  Of a layer with more entries in its interval than its list holds (values
// that came from 16 or 8 bits repeat) every key of the interval is counted, and every slice keeps a list of its own, where its codes
// were; the slices' counts then follow from those (k_sel_recount, usually nothing to do).  No kernel waits on another: offsets
// come from stored counts.
#pragma once
#include "kimad_curve.cuh"

namespace kimad {

// A chunk (at most 32768 elements from its 16-byte aligned start) is cut into 16 slices of 2048 elements; in
// the sweeps of this stage a warp works on a slice by itself, so no sweep needs a block-wide barrier.
constexpr int kSliceElems = 2048;
constexpr int kSlices = 16;
constexpr int kStageCap = 128;    // ... of which a CTA of the counting sweep gathers as many before it appends them

struct ChunkSel { // per (worker, chunk)
    uint16_t above[kSlices];   // per slice: entries whose key lies above the interval, after k_sel_offsets above the threshold
    uint16_t eq[kSlices];      // per slice: entries equal to the threshold; until k_sel_recount, where every slice has a list of its
                               // own: entries inside the interval
    uint4 mask[kSlices];       // per slice: bit g set when the 16-element group g may hold a kept entry (key >= the
                               // interval's lower end); a superset of the groups the write sweep has to read
};

// Everything the write sweep needs to know about a (worker, chunk) besides the data, gathered by k_sel_offsets so
// that the write sweep starts from loads whose addresses depend on the block index only.
struct ChunkJob {
    uint32_t mode;      // 0: nothing of this chunk is kept; 1: threshold tau; 2: the whole layer is kept
    uint32_t tau;
    uint32_t keep_eq;   // entries equal to tau that are kept, over the layer (lowest indices first)
    uint32_t gt_before; // entries above tau in the layer's earlier chunks
    uint32_t eq_before; // entries equal to tau in the layer's earlier chunks
    uint32_t idx0;      // layer-local index of the chunk's aligned start (may wrap; added back by the sweep)
    uint64_t base;      // first output position of the layer in the worker's packed buffers
};

// Entries inside the intervals.  Only layers swept with a histogram have an interval wider than one key; their bin tables
// and bin histograms are free after the DP, and hold the layer's list (kListCap records {chunk of the layer, slice << 16 |
// key - lo}) or, for intervals that may hold more, the count of every key of the interval (clean before and after).
struct Interval {
    uint32_t* n;        // [W][L] entries in the layer's list, then finished chunks of k_sel_recount; zero between steps
    uint32_t* bin_lo;   // [W][R][kMaxBins + 1]
    uint32_t* bh_cnt;   // [W][R][kMaxBins]
    unsigned long long* bh_sum;
    const uint32_t* reg_index;
    uint32_t R;
    __device__ __forceinline__ size_t slot(uint32_t w, uint32_t l) const { return (size_t)w * R + reg_index[l]; }
    __device__ __forceinline__ uint2* list(size_t wr) const {
        return reinterpret_cast<uint2*>((reinterpret_cast<uintptr_t>(bin_lo + wr * (kMaxBins + 1)) + 7u) & ~(uintptr_t)7u);
    }
    __device__ __forceinline__ uint32_t* key_count(size_t wr, uint32_t d) const {
        return d < (uint32_t)kMaxBins ? bh_cnt + wr * kMaxBins + d : reinterpret_cast<uint32_t*>(bh_sum + wr * kMaxBins) + (d - kMaxBins);
    }
};
static_assert(kListCap * 8 + 8 <= (uint32_t)(kMaxBins + 1) * 4 && 3 * kMaxBins >= (1 << kMaxShift), "list and key counts fit the bin arrays");

// The list of a slice: distances (key - lo) of its entries inside the interval, laid over the slice's own codes once its warp has
// read them (units of sixteen codes that the slice shares with another chunk stay).  Nobody reads a code after the counting sweep.
struct SliceList {
    uint16_t* at;
    uint32_t cap; // entries; a slice with more is counted from the inputs
    __device__ __forceinline__ SliceList(const DSource& p, uint32_t w, const ChunkView& cv, uint32_t sl) {
        const uint32_t b = max((cv.first + 15u) & ~15u, sl * kSliceElems), e = min(cv.len & ~15u, (sl + 1) * kSliceElems);
        at = reinterpret_cast<uint16_t*>(p.code + (size_t)w * p.dstride + cv.a0 + b);
        cap = e > b ? (e - b) / 2 : 0u;
    }
};

// chunks of layers whose slices have lists of their own
struct Recount {
    uint32_t n_chunks;
    uint32_t _pad[3];
};

// ------------------------------------------------------------------------------------------------
// Counting sweep: one or two CTAs per chunk, a warp takes one or two slices.
// Bound by the loads of the codes where layers are large, by instructions where most lanes hold a kept entry: a lane's sixteen
// flags are gathered in one word, so that only entries with the interval's own code cost more than a few instructions
// (2 x 1.1 B, 0.7 % kept: 495 -> 479 us; 4 x 124 M, 16 % kept: 166 -> 161; 8 x 25.6 M, 5 %: 78 -> 76, against flags taken word by word).
// ------------------------------------------------------------------------------------------------
__global__ void __launch_bounds__(kThreads, 6)
k_sel_count(DSource dbuf, const Chunk* __restrict__ chunks, uint32_t n_chunks, uint32_t L,
            const Sel* __restrict__ sel, const LayerDesc* __restrict__ layers, ChunkSel* __restrict__ csel, const Interval in,
            Recount* __restrict__ rc, uint32_t w_base) {
    pdl_wait();
    __shared__ uint32_t s_n, s_at, s_in[kThreads / 32]; // s_in: entries in the list of the warp's slice
    __shared__ uint32_t s_low[kStageCap];
    const Chunk ch = chunks[blockIdx.x];
    const uint32_t w = w_base + blockIdx.y;
    const size_t wl = (size_t)w * L + ch.layer;
    const Sel s = sel[wl];
    const LayerDesc ld = layers[ch.layer];
    ChunkSel* out = csel + (size_t)w * n_chunks + blockIdx.x;
    const ChunkView cv(ch, dbuf.phase.at(w));
    const uint32_t lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    if (blockIdx.x == 0 && blockIdx.y == 0 && threadIdx.x == 0) rc->n_chunks = 0; // consumed by the step before
    if (s.k == 0 || (uint64_t)s.k == ld.n) { // nothing / everything kept: no need to look at the data
        if (threadIdx.x < kSlices) {
            const uint32_t lo = max(cv.first, threadIdx.x * kSliceElems), hi = min(cv.len, (threadIdx.x + 1) * kSliceElems);
            out->above[threadIdx.x] = (uint16_t)((s.k && hi > lo) ? hi - lo : 0u);
            out->eq[threadIdx.x] = 0;
        }
        return;
    }
    const uint32_t lo = s.tau, width = 1u << s.shift;
    const bool exact = s.shift == 0, many = !exact && (s.code & kSelMany) != 0;
    const uint32_t rel = blockIdx.x - ld.first_chunk, code = s.code & 127u;
    if (threadIdx.x == 0) s_n = 0;
    __syncthreads();
    const DView dd(dbuf, w, cv.a0);
    auto append = [&](uint32_t at, uint32_t rec) { // one entry of the layer's interval, the at-th
        if (at < kListCap) in.list(in.slot(w, ch.layer))[at] = make_uint2(rel, rec);
    };
    // Codes first: an entry whose code (the byte the sweep left for it) is larger than the code of the interval's
    // keys lies above the interval, one with a smaller code below; only entries with the interval's own code are
    // completed from the inputs.  Codes are 7-bit numbers, so "x >= t" for the four bytes of a word is bit 7 of
    // every byte of x + (0x80 - t) * 0x01010101.
    const uint32_t add_gt = (0x80u - (code + 1u)) * 0x01010101u, add_ge = (0x80u - code) * 0x01010101u;
    for (uint32_t sl = wid + blockIdx.z * (kThreads / 32); sl < (uint32_t)kSlices; sl += gridDim.z * (kThreads / 32)) {
        // low half: entries above the interval; high half: entries equal to an exact threshold, or in the slice's own list
        uint32_t above = 0;
        uint32_t mask[kSliceElems / 512];
        auto visit = [&](uint32_t key, auto many_c) -> bool { // true: the key is not below the interval
            const uint32_t d1 = key - lo; // wraps to >= 2^31 for keys below the interval
            if (d1 < width) {
                if (decltype(many_c)::value) {
                    above += 0x10000u;
                    const SliceList mine(dbuf, w, cv, sl);
                    const uint32_t p = atomicAdd(&s_in[wid], 1u);
                    if (p < mine.cap) mine.at[p] = (uint16_t)d1;
                    if (KIMAD_CHECK(d1 < (1u << kMaxShift), 1)) atomicAdd(in.key_count(in.slot(w, ch.layer), d1), 1u);
                } else if (exact) {
                    // an exact threshold needs no list, only the slice's number of equal entries (there may be millions of
                    // them: the exact zeros of a sparse gradient)
                    above += 0x10000u;
                } else {
                    const uint32_t p = atomicAdd(&s_n, 1u);
                    if (p < (uint32_t)kStageCap) s_low[p] = (sl << 16) | d1;
                    else append(atomicAdd(in.n + wl, 1u), (sl << 16) | d1);
                }
            } else {
                above += d1 < 0x80000000u;
            }
            return d1 < 0x80000000u;
        };
        // a lane takes sixteen consecutive codes (one 128-bit load) of each of the slice's four rows of 512 elements: a group
        constexpr int ROWS = kSliceElems / 512;
        const uint32_t u0 = sl * (kSliceElems / 16) + lane; // this lane's 16-element unit in row 0
        // EDGE: the slice reaches over an end of the chunk; its units there hold codes of the neighbouring chunk, or bytes that
        // nobody wrote
        // MANY: every slice has a list of its own
        auto count = [&](auto edge_c, auto many_c) {
            constexpr bool EDGE = decltype(edge_c)::value, MANY = decltype(many_c)::value;
            uint4 a[ROWS];
#pragma unroll
            for (int r = 0; r < ROWS; ++r) {
                const uint32_t e0 = 16 * (u0 + r * 32);
                if (EDGE) a[r] = make_uint4(0u, 0u, 0u, 0u);
                if (!EDGE || (e0 + 16 > cv.first && e0 < cv.len)) a[r] = __ldcs(reinterpret_cast<const uint4*>(dd.code) + u0 + r * 32);
            }
            if (MANY) { // the list takes the place of the codes
                __syncwarp();
                if (lane == 0) s_in[wid] = 0;
                __syncwarp();
            }
#pragma unroll
            for (int r = 0; r < ROWS; ++r) {
                const uint32_t e0 = 16 * (u0 + r * 32);
                bool f = false; // this lane holds an entry that is not below the interval
                uint32_t in = 0xffffu; // elements of the unit that are the chunk's
                uint32_t x[4] = {a[r].x, a[r].y, a[r].z, a[r].w};
                if (EDGE) {
                    if (e0 < cv.first) in = e0 + 16 > cv.first ? in & (~0u << (cv.first - e0)) : 0u;
                    if (e0 + 16 > cv.len) in = e0 < cv.len ? in & ~(~0u << (cv.len - e0)) : 0u;
#pragma unroll
                    for (int j = 0; j < 4; ++j) x[j] &= 0x7f7f7f7fu;
                }
                uint32_t ge[4];
#pragma unroll
                for (int j = 0; j < 4; ++j) ge[j] = (x[j] + add_ge) & 0x80808080u;
                if ((ge[0] | ge[1] | ge[2] | ge[3]) && in) { // with a sparse budget few lanes hold a code that is not below the interval's
                    // the unit's sixteen flags in one word: bit 8 k + 7 - j -> element 4 j + k
                    uint32_t gt = 0, border = 0;
#pragma unroll
                    for (int j = 0; j < 4; ++j) {
                        gt |= ((x[j] + add_gt) & 0x80808080u) >> j;
                        border |= ge[j] >> j;
                    }
                    border ^= gt; // the interval's own code
                    if (EDGE) {
                        uint32_t m = 0;
#pragma unroll
                        for (int j = 0; j < 4; ++j) {
                            const uint32_t v = in >> (4 * j);
                            m |= (((v & 1u) << 7) | ((v & 2u) << 14) | ((v & 4u) << 21) | ((v & 8u) << 28)) >> j;
                        }
                        gt &= m;
                        border &= m;
                    }
                    above += __popc(gt);
                    f = gt != 0; // entries with the interval's code mark the group only if they are not below it
                    auto take = [&]() { // the next one of them
                        const uint32_t p = __ffs(border) - 1;
                        border &= border - 1;
                        return e0 + 4u * (7u - (p & 7u)) + (p >> 3);
                    };
                    while (border) { // completed from the inputs two at a time: their loads are independent
                        const uint32_t p0 = take(), p1 = border ? take() : p0;
                        const float v0 = dd.at(p0), v1 = dd.at(p1);
                        f |= visit(key_of(v0), many_c);
                        if (p1 != p0) f |= visit(key_of(v1), many_c);
                    }
                }
                mask[r] = __ballot_sync(0xffffffffu, f);
            }
        };
        if (many) count(std::true_type{}, std::true_type{});
        else if (sl * kSliceElems >= cv.first && (sl + 1) * kSliceElems <= cv.len) count(std::false_type{}, std::false_type{});
        else count(std::true_type{}, std::false_type{});
#pragma unroll
        for (int o = 16; o; o >>= 1) above += __shfl_xor_sync(0xffffffffu, above, o);
        if (lane == 0) { out->above[sl] = (uint16_t)above; out->eq[sl] = (uint16_t)(above >> 16); out->mask[sl] = make_uint4(mask[0], mask[1], mask[2], mask[3]); }
    }
    __syncthreads();
    const uint32_t n_in = min(s_n, (uint32_t)kStageCap);
    if (n_in) {
        if (threadIdx.x == 0) s_at = atomicAdd(in.n + wl, n_in);
        __syncthreads();
        if (threadIdx.x < n_in) append(s_at + threadIdx.x, s_low[threadIdx.x]);
    }
}

// Job records of a layer's chunks: exclusive prefix of the chunk totals over the layer's earlier chunks, stored with the
// layer's threshold.  The whole CTA works on it.
template <int NT>
__device__ __forceinline__ void sel_scan_layer(const LayerDesc& ld, const Sel& s, const Chunk* __restrict__ chunks,
                                               uint32_t phase, const ChunkSel* cs /* the layer's */, ChunkJob* __restrict__ jb,
                                               uint32_t* s_w) {
    const bool all = (uint64_t)s.k == ld.n;
    uint32_t run_g = 0, run_e = 0;
    for (uint32_t base = 0; base < ld.n_chunks; base += NT) {
        const uint32_t i = base + threadIdx.x;
        uint32_t g = 0, q = 0;
        if (i < ld.n_chunks) { // sixteen 16-bit counts each
            const uint4* p = reinterpret_cast<const uint4*>(cs + i);
            const uint4 a = __ldcg(p), b = __ldcg(p + 1), c = __ldcg(p + 2), d = __ldcg(p + 3);
            auto sum = [](const uint4& x, const uint4& y) {
                const uint32_t t = (x.x & 0xffffu) + (x.y & 0xffffu) + (x.z & 0xffffu) + (x.w & 0xffffu) + (y.x & 0xffffu) +
                                   (y.y & 0xffffu) + (y.z & 0xffffu) + (y.w & 0xffffu);
                return t + (x.x >> 16) + (x.y >> 16) + (x.z >> 16) + (x.w >> 16) + (y.x >> 16) + (y.y >> 16) + (y.z >> 16) + (y.w >> 16);
            };
            g = sum(a, b);
            q = sum(c, d);
        }
        uint32_t tg, te;
        const uint32_t eg = block_excl_scan<uint32_t, NT>(g, s_w, &tg);
        const uint32_t ee = block_excl_scan<uint32_t, NT>(q, s_w, &te);
        if (i < ld.n_chunks) {
            const ChunkView cv(chunks[ld.first_chunk + i], phase);
            ChunkJob j;
            j.tau = s.tau;
            j.keep_eq = s.keep_eq;
            j.gt_before = run_g + eg;
            j.eq_before = run_e + ee;
            j.idx0 = (uint32_t)(cv.a0 - phase - ld.begin);
            j.base = s.base;
            const bool none = s.k == 0 || (!all && g == 0 && (q == 0 || j.eq_before >= s.keep_eq));
            j.mode = none ? 0u : (all ? 2u : 1u);
            jb[i] = j;
        }
        run_g += tg;
        run_e += te;
    }
}

// Exact per-slice (gt, eq) of a chunk whose slices have lists of their own, by a warp: from the lists, or from the inputs where a slice
// has more entries inside the interval than its list holds.  The first 32 entries of AHEAD lists are requested together.
template <int AHEAD>
__device__ __forceinline__ void recount_chunk(const DSource& dbuf, uint32_t w, const Chunk& ch, const Sel& s, ChunkSel* out) {
    const uint32_t lane = threadIdx.x & 31;
    const ChunkView cv(ch, dbuf.phase.at(w));
    const uint32_t my_in = lane < (uint32_t)kSlices ? out->eq[lane] : 0u; // lane i: slice i
    uint32_t my_gt = lane < (uint32_t)kSlices ? out->above[lane] : 0u, my_eq = 0;
#pragma unroll 1
    for (int sl0 = 0; sl0 < kSlices; sl0 += AHEAD) {
        uint32_t first[AHEAD]; // the slices' first entries, a lane each
#pragma unroll
        for (int i = 0; i < AHEAD; ++i) {
            const SliceList list(dbuf, w, cv, sl0 + i);
            const uint32_t n_in = __shfl_sync(0xffffffffu, my_in, sl0 + i);
            first[i] = lane < n_in && n_in <= list.cap ? list.at[lane] : 0xffffffffu;
        }
#pragma unroll
        for (int i = 0; i < AHEAD; ++i) {
            const uint32_t sl = sl0 + i;
            const SliceList list(dbuf, w, cv, sl);
            const uint32_t n_in = __shfl_sync(0xffffffffu, my_in, sl);
            if (n_in == 0) continue;
            uint32_t gt = 0, eq = 0;
            if (n_in <= list.cap) {
                auto count = [&](uint32_t d) {
                    gt += __popc(__ballot_sync(0xffffffffu, d != 0xffffffffu && d > s.tau_low));
                    eq += __popc(__ballot_sync(0xffffffffu, d == s.tau_low));
                };
                count(first[i]);
                for (uint32_t x = 32; x < n_in; x += 32) count(x + lane < n_in ? list.at[x + lane] : 0xffffffffu);
                gt += __shfl_sync(0xffffffffu, my_gt, sl);
            } else {
                const DView dd(dbuf, w, cv.a0);
                const uint32_t x0 = max(cv.first, sl * kSliceElems), x1 = min(cv.len, (sl + 1) * kSliceElems);
                for (uint32_t x = x0 + lane; x < x1; x += 32) {
                    const uint32_t key = key_of(dd.at(x));
                    gt += key > s.tau;
                    eq += key == s.tau;
                }
#pragma unroll
                for (int o = 16; o; o >>= 1) {
                    gt += __shfl_xor_sync(0xffffffffu, gt, o);
                    eq += __shfl_xor_sync(0xffffffffu, eq, o);
                }
            }
            if (lane == sl) { my_gt = gt; my_eq = eq; }
        }
    }
    if (lane < (uint32_t)kSlices) { out->above[lane] = (uint16_t)my_gt; out->eq[lane] = (uint16_t)my_eq; }
}

// Exact threshold and job records, one CTA per (layer, worker).  The listed entries (16-bit distances from the interval's
// lower key) are ranked by two 8-bit digits; each then joins its slice's counts.  Bound by the latency of a few dependent
// rounds per layer: NT = 512 where a layer has thousands of chunks, 128 where none has more than 256 (1995 layers of two
// two chunks: 40 us with 512 threads, which need two waves of CTAs).
// HERE: layers with repeated values count their chunks here (at most kInlineChunks of them: a kernel less in the step's chain);
// else they are listed for k_sel_recount.  (Ten CTAs of 128 threads per SM.)
template <int NT, bool HERE>
__global__ void __launch_bounds__(NT, NT == 512 ? 3 : 10)
k_sel_offsets(const DSource dbuf, const LayerDesc* __restrict__ layers, const Chunk* __restrict__ chunks, uint32_t n_chunks, uint32_t L,
              Sel* __restrict__ sel, ChunkSel* __restrict__ csel, ChunkJob* __restrict__ jobs, const Interval in, FbList* __restrict__ fb,
              Recount* __restrict__ rc, uint2* __restrict__ rc_chunks, uint32_t list_cap, uint32_t w_base) {
    pdl_wait();
    __shared__ uint32_t s_w[NT / 32], s_h[256], s_digit, s_gt, s_at;
    __shared__ uint16_t s_key[kListCap];
    const uint32_t l = blockIdx.x, w = w_base + blockIdx.y;
    const size_t wl = (size_t)w * L + l;
    const LayerDesc ld = layers[l];
    Sel s = sel[wl];
    if (blockIdx.x == 0 && blockIdx.y == 0 && threadIdx.x == 0) { // the curve stage's lists (of these workers) have been consumed
        fb->n_chunks = 0;
        fb->n_layers = 0;
        fb->rf_chunks = 0;
        fb->rf_layers = 0;
    }
    ChunkSel* cs = csel + (size_t)w * n_chunks + ld.first_chunk;
    if (s.k != 0 && (uint64_t)s.k != ld.n && s.shift != 0) {
        const size_t wr = in.slot(w, l);
        const uint2* list = in.list(wr);
        const uint32_t cnt = min(in.n[wl], kListCap);
        const bool over = (s.code & kSelMany) != 0;
        if (!over) {
            for (uint32_t i = threadIdx.x; i < cnt; i += NT) s_key[i] = (uint16_t)(list[i].y & 0xffffu);
            uint32_t rank = s.keep_eq, hi_digit = 0, greater = 0; // rank <= cnt by construction
            for (int pass = 0; pass < 2; ++pass) {
                for (uint32_t i = threadIdx.x; i < 256; i += NT) s_h[i] = 0;
                __syncthreads();
                for (uint32_t i = threadIdx.x; i < cnt; i += NT) {
                    const uint32_t k = s_key[i];
                    if (pass == 0) atomicAdd(&s_h[k >> 8], 1u);
                    else if ((k >> 8) == hi_digit) atomicAdd(&s_h[k & 255u], 1u);
                }
                __syncthreads();
                if (threadIdx.x < 32) { // warp 0: lane L takes the digits 255 - 8 L down to 248 - 8 L
                    const uint32_t lane = threadIdx.x, top = 255u - 8u * lane;
                    uint32_t mine = 0;
#pragma unroll
                    for (uint32_t j = 0; j < 8; ++j) mine += s_h[top - j];
                    uint32_t incl = mine;
#pragma unroll
                    for (int o = 1; o < 32; o <<= 1) {
                        const uint32_t y = __shfl_up_sync(0xffffffffu, incl, o);
                        if (lane >= (uint32_t)o) incl += y;
                    }
                    const uint32_t hit = __ballot_sync(0xffffffffu, incl >= rank);
                    if (hit && lane == (uint32_t)(__ffs(hit) - 1)) {
                        uint32_t acc = incl - mine, d = top;
                        while (acc + s_h[d] < rank) { acc += s_h[d]; --d; }
                        s_digit = d;
                        s_gt = acc; // entries of this pass's candidates with a larger digit
                    }
                }
                __syncthreads();
                if (pass == 0) { hi_digit = s_digit; greater = s_gt; rank -= s_gt; }
                else { greater += s_gt; }
            }
            s.tau_low = (hi_digit << 8) | s_digit;
            s.keep_eq -= greater; // rank among the entries equal to the threshold: those above it come first
            for (uint32_t i = threadIdx.x; i < cnt; i += NT) {
                const uint2 e = list[i];
                const uint32_t k = e.y & 0xffffu, sl = e.y >> 16;
                if (k < s.tau_low || !KIMAD_CHECK(e.x < ld.n_chunks && sl < (uint32_t)kSlices, 6)) continue;
                uint32_t* c = reinterpret_cast<uint32_t*>(k > s.tau_low ? cs[e.x].above : cs[e.x].eq) + (sl >> 1);
                atomicAdd(c, 1u << (16u * (sl & 1u)));
            }
            __threadfence(); // the counts are read back below by other threads of this CTA
        } else { // every key of the interval was counted
            // thread t takes the keys [k0, k1), descending with t
            const uint32_t width = 1u << s.shift, per = (width + NT - 1) / NT;
            const uint32_t k1 = threadIdx.x * per < width ? width - threadIdx.x * per : 0u, k0 = k1 > per ? k1 - per : 0u;
            uint32_t mine = 0;
            for (uint32_t k = k0; k < k1; ++k) mine += __ldcg(in.key_count(wr, k));
            uint32_t before = block_excl_scan<uint32_t, NT>(mine, s_w, nullptr);
            if (before < s.keep_eq && before + mine >= s.keep_eq) {
                uint32_t k = k1 - 1;
                for (;; --k) {
                    const uint32_t c = __ldcg(in.key_count(wr, k));
                    if (before + c >= s.keep_eq) break;
                    before += c;
                }
                s_digit = k;
                s_gt = before;
            }
            __syncthreads();
            s.tau_low = s_digit;
            s.keep_eq -= s_gt;
            for (uint32_t k = k0; k < k1; ++k) *in.key_count(wr, k) = 0; // clean for the next use
            if (!HERE && threadIdx.x == 0) s_at = atomicAdd(&rc->n_chunks, ld.n_chunks);
        }
        s.tau += s.tau_low;
        s.shift = 0;
        __syncthreads();
        if (threadIdx.x == 0) { sel[wl] = s; in.n[wl] = 0; }
        if (over && HERE) {
            for (uint32_t i = threadIdx.x >> 5; i < ld.n_chunks; i += NT / 32) recount_chunk<4>(dbuf, w, chunks[ld.first_chunk + i], s, cs + i);
            __threadfence();
            __syncthreads();
        } else if (over) { // its chunks are counted again
            for (uint32_t i = threadIdx.x; i < ld.n_chunks; i += NT)
                if (KIMAD_CHECK(s_at + i < list_cap, 2)) rc_chunks[s_at + i] = make_uint2(w, ld.first_chunk + i);
            return;
        }
    }
    sel_scan_layer<NT>(ld, s, chunks, dbuf.phase.at(w), cs, jobs + (size_t)w * n_chunks + ld.first_chunk, s_w);
}

// The listed chunks, a warp each.  The CTA that finishes the last chunk of a layer makes the layer's job records (Interval::n counts the
// finished ones).  Bound by latency.  Values of bf16 gradients (4 x 124 M, 0.6 % kept): offsets 1226 us with every chunk counted
// again from the inputs, 77 so, and 22 where nothing repeats.
__global__ void __launch_bounds__(kThreads)
k_sel_recount(DSource dbuf, const LayerDesc* __restrict__ layers, const Chunk* __restrict__ chunks, uint32_t n_chunks,
              uint32_t L, const Sel* __restrict__ sel, ChunkSel* __restrict__ csel, ChunkJob* __restrict__ jobs, const Interval in,
              const Recount* __restrict__ rc, const uint2* __restrict__ rc_chunks) {
    pdl_wait();
    constexpr uint32_t kWarps = kThreads / 32;
    __shared__ uint32_t s_w[kWarps], s_last[kWarps]; // s_last: the warp's chunk was the last one of its layer
    const uint32_t n = rc->n_chunks;
    const uint32_t lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    for (uint32_t base = blockIdx.x * kWarps; base < n; base += gridDim.x * kWarps) {
        if (lane == 0) s_last[wid] = 0;
        if (base + wid < n) {
            const uint2 e = rc_chunks[base + wid];
            const Chunk ch = chunks[e.y];
            const size_t wl = (size_t)e.x * L + ch.layer;
            const Sel s = sel[wl];
            recount_chunk<kSlices>(dbuf, e.x, ch, s, csel + (size_t)e.x * n_chunks + e.y);
            __threadfence();
            __syncwarp();
            if (lane == 0) s_last[wid] = atomicAdd(in.n + wl, 1u) + 1u == layers[ch.layer].n_chunks;
        }
        __syncthreads();
        for (uint32_t i = 0; i < kWarps; ++i) {
            if (!s_last[i]) continue;
            const uint2 e = rc_chunks[base + i];
            const uint32_t l = chunks[e.y].layer;
            const size_t wl = (size_t)e.x * L + l;
            const LayerDesc ld = layers[l];
            __threadfence();
            sel_scan_layer<kThreads>(ld, sel[wl], chunks, dbuf.phase.at(e.x), csel + (size_t)e.x * n_chunks + ld.first_chunk,
                                     jobs + (size_t)e.x * n_chunks + ld.first_chunk, s_w);
            if (threadIdx.x == 0) in.n[wl] = 0;
        }
        __syncthreads();
    }
}

// ------------------------------------------------------------------------------------------------
// (e) + (f).  A warp compacts a slice by itself, 512 elements a round.  Bound by memory: both inputs are read, and every
// 32-byte sector of the estimator with a kept entry is written.  A round is four rows of 128 elements, so that the lanes of an
// access lie side by side; positions in index order come from one warp scan of the four rows' counts, a byte each.  (Sixteen
// consecutive elements per lane, whose lanes lie 64 bytes apart, took 117 instead of 109 us for 4 x 11.7 M elements of which 6.5 %
// are kept, 657 instead of 582 us for 4 x 124 M of which 16 % are kept, and 177 instead of 109 us for 2 x 25.6 M at odd distances.)
// ------------------------------------------------------------------------------------------------
// DENSE: tuned for steps whose budget keeps more than a few per cent of the entries (the host picks the
// instantiation from the budgets; both are correct for any input).
// A slice is read group by group where at most kSparseGroups of its 128 groups are marked.  Write stage with 48 / 64 / 96 / 128:
// sparse (4 x 124 M, 0.6 % kept) 148 / 141 / 137 / 138 us, (1.1 B, half of it zero) 145 / 145 / 144 / 150; dense (4 x 124 M, 16 %)
// 558 / 553 / 561 / 728, (8 x 25.6 M, 5 %) 201 / 200 / 213 / 244.  Groups of 32 elements instead of 16 (steps): 1201 -> 1178 us
// (4 x 124 M, 0.6 %), 4740 -> 4620 (2 x 1.1 B, 0.7 %), 925 -> 910 (8 x 25.6 M).
template <bool BF16, bool DENSE>
__global__ void __launch_bounds__(kThreads, DENSE ? 3 : 8)
k_sel_write(const float* __restrict__ grads, float* __restrict__ state, const Chunk* __restrict__ chunks,
            uint32_t n_chunks, uint64_t stride, const Phase phase, const ChunkSel* __restrict__ csel,
            const ChunkJob* __restrict__ jobs, uint64_t cap, uint32_t* __restrict__ out_idx, void* __restrict__ out_val,
            uint32_t w_base) {
    pdl_wait();
    const uint32_t w = w_base + blockIdx.y;
    const ChunkJob jb = jobs[(size_t)w * n_chunks + blockIdx.x];
    if (jb.mode == 0) return; // nothing kept in this chunk
    const Chunk ch = chunks[blockIdx.x];
    const ChunkSel& cs = csel[(size_t)w * n_chunks + blockIdx.x];
    const bool all = jb.mode == 2;
    const uint32_t keep_eq = jb.keep_eq;
    const uint32_t tau = jb.tau;
    const ChunkView cv(ch, phase.at(w));
    // d is recomputed from the inputs; every element of the estimator is read before this kernel updates it
    const float* gr = grads + (size_t)w * stride + cv.a0 - phase.at(w);
    float* st = state + (size_t)w * stride + cv.a0 - phase.at(w);
    uint32_t* oi = out_idx + (size_t)w * cap + jb.base;
    float* ov32 = reinterpret_cast<float*>(out_val) + (size_t)w * cap + jb.base;
    __nv_bfloat16* ov16 = reinterpret_cast<__nv_bfloat16*>(out_val) + (size_t)w * cap + jb.base;
    const uint32_t idx0 = jb.idx0;
    const uint32_t lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const bool st_vec = ((reinterpret_cast<uintptr_t>(st) | reinterpret_cast<uintptr_t>(gr)) & 15u) == 0; // 128-bit access to both
    // entries above (low half) and equal to tau (high half) in the chunk's slices up to the one of lane i
    uint32_t upto = lane < (uint32_t)kSlices ? cs.above[lane] | (uint32_t)cs.eq[lane] << 16 : 0u;
#pragma unroll
    for (int o = 1; o < kSlices; o <<= 1) {
        const uint32_t y = __shfl_up_sync(0xffffffffu, upto, o);
        if (lane >= (uint32_t)o) upto += y;
    }
    constexpr uint32_t kSparseGroups = DENSE ? 64 : 96;
    __shared__ uint8_t s_pos[kThreads / 32][kSparseGroups]; // per warp: the marked groups of a slice, ascending
    __shared__ uint32_t s_stage[DENSE ? kThreads / 32 : 1][DENSE ? 2 * 16 * 32 : 1]; // per warp: a round's indices, values

    for (uint32_t sl = wid + blockIdx.z * (kThreads / 32); sl < (uint32_t)kSlices; sl += gridDim.z * (kThreads / 32)) {
        const uint32_t x0 = sl * kSliceElems;
        if (x0 >= cv.len) break;
        // entries equal to tau are kept while their rank among equals (ascending index) is below keep_eq
        const uint32_t ahead = sl ? __shfl_sync(0xffffffffu, upto, sl - 1) : 0u, here = __shfl_sync(0xffffffffu, upto, sl) - ahead;
        const uint32_t gt_before = jb.gt_before + (ahead & 0xffffu), eq_before = jb.eq_before + (ahead >> 16);
        const uint32_t gt_here = here & 0xffffu, eq_here = here >> 16;
        // eq_mode 0: none of this slice's equals is kept; 1: all are; 2: ranks must be counted
        const int eq_mode = (all || eq_here == 0 || eq_before >= keep_eq) ? 0 : (eq_before + eq_here <= keep_eq ? 1 : 2);
        if (!all && gt_here == 0 && eq_mode == 0) continue; // nothing kept in this slice
        uint32_t eq_seen = eq_before;
        uint32_t pos = gt_before + min(eq_before, keep_eq); // position of the slice's first kept entry in the layer
        const uint4 gm = cs.mask[sl];
        const uint32_t n_groups = __popc(gm.x) + __popc(gm.y) + __popc(gm.z) + __popc(gm.w);
        if (!all && n_groups <= kSparseGroups) {
            // sparse slice: read only the 16-element groups the counting sweep marked; four lanes per group,
            // eight groups per pass, in ascending order, so that lane order is index order
            uint8_t* sp = s_pos[wid];
            const uint32_t lt = (1u << lane) - 1u, g4[4] = {gm.x, gm.y, gm.z, gm.w};
            __syncwarp();
            uint32_t at = 0;
#pragma unroll
            for (uint32_t q = 0; q < 4; ++q) {
                if ((g4[q] >> lane) & 1u) sp[at + __popc(g4[q] & lt)] = (uint8_t)(32u * q + lane);
                at += __popc(g4[q]);
            }
            __syncwarp();
            for (uint32_t it = 0; it < n_groups; it += 8) {
                const uint32_t r = it + (lane >> 2);
                uint32_t keepm = 0, eqm = 0, e0 = 0;
                auto classify = [&](float v, int i) {
                    const uint32_t key = key_of(v);
                    if (key > tau || (eq_mode == 1 && key == tau)) keepm |= 1u << i;
                    if (eq_mode == 2 && key == tau) eqm |= 1u << i;
                };
                float vq[4] = {0.f, 0.f, 0.f, 0.f}, sq[4] = {0.f, 0.f, 0.f, 0.f}; // d and the state of this lane's quad
                if (r < n_groups) {
                    e0 = x0 + (uint32_t)sp[r] * 16u + (lane & 3u) * 4u;
                    if (e0 >= cv.first && e0 + 4 <= cv.len) {
                        // the state is requested together with d: a kept entry's update then waits for one
                        // memory round trip, not two
                        float gq[4];
                        if (st_vec) {
                            const float4 a = __ldg(reinterpret_cast<const float4*>(gr + e0));
                            const float4 b = *reinterpret_cast<const float4*>(st + e0);
                            gq[0] = a.x; gq[1] = a.y; gq[2] = a.z; gq[3] = a.w;
                            sq[0] = b.x; sq[1] = b.y; sq[2] = b.z; sq[3] = b.w;
                        } else {
#pragma unroll
                            for (int i = 0; i < 4; ++i) { gq[i] = __ldg(gr + e0 + i); sq[i] = st[e0 + i]; }
                        }
#pragma unroll
                        for (int i = 0; i < 4; ++i) { vq[i] = __fsub_rn(gq[i], sq[i]); classify(vq[i], i); }
                    } else {
#pragma unroll
                        for (int i = 0; i < 4; ++i)
                            if (e0 + i >= cv.first && e0 + i < cv.len) {
                                sq[i] = st[e0 + i];
                                vq[i] = __fsub_rn(__ldg(gr + e0 + i), sq[i]);
                                classify(vq[i], i);
                            }
                    }
                }
                if (eq_mode == 2) { // uniform over the warp
                    uint32_t incl = __popc(eqm);
#pragma unroll
                    for (int o = 1; o < 32; o <<= 1) {
                        const uint32_t y = __shfl_up_sync(0xffffffffu, incl, o);
                        if (lane >= (uint32_t)o) incl += y;
                    }
                    uint32_t eq_rank = eq_seen + incl - __popc(eqm);
                    for (uint32_t m = eqm; m; m &= m - 1) {
                        if (eq_rank < keep_eq) keepm |= m & (0u - m);
                        ++eq_rank;
                    }
                    eq_seen += __shfl_sync(0xffffffffu, incl, 31);
                }
                uint32_t incl = __popc(keepm);
#pragma unroll
                for (int o = 1; o < 32; o <<= 1) {
                    const uint32_t y = __shfl_up_sync(0xffffffffu, incl, o);
                    if (lane >= (uint32_t)o) incl += y;
                }
                uint32_t o = pos + incl - __popc(keepm);
                pos += __shfl_sync(0xffffffffu, incl, 31);
#pragma unroll
                for (int i = 0; i < 4; ++i)
                    if (((keepm >> i) & 1u) && KIMAD_CHECK(jb.base + o < cap, 3)) {
                        oi[o] = idx0 + e0 + i;
                        float sent;
                        if (BF16) {
                            const __nv_bfloat16 h = __float2bfloat16_rn(vq[i]);
                            ov16[o] = h;
                            sent = __bfloat162float(h);
                        } else {
                            ov32[o] = vq[i];
                            sent = vq[i];
                        }
                        st[e0 + i] = __fadd_rn(sq[i], sent);
                        ++o;
                    }
            }
            continue;
        }
        // a round is four rows of 128 elements, a lane takes four consecutive ones of each: bit 4 u + i of a lane's masks
        // stands for the element 128 u + 4 lane + i of the round
        constexpr int E = 16;
        // counts of a mask's rows, one byte each
        auto rows_of = [](uint32_t m) {
            m = (m & 0xfu) | (m & 0xf0u) << 4 | (m & 0xf00u) << 8 | (m & 0xf000u) << 12;
            m -= (m >> 1) & 0x05050505u;
            return (m & 0x03030303u) + ((m >> 2) & 0x03030303u);
        };
        // ranks (over the warp's round, in index order) of each row's first marked element in this lane, and the round's total
        auto ranks_of = [&](uint32_t m, uint32_t (&first)[4]) {
            const uint32_t own = rows_of(m);
            uint32_t incl = own; // (a row's count is at most 128)
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const uint32_t y = __shfl_up_sync(0xffffffffu, incl, o);
                if (lane >= (uint32_t)o) incl += y;
            }
            const uint32_t tot = __shfl_sync(0xffffffffu, incl, 31), excl = incl - own;
            uint32_t base = 0;
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                first[u] = base + ((excl >> (8 * u)) & 255u);
                base += (tot >> (8 * u)) & 255u;
            }
            return base;
        };
        for (uint32_t rb = x0; rb < min(cv.len, x0 + kSliceElems); rb += E * 32) {
            const uint32_t t0 = rb + 4 * lane;
            uint32_t keepm = 0, eqm = 0;
            const bool full = rb >= cv.first && rb + E * 32 <= cv.len; // round fully inside the chunk
            float v[E];
            float sv[DENSE ? E : 1]; // the dense instantiation keeps the estimator's values for its update
            if (full) {
                if (st_vec) {
#pragma unroll
                    for (int u = 0; u < 4; ++u) {
                        const float4 a = __ldg(reinterpret_cast<const float4*>(gr + t0 + 128 * u));
                        const float4 b = *reinterpret_cast<const float4*>(st + t0 + 128 * u);
                        v[4 * u] = __fsub_rn(a.x, b.x); v[4 * u + 1] = __fsub_rn(a.y, b.y);
                        v[4 * u + 2] = __fsub_rn(a.z, b.z); v[4 * u + 3] = __fsub_rn(a.w, b.w);
                        if (DENSE) { sv[4 * u] = b.x; sv[4 * u + 1] = b.y; sv[4 * u + 2] = b.z; sv[4 * u + 3] = b.w; }
                    }
                } else {
#pragma unroll
                    for (int i = 0; i < E; ++i) {
                        const uint32_t e = t0 + 128 * (i >> 2) + (i & 3);
                        const float b = st[e];
                        v[i] = __fsub_rn(__ldg(gr + e), b);
                        if (DENSE) sv[i] = b;
                    }
                }
#pragma unroll
                for (int i = 0; i < E; ++i) {
                    const uint32_t key = key_of(v[i]);
                    if (all || key > tau || (eq_mode == 1 && key == tau)) keepm |= 1u << i;
                    if (eq_mode == 2 && key == tau) eqm |= 1u << i;
                }
            } else {
#pragma unroll
                for (int i = 0; i < E; ++i) {
                    const uint32_t e = t0 + 128 * (i >> 2) + (i & 3);
                    const bool in = e >= cv.first && e < cv.len;
                    const uint32_t key = key_of(in ? __fsub_rn(__ldg(gr + e), st[e]) : 0.f);
                    if (in && (all || key > tau || (eq_mode == 1 && key == tau))) keepm |= 1u << i;
                    if (in && eq_mode == 2 && key == tau) eqm |= 1u << i;
                }
            }
            uint32_t ol[4]; // position of each row's first kept entry inside the round
            if (eq_mode == 2) { // uniform over the warp
                const uint32_t n_eq = ranks_of(eqm, ol);
                uint32_t m = eqm;
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    uint32_t eq_rank = eq_seen + ol[u];
                    for (uint32_t x = (m >> (4 * u)) & 15u; x; x &= x - 1) {
                        if (eq_rank < keep_eq) keepm |= (x & (0u - x)) << (4 * u);
                        ++eq_rank;
                    }
                }
                eq_seen += n_eq;
            }
            const uint32_t round_total = ranks_of(keepm, ol), round_pos = pos;
            pos += round_total;
            if (DENSE && full && round_total >= 48u) {
                // many kept entries: values come from the registers and the state is read before it is needed,
                // so that no store waits for a load of its own
                // the round's entries are laid out in shared memory first, so that the packed buffers are written
                // with consecutive lanes on consecutive entries
                uint32_t* sg_idx = s_stage[wid];
                uint32_t* sg_val = sg_idx + E * 32;
#pragma unroll
                for (int i = 0; i < E; ++i)
                    if ((keepm >> i) & 1u) {
                        const uint32_t at = ol[i >> 2]++;
                        sg_idx[at] = idx0 + t0 + 128 * (i >> 2) + (i & 3);
                        float sent;
                        if (BF16) {
                            const __nv_bfloat16 h = __float2bfloat16_rn(v[i]);
                            sg_val[at] = (uint32_t)__bfloat16_as_ushort(h);
                            sent = __bfloat162float(h);
                        } else {
                            sg_val[at] = __float_as_uint(v[i]);
                            sent = v[i];
                        }
                        sv[i] = __fadd_rn(sv[i], sent);
                    }
                __syncwarp();
                for (uint32_t q = lane; q < round_total; q += 32) {
                    if (!KIMAD_CHECK(jb.base + round_pos + q < cap, 3)) continue;
                    oi[round_pos + q] = sg_idx[q];
                    if (BF16) ov16[round_pos + q] = __ushort_as_bfloat16((unsigned short)sg_val[q]);
                    else ov32[round_pos + q] = __uint_as_float(sg_val[q]);
                }
                __syncwarp();
                if (st_vec) {
#pragma unroll
                    for (int u = 0; u < 4; ++u)
                        if ((keepm >> (4 * u)) & 15u)
                            *reinterpret_cast<float4*>(st + t0 + 128 * u) = make_float4(sv[4 * u], sv[4 * u + 1], sv[4 * u + 2], sv[4 * u + 3]);
                } else {
#pragma unroll
                    for (int i = 0; i < E; ++i)
                        if ((keepm >> i) & 1u) st[t0 + 128 * (i >> 2) + (i & 3)] = sv[i];
                }
                continue;
            }
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                uint32_t o = round_pos + ol[u];
                for (uint32_t m = (keepm >> (4 * u)) & 15u; m; m &= m - 1) {
                    const uint32_t e = t0 + 128 * u + (uint32_t)__ffs(m) - 1u;
                    if (!KIMAD_CHECK(jb.base + o < cap && e >= cv.first && e < cv.len, 3)) { ++o; continue; }
                    const float was = st[e];
                    const float val = __fsub_rn(__ldg(gr + e), was); // both loaded a moment ago: L1 hits
                    oi[o] = idx0 + e;
                    float sent;
                    if (BF16) {
                        const __nv_bfloat16 h = __float2bfloat16_rn(val);
                        ov16[o] = h;
                        sent = __bfloat162float(h);
                    } else {
                        ov32[o] = val;
                        sent = val;
                    }
                    st[e] = __fadd_rn(was, sent);
                    ++o;
                }
            }
        }
    }
}

} // namespace kimad
