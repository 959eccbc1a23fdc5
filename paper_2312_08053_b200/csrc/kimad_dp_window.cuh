// The knapsack's search over windows of the rows (see kimad_dp.cuh for the recursion itself): the same values, candidates and
// total as the recursion over whole rows, from the few cells of each row that the chosen path can pass through.
//
// Eq. 2 relaxed with a price per cell: for any price x, the errors of the layers 1..l on the way to cell b are at least
// M_l(x) - x b with M_l(x) = sum_{i<=l} min_j (e_ij + x u_ij), those of the layers behind at least (T(x) - M_l(x)) - x (C - b), and a
// candidate adds what its e + x u lies above the layer's smallest one.  A path whose binary32 total is U has errors of at most
// U (1 + (L + 16) 2^-24) in all, so neither the chosen path nor any other with the same total visits a cell, or takes a candidate,
// with which the bounds add up to more: over the other cells and candidates the recursion, its ties included, is the same.
//
//   1. The price at which the relaxed choice fills the axis: rounds of 8 to 24 prices at a time.
//   2. Smallest priced errors summed up layer by layer (binary64) at eight prices around it, and the cells that the relaxed choice
//      takes: two neighbouring prices, weighted so that the axis is filled.
//   3. The recursion in windows of 64 cells around that line (128 where the records of all layers are not staged at once, 256 where the
//      two prices are far apart in cells), over the candidates that cost little at this price, one warp per 64 cells: a total U, nearly
//      always the smallest one already.
//   4. Do the bounds at U rule out every cell outside the windows and every candidate left out?  Nearly always; else the
//      recursion once more in windows around the cells they leave open (64, 128 or 256), with the candidates they leave.  More than
//      256 cells: whole rows.
//   5. The way back along one byte per cell of the window (the cell it came from), a piece of the layers per warp.
//
// Bound by chains of latencies: about 130 cycles per four candidates of a layer in the recursion (row to shared memory, cells back, sums,
// minimum), a few thousand for each of the steps around it, whose instructions are fetched anew in every step.  GPT-2 small's 148 layers
// leave at most 35 cells of 852 open, 1995 blocks of it 33 of 1996, ResNet-50's 161 layers 127 of 835.  Against whole rows: 148 layers, 16
// candidates 68 -> 46 us, 161 layers, 7 candidates 70 -> 52, 201 layers 150 -> 56, 1995 blocks 1732 -> 465 to 480, and 790 where the
// bounds leave the first windows.  (A kernel of 512 threads of its own: inside the whole rows' kernel the search took 57 us on the 148 layers, and
// spilled where that has 1024 threads.)
#pragma once
#include "kimad_kernels.cuh"

namespace kimad {

constexpr uint32_t kWindowMost = 256;             // cells of a window at most (a byte names one of them)
constexpr uint32_t kWindowPiece = 32 * 1024;      // shared memory for the steps back where not all of them fit
// Windows are tried from so many layers on.  They take about 20 us and 0.2 us per layer (16 candidates), whole rows 10 us and 0.4 to 0.7 us (up
// to 1024 cells) or 0.85 us and more.  With fewer layers the cells of one candidate are many and windows seldom decide: ResNet-18's 62
// layers, 7 candidates, 939 cells leave too much open in every step, and whole rows take 31 us alone, 38 beside windows; 40 to 64
// layers on 2000 cells and more are decided on half of the curves tried, 2 to 5 times as fast.
KIMAD_HD uint32_t window_layers(uint32_t cells) { return cells <= 1024u ? 100u : 40u; }
constexpr uint32_t kWindowJump = 100;             // cells between two neighbouring prices' choices up to which 64 cells are tried first
constexpr uint32_t kPrices = 8, kSearchRounds = 20, kSearchPrices = 24;
// Where the records are not staged at once, a sample of the layers tells the price first: what it may be off (bits of a binary32: 3/32 to 3/16
// of the price), after which two rounds over all layers find it.  (Stopped at 3 % after one round, 12 us less, the first windows are too narrow
// or off more often.)
constexpr uint32_t kThinSpread = 3u << 19;
constexpr int kWindowThreads = 512;
constexpr uint32_t kPriceThreads = 64;            // threads that share a price's layers
constexpr uint32_t kBackWarps = 16;
constexpr uint32_t kWindowChunk = kDpMaxChunkLayers;

// What the warps of the recursion are told to do, in the order of the layers: errors to be added at every cell (layers with one
// candidate left that stays at its cell; filled up with +0, which changes nothing), then candidates, four per operation: distances
// in cells to those read (one window: +inf is read) and errors.  Cells that are only added to are exchanged at distance 0.
// Nothing in the recursion's loop branches (an inner loop over a layer's operations took 280 cycles per operation, this 130): an
// operation that is not its layer's first one exchanges the same row again.
struct WindowOp {
    uint32_t first;   // of its layer
    float own[2];
    uint32_t exchange; // which one of the chunk
    int dist[4];
    float err[4];
};

// budget_cells = (bytes D + c - 1) / c in binary64: everything is an integer below 2^50 (bytes < 2^35, D < 2^13, c below the sum of
// the layers' sizes), the quotient from the reciprocal is off by one at most and the remainder is exact.  D + 1 where it is more.
struct CellsOf {
    double cd, inv_c, c_1, most;
    uint32_t D;
    __device__ __forceinline__ CellsOf(uint64_t c, uint32_t D_) : cd((double)c), inv_c(1.0 / (double)c), c_1((double)c - 1.0), most((double)(D_ + 1u)), D(D_) {}
    __device__ __forceinline__ uint32_t operator()(double cost) const {
        const double num = fabs(cost) + c_1;
        const uint32_t u = (uint32_t)fmin(num * inv_c, most);
        const double rest = fma(-(double)u, cd, num);
        return min(rest < 0.0 ? u - 1u : (rest >= cd ? u + 1u : u), D + 1u);
    }
};

struct WindowScratch { // shared memory
    double run[2][kPrices], warp_sum[kPrices][kWindowChunk / kPriceThreads][2];
    float price[kPrices], all[kPrices];
    int cells[2][2], warp_cells[2][kWindowChunk / kPriceThreads][2]; // of the two middle prices: so far (two turns), of the price's two warps
    uint32_t mask[2 * kWindowChunk / 32], count[2 * kWindowChunk / 32]; // layers of a chunk that exchange their rows; operations per warp
    uint32_t listed[kWindowChunk]; // layers whose candidates take different numbers of cells
    uint32_t used[kSearchRounds][kSearchPrices];
    float rows[2 * 3 * kWindowMost];   // two rows with a window of +inf on either side; later the pieces of the way back
};
static_assert(sizeof(WindowScratch) % 16 == 0 && kBackWarps * kWindowMost <= sizeof(float) * 6 * kWindowMost, "layout of the scratch memory");
constexpr uint32_t kWindowTables = 40; // bytes per layer: sums at the eight prices, cells at the middle ones

// A layer's record, rw = 2 kr + 4 words: {cells above the smallest candidate's, as binary32 [kr] | errors [kr] | entries, the smallest
// candidate's cells}: of the usable candidates that take the same cells the smallest error; the last eight are filled up with entry 0.
// Shared memory (offsets): records at 0, those of all layers or [2][chunk_layers]; mem: scratch | operations of a chunk (before them
// what its records are made of) | word per layer | windows' ends [L + 1] | tables and steps back, where all records are there at once
// (else these are in the workspace, and pieces of the steps are staged here).
// Workspace (window_mem_bytes): [records | tables | steps back], nothing where all records are staged at once.
struct WindowArgs {
    uint32_t L, K, D, kr, rw;
    uint64_t c;            // budget in bytes
    const double* cost;    // [L][K] and the worker's errors
    const float* err;
    uint32_t chunk_layers;
    uint32_t mem, mem_bytes;
    unsigned char* g_mem;  // on a 16-byte boundary
    size_t g_bytes;
    const uint32_t* flags; // of the worker: kFlagChosen once the whole rows have the answer
    uint32_t p, x, j;      // offsets of: float [L] scratch; uint16_t [L] scratch; uint8_t [L] out: the chosen candidates
};
KIMAD_HD uint32_t window_op_bytes(uint32_t chunk_layers, uint32_t kr) { return chunk_layers * (kr / 4u) * (uint32_t)sizeof(WindowOp); }
KIMAD_HD size_t window_table_bytes(uint32_t L, uint32_t rw) { return ((size_t)L * (rw * 4u + kWindowTables) + 15u) & ~(size_t)15u; }
KIMAD_HD size_t window_mem_bytes(uint32_t L, uint32_t rw, uint32_t chunk_layers) {
    return chunk_layers >= L ? 0u : window_table_bytes(L, rw) + (size_t)L * kWindowMost;
}
// What a search came to: nothing, the answer in the first or the second windows, or nothing since it was no longer needed.
enum : uint32_t { kWindowNone = 0, kWindowFirst = 1, kWindowSecond = 2, kWindowStopped = 3 };
constexpr uint32_t kWindowPoll = 64; // operations of the recursion between two looks at the worker's flags

// Selections, written out: as conditional expressions they become branches, which cost the recursion's loop 130 cycles of 285 per operation.
__device__ __forceinline__ void take_less(float v, float& least, float x, float& with) { // the smaller value and what came with it
    asm("{.reg .pred p; setp.lt.f32 p, %2, %0; selp.f32 %0, %2, %0, p; selp.f32 %1, %3, %1, p;}" : "+f"(least), "+f"(with) : "f"(v), "f"(x));
}
__device__ __forceinline__ int pick_equal(float a, float b, int x, int y) { // a == b ? x : y
    int r;
    asm("{.reg .pred p; setp.eq.f32 p, %1, %2; selp.b32 %0, %3, %4, p;}" : "=r"(r) : "f"(a), "f"(b), "r"(x), "r"(y));
    return r;
}
__device__ __forceinline__ float pick_if(int c, float x, float y) { // c != 0 ? x : y
    float r;
    asm("{.reg .pred p; setp.ne.s32 p, %1, 0; selp.f32 %0, %2, %3, p;}" : "=f"(r) : "r"(c), "f"(x), "f"(y));
    return r;
}

__device__ __forceinline__ void store_if(int c, uint32_t at, uint32_t x) { // to shared memory
    asm volatile("{.reg .pred p; setp.ne.s32 p, %0, 0; @p st.shared.u32 [%1], %2;}" ::"r"(c), "r"(at), "r"(x) : "memory");
}

__device__ __forceinline__ void window_sync(uint32_t warps) { // the warps that carry the recursion (all of them get here)
    if (warps == 1u) __syncwarp();
    else asm volatile("bar.sync 1, %0;" ::"r"(32u * warps) : "memory");
}
__device__ __forceinline__ bool window_any(uint32_t warps, uint32_t x) { // x != 0 in any of these warps' threads
    if (warps == 1u) return __any_sync(0xffffffffu, x);
    uint32_t r;
    asm volatile("{.reg .pred p, q; setp.ne.u32 q, %1, 0; barrier.cta.red.or.pred p, 1, %2, q; selp.u32 %0, 1, 0, p;}" : "=r"(r) : "r"(x), "r"(32u * warps) : "memory");
    return r != 0u;
}

// kWindowFirst, kWindowSecond: the candidates and *total are the knapsack's.  Else nothing but scratch was written.  By the whole
// CTA (kWindowThreads).  ONE: the records of all layers are staged at once.  (Loops are not unrolled over candidates or layers: in a
// step, every instruction is fetched anew.)
template <bool ONE>
__device__ __forceinline__ uint32_t window_search(const WindowArgs& a, float* total) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ uint32_t s_top, s_bad, s_most, s_at, s_stop;
    __shared__ __align__(16) uint32_t s_seen[4];
    __shared__ unsigned long long s_least;
    __shared__ float s_bestv[kWindowMost / 64];
    __shared__ uint32_t s_bestb[kWindowMost / 64];
    const uint32_t t = threadIdx.x, T = blockDim.x, lane = t & 31u, wid = t >> 5;
    const uint32_t L = a.L, K = a.K, D = a.D, kr = a.kr, rw = a.rw, rec16 = rw / 4u, CL = a.chunk_layers;
    const float kInf = __int_as_float(0x7f800000);
    WindowScratch& sc = *reinterpret_cast<WindowScratch*>(smem_raw + a.mem);
    float* s_p = reinterpret_cast<float*>(smem_raw + a.p);
    uint16_t* s_x = reinterpret_cast<uint16_t*>(smem_raw + a.x);
    const uint32_t at_ops = a.mem + (uint32_t)sizeof(WindowScratch), at_meta = at_ops + window_op_bytes(CL, kr), at_lo = at_meta + 4u * L;
    const uint32_t at_tables = (at_lo + 2u * (L + 1u) + 15u) & ~15u, at_back = at_tables + (ONE ? kWindowTables * L : 0u);
    const uint32_t back_bytes = a.mem + a.mem_bytes - at_back;
    WindowOp* ops = reinterpret_cast<WindowOp*>(smem_raw + at_ops);
    uint32_t* meta = reinterpret_cast<uint32_t*>(smem_raw + at_meta);
    int16_t* s_lo = reinterpret_cast<int16_t*>(smem_raw + at_lo); // lowest cell of the window before layer 0, after layer 0, ...
    uint32_t* tab = reinterpret_cast<uint32_t*>(a.g_mem); // [L][rw]
    float* sums = reinterpret_cast<float*>(ONE ? smem_raw + at_tables : a.g_mem + (size_t)L * rw * 4u); // [L][kPrices]
    int2* cells = reinterpret_cast<int2*>(sums + (size_t)L * kPrices);                                  // [L]
    uint8_t* back = ONE ? smem_raw + at_back : a.g_mem + window_table_bytes(L, rw); // [exchanges][W]; in the workspace staged in units of 16 bytes
    const uint32_t n_chunks = ONE ? 1u : (L + CL - 1u) / CL;
    if (t == 0)
        (void)KIMAD_CHECK(at_back + (ONE ? L * kWindowMost : kWindowPiece) <= a.mem + a.mem_bytes && T >= kPrices * kPriceThreads && CL <= kWindowChunk &&
                          window_mem_bytes(L, rw, CL) <= a.g_bytes, 4);
    auto stage = [&](uint32_t buf, uint32_t first, uint32_t step, uint32_t n) { // records first, first + step, ...
        const uint32_t dst = smem_u32(smem_raw) + buf * CL * rw * 4u;
        for (uint32_t i = t; i < n * rec16; i += T) {
            const uint32_t r = i / rec16;
            cp_async_16(dst + 16u * i, reinterpret_cast<const uint4*>(tab + (size_t)(first + r * step) * rw) + (i - r * rec16));
        }
    };
    // f(records, first layer, layers) for the layers in order, chunk by chunk, by the whole CTA (up to the chunk in which it is stopped)
    auto for_chunks = [&](auto f) {
        if (ONE) {
            f(reinterpret_cast<const uint32_t*>(smem_raw), 0u, L);
            return;
        }
        stage(0, 0, 1, CL);
        for (uint32_t ch = 0; ch < n_chunks; ++ch) {
            cp_async_wait();
            __syncthreads(); // this chunk's records are there, nobody reads the other buffer any more
            if (ch + 1u < n_chunks) stage((ch + 1u) & 1u, (ch + 1u) * CL, 1, min(CL, L - (ch + 1u) * CL));
            f(reinterpret_cast<const uint32_t*>(smem_raw) + (ch & 1u) * CL * rw, ch * CL, min(CL, L - ch * CL));
            if (s_stop) break;
        }
        cp_async_wait(); // (the next chunk's, where it was stopped)
        __syncthreads();
    };
    // f(cells above the smallest candidate's, error) for a record's candidates, eight at a time (the last ones repeat candidate 0)
    auto for_candidates = [&](const uint32_t* rec, auto f) {
        const uint32_t nd = rec[2u * kr];
#pragma unroll 1
        for (uint32_t j = 0; j < nd; j += 8u) {
            const float4 u = *reinterpret_cast<const float4*>(rec + j), v = *reinterpret_cast<const float4*>(rec + j + 4u);
            const float4 e = *reinterpret_cast<const float4*>(rec + kr + j), g = *reinterpret_cast<const float4*>(rec + kr + j + 4u);
            f(u.x, e.x); f(u.y, e.y); f(u.z, e.z); f(u.w, e.w);
            f(v.x, g.x); f(v.y, g.y); f(v.z, g.z); f(v.w, g.w);
        }
    };

    // ---- 0. the records: cells and errors of a chunk's candidates, a thread each, then a thread per layer
    const CellsOf cells_of(a.c, D);
    auto error_of = [](double cost, float e) { return cost < 0.0 ? 0.f : e; }; // a layer sent densely (negative cost) loses nothing
    if (t == 0) { s_top = 0; s_bad = 0; s_most = 0; s_least = 0ull; s_stop = 0; }
    if (t < 4u) s_seen[t] = 0;
    const FlagsCopy copy(a.flags, s_seen);
    for (uint32_t i = t; i < kSearchRounds * kSearchPrices; i += T) (&sc.used[0][0])[i] = 0;
    float2* raw = reinterpret_cast<float2*>(ops); // [chunk_layers][K + 1]
    for (uint32_t ch = 0; ch < n_chunks; ++ch) {
        const uint32_t l0 = ch * CL, nl = min(CL, L - l0);
        uint32_t* recs = reinterpret_cast<uint32_t*>(smem_raw);
        for (uint32_t i0 = t; i0 < nl * K; i0 += 4u * T) { // loads of four requested together: they come from DRAM on most steps
            double cost[4];
            float e[4];
#pragma unroll
            for (uint32_t q = 0; q < 4u; ++q) {
                const uint32_t i = min(i0 + q * T, nl * K - 1u);
                cost[q] = a.cost[(size_t)l0 * K + i];
                e[q] = a.err[(size_t)l0 * K + i];
            }
#pragma unroll
            for (uint32_t q = 0; q < 4u; ++q) {
                const uint32_t i = i0 + q * T, l = i / K;
                if (i < nl * K) raw[i + l] = make_float2((float)cells_of(cost[q]), error_of(cost[q], e[q]));
            }
        }
        __syncthreads();
        uint32_t least = 0, top = 0, odd = 0;
        if (t < nl) {
            const float2* in = raw + t * (K + 1u);
            uint32_t* rec = recs + t * rw;
            const float u0 = in[0].x, most = (float)D;
            uint32_t at = 0; // the entry being made; stored when the next one is met
            const uint32_t to = smem_u32(rec);
            float du = 0.f, e = in[0].y;
            odd |= (uint32_t)(u0 > most) | (uint32_t)!(e >= 0.f && e < kInf); // (not even the smallest candidate fits)
#pragma unroll 4
            for (uint32_t j = 1; j < K; ++j) { // sizes ascend with j: the usable candidates come first
                const float2 y = in[j];
                const int ok = y.x <= most;
                odd |= (uint32_t)ok & ((uint32_t)!(y.y >= 0.f) | (uint32_t)!(y.y < kInf));
                const float d = fminf(y.x - u0, 8192.f);
                const int fresh = ok & (int)(d != du);
                store_if(fresh, to + 4u * at, __float_as_uint(du));
                store_if(fresh, to + 4u * (kr + at), __float_as_uint(e));
                at += fresh;
                du = pick_if(fresh, d, du);
                e = pick_if(fresh, y.y, pick_if(ok, fminf(e, y.y), e));
            }
            rec[at] = __float_as_uint(du);
            rec[kr + at] = __float_as_uint(e);
            const uint32_t nd = at + 1u;
            const uint32_t r0 = rec[0], r1 = rec[kr];
            for (uint32_t x = nd; x < ((nd + 7u) & ~7u); ++x) { rec[x] = r0; rec[kr + x] = r1; }
            rec[2u * kr] = nd;
            rec[2u * kr + 1u] = (uint32_t)u0;
            least = (uint32_t)u0;
            top = r1;
        }
        least = __reduce_add_sync(0xffffffffu, least);
        top = __reduce_max_sync(0xffffffffu, top); // (errors are not negative: ordered as their bits)
        if (lane == 0 && t < nl) { atomicAdd(&s_least, (unsigned long long)least); atomicMax(&s_top, top); }
        if (odd) s_bad = 1u;
        __syncthreads();
        if (!ONE) {
            for (uint32_t i = t; i < nl * rec16; i += T) reinterpret_cast<uint4*>(tab + (size_t)l0 * rw)[i] = reinterpret_cast<const uint4*>(recs)[i];
            __syncthreads();
        }
    }
    if (s_bad || s_top == 0u || s_least > D) return kWindowNone; // (errors of any sign, infinite ones, no room: whole rows)
    const uint32_t C = D - (uint32_t)s_least;              // cells of the row are 0 .. C
    __syncthreads();
    const uint32_t thin = ONE ? 1u : (L + CL - 1u) / CL, n_thin = (L + thin - 1u) / thin; // every thin-th layer
    if (!ONE) {
        stage(0, 0, thin, n_thin);
        cp_async_wait();
    }

    // ---- 1. the price: bits of a binary32 number, cut into equal pieces (about equal ratios).  Above the largest error nothing
    // but the smallest candidates is taken.  Records that are not staged at once: those of every thin-th layer first.
    const uint32_t highest = s_top + 1u, lowest = highest > (40u << 23) ? highest - (40u << 23) : 1u;
    uint32_t lo = lowest, hi = highest, round = 0;
    bool lo_sure = ONE, hi_sure = ONE; // the answer is known to lie on this side
    // of the staged records, those that matter
    if (t == 0) s_at = 0;
    __syncthreads();
    if (t < n_thin && reinterpret_cast<const uint32_t*>(smem_raw)[t * rw + 2u * kr] > 1u) sc.listed[atomicAdd(&s_at, 1u)] = t;
    __syncthreads();
    const uint32_t n_listed = s_at;
    // Rounds of prices, eight per thread; groups of whole warps take different prices (three at most: more warps take longer than a
    // round less would save).  The prices below the answer are those at which more than `most` cells are taken.
    auto rounds = [&](bool listed, uint32_t most, uint32_t until) {
        const uint32_t n = listed ? n_listed : CL, wide = max(32u, (n + 31u) & ~31u);
        const uint32_t groups = max(1u, min(kSearchPrices / 8u, T / wide)), n_try = 8u * groups;
        const uint32_t group = groups > 1u ? t / wide : 0u, slot = groups > 1u ? t - group * wide : t, slots = groups > 1u ? wide : T;
        while (hi - lo > until && round < kSearchRounds) {
            const uint32_t step = (hi - lo) / (n_try + 1u), from = lo;
            float x[8];
            int used[8];
#pragma unroll
            for (int i = 0; i < 8; ++i) { x[i] = __uint_as_float(from + step * (group * 8u + i + 1u)); used[i] = 0; }
            auto take = [&](const uint32_t* rec) {
                float best[8], taken[8];
#pragma unroll
                for (int i = 0; i < 8; ++i) { best[i] = kInf; taken[i] = 0.f; }
                for_candidates(rec, [&](float du, float e) {
#pragma unroll
                    for (int i = 0; i < 8; ++i) take_less(fmaf(x[i], du, e), best[i], du, taken[i]);
                });
#pragma unroll
                for (int i = 0; i < 8; ++i) used[i] += (int)taken[i];
            };
            if (listed) {
                if (group < groups && slot < n) take(reinterpret_cast<const uint32_t*>(smem_raw) + sc.listed[slot] * rw);
            } else {
                for_chunks([&](const uint32_t* recs, uint32_t, uint32_t nl) {
                    if (group < groups)
                        for (uint32_t l = slot; l < nl; l += slots) take(recs + l * rw);
                });
            }
            if (group < groups) { // (whole warps)
                uint32_t mine = 0;
#pragma unroll
                for (int i = 0; i < 8; ++i) {
                    const uint32_t y = __reduce_add_sync(0xffffffffu, (uint32_t)used[i]);
                    if (lane == (uint32_t)i) mine = y;
                }
                if (lane < 8u && mine) atomicAdd(&sc.used[round][group * 8u + lane], mine);
            }
            __syncthreads();
            const uint32_t over = __popc(__ballot_sync(0xffffffffu, lane < n_try && sc.used[round][lane] > most));
            if (over) lo = from + step * over;
            if (over < n_try) hi = from + step * (over + 1u);
            ++round;
            if (!ONE && listed) continue;
            lo_sure |= over != 0u;
            hi_sure |= over != n_try;
            if (!lo_sure) lo = lo > lowest + (1u << 23) ? lo - (1u << 23) : lowest; // the sample of layers misled: a factor of two further
            if (!hi_sure) hi = highest - hi > (1u << 23) ? hi + (1u << 23) : highest;
            lo_sure |= lo == lowest;
            hi_sure |= hi == highest;
        }
    };
    if (!ONE) {
        rounds(true, (uint32_t)((uint64_t)C * n_thin / L), 1u << 18);
        lo = lo > lowest + kThinSpread ? lo - kThinSpread : lowest;
        hi = min(hi + kThinSpread, highest);
        __syncthreads(); // the staged records make room
    }
    rounds(ONE, C, 1u << 15);
    if (hi >= 0x7f000000u) return kWindowNone; // (twice the price is finite)

    // ---- 2. sums of the smallest priced errors; 64 threads share a price, a layer each and up to four times (side by side:
    // consecutive layers per thread lie on the same banks)
    // (prices at factors of 0.7 .. 1.4 or 0.3 .. 3.3 around the two middle ones leave up to three times as many cells open)
    const uint32_t pi = t / kPriceThreads, pg = t % kPriceThreads;
    const float x_hi = __uint_as_float(hi);
    if (t < kPrices) {
        const float f = t < 4u ? (t < 2u ? (t == 0u ? 0.5f : 0.8f) : (t == 2u ? 0.95f : 1.f)) : (t < 6u ? (t == 4u ? 1.f : 1.05f) : (t == 6u ? 1.25f : 2.f));
        sc.price[t] = f * (t <= 3u ? __uint_as_float(lo) : x_hi);
        sc.run[0][t] = 0.0;
        if (t < 2u) sc.cells[0][t] = 0;
    }
    __syncthreads();
    {
        const float x = pi < kPrices ? sc.price[pi] : 0.f;
        const bool middle = pi == 3u || pi == 4u;
        uint32_t turn = 0;
        for_chunks([&](const uint32_t* recs, uint32_t l0, uint32_t nl) {
            constexpr uint32_t Q = kWindowChunk / kPriceThreads;
            double incl[Q];
            int ic[Q];
#pragma unroll
            for (uint32_t i = 0; i < Q; ++i) {
                const uint32_t l = i * kPriceThreads + pg;
                float m = 0.f, u = 0.f;
                if (pi < kPrices && l < nl) { // (a product and a sum in binary32 per layer)
                    m = kInf;
                    for_candidates(recs + l * rw, [&](float du, float e) { take_less(fmaf(x, du, e), m, du, u); });
                }
                incl[i] = (double)m;
                ic[i] = (int)u;
            }
#pragma unroll
            for (int o = 1; o < 32; o <<= 1)
#pragma unroll
                for (uint32_t i = 0; i < Q; ++i) {
                    const double y = __shfl_up_sync(0xffffffffu, incl[i], o);
                    const int yc = __shfl_up_sync(0xffffffffu, ic[i], o);
                    if (lane >= (uint32_t)o) { incl[i] += y; ic[i] += yc; }
                }
            if (lane == 31u && pi < kPrices) {
#pragma unroll
                for (uint32_t i = 0; i < Q; ++i) {
                    sc.warp_sum[pi][i][wid & 1u] = incl[i];
                    if (middle) sc.warp_cells[pi - 3u][i][wid & 1u] = ic[i];
                }
            }
            __syncthreads();
            if (pi < kPrices) {
                double base = sc.run[turn][pi];
                int cbase = middle ? sc.cells[turn][pi - 3u] : 0;
#pragma unroll
                for (uint32_t i = 0; i < Q; ++i) {
                    const size_t l = l0 + i * kPriceThreads + pg;
                    const double a0 = sc.warp_sum[pi][i][0], a1 = sc.warp_sum[pi][i][1];
                    int c0 = 0, c1 = 0;
                    if (middle) { c0 = sc.warp_cells[pi - 3u][i][0]; c1 = sc.warp_cells[pi - 3u][i][1]; }
                    if (i * kPriceThreads + pg < nl) {
                        sums[l * kPrices + pi] = (float)(base + (pg < 32u ? 0.0 : a0) + incl[i]);
                        const int c = cbase + (pg < 32u ? 0 : c0) + ic[i];
                        if (pi == 3u) cells[l].x = c;
                        if (pi == 4u) cells[l].y = c;
                    }
                    base += a0 + a1;
                    cbase += c0 + c1;
                }
                if (pg == 0u) { // of all layers so far
                    sc.run[turn ^ 1u][pi] = base;
                    sc.all[pi] = (float)base;
                    if (middle) sc.cells[turn ^ 1u][pi - 3u] = cbase;
                }
            }
            turn ^= 1u;
            __syncthreads();
        });
        if (t < 2u) s_bestb[t] = (uint32_t)sc.cells[turn][t];
    }
    __syncthreads();
    const int below_all = (int)s_bestb[0], above_all = (int)s_bestb[1]; // cells taken at the lower, the higher middle price
    const float part = below_all > above_all ? fminf(fmaxf((float)((int)C - above_all) / (float)(below_all - above_all), 0.f), 1.f) : 0.f;

    // ---- 3. the recursion inside windows of W cells, over the candidates that cost at most `cost` at the higher middle price.  A
    // path that takes the relaxed choice at that price costs x_hi (C - above_all); the best one is nearly always far below.
    // (Many layers wander further from the line: of 1995 blocks most steps need more than 64 cells, and starting with 64 the search is a
    // tenth faster where they are enough and a quarter slower where they are not.)
    uint32_t W = below_all - above_all <= (int)kWindowJump ? (ONE ? 64u : 128u) : kWindowMost;
    float most = 0.f;
    for (uint32_t i = 0; i < kPrices; ++i) most = fmaxf(most, sc.all[i] + sc.price[i] * (float)C);
    if (!(most < 1e37f)) return kWindowNone;
    const float binary32 = (float)(L + 16u) * 0x1p-24f; // relative error of a path's sum at most
    const float rounded = most * 0x1p-19f;              // of what is computed here from the sums: 32 roundings
    float cost = x_hi * (3.f + 0.4f * (float)max((int)C - above_all, 0)) + 2.f * binary32 * fmaxf(sc.all[4] - x_hi * (float)C, 0.f) + 4.f * rounded;
    float best = kInf;
    uint32_t best_b = 0xffffffffu, n_ex = 0;
    auto windows_on_line = [&]() {
        for (uint32_t l = t; l < L; l += T) {
            const int2 c = cells[l];
            s_lo[l + 1u] = (int16_t)(c.y + __float2int_rd(part * (float)(c.x - c.y)) - (int)(W / 2u));
        }
        if (t == 0) s_lo[0] = (int16_t)(-(int)(W / 2u));
    };
    auto recursion = [&]() -> bool { // false: stopped
        const uint32_t warps = W / 64u;
        for (uint32_t i = t; i < 6u * W; i += T) sc.rows[i] = kInf;
        float v0 = kInf, v1 = kInf;
        const uint32_t x0 = wid * 64u + lane, x1 = x0 + 32u; // the thread's cells of the window
        if (x0 == W / 2u) v0 = 0.f;
        if (x1 == W / 2u) v1 = 0.f;
        uint32_t buf = 0;
        n_ex = 0;
        __syncthreads(); // (the windows' lower ends are written)
        for_chunks([&](const uint32_t* recs, uint32_t l0, uint32_t nl) {
            // ---- the chunk's operations, two threads per layer (the first and the second half of its candidates)
            const uint32_t i = t >> 1, half = t & 1u, l = l0 + i;
            const bool have = i < nl;
            const uint32_t* rec = recs + min(i, nl - 1u) * rw;
            const uint32_t nd = rec[2u * kr], mid = ((nd + 7u) >> 3) << 2, j0 = half ? mid : 0u, j1 = half ? nd : min(mid, nd);
            // f(cells above the smallest candidate's, error); past the end of the list the errors are infinite
            auto my_candidates = [&](auto f) {
#pragma unroll 1
                for (uint32_t j = j0; j < j1; j += 4u) {
                    const float4 u = *reinterpret_cast<const float4*>(rec + j);
                    const float4 e = *reinterpret_cast<const float4*>(rec + kr + j);
                    f(u.x, e.x);
                    f(u.y, pick_if(j + 1u < j1, e.y, kInf));
                    f(u.z, pick_if(j + 2u < j1, e.z, kInf));
                    f(u.w, pick_if(j + 3u < j1, e.w, kInf));
                }
            };
            const int move = (int)s_lo[min(l, L - 1u) + 1u] - (int)s_lo[min(l, L - 1u)];
            float least = kInf;
            my_candidates([&](float du, float e) { least = fminf(least, fmaf(x_hi, du, e)); });
            least = fminf(least, __shfl_xor_sync(0xffffffffu, least, 1));
            const float dearest = least + cost;
            const float d_min = (float)(move - (int)W), d_max = (float)(move + (int)W);
            auto leads = [&](float du, float e) { // from a cell of the window into the next one, and not too dear
                return (int)(du > d_min) & (int)(du < d_max) & (int)(fmaf(x_hi, du, e) <= dearest);
            };
            uint32_t n_half = 0;
            float own = 0.f, du_last = 0.f; // (of the last one)
            my_candidates([&](float du, float e) {
                const int yes = leads(du, e);
                n_half += yes;
                du_last = pick_if(yes, du, du_last);
                own = pick_if(yes, e, own);
            });
            const bool stays = (int)du_last == move;
            const uint32_t n_other = __shfl_xor_sync(0xffffffffu, n_half, 1), n = n_half + n_other;
            const bool keeps = have && n == 1u && n_half == 1u && stays; // (in the thread that holds the candidate)
            if (keeps) s_p[l] = own;
            const uint32_t kept = __ballot_sync(0xffffffffu, keeps);
            const bool exchanges = have && ((kept >> (lane & ~1u)) & 3u) == 0u;
            const uint32_t ex_bits = __ballot_sync(0xffffffffu, exchanges); // two equal bits per layer
            if (lane == 0 && wid < 2u * kWindowChunk / 32u) sc.mask[wid] = ex_bits;
            __syncthreads();
            uint32_t run = 0; // layers that keep their cells since the last exchange
            if (have) {
                const uint32_t low = sc.mask[wid] & ((1u << (lane & ~1u)) - 1u);
                uint32_t last = low ? wid * 16u + (33u - __clz(low)) / 2u : 0u; // one past the last exchange
                for (uint32_t v = wid; v-- > 0u && last == 0u;) {
                    const uint32_t m = sc.mask[v];
                    if (m) last = v * 16u + (33u - __clz(m)) / 2u;
                }
                run = i - last;
            }
            // own errors go with the next exchange, two at most: a run's layers 1, 3, ... (and the chunk's last) are an exchange at distance 0
            const uint32_t n_ops = !have ? 0u : (exchanges ? max(1u, (n + 3u) / 4u) : ((run & 1u) || i == nl - 1u ? 1u : 0u));
            uint32_t incl = half ? 0u : n_ops | (n_ops ? 0x10000u : 0u); // operations | exchanges << 16
            const uint32_t mine = incl;
#pragma unroll
            for (int o = 2; o < 32; o <<= 1) {
                const uint32_t y = __shfl_up_sync(0xffffffffu, incl, o);
                if (lane >= (uint32_t)o) incl += y;
            }
            if (lane == 30u && wid < 2u * kWindowChunk / 32u) sc.count[wid] = incl;
            incl = __shfl_sync(0xffffffffu, incl - mine, lane & ~1u); // before the layer
            __syncthreads();
            uint32_t total = 0; // operations | exchanges << 16 of the chunk
            {
                uint32_t before = incl;
                for (uint32_t v = 0; v < 2u * kWindowChunk / 32u; ++v) {
                    if (v < wid) before += sc.count[v];
                    total += sc.count[v];
                }
                const uint32_t at = before & 0xffffu;
                if (have && half == 0u) {
                    (void)KIMAD_CHECK((at + n_ops) * sizeof(WindowOp) <= window_op_bytes(CL, kr), 4);
                    meta[l] = (n_ex + (before >> 16)) | (exchanges ? 0x80000000u : 0u);
                    if (n_ops) {
                        const uint32_t held = exchanges ? run & 1u : (run & 1u) + 1u, from = l + (exchanges ? 0u : 1u) - held;
                        const float o0 = held ? s_p[from] : 0.f, o1 = held > 1u ? s_p[from + 1u] : 0.f;
                        for (uint32_t b = 0; b < n_ops; ++b)
                            *reinterpret_cast<uint4*>(&ops[at + b]) = make_uint4(b == 0u ? 1u : 0u, __float_as_uint(o0), __float_as_uint(o1), before >> 16);
                    }
                    if (!exchanges && n_ops) ops[at].dist[0] = 0, ops[at].err[0] = 0.f;
                }
                if (have && n_ops) {
                    uint32_t c = half ? n_other : 0u;
                    if (exchanges)
                        my_candidates([&](float du, float e) {
                            const int yes = leads(du, e);
                            const uint32_t to = smem_u32(&ops[at + c / 4u].dist[c & 3u]);
                            store_if(yes, to, (uint32_t)((int)du - move));
                            store_if(yes, to + 16u, __float_as_uint(e)); // (err lies behind dist)
                            c += yes;
                        });
                    if (half) // the rest of the last operation
                        for (c = exchanges ? n : 1u; c < 4u * n_ops; ++c) { ops[at + c / 4u].dist[c & 3u] = (int)W; ops[at + c / 4u].err[c & 3u] = 0.f; }
                }
            }
            __syncthreads();
            // ---- the recursion over them
            auto carry = [&](auto one_warp) {
                uint8_t* to = back + (size_t)n_ex * W + x0;
                const uint4* op = reinterpret_cast<const uint4*>(ops);
                uint4 h = op[0];
                int4 d = *reinterpret_cast<const int4*>(op + 1);
                float4 e = *reinterpret_cast<const float4*>(op + 2);
                float* row = sc.rows + (buf ? 4u : 1u) * W + x0;
                int other = buf ? -3 * (int)W : 3 * (int)W; // from row to row
                float p0 = v0, p1 = v1; // the row before the layer
                int y0 = 0, y1 = 0;     // distances to the cells that the values come from
                bool stop = false;
#pragma unroll 1
                for (uint32_t left = total & 0xffffu; left && !stop;) {
                    const uint32_t until = left > kWindowPoll ? left - kWindowPoll : 0u;
                    if (t == 0) copy.ask();
#pragma unroll 1
                    for (; left > until; --left) {
                        const bool first = h.x != 0u;
                        const float own0 = __uint_as_float(h.y), own1 = __uint_as_float(h.z);
                        uint8_t* at = to + h.w * W;
                        p0 = first ? __fadd_rn(__fadd_rn(v0, own0), own1) : p0;
                        p1 = first ? __fadd_rn(__fadd_rn(v1, own0), own1) : p1;
                        v0 = first ? kInf : v0;
                        v1 = first ? kInf : v1;
                        row[0] = p0;
                        row[32] = p1;
                        if (decltype(one_warp)::value) __syncwarp();
                        else window_sync(warps);
                        const float *r0 = row - d.x, *r1 = row - d.y, *r2 = row - d.z, *r3 = row - d.w;
                        float a0 = r0[0], a1 = r1[0], a2 = r2[0], a3 = r3[0], b0 = r0[32], b1 = r1[32], b2 = r2[32], b3 = r3[32];
                        const int4 dc = d;
                        const float4 ec = e;
                        op += 3; // (the last one read lies behind the operations, in the same memory)
                        h = op[0];
                        d = *reinterpret_cast<const int4*>(op + 1);
                        e = *reinterpret_cast<const float4*>(op + 2);
                        a0 = __fadd_rn(a0, ec.x); a1 = __fadd_rn(a1, ec.y); a2 = __fadd_rn(a2, ec.z); a3 = __fadd_rn(a3, ec.w);
                        b0 = __fadd_rn(b0, ec.x); b1 = __fadd_rn(b1, ec.y); b2 = __fadd_rn(b2, ec.z); b3 = __fadd_rn(b3, ec.w);
                        const float m0 = min3(min3(a0, a1, a2), a3, v0), m1 = min3(min3(b0, b1, b2), b3, v1);
                        // the first candidate that attains the minimum (beside the chain of the values)
                        y0 = pick_equal(v0, m0, y0, pick_equal(a0, m0, dc.x, pick_equal(a1, m0, dc.y, pick_equal(a2, m0, dc.z, dc.w))));
                        y1 = pick_equal(v1, m1, y1, pick_equal(b0, m1, dc.x, pick_equal(b1, m1, dc.y, pick_equal(b2, m1, dc.z, dc.w))));
                        v0 = m0;
                        v1 = m1;
                        at[0] = (uint8_t)(x0 - (uint32_t)y0);
                        at[32] = (uint8_t)(x1 - (uint32_t)y1);
                        row += other;
                        other = -other;
                    }
                    stop = window_any(decltype(one_warp)::value ? 1u : warps, copy.chosen()); // (the same for all of these warps)
                }
                if (stop && t == 0) s_stop = 1u;
                buf ^= total & 1u;
            };
            if (wid < warps) {
                if (warps == 1u) carry(std::true_type{});
                else carry(std::false_type{});
            }
            n_ex += total >> 16;
            __syncthreads();
        });
        if (s_stop) return false;
        // lowest cell attaining the minimum
        if (wid < warps) {
            const int end = (int)s_lo[L];
            const int b0 = end + (int)x0, b1 = end + (int)x1;
            float bv = b0 <= (int)C ? v0 : kInf;
            int bb = b0;
            if (b1 <= (int)C && v1 < bv) { bv = v1; bb = b1; }
#pragma unroll
            for (int o = 16; o; o >>= 1) {
                const float ov = __shfl_xor_sync(0xffffffffu, bv, o);
                const int ob = __shfl_xor_sync(0xffffffffu, bb, o);
                if (ov < bv || (ov == bv && ob < bb)) { bv = ov; bb = ob; }
            }
            if (lane == 0) { s_bestv[wid] = bv; s_bestb[wid] = (uint32_t)bb; }
        }
        __syncthreads();
        best = s_bestv[0]; best_b = s_bestb[0];
        for (uint32_t i = 1; i < warps; ++i)
            if (s_bestv[i] < best) { best = s_bestv[i]; best_b = s_bestb[i]; } // (cells ascend with the warp)
        return true;
    };
    uint32_t found = kWindowFirst;
    windows_on_line();
    if (!recursion()) return kWindowStopped;
    if (!(best < kInf) && W < kWindowMost) {
        __syncthreads();
        W = kWindowMost;
        windows_on_line();
        if (!recursion()) return kWindowStopped;
    }
    if (!(best < kInf)) return kWindowNone;

    // ---- 4. the bounds at a total of `best`
    const float limit = best + best * binary32 + rounded;
    const float dear = limit - (sc.all[4] - x_hi * (float)C) + rounded; // what a candidate can cost on such a path
    {
        bool outside = !(dear <= cost);
        for (uint32_t l = t; l < L; l += T) {
            float m[kPrices];
            const float4 ma = *reinterpret_cast<const float4*>(sums + (size_t)l * kPrices), mb = *reinterpret_cast<const float4*>(sums + (size_t)l * kPrices + 4);
            m[0] = ma.x; m[1] = ma.y; m[2] = ma.z; m[3] = ma.w; m[4] = mb.x; m[5] = mb.y; m[6] = mb.z; m[7] = mb.w;
            // (convex in the cell, and some cell of the window is below the limit: the ends decide)
            auto bound = [&](int b) {
                float pre = -kInf, rest = -kInf;
#pragma unroll
                for (uint32_t i = 0; i < kPrices; ++i) {
                    pre = fmaxf(pre, m[i] - sc.price[i] * (float)b);
                    rest = fmaxf(rest, (sc.all[i] - m[i]) - sc.price[i] * (float)((int)C - b));
                }
                return pre + rest;
            };
            const int from = (int)s_lo[l + 1u] - 1, to = from + 1 + (int)W;
            outside |= (from >= 0 && !(bound(from) > limit)) || (to <= (int)C && !(bound(to) > limit));
        }
        if (outside) s_bad = 1u;
    }
    __syncthreads();
    if (s_bad) {
        uint32_t widest = 0;
        for (uint32_t l = t; l < L; l += T) {
            const float* m = sums + (size_t)l * kPrices;
            float b_lo = 0.f, b_hi = (float)C;
#pragma unroll 1
            for (uint32_t i = 0; i < kPrices; ++i) {
#pragma unroll 1
                for (uint32_t k = i + 1u; k < kPrices; ++k) {
                    const float xi = sc.price[i], xk = sc.price[k], width = xk - xi;
                    if (!(width > 0.01f * xk)) continue; // (the middle two)
                    // layers so far at price i, the rest at price k: grows with the cell; the other way round: falls
                    b_hi = fminf(b_hi, (limit - m[i] - (sc.all[k] - m[k]) + xk * (float)C) / width);
                    b_lo = fmaxf(b_lo, (m[k] + (sc.all[i] - m[i]) - xi * (float)C - limit) / width);
                }
            }
            const int c_lo = (int)ceilf(fminf(b_lo, (float)C + 1.f) - 0.1f), c_hi = (int)floorf(fmaxf(b_hi, -1.f) + 0.1f);
            widest = max(widest, c_hi >= c_lo ? (uint32_t)(c_hi - c_lo + 1) : 0x7fffffffu);
            meta[l] = (uint32_t)(uint16_t)c_lo | (uint32_t)(uint16_t)c_hi << 16;
        }
        widest = __reduce_max_sync(0xffffffffu, widest);
        if (lane == 0) atomicMax(&s_most, widest);
        __syncthreads();
        if (s_most > kWindowMost) return kWindowNone;
        W = s_most <= 64u ? 64u : (s_most <= 128u ? 128u : kWindowMost);
        for (uint32_t l = t; l < L; l += T) {
            const int c_lo = (int)(meta[l] & 0xffffu), c_hi = (int)(meta[l] >> 16);
            s_lo[l + 1u] = (int16_t)(c_lo - ((int)W - (c_hi - c_lo + 1)) / 2);
        }
        if (t == 0) s_lo[0] = (int16_t)(-(int)(W / 2u));
        cost = dear;
        __syncthreads();
        if (!recursion()) return kWindowStopped;
        if (!(best < kInf)) return kWindowNone;
        found = kWindowSecond;
    }

    // ---- 5. the way back over the exchanges.  Every warp takes a piece of them: first from all cells of its last window, then, once the
    // pieces behind it have told where the path enters, along the path.  s_x: the path's cell of the window before every exchange.
    uint8_t* s_map = reinterpret_cast<uint8_t*>(sc.rows); // [kBackWarps][W]
    const uint32_t end = (uint32_t)((int)best_b - (int)s_lo[L]);
    if (t == 0) s_at = end;
    const uint32_t most_rows = ONE ? L : back_bytes / W;
    for (uint32_t l1 = n_ex; l1;) {
        const uint32_t l0 = l1 > most_rows ? l1 - most_rows : 0u;
        if (!ONE) {
            __syncthreads(); // nobody reads the rows before
            for (uint32_t i = t; i < (l1 - l0) * W / 16u; i += T) cp_async_16(smem_u32(smem_raw + at_back) + 16u * i, back + (size_t)l0 * W + 16u * i);
            cp_async_wait();
        }
        __syncthreads();
        const uint8_t* steps = smem_raw + at_back; // of exchange l0, ...
        const uint32_t n = l1 - l0, per = (n + kBackWarps - 1u) / kBackWarps, from = min(wid * per, n), upto = min(from + per, n);
        if (wid < kBackWarps)
            for (uint32_t c = lane; c < W; c += 64u) {
                uint32_t x = c, y = c + 32u;
#pragma unroll 1
                for (uint32_t l = upto; l-- > from;) {
                    x = steps[l * W + x] & (W - 1u); // (cells without a value hold anything)
                    y = steps[l * W + y] & (W - 1u);
                }
                s_map[wid * W + c] = (uint8_t)x;
                s_map[wid * W + c + 32u] = (uint8_t)y;
            }
        __syncthreads();
        uint32_t x = s_at;
        if (wid < kBackWarps) {
            for (uint32_t v = kBackWarps - 1u; v > wid; --v) x = s_map[v * W + x];
            if (lane == 0) {
#pragma unroll 1
                for (uint32_t l = upto; l-- > from;) {
                    x = KIMAD_CHECK(x < W, 5) ? steps[l * W + x] : 0u;
                    s_x[l0 + l] = (uint16_t)x;
                }
            }
        }
        __syncthreads();
        if (t == 0) s_at = x;
        l1 = l0;
    }
    __syncthreads();
    // every layer's cells and the smallest error they cost; word: cells << 8 | candidate (none yet)
    for_chunks([&](const uint32_t* recs, uint32_t l0, uint32_t nl) {
        for (uint32_t i = t; i < nl; i += T) {
            const uint32_t l = l0 + i, k = meta[l] & 0x7fffffffu, k1 = k + (meta[l] >> 31);
            auto cell = [&](uint32_t k) { return (int)(k < n_ex ? s_x[k] : end); };
            const float du = (float)((int)s_lo[l + 1u] + cell(k1) - ((int)s_lo[l] + cell(k)));
            float e = kInf;
            for_candidates(recs + i * rw, [&](float u, float err) { e = fminf(e, u == du ? err : kInf); });
            (void)KIMAD_CHECK(e < kInf, 5);
            s_p[l] = e;
            meta[l] = (recs[i * rw + 2u * kr + 1u] + (uint32_t)du) << 8 | 0xffu;
        }
    });
    __syncthreads();
    if (t == 0) { // the values along the path, in the order of the layers
        float p = 0.f;
        uint32_t l = 0;
#pragma unroll 1
        for (; l + 8u <= L; l += 8u) {
            float e[8];
#pragma unroll
            for (int i = 0; i < 8; ++i) e[i] = s_p[l + i];
#pragma unroll
            for (int i = 0; i < 8; ++i) { s_p[l + i] = p; p = __fadd_rn(p, e[i]); }
        }
        for (; l < L; ++l) { const float e = s_p[l]; s_p[l] = p; p = __fadd_rn(p, e); }
        (void)KIMAD_CHECK(p == best, 5);
    }
    __syncthreads();
    // the first candidate with these cells that attains the value after the layer
    for (uint32_t i0 = t; i0 < L * K; i0 += 4u * T) {
        double cost[4];
        float e[4];
#pragma unroll
        for (uint32_t q = 0; q < 4u; ++q) {
            const uint32_t i = min(i0 + q * T, L * K - 1u);
            cost[q] = a.cost[i];
            e[q] = a.err[i];
        }
#pragma unroll
        for (uint32_t q = 0; q < 4u; ++q) {
            const uint32_t i = min(i0 + q * T, L * K - 1u), l = i / K, word = cells_of(cost[q]) << 8;
            const float after = l + 1u < L ? s_p[l + 1u] : best;
            if (((meta[l] ^ word) & ~0xffu) == 0u && __fadd_rn(s_p[l], error_of(cost[q], e[q])) == after) atomicMin(&meta[l], word | (i - l * K));
        }
    }
    __syncthreads();
    for (uint32_t l = t; l < L; l += T) {
        const uint32_t j = meta[l] & 0xffu;
        smem_raw[a.j + l] = (uint8_t)(KIMAD_CHECK(j < K, 5) ? j : 0u);
    }
    *total = best;
    __syncthreads();
    return found;
}

} // namespace kimad
