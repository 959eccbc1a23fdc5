// Plain structs and integer helpers shared by the host planner and the kernels of the CUDA library.
#pragma once
#include <math.h>
#include <stdint.h>

#include "kimad.h"

#if defined(__CUDACC__)
#define KIMAD_HD __host__ __device__ __forceinline__
#else
#define KIMAD_HD inline
#endif

// Checked build (-DKIMAD_CHECKED): indices into the workspace and the output buffers are tested before use; a failed
// test sets its bit in a status word that the host reads (kimad_debug_check) and the access is skipped -- nothing
// traps.  Bits: 0 sweep: bin outside the layer's histogram; 1 counting sweep: key outside its interval;
// 2 a work list (exact path, recount) appended beyond its capacity; 3 write sweep: packed position beyond the capacity or element
// outside its chunk; 4 knapsack: a record, row or exchange outside the memory it lies in; 5 knapsack: a cell outside its row;
// 6 selection: a listed entry outside its layer's chunks; 7 curve: the pieces of a refined bin do not add up to the bin.
// In the ordinary build KIMAD_CHECK(cond, bit) is `true`.
#if defined(KIMAD_CHECKED) && defined(__CUDACC__)
__device__ unsigned int g_kimad_check_word;
#define KIMAD_CHECK(cond, bit) ((cond) ? true : (atomicOr(&g_kimad_check_word, 1u << (bit)), false))
#else
#define KIMAD_CHECK(cond, bit) (true)
#endif

namespace kimad {

// A chunk is the part of one layer that falls inside one aligned window of the flat per-worker vector.  One CTA streams
// one chunk.  Contexts whose workers start at different distances from a 128-bit boundary (unpadded strides) have windows of
// kChunkElemsOdd elements: a chunk that starts up to three elements past a boundary then still has at most kChunkElems from
// the boundary on, and windows start on 128-byte lines of the code plane (with windows of 32752 the counting sweep took
// 12-20 % longer).
constexpr uint64_t kChunkElems = 32768;
constexpr uint64_t kChunkElemsOdd = 32640;
constexpr int kDpWorkersPerLaunch = 32;

struct Chunk {
    uint32_t layer;
    uint32_t _pad;
    uint64_t begin; // flat element index inside the worker's vector
    uint64_t end;
};

struct LayerDesc {
    uint64_t begin;
    uint64_t n;
    uint32_t first_chunk;
    uint32_t n_chunks;
};

// Radix-select state of one (worker, layer, candidate) between digit passes.
struct Cand {
    double err_low;  // sum of squares of everything known to lie below the current bin
    uint32_t rank;   // 1-based rank of the wanted key inside the current bin, counted from the top
    uint32_t gt;     // keys known to be larger than everything in the current bin
    uint32_t slot;   // which histogram slot of this (worker, layer) refines the current bin
    uint32_t prefix; // the bin: top 11 / 21 / 31 bits of the key after digit 1 / 2 / 3
};

struct SlotTab {
    uint32_t n;
    uint32_t prefix[KIMAD_MAX_RATIOS];
};

// Entries inside a layer's key interval that the select stage lists in one place; the curve stage marks an interval that may
// hold more (kSelMany, beside the code of its keys).
constexpr uint32_t kListCap = 4096;
constexpr uint32_t kSelMany = 256;

// What the select kernels need to know about one (worker, layer) after the DP.  The threshold lies in
// the key interval [tau, tau + 2^shift) and is the keep_eq-th largest key inside it; k_sel_offsets
// narrows that to the exact threshold (shift = 0) and to the number of ties kept.
struct Sel {
    uint32_t tau;     // lower key of the interval, then the exact threshold key
    uint32_t keep_eq; // rank inside the interval, then: entries equal to tau that are kept (lowest indices first)
    uint32_t k;       // 0: nothing to pack for this layer (the worker failed)
    uint32_t shift;   // log2 of the interval width (<= 10)
    uint32_t tau_low; // exact threshold minus the interval's lower key
    uint32_t code;    // the code (byte plane of the sweep) of the keys of the interval: entries with a larger code lie
                      // above the interval, entries with a smaller one below; | kSelMany
    uint64_t base;    // first output position of the layer in the worker's packed buffers
};

// The candidate table k_{l,j}: one table for all workers (wstride = 0: the ratio grid applied to the layer sizes), or
// one per worker (the ratio fitted to each worker's budget).
struct KTab {
    const uint64_t* p;
    uint64_t wstride;
    KIMAD_HD uint64_t at(uint32_t w, size_t i) const { return p[(size_t)w * wstride + i]; }
};

// Size in bytes of candidate k of a layer of n elements and the entries it keeps (Eq. 3's b_ij; the paper fixes no
// encoding).  cost model 0: k (4 + vb).  cost model 1: once the sparse size reaches the dense size vb n the layer is
// sent densely: every value, no indices; it then keeps all n entries and loses nothing.
KIMAD_HD uint64_t candidate_bytes(uint64_t n, uint64_t k, uint32_t bpe, uint32_t cost_model, bool* dense) {
    const uint64_t vb = bpe - 4;
    const bool d = cost_model == 1 && k * bpe >= vb * n;
    if (dense) *dense = d;
    return d ? vb * n : k * bpe;
}

// Budget cells a candidate of `bytes` occupies when c bytes are split into D cells (rounded up, so
// the byte constraint of Eq. 3 can never be exceeded).  c > 0.
KIMAD_HD uint64_t budget_cells(uint64_t bytes, uint32_t D, uint64_t c) { return (bytes * (uint64_t)D + c - 1) / c; }

// The numerator's share of that for a candidate, bytes * D, as the knapsack kernel reads it (binary64, exact: below 2^48);
// negative where the layer is sent densely.
inline double candidate_cost(uint64_t n, uint64_t k, uint32_t bpe, uint32_t cost_model, uint32_t D) {
    bool dense;
    const double x = (double)(candidate_bytes(n, k, bpe, cost_model, &dense) * (uint64_t)D);
    return dense ? -x : x;
}

// ---- The sample of a layer (k_sample) is read in units of consecutive elements, a warp each.  Half of the layer is enough: drawn without
// replacement its ranks are as certain as those of kSampleUnits units of a large layer.  Up to kWholeUnits the layer is taken whole
// (exact ranks, bands of one cell).
constexpr int kSampleUnit = 32;    // elements (128 bytes)
constexpr int kSampleUnits = 2047; // of a sample at most (65504 elements: the u16 cell counters cannot overflow)
constexpr int kWholeUnits = 1024;
constexpr uint32_t kSampleRound = 256; // units that a CTA has in flight together
KIMAD_HD uint32_t sample_units(uint32_t units) {
    const uint32_t half = units / 2u > (uint32_t)kWholeUnits ? units / 2u : (uint32_t)kWholeUnits;
    return units <= (uint32_t)kWholeUnits ? units : (half < (uint32_t)kSampleUnits ? half : (uint32_t)kSampleUnits);
}

// CTAs that read a layer's sample together: `layers` of them (over all workers), the largest with `most` elements; resident[i]: clusters of
// 2^i CTAs that the GPU holds at once (148, 74, 33 and 15 on a B200).  A second wave of clusters costs more than they save (16 layers of
// 1 M elements: 37.4 us with one CTA each, 29.4 with four, 37.6 with eight), and so does every CTA of a cluster beyond the rounds of the largest
// layer, for clearing its counters and meeting the others (stage in us with 1 / 2 / 4 / 8 CTAs, eight layers of 8 K elements:
// 18.2 / 20.3 / 21.4 / 21.1, 16 K: 19.7 / 23.3 / 23.5 / 23.6, 32 K: 24.6 / 25.7 / 23.3 / 24.5, 70 K: 27.4 / 25.6 / 23.8 / 25.6,
// 110 K: 31.8 / 27.7 / 25.2 / 25.5, 1 M: 36.0 / 31.5 / 27.9 / 25.7).
constexpr uint32_t kSampleClusterMost = 8;
KIMAD_HD uint32_t sample_cluster(uint64_t most, uint64_t layers, const uint32_t* resident) {
    const uint32_t units = sample_units((uint32_t)((most + kSampleUnit - 1) / kSampleUnit)), rounds = (units + kSampleRound - 1) / kSampleRound;
    if (rounds >= 7u && layers <= resident[3]) return 8u;
    if (rounds >= 4u && layers <= resident[2]) return 4u;
    if (rounds >= 5u && layers <= resident[1]) return 2u;
    return 1u;
}

// ---- Planning of the sweep's bins from the sample (k_sample).  A fine bin is 2^shift keys wide, between kMinShift and a cell.
constexpr uint32_t kMinShift = 5, kCellShift = 15;
constexpr float kMostBins = 1024.f; // ... and a cell is cut into at most that many

// Bins per cell that a candidate needs: at most ~2048 entries per bin (`dens`: entries per cell), and bins narrow enough that the
// uncertainty of the one holding the threshold (its entries times its spread of squares, 2^-7 of v^2 for a whole cell;
// `load`: entries per cell times v^2) stays below ~3e-6 of the error.  Finite whatever the estimates are, and never more than a cell
// can be cut into: an error that vanishes in binary32 beside `load` asks for all a cell can get.
KIMAD_HD float bins_needed(float dens, float load, float error) {
    const float cert = error > 0.f ? sqrtf(load / error * (0.0078125f / 3e-6f)) : kMostBins;
    const float bins = fmaxf(dens * (1.f / 2048.f), cert);
    return bins < kMostBins ? bins : kMostBins; // (also where it is not a number)
}

// What coarsen_groups() wants to know about the threads that run it together: one, or a warp (WarpLanes).
struct OneLane {
    uint32_t lane = 0, lanes = 1;
    KIMAD_HD uint32_t sum(uint32_t x) const { return x; }
    KIMAD_HD void sync() const {}
};

// Where the groups of bands together have more fine bins than there is room for (`fine` of them, `most` allowed), groups are
// coarsened one step at a time, always the one that stays closest to what its candidates need (bins per cell are powers of two, so many
// have more than they need); every group keeps at least one bin per cell.  Group g has the cells bot[g] .. top[g], bins of
// 2^shift[g] keys and needs need[g] bins per cell.  A group's steps double its need over bins per cell, so the steps taken are
// all those below some value of it, which is found by bisection over the bits of that value (31 rounds, whatever the needs are), and some
// of those at that value.  false: one bin per cell everywhere is still too much.
// (A thread alone, step by step: 60 us of the sample kernel for thirty groups over 150 octaves.)
template <typename Lanes>
KIMAD_HD bool coarsen_groups(const Lanes& t, const uint32_t* bot, const uint32_t* top, uint32_t* shift, const float* need, uint32_t n,
                             uint32_t fine, uint32_t most, uint32_t* left) {
    auto value = [&](uint32_t g) { // need over bins per cell, up to a common factor: ordered as its bits, a step adds one to the exponent
        union { float f; uint32_t u; } x;
        x.f = need[g] > 1e-18f ? (need[g] < 1e18f ? need[g] : 1e18f) : 1e-18f;
        return x.u + (shift[g] << 23);
    };
    auto steps = [&](uint32_t g, uint32_t below) { // of group g, those at values below `below`
        const uint32_t v = value(g), all = kCellShift - shift[g];
        const uint32_t k = v < below ? ((below - 1u - v) >> 23) + 1u : 0u;
        return k < all ? k : all;
    };
    auto freed = [&](uint32_t below) {
        uint32_t x = 0;
        for (uint32_t g = t.lane; g < n; g += t.lanes) {
            const uint32_t room = kCellShift - shift[g];
            x += (top[g] - bot[g] + 1u) * ((1u << room) - (1u << (room - steps(g, below))));
        }
        return t.sum(x);
    };
    if (fine > most) {
        uint32_t lo = 0, hi = 0x7fffffffu; // too little is freed below lo, enough below hi (if at all)
        const bool fits = fine - freed(hi) <= most;
        while (fits && hi - lo > 1u) {
            const uint32_t mid = (lo + hi) >> 1;
            if (fine - freed(mid) <= most) hi = mid;
            else lo = mid;
        }
        if (!fits) lo = hi;
        fine -= freed(lo);
        for (uint32_t g = t.lane; g < n; g += t.lanes) shift[g] += steps(g, lo);
        t.sync();
        if (!fits) return false;
        for (uint32_t g = 0; g < n && fine > most; ++g) // the steps at that very value, one by one
            if (shift[g] < kCellShift && value(g) == lo) {
                fine -= (top[g] - bot[g] + 1u) << (kCellShift - 1u - shift[g]);
                t.sync();
                if (t.lane == 0) shift[g] += 1u;
            }
        t.sync();
    }
    *left = most - fine;
    return true;
}

} // namespace kimad
