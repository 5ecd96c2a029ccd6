// lc_partition.cuh -- host side of the measure's work partition, shared by
// the contexts (lc_api.cu) and the allocation-free measure (lc_noalloc.cu).
#pragma once

#include "lc_internal.cuh"

#include <stddef.h>
#include <stdint.h>

// CTAs of a bulk-engine measure, in waves of one CTA per resident slot.
#ifndef LC_MEASURE_BULK_WAVES
#define LC_MEASURE_BULK_WAVES 1
#endif
// The bulk measure (and the fused step on its partition): a CTA walks an
// equal share of the first (100 - LC_MEASURE_POOL_PCT)% of the work space,
// then takes small units of the rest, LC_MEASURE_POOL_UNITS per CTA in all,
// from a counter.  CTAs that stream faster take more units, so the launch
// ends when the pool runs dry rather than when its slowest share is done.
// A unit is at least LC_MEASURE_POOL_MIN granules (64 KB of W: it costs a
// counter fetch, a table lookup and a flush); a pool too small to give every
// CTA a unit on average is not used.  With units of 512 KB (before a flush
// cost five fp64 adds a warp instead of ten) the fused step over 1.2 G
// parameters takes 5196 instead of 5162 us, the measure of 412 M 256 instead of
// 253, of 138 M fp32 parameters 179 instead of 177; 64 to 256 KB are alike.
#ifndef LC_MEASURE_POOL_PCT
#define LC_MEASURE_POOL_PCT 10
#endif
#ifndef LC_MEASURE_POOL_MIN
#define LC_MEASURE_POOL_MIN 128
#endif
#ifndef LC_MEASURE_POOL_UNITS
#define LC_MEASURE_POOL_UNITS 8
#endif
// Runs whose R is shifted cost the consumers more than aligned ones of the
// same bytes, so equal shares take unequal times and the pool is larger where
// they are a quarter of the vectors or more.  Decisions over 412 M parameters,
// nearly all shifted: bf16 304 us (332 with the usual pool), accumulate mode
// 413 (460), fp32 480 (481), accumulate mode 742 (811).  With fewer than 4
// smallest units a CTA it shares worse than the usual pool (46 M parameters 57
// instead of 55 us).
#ifndef LC_MEASURE_POOL_PCT_SHIFTED
#define LC_MEASURE_POOL_PCT_SHIFTED 30
#endif

namespace lc {

// What a segment costs a CTA beside its bytes, in vectors: a job of its own
// (and its edges), however small it is.  The CTAs' own ranges share the work
// space by that measure, so that a range of several small tensors has fewer
// bytes.  6 M parameters in 38 tensors: that took the decision from 26.0 us
// (equal vectors) to 23.9 (25.2 with a cost of 768, 23.8 with 3072; 22 now, with
// the select as it is), with every tensor a layer from 29.5 to 26; large models
// are the same.
#ifndef LC_MEASURE_SEG_COST
#define LC_MEASURE_SEG_COST 1536
#endif

// G equal shares of the work space in granules of LC_MEASURE_ALIGN_VECS and,
// with a pool, `units` ranges over what the shares leave.
struct PartitionShape {
    int64_t V = 0;        // vectors of the work space
    int64_t ngran = 0;    // granules
    int64_t pool = 0;     // granules in the pool
    int64_t G = 1;        // ranges that are a CTA's own
    int64_t units = 0;    // ranges in the pool
    int64_t ranges() const { return G + units; }
};

// `units_per_cta`: at most so many pool units a CTA on average (0: no pool).
// `shifted`: vectors of the segments whose R is shifted.
inline PartitionShape partition_shape(int64_t V, int64_t grid, int64_t units_per_cta, int64_t shifted) {
    PartitionShape s;
    s.V = V;
    s.ngran = (V + LC_MEASURE_ALIGN_VECS - 1) / LC_MEASURE_ALIGN_VECS;
    s.G = s.ngran < grid ? s.ngran : grid;
    if (s.G < 1) s.G = 1;
    if (units_per_cta > 0) {
        const int64_t more = s.ngran * LC_MEASURE_POOL_PCT_SHIFTED / 100, most = s.G * units_per_cta;
        const int64_t pool = 4 * shifted >= V && more >= s.G * 4 * LC_MEASURE_POOL_MIN ? more
                                                                              : s.ngran * LC_MEASURE_POOL_PCT / 100;
        if (pool >= s.G * LC_MEASURE_POOL_MIN) {
            s.units = pool / LC_MEASURE_POOL_MIN < most ? pool / LC_MEASURE_POOL_MIN : most;
            s.pool = pool;
        }
    }
    return s;
}

// Fills the ranges' tables (vec: ranges() + 1; seg0, slot0: ranges()) and the
// layers' slots (layer_slot: nlayers + 1) for segments in measure order;
// returns the number of slots, at most ranges() + nlayers.  One slot per
// (range, layer) run: ranges and layers both follow the work space, so a
// layer's slots are contiguous, and a range's are fixed whichever CTA walks it.
inline int32_t partition_fill(const PartitionShape& sh, const SegDev* sd, int32_t nseg, int32_t nlayers, int64_t* vec,
                              int32_t* seg0, int32_t* slot0, int32_t* layer_slot) {
    const int64_t gran = LC_MEASURE_ALIGN_VECS, own = sh.ngran - sh.pool, R = sh.ranges();
    auto at = [&](int64_t g) { return g * gran < sh.V ? g * gran : sh.V; };
    // the CTAs' own ranges: equal shares of vectors and costs
    const int64_t own_end = at(own);
    int64_t total = own_end;
    for (int32_t i = 0; i < nseg && sd[i].vec_begin < own_end; ++i) total += LC_MEASURE_SEG_COST;
    vec[0] = 0;
    int32_t i = 0;
    int64_t spent = LC_MEASURE_SEG_COST;                           // costs up to segment i's own
    for (int64_t b = 1; b < sh.G; ++b) {
        const int64_t t = total / sh.G * b + total % sh.G * b / sh.G;
        while (i + 1 < nseg && sd[i + 1].vec_begin < own_end && sd[i + 1].vec_begin + spent <= t) {
            ++i;
            spent += LC_MEASURE_SEG_COST;
        }
        int64_t v = t - spent < sd[i].vec_begin ? sd[i].vec_begin : t - spent;
        v = (v + gran / 2) / gran * gran;
        vec[b] = v < vec[b - 1] ? vec[b - 1] : v > own_end ? own_end : v;
    }
    vec[sh.G] = own_end;
    for (int64_t u = 1; u <= sh.units; ++u) vec[sh.G + u] = at(own + sh.pool * u / sh.units);
    for (int32_t l = 0; l < nlayers; ++l) layer_slot[l] = -1;
    int32_t slot = 0, s = 0;
    for (int64_t b = 0; b < R; ++b) {
        const int64_t v0 = vec[b], v1 = vec[b + 1];
        while (s < nseg && sd[s].vec_begin + sd[s].nvec <= v0) ++s;
        seg0[b] = s;
        slot0[b] = slot;
        for (int32_t t = s; v0 < v1 && t < nseg && sd[t].vec_begin < v1; ++t) {
            if (t > s && sd[t].layer == sd[t - 1].layer) continue;
            if (layer_slot[sd[t].layer] < 0) layer_slot[sd[t].layer] = slot;
            ++slot;
        }
    }
    layer_slot[nlayers] = slot;
    for (int32_t l = nlayers - 1; l >= 0; --l)
        if (layer_slot[l] < 0) layer_slot[l] = layer_slot[l + 1];
    return slot;
}

}  // namespace lc
