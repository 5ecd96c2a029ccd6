// lc_measure.cu -- Eq. 1 (§3.2) on sm_103a: per layer sum|W - R|, sum|R| and
// the element count.
//
// Work decomposition: every segment is covered by 16-byte "virtual vectors"
// aligned to absolute addresses (lc_internal.cuh).  All vectors of all
// segments, layers ascending, form one linear work space that is cut into
// contiguous ranges: G equal ones, one per CTA, with G = resident CTAs on
// the device (one wave), and for the bulk kernel a pool of small ones after
// them.  A CTA streams its range(s) (the thread kernel: 128-bit
// non-allocating loads of W and R, several in flight per thread) and writes
// one fp64 partial per (range, layer) run.  The last CTA to finish (atomic
// ticket, no spinning) adds the partials of each layer in a fixed order, so
// the result is deterministic for a layout.
//
// Precision: per-thread fp32 accumulators take at most kUnroll * kFlush
// terms each before they are added (fixed tree) into per-thread fp64 sums;
// the relative error of a layer sum is below about 2e-6 (all terms >= 0).
#include "lc_bulk.cuh"
#include "lc_reduce.cuh"

#include <type_traits>

namespace lc {
namespace {

#ifndef LC_MEASURE_UNROLL
#define LC_MEASURE_UNROLL 4
#endif
#ifndef LC_MEASURE_FLUSH
#define LC_MEASURE_FLUSH 4
#endif
constexpr int kUnroll = LC_MEASURE_UNROLL;   // vectors of W (and of R) in flight per thread
constexpr int kFlush = LC_MEASURE_FLUSH;     // unrolled iterations between fp64 flushes
static_assert(kUnroll * kFlush <= 32, "fp32 partial sums are bounded to 32 terms");

// Adds one 16-byte vector pair into 8 fp32 lane accumulators.
template <int ESZ_LOG2>
__device__ __forceinline__ void accumulate(const uint4& w, const uint4& r, float (&ad)[8], float (&aa)[8]) {
    const uint32_t wv[4] = {w.x, w.y, w.z, w.w};
    const uint32_t rv[4] = {r.x, r.y, r.z, r.w};
    if constexpr (ESZ_LOG2 == 1) {
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const float w0 = bf16_lo(wv[j]), w1 = bf16_hi(wv[j]);
            const float r0 = bf16_lo(rv[j]), r1 = bf16_hi(rv[j]);
            ad[2 * j] += fabsf(w0 - r0);
            ad[2 * j + 1] += fabsf(w1 - r1);
            aa[2 * j] += fabsf(r0);
            aa[2 * j + 1] += fabsf(r1);
        }
    } else {
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const float w0 = __uint_as_float(wv[j]), r0 = __uint_as_float(rv[j]);
            ad[j] += fabsf(w0 - r0);
            aa[j] += fabsf(r0);
        }
    }
}

__device__ __forceinline__ float tree8(const float (&a)[8]) {
    return ((a[0] + a[1]) + (a[2] + a[3])) + ((a[4] + a[5]) + (a[6] + a[7]));
}

// Full, co-aligned vectors [k0, k1) of one segment.
template <int ESZ_LOG2, bool WRITE_R>
__device__ __forceinline__ void run_vectors(const SegDev& sd, int64_t k0, int64_t k1,
                                            double& dd, double& da) {
    constexpr int BS = kMeasureThreads;
    const uint8_t* wb = sd.w - (int64_t(sd.lead) << ESZ_LOG2);
    uint8_t* rb = sd.r - (int64_t(sd.lead) << ESZ_LOG2);
    int64_t k = k0 + threadIdx.x;
    while (k < k1) {
        float ad[8], aa[8];
#pragma unroll
        for (int j = 0; j < 8; ++j) { ad[j] = 0.f; aa[j] = 0.f; }
#pragma unroll 1
        for (int f = 0; f < kFlush && k < k1; ++f) {
            if (k + int64_t(kUnroll - 1) * BS < k1) {
                uint4 w[kUnroll], r[kUnroll];
#pragma unroll
                for (int u = 0; u < kUnroll; ++u) {
                    w[u] = ld_stream(wb + 16 * (k + int64_t(u) * BS));
                    r[u] = WRITE_R ? ld_coherent(rb + 16 * (k + int64_t(u) * BS))
                                   : ld_stream(rb + 16 * (k + int64_t(u) * BS));
                }
                if constexpr (WRITE_R) {
#pragma unroll
                    for (int u = 0; u < kUnroll; ++u) st_vec(rb + 16 * (k + int64_t(u) * BS), w[u]);
                }
#pragma unroll
                for (int u = 0; u < kUnroll; ++u) accumulate<ESZ_LOG2>(w[u], r[u], ad, aa);
                k += int64_t(kUnroll) * BS;
            } else {
                const uint4 w = ld_stream(wb + 16 * k);
                const uint4 r = WRITE_R ? ld_coherent(rb + 16 * k) : ld_stream(rb + 16 * k);
                if constexpr (WRITE_R) st_vec(rb + 16 * k, w);
                accumulate<ESZ_LOG2>(w, r, ad, aa);
                k += BS;
            }
        }
        dd += double(tree8(ad));
        da += double(tree8(aa));
    }
}

__device__ __forceinline__ float load_elem(const uint8_t* base, int esz_log2, int64_t e) {
    if (esz_log2 == 1) {
        const uint16_t x = *reinterpret_cast<const uint16_t*>(base + 2 * e);
        return __uint_as_float(uint32_t(x) << 16);
    }
    return *reinterpret_cast<const float*>(base + 4 * e);
}

// Vector k of a segment element by element (partial edge vectors, and every
// vector of a segment whose W and R are not co-aligned).
template <bool WRITE_R>
__device__ void scalar_vector(const SegDev& sd, int64_t k, double& dd, double& da) {
    const int ve = 16 >> sd.esz_log2;
    for (int j = 0; j < ve; ++j) {
        const int64_t e = k * ve - sd.lead + j;
        if (e < 0 || e >= sd.numel) continue;
        const float w = load_elem(sd.w, sd.esz_log2, e);
        const float r = load_elem(sd.r, sd.esz_log2, e);
        dd += double(fabsf(w - r));
        da += double(fabsf(r));
        if constexpr (WRITE_R) {
            if (sd.esz_log2 == 1)
                reinterpret_cast<uint16_t*>(sd.r)[e] = reinterpret_cast<const uint16_t*>(sd.w)[e];
            else
                reinterpret_cast<float*>(sd.r)[e] = reinterpret_cast<const float*>(sd.w)[e];
        }
    }
}

// The terms of element e of a segment.
template <bool WRITE_R>
__device__ __forceinline__ void edge_element(const SegDev& sd, int64_t e, float& xd, float& xa) {
    const float w = load_elem(sd.w, sd.esz_log2, e);
    const float r = load_elem(sd.r, sd.esz_log2, e);
    xd = fabsf(w - r);
    xa = fabsf(r);
    if constexpr (WRITE_R) {
        if (sd.esz_log2 == 1)
            reinterpret_cast<uint16_t*>(sd.r)[e] = reinterpret_cast<const uint16_t*>(sd.w)[e];
        else
            reinterpret_cast<float*>(sd.r)[e] = reinterpret_cast<const float*>(sd.w)[e];
    }
}

// Vectors [lo, hi) of one segment into the calling thread's fp64 sums.
template <bool WRITE_R>
__device__ void process_run(const SegDev& sd, int64_t lo, int64_t hi, double& dd, double& da) {
    const int ve = 16 >> sd.esz_log2;
    const bool head_partial = sd.lead > 0;
    const bool tail_partial = ((int64_t(sd.lead) + sd.numel) % ve) != 0;
    if (sd.rshift == 0) {
        const int64_t kf0 = head_partial ? 1 : 0;
        const int64_t kf1 = tail_partial ? sd.nvec - 1 : sd.nvec;
        const int64_t a = lo > kf0 ? lo : kf0;
        const int64_t b = hi < kf1 ? hi : kf1;
        if (a < b) {
            if (sd.esz_log2 == 1) run_vectors<1, WRITE_R>(sd, a, b, dd, da);
            else run_vectors<2, WRITE_R>(sd, a, b, dd, da);
        }
        if (threadIdx.x == 0) {
            if (head_partial && lo <= 0 && 0 < hi) scalar_vector<WRITE_R>(sd, 0, dd, da);
            const int64_t last = sd.nvec - 1;
            if (tail_partial && last >= lo && last < hi && !(head_partial && last == 0))
                scalar_vector<WRITE_R>(sd, last, dd, da);
        }
    } else {
        for (int64_t k = lo + threadIdx.x; k < hi; k += kMeasureThreads)
            scalar_vector<WRITE_R>(sd, k, dd, da);
    }
}

template <bool WRITE_R>
__global__ void __launch_bounds__(kMeasureThreads) measure_kernel(const MeasureParams p) {
    __shared__ double red_d[kMeasureThreads / 32];
    __shared__ double red_a[kMeasureThreads / 32];
    __shared__ unsigned int s_ticket;

    const int b = blockIdx.x;
    int64_t v0 = p.cta_vec_begin[b];
    const int64_t v1 = p.cta_vec_begin[b + 1];
    int s = p.cta_seg0[b];
    int slot = p.cta_slot0[b];
    double dd = 0.0, da = 0.0;
    while (v0 < v1 && s < p.nseg) {
        const SegDev sd = p.segs[s];
        const int64_t seg_end = sd.vec_begin + sd.nvec;
        const int64_t lo = v0 - sd.vec_begin;
        const int64_t hi = (v1 < seg_end ? v1 : seg_end) - sd.vec_begin;
        process_run<WRITE_R>(sd, lo, hi, dd, da);
        ++s;
        v0 = sd.vec_begin + hi;
        if (v0 < v1 && s < p.nseg && p.segs[s].layer == sd.layer) continue;
        block_sum(dd, da, red_d, red_a);
        if (threadIdx.x == 0) p.partials[slot] = make_double2(dd, da);
        ++slot;
        dd = 0.0;
        da = 0.0;
    }

    if (threadIdx.x == 0) {
        __threadfence();
        s_ticket = atomicAdd(p.ticket, 1u);
    }
    __syncthreads();
    if (s_ticket != gridDim.x - 1) return;
    __threadfence();
    finalize(p);
}

// ---------------------------------------------------------------------------
// Bulk-load measure.  The CTA walks its own range of the work space and
// then units of a pool of small ranges, each taken from a counter
// (next_pool_range), so that CTAs streaming faster take more of the work.
// Each range is the same walk over segment runs as above, turned into a
// sequence of jobs by one producer thread (warp 0): for the vectors of a run
// that lie inside W and whose R windows (below) lie inside R, chunks of up to
// kMChunk bytes of W and the same bytes of R loaded by cp.async.bulk into a
// ring of kMStages buffers (one "full" mbarrier per buffer, completed by the
// loads' byte count); with a run's first job come the few elements at the
// segment's edges, which the consumers read from global memory, one a thread;
// with its last the flush.
//
// W and R at different offsets from a 16-byte boundary (rshift != 0: weights
// that are views of a flat buffer, snapshots that are tensors of their own):
// a bulk load starts on 16 bytes, so R's chunk is loaded from the boundary
// below its first byte, one vector longer, and the consumers take R's vector
// v from the staged vectors v and v + 1, shifted by rshift bytes.  The shift
// is the same for the whole segment, so it is a template parameter of the
// loop.  A run like that used to be read element by element, two fp64 adds
// each: a decision over 412 M bf16 parameters in 146 such segments took
// 3110 us and takes 304 (0.53 and 5.4 TB/s; the same parameters co-aligned
// 255).  What bounds the shifted bf16 runs is the consumers' arithmetic: plain
// fp32 chains, as in the aligned runs, would be a sixth faster, but these sums
// had fp64's precision and plain chains lose it (6e-12 off the 64-bit sums of
// ordinary weights instead of 3e-12).  With chains that recovered an error only
// where the sum was the larger operand a decision took 271 us, and the sums
// were 4e-13 off the exact ones of ordinary weights (now 0) and 7e-10 with
// magnitudes over 30 binades (now 8e-17).  The loops are short, unrolled twice
// over one pair of chains: with four pairs 345 us, unrolled four times 406 (both
// with the usual pool of ranges, the present loop 332), seven times 590.
//
// Warps 1..7 consume every job in order: each thread adds its 16-byte vectors
// of the chunk into fp32 lanes (at most ceil(chunk vectors / 224) terms before
// they go to fp64), and at a flush each warp reduces its threads' fp64 sums in
// a fixed order into the run box; the last warp to arrive adds the warps' sums
// in warp order and writes the run's partial slot (run_flush), so no warp
// waits for another and no barrier spans warps.  Each warp hands a buffer back
// on its "empty" mbarrier (7 arrivals) before it turns to fp64.  Every wait is
// bounded; a wait that runs out raises the fault word.  A warp's lanes wait
// together and take the outcome together, so they never part ways.
// ---------------------------------------------------------------------------
#ifndef LC_MEASURE_BULK_STAGES
#define LC_MEASURE_BULK_STAGES 2
#endif
#ifndef LC_MEASURE_BULK_CHUNK
#define LC_MEASURE_BULK_CHUNK 24576
#endif
constexpr int kMStages = LC_MEASURE_BULK_STAGES;
constexpr uint32_t kMChunk = LC_MEASURE_BULK_CHUNK;      // bytes of W (and of R) per buffer
// In accumulate mode a buffer that goes back to R by bulk store is filled less:
// its next load waits for the store to have read it, and DRAM likes the loads
// and stores in shorter turns.  1.2 G bf16 parameters in 146 layers: 1075 us
// (6.9 TB/s; 1133 with full buffers of 24 KB, 1135 with 18, 1082 with 16, 1074
// with 13 or 14, 1179 with 8), fp32 2128 (2205), 138 M 150.5 (156), 6 M 28.6
// (29.0; 29.8 with 14 KB).
#ifndef LC_MEASURE_ACC_CHUNK
#define LC_MEASURE_ACC_CHUNK 15360
#endif
constexpr int kMConsumerWarps = kMeasureThreads / 32 - 1;   // warps 1.. consume (2.. in accumulate mode)
constexpr uint32_t kMStage = 2 * kMChunk + 128;          // R's part has room for the window's extra vector
constexpr size_t kMeasureBulkSmem = size_t(kMStages) * kMStage;
static_assert(kMChunk % 16 == 0 && LC_MEASURE_ACC_CHUNK % 16 == 0 && LC_MEASURE_ACC_CHUNK <= kMChunk && kMStages >= 2,
              "measure ring shape");

// One job of a run: a chunk of n staged vectors (n may be 0), the elements at
// the segment's edges (with the run's first job) and the flush (with its
// last), so that a run of one chunk costs one turn of the ring.  What the
// producer knows of the chunk travels with it: consumers and storer read no
// table in global memory for it.
struct MJob {
    int64_t ea, eb;     // elements [ea, ea + na) and [eb, eb + nb) of segment seg
    uint8_t* r_out;     // the granule of R that holds the chunk's first byte
    int32_t na, nb;
    int32_t n;          // staged vectors; -1: no more jobs
    int32_t esz_log2;
    int32_t rshift;
    int32_t seg;
    int32_t slot;       // flush the run into this partial slot (-1: not yet)
    int32_t pad;
};

// A warp hands a job's buffer back before it flushes, so the flush's shuffles
// and fp64 adds overlap the buffer's next load.  The producer is then up to
// kMStages jobs ahead of a warp's last flush, hence one box more than stages.
constexpr int kMBoxes = kMStages + 1;

struct MRing {
    uint64_t full[kMStages];
    uint64_t empty[kMStages];
    MJob jobs[kMStages];
    RunBox<kMBoxes, kMConsumerWarps> box;
};

template <bool WRITE_R>
__device__ void measure_produce(const MeasureParams& p, uint8_t* ring, MRing& r) {
    const uint32_t ring_s = smem_addr(ring);
    const uint32_t full_s = smem_addr(r.full), empty_s = smem_addr(r.empty);
    uint64_t k = 0;
    uint32_t extra = p.stall_first ? 16u : 0u;   // bytes announced beyond the first load's
    // the ring's next stage once its previous job has been handed back, or -1
    auto stage = [&]() -> int {
        const int st = int(k % kMStages);
        if (k >= uint64_t(kMStages) &&
            !mbar_wait_bounded(empty_s + 8 * st, uint32_t((k / kMStages - 1) & 1), kWaitNs))
            return -1;
        ++k;
        return st;
    };
    int st = 0;
    // the CTA's own range, then units of the pool until it is empty
    for (int rng = int(blockIdx.x); st >= 0 && rng >= 0; rng = st >= 0 ? next_pool_range(p) : -1) {
        int64_t v0 = p.cta_vec_begin[rng];
        const int64_t v1 = p.cta_vec_begin[rng + 1];
        int s = p.cta_seg0[rng];
        int slot = p.cta_slot0[rng];
        SegDev sd;
        if (v0 < v1 && s < p.nseg) sd = p.segs[s];
        while (st >= 0 && v0 < v1 && s < p.nseg) {
            const int64_t seg_end = sd.vec_begin + sd.nvec;
            const int64_t lo = v0 - sd.vec_begin;
            const int64_t hi = (v1 < seg_end ? v1 : seg_end) - sd.vec_begin;
            // the next segment is fetched while this one streams; the run ends with its layer
            SegDev next;
            const bool more = seg_end < v1 && s + 1 < p.nseg;
            if (more) next = p.segs[s + 1];
            const bool run_ends = !more || next.layer != sd.layer;
            // vectors [kf0, kf1) lie inside W with their R windows inside R
            const int64_t lead_b = (int64_t(sd.lead) << sd.esz_log2) + sd.rshift;
            const int64_t kf0 = (lead_b + 15) >> 4;
            int64_t kf1 = ((lead_b + (sd.numel << sd.esz_log2)) >> 4) - (sd.rshift ? 1 : 0);
            if (kf1 < kf0) kf1 = kf0;
            int64_t x = lo > kf0 ? lo : kf0;
            const int64_t e = hi < kf1 ? hi : kf1;
            // vectors [a, b) of the edges as elements of the segment
            const int ve_log2 = 4 - sd.esz_log2;
            auto first_elem = [&](int64_t a) { return a > 0 ? (a << ve_log2) - sd.lead : int64_t(0); };
            auto end_elem = [&](int64_t b) {
                const int64_t q = (b << ve_log2) - sd.lead;
                return q < sd.numel ? q : sd.numel;
            };
            const int64_t most = (WRITE_R && sd.rshift == 0 ? LC_MEASURE_ACC_CHUNK : kMChunk) / 16;
            bool edges = true;
            do {
                st = stage();
                if (st < 0) break;
                MJob& j = r.jobs[st];
                const int64_t n = x < e ? (e - x < most ? e - x : most) : 0;
                j.na = j.nb = 0;
                if (edges && lo < kf0) {
                    j.ea = first_elem(lo);
                    j.na = int32_t(end_elem(hi < kf0 ? hi : kf0) - j.ea);
                }
                if (edges && hi > kf1) {
                    j.eb = first_elem(lo > kf1 ? lo : kf1);
                    j.nb = int32_t(end_elem(hi) - j.eb);
                }
                edges = false;
                j.n = int32_t(n);
                j.esz_log2 = sd.esz_log2;
                j.rshift = sd.rshift;
                j.seg = s;
                j.slot = run_ends && x + n >= e ? slot : -1;
                if (n > 0) {
                    const uint32_t bytes = uint32_t(n) * 16u, rbytes = bytes + (sd.rshift ? 16u : 0u);
                    const int64_t at = 16 * x - (int64_t(sd.lead) << sd.esz_log2);
                    j.r_out = sd.r + at - sd.rshift;
                    mbar_expect_tx(full_s + 8 * st, bytes + rbytes + extra);
                    extra = 0;
                    bulk_g2s(ring_s + uint32_t(st) * kMStage, sd.w + at, bytes, full_s + 8 * st);
                    bulk_g2s(ring_s + uint32_t(st) * kMStage + kMChunk, j.r_out, rbytes, full_s + 8 * st);
                } else {
                    mbar_arrive(full_s + 8 * st);
                }
                x += n;
            } while (x < e);
            if (run_ends) ++slot;
            ++s;
            v0 = sd.vec_begin + hi;
            sd = next;
        }
    }
    if (st >= 0) st = stage();
    if (st >= 0) {
        r.jobs[st].n = -1;
        mbar_arrive(full_s + 8 * st);
    } else {
        raise_fault(p.fault);
        // the loads of the last kMStages jobs may still be landing in shared memory
        const uint64_t first = k > uint64_t(kMStages) ? k - kMStages : 0;
        for (uint64_t c = first; c < k; ++c)
            mbar_wait_bounded(full_s + 8 * int(c % kMStages), uint32_t((c / kMStages) & 1), kDrainNs);
    }
}

template <int ESZ_LOG2>
__device__ __forceinline__ void accumulate_comp(const uint4& w, const uint4& r, CompSum& cd, CompSum& ca) {
    const uint32_t wv[4] = {w.x, w.y, w.z, w.w};
    const uint32_t rv[4] = {r.x, r.y, r.z, r.w};
    auto pair = [](const uint32_t (&x)[4], int j) {
        return ESZ_LOG2 == 1 ? F2::of(bf16_lo(x[j]), bf16_hi(x[j]))
                             : F2::of(__uint_as_float(x[2 * j]), __uint_as_float(x[2 * j + 1]));
    };
#pragma unroll
    for (int j = 0; j < (8 >> ESZ_LOG2); ++j) {
        const F2 w2 = pair(wv, j), r2 = pair(rv, j);
        cd.add((w2 - r2).abs());
        ca.add(r2.abs());
    }
}

// The same vectors element by element in fp64, for a chain that is not
// finite: terms near the end of fp32's range, an infinity or a NaN.
template <int ESZ_LOG2>
__device__ __noinline__ double2 staged_elements(const uint8_t* W, const uint8_t* R, int n, int tid, int nt) {
    double dd = 0.0, da = 0.0;
    for (int v = tid; v < n; v += nt) {
        for (int i = 0; i < (16 >> ESZ_LOG2); ++i) {
            const int64_t e = int64_t(v) * (16 >> ESZ_LOG2) + i;
            const float w = load_elem(W, ESZ_LOG2, e), r = load_elem(R, ESZ_LOG2, e);
            dd += double(fabsf(w - r));
            da += double(fabsf(r));
        }
    }
    return make_double2(dd, da);
}

// n staged vectors of a run whose R bytes start SH bytes into their windows.
// In accumulate mode R's 16-byte vector v of the chunk (at r_out + 16 v)
// takes the end of W's vector v - 1 and the start of vector v; the chunk's
// first and last R vectors are only partly its own and are stored by
// elements.  No other chunk reads or writes those elements of R.
//
// The fp32 chains keep their rounding errors (CompSum): these runs used to be
// added element by element in fp64.  Against the exact sums of the same fp32
// terms, tensors of 100 to 1 M elements, both ways give bf16 sums without any
// error for normally distributed weights, and up to 4e-16 for magnitudes
// spread over 30 to 36 binades; fp32 sums 2e-16 and up to 6e-16 (4e-16 in fp64).
template <int ESZ_LOG2, int SH, bool WRITE_R, int NT>
__device__ __forceinline__ void shifted_run(const uint4* W, const uint4* R, int n, int tid, uint8_t* r_out,
                                            double& dd, double& da, float& td, float& ta) {
    CompSum cd, ca;
#pragma unroll 2
    for (int v = tid; v < n; v += NT) {
        const uint4 w = W[v];
        accumulate_comp<ESZ_LOG2>(w, window16<SH>(R[v], R[v + 1]), cd, ca);
        if constexpr (WRITE_R) {
            using T = typename std::conditional<ESZ_LOG2 == 1, uint16_t, uint32_t>::type;
            constexpr int kE = 16 >> ESZ_LOG2, kSplit = kE - (SH >> ESZ_LOG2);
            const uint32_t x[4] = {w.x, w.y, w.z, w.w};
            auto elem = [&](int i) {
                return T(ESZ_LOG2 == 1 ? x[i >> 1] >> (16 * (i & 1)) : x[ESZ_LOG2 == 1 ? 0 : i]);
            };
            if (v > 0) {
                st_vec(r_out + 16 * v, window16<16 - SH>(W[v - 1], w));
            } else {
                T* first = reinterpret_cast<T*>(r_out + SH);
#pragma unroll
                for (int i = 0; i < kSplit; ++i) first[i] = elem(i);
            }
            if (v == n - 1) {
                T* last = reinterpret_cast<T*>(r_out + 16 * n);
#pragma unroll
                for (int i = kSplit; i < kE; ++i) last[i - kSplit] = elem(i);
            }
        }
    }
    float ed, ea;
    cd.total(td, ed);
    ca.total(ta, ea);
    if (isfinite(td) && isfinite(ta)) {
        dd += double(ed);
        da += double(ea);
    } else {
        td = ta = 0.f;
        const double2 x = staged_elements<ESZ_LOG2>(reinterpret_cast<const uint8_t*>(W),
                                                    reinterpret_cast<const uint8_t*>(R) + SH, n, tid, NT);
        dd += x.x;
        da += x.y;
    }
}

template <bool WRITE_R, int NT>
__device__ __forceinline__ void shifted_chunk(int esz_log2, int rshift, const uint4* W, const uint4* R, int n,
                                              int tid, uint8_t* r_out, double& dd, double& da, float& td, float& ta) {
    if (esz_log2 == 1) {
        switch (rshift) {
            case 2: shifted_run<1, 2, WRITE_R, NT>(W, R, n, tid, r_out, dd, da, td, ta); break;
            case 4: shifted_run<1, 4, WRITE_R, NT>(W, R, n, tid, r_out, dd, da, td, ta); break;
            case 6: shifted_run<1, 6, WRITE_R, NT>(W, R, n, tid, r_out, dd, da, td, ta); break;
            case 8: shifted_run<1, 8, WRITE_R, NT>(W, R, n, tid, r_out, dd, da, td, ta); break;
            case 10: shifted_run<1, 10, WRITE_R, NT>(W, R, n, tid, r_out, dd, da, td, ta); break;
            case 12: shifted_run<1, 12, WRITE_R, NT>(W, R, n, tid, r_out, dd, da, td, ta); break;
            default: shifted_run<1, 14, WRITE_R, NT>(W, R, n, tid, r_out, dd, da, td, ta); break;
        }
    } else {
        switch (rshift) {
            case 4: shifted_run<2, 4, WRITE_R, NT>(W, R, n, tid, r_out, dd, da, td, ta); break;
            case 8: shifted_run<2, 8, WRITE_R, NT>(W, R, n, tid, r_out, dd, da, td, ta); break;
            default: shifted_run<2, 12, WRITE_R, NT>(W, R, n, tid, r_out, dd, da, td, ta); break;
        }
    }
}

// Consumers: warps 1.. (warps 2.. in accumulate mode, where warp 1 writes R).
template <bool WRITE_R>
__device__ void measure_consume(const MeasureParams& p, const uint8_t* ring, MRing& r) {
    constexpr int kFirstWarp = WRITE_R ? 2 : 1;
    constexpr int kThreads = 32 * (kMeasureThreads / 32 - kFirstWarp);
    const uint32_t full_s = smem_addr(r.full), empty_s = smem_addr(r.empty);
    const int tid = int(threadIdx.x) - 32 * kFirstWarp;
    const int warp = tid >> 5, lane = tid & 31;
    double dd = 0.0, da = 0.0;
    int box = 0;                // of the next flush, the same in every warp
    for (uint64_t k = 0;; ++k) {
        const int st = int(k % kMStages);
        const uint32_t parity = uint32_t((k / kMStages) & 1);
        if (!mbar_wait_warp(full_s + 8 * st, parity)) {
            if (lane == 0) raise_fault(p.fault);
            break;
        }
        const MJob j = r.jobs[st];
        if (j.n < 0) break;
        float xd = 0.f, xa = 0.f;   // this thread's element of the segment's edges
        if (tid < j.na + j.nb) edge_element<WRITE_R>(p.segs[j.seg], tid < j.na ? j.ea + tid : j.eb + (tid - j.na), xd, xa);
        float td = 0.f, ta = 0.f;     // and its chunk's sums
        if (j.n > 0) {
            const uint4* W = reinterpret_cast<const uint4*>(ring + size_t(st) * kMStage);
            const uint4* R = W + kMChunk / 16;
            if (j.rshift) {
                shifted_chunk<WRITE_R, kThreads>(j.esz_log2, j.rshift, W, R, j.n, tid, j.r_out, dd, da, td, ta);
            } else {
                float ad[8], aa[8];
#pragma unroll
                for (int q = 0; q < 8; ++q) { ad[q] = 0.f; aa[q] = 0.f; }
                if (j.esz_log2 == 1) {
#pragma unroll 4
                    for (int v = tid; v < j.n; v += kThreads) accumulate<1>(W[v], R[v], ad, aa);
                } else {
#pragma unroll 4
                    for (int v = tid; v < j.n; v += kThreads) accumulate<2>(W[v], R[v], ad, aa);
                }
                td = tree8(ad);
                ta = tree8(aa);
            }
        }
        mbar_arrive_warp(empty_s + 8 * st, lane);
        after_handback(td, ta);
        dd += double(td);
        da += double(ta);
        if (tid < j.na + j.nb) {
            dd += double(xd);
            da += double(xa);
        }
        if (j.slot >= 0) {   // flush: this warp's share of the run
            run_flush<kMConsumerWarps - (WRITE_R ? 1 : 0)>(r.box, box, warp, lane, dd, da, p.partials + j.slot);
            box = box + 1 < kMBoxes ? box + 1 : 0;
            dd = 0.0;
            da = 0.0;
        }
    }
}

// Accumulate mode (R <- W after the measure, Eq. 1 against W(t-1)): one
// thread stores every staged W chunk to R with a bulk store once the chunk
// (and with it the old R) has landed, and hands the buffer back when the
// store has read it.
__device__ void measure_store_r(const MeasureParams& p, const uint8_t* ring, MRing& r) {
    const uint32_t full_s = smem_addr(r.full), empty_s = smem_addr(r.empty);
    const uint32_t ring_s = smem_addr(ring);
    for (uint64_t k = 0;; ++k) {
        const int st = int(k % kMStages);
        if (!mbar_wait_bounded(full_s + 8 * st, uint32_t((k / kMStages) & 1), kWaitNs)) {
            raise_fault(p.fault);
            break;
        }
        const MJob& j = r.jobs[st];
        if (j.n < 0) break;
        if (j.n > 0 && j.rshift == 0) {
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            bulk_s2g(j.r_out, ring_s + uint32_t(st) * kMStage, uint32_t(j.n) * 16u);
            asm volatile("cp.async.bulk.commit_group;" ::: "memory");
            asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory");
        }
        mbar_arrive(empty_s + 8 * st);
    }
    asm volatile("cp.async.bulk.wait_group 0;" ::: "memory");
}

template <bool WRITE_R>
__global__ void __launch_bounds__(kMeasureThreads, 1) measure_bulk_kernel(const MeasureParams p) {
    extern __shared__ __align__(128) uint8_t ring[];
    __shared__ __align__(8) MRing r;
    __shared__ unsigned int s_ticket;
    __shared__ __align__(8) FinTables tables;
    if (threadIdx.x == 0) {
        for (int st = 0; st < kMStages; ++st) {
            mbar_init(smem_addr(&r.full[st]), 1);
            mbar_init(smem_addr(&r.empty[st]), kMConsumerWarps);
        }
        for (int b = 0; b < kMBoxes; ++b) r.box.count[b] = 0u;
        mbar_init_fence();
    }
    fin_prefetch(p, tables);   // before the wait: see static_tables
    dependents_may_start();
    dependency_wait();
    __syncthreads();
    if (threadIdx.x == 0) {
        measure_produce<WRITE_R>(p, ring, r);
    } else if (WRITE_R && threadIdx.x < 64) {
        if (threadIdx.x == 32) measure_store_r(p, ring, r);
    } else if (threadIdx.x >= 32) {
        measure_consume<WRITE_R>(p, ring, r);
    }
    fin_prefetch_wait();
    __syncthreads();
    if (threadIdx.x == 0) {
        __threadfence();
        s_ticket = atomicAdd(p.ticket, 1u);
    }
    __syncthreads();
    if (s_ticket != gridDim.x - 1) return;
    __threadfence();
    // the ring's loads have all landed (or the CTA gave up): it stages the combine
    finalize(p, reinterpret_cast<double2*>(ring), int32_t(kMeasureBulkSmem / sizeof(double2)), &tables);
    if (p.nan_on_fault && *reinterpret_cast<volatile const uint32_t*>(p.fault)) {
        __syncthreads();
        for (int i = threadIdx.x; i < 3 * p.nlayers; i += blockDim.x) p.sums[i] = __longlong_as_double(-1);
    }
}

}  // namespace

cudaError_t launch_measure(const MeasureParams& p, int grid, bool write_ref, cudaStream_t s) {
    cudaGetLastError();  // a stale non-sticky status must not be blamed on this launch
    if (write_ref) measure_kernel<true><<<grid, kMeasureThreads, 0, s>>>(p);
    else measure_kernel<false><<<grid, kMeasureThreads, 0, s>>>(p);
    return cudaGetLastError();
}

cudaError_t launch_measure_bulk(const MeasureParams& p, int grid, bool write_ref, cudaStream_t s) {
    if (!p.static_tables) {   // the kernel before this one writes the tables: nothing could start early
        if (write_ref) return cudaErrorInvalidValue;   // no caller has such tables and an R to write
        cudaGetLastError();
        measure_bulk_kernel<false><<<grid, kMeasureThreads, kMeasureBulkSmem, s>>>(p);
        return cudaGetLastError();
    }
    return launch_dependent(write_ref ? measure_bulk_kernel<true> : measure_bulk_kernel<false>, grid, kMeasureThreads,
                            kMeasureBulkSmem, s, p);
}

cudaError_t measure_bulk_prepare(int* blocks_per_sm) {
    cudaError_t e = cudaFuncSetAttribute(measure_bulk_kernel<false>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         int(kMeasureBulkSmem));
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(measure_bulk_kernel<true>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 int(kMeasureBulkSmem));
    if (e != cudaSuccess) return e;
    return cudaOccupancyMaxActiveBlocksPerMultiprocessor(blocks_per_sm, measure_bulk_kernel<false>,
                                                         kMeasureThreads, kMeasureBulkSmem);
}

cudaError_t measure_occupancy(int* blocks_per_sm) {
    return cudaOccupancyMaxActiveBlocksPerMultiprocessor(blocks_per_sm, measure_kernel<false>,
                                                         kMeasureThreads, 0);
}

}  // namespace lc
