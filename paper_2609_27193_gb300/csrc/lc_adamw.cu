// lc_adamw.cu -- one AdamW step fused with the Eq. 1 sums of its update
// (§3.4.2: the drift is computed on the optimizer update path, so W(t-1) is
// read once, by the optimizer).  W is fp32 master weights here, so a
// 16-byte vector holds 4 parameters; the work partition, the partial slots
// and the fixed-order finalize are those of the measure scan.
#include "lc_bulk.cuh"
#include "lc_reduce.cuh"

#include <cuda_bf16.h>

namespace lc {
namespace {

#ifndef LC_ADAM_UNROLL
#define LC_ADAM_UNROLL 2
#endif
#ifndef LC_ADAM_MIN_BLOCKS
#define LC_ADAM_MIN_BLOCKS 2
#endif
constexpr int kAdamUnroll = LC_ADAM_UNROLL;      // vectors in flight per thread (5 arrays each)
constexpr int kAdamFlush = 16 / LC_ADAM_UNROLL;  // fp32 chains of 16 terms

__device__ __forceinline__ float adam_elem(float p, float& m, float& v, float g, const AdamConsts& c,
                                           float& p_out) {
    const float p_decayed = __fmul_rn(p, c.decay);
    const float m_new = __fadd_rn(__fmul_rn(c.b1, m), __fmul_rn(c.omb1, g));
    const float v_new = __fadd_rn(__fmul_rn(c.b2, v), __fmul_rn(c.omb2, __fmul_rn(g, g)));
    const float v_hat = __fmul_rn(v_new, c.rbc2);
    const float denom = __fadd_rn(__fsqrt_rn(v_hat), c.eps);
    const float step = __fdiv_rn(__fmul_rn(m_new, c.step_size), denom);
    p_out = __fsub_rn(p_decayed, step);
    m = m_new;
    v = v_new;
    return p_out;
}

__device__ __forceinline__ uint32_t bf16_pair(float lo, float hi) {
    const __nv_bfloat162 b = __floats2bfloat162_rn(lo, hi);
    return *reinterpret_cast<const uint32_t*>(&b);
}

__device__ __forceinline__ uint2 ld_u2(const void* p) {
    uint2 v;
    asm volatile("ld.global.nc.L1::no_allocate.v2.u32 {%0,%1}, [%2];" : "=r"(v.x), "=r"(v.y) : "l"(p));
    return v;
}

// Coherent load of data this kernel rewrites (volatile: kept in program
// order with the stores, which all come after the loads they follow).
__device__ __forceinline__ uint4 ld_rw(const void* p) {
    uint4 v;
    asm volatile("ld.global.L1::no_allocate.v4.u32 {%0,%1,%2,%3}, [%4];"
                 : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w)
                 : "l"(p));
    return v;
}

__device__ __forceinline__ void st_u2(void* p, uint2 v) {
    asm volatile("st.global.v2.u32 [%0], {%1,%2};" : : "l"(p), "r"(v.x), "r"(v.y) : "memory");
}

// kAdamUnroll aligned vectors (4 parameters each) of a fast segment: all
// loads first, then the arithmetic, then all stores.
template <bool GRAD_BF16>
__device__ __forceinline__ void adam_vectors(const SegDev& sd, const OptSegDev& od, int64_t k,
                                             int64_t kend, const AdamConsts& c, float (&ad)[4],
                                             float (&aa)[4]) {
    constexpr int BS = kMeasureThreads;
    constexpr int U = kAdamUnroll;
    uint8_t* wb = const_cast<uint8_t*>(sd.w) - 4 * int64_t(sd.lead);
    uint8_t* mb = reinterpret_cast<uint8_t*>(od.m) - 4 * int64_t(sd.lead);
    uint8_t* vb = reinterpret_cast<uint8_t*>(od.v) - 4 * int64_t(sd.lead);
    const uint8_t* gb = od.grad - (GRAD_BF16 ? 2 : 4) * int64_t(sd.lead);
    uint4 pw[U], mw[U], vw[U];
    uint4 gw[U];
#pragma unroll
    for (int u = 0; u < U; ++u) {
        const int64_t kk = k + int64_t(u) * BS;
        if (kk < kend) {
            pw[u] = ld_rw(wb + 16 * kk);
            mw[u] = ld_rw(mb + 16 * kk);
            vw[u] = ld_rw(vb + 16 * kk);
            if (GRAD_BF16) {
                const uint2 g2 = ld_u2(gb + 8 * kk);
                gw[u] = make_uint4(g2.x, g2.y, 0u, 0u);
            } else {
                gw[u] = ld_stream(gb + 16 * kk);
            }
        }
    }
#pragma unroll
    for (int u = 0; u < U; ++u) {
        const int64_t kk = k + int64_t(u) * BS;
        if (kk >= kend) continue;
        float g[4];
        if (GRAD_BF16) {
            g[0] = bf16_lo(gw[u].x); g[1] = bf16_hi(gw[u].x); g[2] = bf16_lo(gw[u].y); g[3] = bf16_hi(gw[u].y);
        } else {
            g[0] = __uint_as_float(gw[u].x); g[1] = __uint_as_float(gw[u].y);
            g[2] = __uint_as_float(gw[u].z); g[3] = __uint_as_float(gw[u].w);
        }
        float p[4] = {__uint_as_float(pw[u].x), __uint_as_float(pw[u].y), __uint_as_float(pw[u].z),
                      __uint_as_float(pw[u].w)};
        float m[4] = {__uint_as_float(mw[u].x), __uint_as_float(mw[u].y), __uint_as_float(mw[u].z),
                      __uint_as_float(mw[u].w)};
        float v[4] = {__uint_as_float(vw[u].x), __uint_as_float(vw[u].y), __uint_as_float(vw[u].z),
                      __uint_as_float(vw[u].w)};
        float pn[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            adam_elem(p[j], m[j], v[j], g[j], c, pn[j]);
            ad[j] += fabsf(pn[j] - p[j]);
            aa[j] += fabsf(p[j]);
        }
        st_vec(wb + 16 * kk, make_uint4(__float_as_uint(pn[0]), __float_as_uint(pn[1]),
                                        __float_as_uint(pn[2]), __float_as_uint(pn[3])));
        st_vec(mb + 16 * kk, make_uint4(__float_as_uint(m[0]), __float_as_uint(m[1]),
                                        __float_as_uint(m[2]), __float_as_uint(m[3])));
        st_vec(vb + 16 * kk, make_uint4(__float_as_uint(v[0]), __float_as_uint(v[1]),
                                        __float_as_uint(v[2]), __float_as_uint(v[3])));
        if (od.model)
            st_u2(od.model - 2 * int64_t(sd.lead) + 8 * kk,
                  make_uint2(bf16_pair(pn[0], pn[1]), bf16_pair(pn[2], pn[3])));
    }
}

// Element-wise path: partial edge vectors and segments that do not line up.
__device__ void adam_scalar_vector(const SegDev& sd, const OptSegDev& od, int64_t k,
                                   const AdamConsts& c, double& dd, double& da) {
    float* w = reinterpret_cast<float*>(const_cast<uint8_t*>(sd.w));
    for (int j = 0; j < 4; ++j) {
        const int64_t e = 4 * k - sd.lead + j;
        if (e < 0 || e >= sd.numel) continue;
        const float g = od.grad_bf16
                            ? __uint_as_float(uint32_t(reinterpret_cast<const uint16_t*>(od.grad)[e]) << 16)
                            : reinterpret_cast<const float*>(od.grad)[e];
        const float p = w[e];
        float m = od.m[e], v = od.v[e], pn;
        adam_elem(p, m, v, g, c, pn);
        w[e] = pn;
        od.m[e] = m;
        od.v[e] = v;
        if (od.model) reinterpret_cast<__nv_bfloat16*>(od.model)[e] = __float2bfloat16_rn(pn);
        dd += double(fabsf(pn - p));
        da += double(fabsf(p));
    }
}

__device__ void adam_run(const SegDev& sd, const OptSegDev& od, int64_t lo, int64_t hi,
                         const AdamConsts& c, double& dd, double& da) {
    constexpr int BS = kMeasureThreads;
    const bool head_partial = sd.lead > 0;
    const bool tail_partial = ((int64_t(sd.lead) + sd.numel) % 4) != 0;
    if (!od.fast) {
        for (int64_t k = lo + threadIdx.x; k < hi; k += BS) adam_scalar_vector(sd, od, k, c, dd, da);
        return;
    }
    const int64_t kf0 = head_partial ? 1 : 0;
    const int64_t kf1 = tail_partial ? sd.nvec - 1 : sd.nvec;
    const int64_t a = lo > kf0 ? lo : kf0;
    const int64_t b = hi < kf1 ? hi : kf1;
    int64_t k = a + threadIdx.x;
    while (k < b) {
        float ad[4] = {0.f, 0.f, 0.f, 0.f}, aa[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll 1
        for (int f = 0; f < kAdamFlush && k < b; ++f) {
            if (od.grad_bf16) adam_vectors<true>(sd, od, k, b, c, ad, aa);
            else adam_vectors<false>(sd, od, k, b, c, ad, aa);
            k += int64_t(kAdamUnroll) * BS;
        }
        dd += double((ad[0] + ad[1]) + (ad[2] + ad[3]));
        da += double((aa[0] + aa[1]) + (aa[2] + aa[3]));
    }
    if (threadIdx.x == 0) {
        if (head_partial && lo <= 0 && 0 < hi) adam_scalar_vector(sd, od, 0, c, dd, da);
        const int64_t last = sd.nvec - 1;
        if (tail_partial && last >= lo && last < hi && !(head_partial && last == 0))
            adam_scalar_vector(sd, od, last, c, dd, da);
    }
}

__global__ void __launch_bounds__(kMeasureThreads, LC_ADAM_MIN_BLOCKS) adamw_measure_kernel(const MeasureParams p,
                                                                        const OptSegDev* opt,
                                                                        const AdamConsts c) {
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
        const OptSegDev od = opt[s];
        const int64_t seg_end = sd.vec_begin + sd.nvec;
        const int64_t lo = v0 - sd.vec_begin;
        const int64_t hi = (v1 < seg_end ? v1 : seg_end) - sd.vec_begin;
        adam_run(sd, od, lo, hi, c, dd, da);
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
// Bulk-load form.  A per-thread step keeps only a few vectors of each array
// in flight (registers bound it).  Here one producer thread (warp 0) streams
// chunks of kAChunkVec vectors of w, m, v and the gradient into a ring of
// kAStages shared-memory buffers with cp.async.bulk, so the bytes in flight
// no longer cost registers; six consumer warps (2..7) take each chunk from
// shared memory, run the same element step, put the updated w, m and v back
// into the buffer, store the bf16 model copy themselves and add the Eq. 1
// sums of the update; warp 1 writes the buffer's w, m and v with bulk stores.
// A bulk copy starts on 16 bytes: an array that does not line up with w's
// vectors is loaded from the granule below its chunk (Window).  Vectors at a
// segment's edges whose windows would leave an array go element by element.
// Partition (with its pool of units), jobs, the run
// box that combines the warps' partial sums, and bounded waits are those of
// the bulk-load measure.
// ---------------------------------------------------------------------------
#ifndef LC_ADAM_BULK_STAGES
#define LC_ADAM_BULK_STAGES 2
#endif
// A step over 1.2 G parameters with its decision takes 5163 us with 512
// vectors, 5218 with 480 and 5146 with 544.  But the chunk is also the length
// of a thread's fp32 chains between two fp64 adds: with 544 the sums are 3.8e-10
// off their 64-bit values (root mean square over 16000 tensors, scaled to
// 100,000 elements), with 512 3.5e-10.
#ifndef LC_ADAM_BULK_VECS
#define LC_ADAM_BULK_VECS 512
#endif
constexpr int kAStages = LC_ADAM_BULK_STAGES;
constexpr int kAChunkVec = LC_ADAM_BULK_VECS;                 // vectors of 4 parameters per chunk
constexpr uint32_t kAPart = 16u * uint32_t(kAChunkVec) + 16u;   // an array's chunk, and a window's extra vector
constexpr uint32_t kAStage = 4u * kAPart;                     // w, m, v and gradient
constexpr size_t kAdamBulkSmem = size_t(kAStages) * kAStage;
constexpr int kAFirstConsumerWarp = 2;     // warp 0 loads, warp 1 stores
constexpr int kAConsumerWarps = kMeasureThreads / 32 - kAFirstConsumerWarp;
constexpr int kAConsumers = 32 * kAConsumerWarps;
static_assert(kAChunkVec % 2 == 0 && kAStages >= 2, "fused ring shape");

enum : int32_t { kAJobChunk = 0, kAJobScalar = 1, kAJobFlush = 2, kAJobEnd = 3 };
// Which arrays line up with w's vectors: m, v, gradient and model copy; m and v; not even those.
enum : int32_t { kALined = 0, kAMoments = 1, kALoose = 2 };

// What the producer knows of a job travels with it: the consumers and the
// storer read no table in global memory per chunk.
struct AJob {
    int64_t k0, k1;      // element-wise job: vectors [k0, k1) of the segment
    uint8_t *w, *m, *v;  // chunk: where its vectors go
    uint8_t* model;      // or null
    int32_t kind;
    int32_t seg;
    int32_t slot;
    int32_t n;           // chunk: vectors
    int32_t form;        // chunk: kALined, kAMoments or kALoose
    int32_t grad_bf16;
    int32_t grad_off;    // chunk: place of its first gradient in the first staged granule
    int32_t pad;
};

struct ARing {
    uint64_t full[kAStages];
    uint64_t computed[kAStages];   // consumers done with the buffer
    uint64_t empty[kAStages];
    AJob jobs[kAStages];
    RunBox<kAStages, kAConsumerWarps> box;
};

// Vectors [k0, k0 + n) of an array of `per_vec` bytes a vector whose first
// element belongs to vector 0 at place `lead`: the 16-byte granules that hold
// them, and how far into the first one they start.
struct Window {
    const uint8_t* from;
    uint32_t off, bytes;
    __device__ __forceinline__ Window(const uint8_t* base, int64_t lead, int per_vec, int64_t k0, uint32_t n) {
        const uint8_t* first = base - lead * (per_vec / 4) + per_vec * k0;
        off = uint32_t(uintptr_t(first) & 15);
        from = first - off;
        bytes = (off + uint32_t(per_vec) * n + 15u) & ~15u;
    }
};

// Narrows [kf0, kf1) to the vectors whose windows lie inside the array.
__device__ __forceinline__ void window_bounds(const void* array, const SegDev& sd, int per_vec, int64_t& kf0,
                                              int64_t& kf1) {
    const int64_t at = int64_t(uintptr_t(array) & 15);                  // addresses relative to the granule below
    const int64_t zero = at - int64_t(sd.lead) * (per_vec / 4);         // of vector 0
    const int64_t lo = ((at + 15) & ~int64_t(15)) - zero + per_vec - 1;
    const int64_t hi = ((at + sd.numel * (per_vec / 4)) & ~int64_t(15)) - zero;
    if (lo / per_vec > kf0) kf0 = lo / per_vec;
    if (hi / per_vec < kf1) kf1 = hi / per_vec;
}

__device__ void adam_produce(const MeasureParams& p, const OptSegDev* opt, uint8_t* ring, ARing& r) {
    const uint32_t ring_s = smem_addr(ring);
    const uint32_t full_s = smem_addr(r.full), empty_s = smem_addr(r.empty);
    uint64_t k = 0;
    bool stall = p.stall_first != 0;
    SegDev sd{};
    OptSegDev od{};
    auto post = [&](int32_t kind, int32_t s, int32_t slot, int64_t k0, int64_t k1) -> bool {
        const int st = int(k % kAStages);
        if (k >= uint64_t(kAStages) &&
            !mbar_wait_bounded(empty_s + 8 * st, uint32_t((k / kAStages - 1) & 1), kWaitNs))
            return false;
        AJob& j = r.jobs[st];
        j.kind = kind;
        j.seg = s;
        j.slot = slot;
        if (kind == kAJobChunk) {
            const uint32_t n = uint32_t(k1 - k0);
            const int64_t lead = sd.lead;
            const uint32_t buf = ring_s + uint32_t(st) * kAStage;
            const Window wm(reinterpret_cast<const uint8_t*>(od.m), lead, 16, k0, n);
            const Window wv(reinterpret_cast<const uint8_t*>(od.v), lead, 16, k0, n);
            const Window wg(od.grad, lead, od.grad_bf16 ? 8 : 16, k0, n);
            j.w = const_cast<uint8_t*>(sd.w) - 4 * lead + 16 * k0;
            j.m = const_cast<uint8_t*>(wm.from) + wm.off;
            j.v = const_cast<uint8_t*>(wv.from) + wv.off;
            j.model = od.model ? od.model - 2 * lead + 8 * k0 : nullptr;
            j.n = int32_t(n);
            j.form = od.fast ? kALined : (wm.off | wv.off) == 0 ? kAMoments : kALoose;
            j.grad_bf16 = od.grad_bf16;
            j.grad_off = int32_t(wg.off);
            mbar_expect_tx(full_s + 8 * st, 16 * n + wm.bytes + wv.bytes + wg.bytes + (stall ? 16u : 0u));
            stall = false;
            bulk_g2s(buf, j.w, 16 * n, full_s + 8 * st);
            bulk_g2s(buf + kAPart, wm.from, wm.bytes, full_s + 8 * st);
            bulk_g2s(buf + 2 * kAPart, wv.from, wv.bytes, full_s + 8 * st);
            bulk_g2s(buf + 3 * kAPart, wg.from, wg.bytes, full_s + 8 * st);
        } else {
            j.k0 = k0;
            j.k1 = k1;
            mbar_arrive(full_s + 8 * st);
        }
        ++k;
        return true;
    };
    bool ok = true;
    // the CTA's own range, then units of the pool until it is empty
    for (int rng = int(blockIdx.x); ok && rng >= 0; rng = ok ? next_pool_range(p) : -1) {
        int64_t v0 = p.cta_vec_begin[rng];
        const int64_t v1 = p.cta_vec_begin[rng + 1];
        int s = p.cta_seg0[rng];
        int slot = p.cta_slot0[rng];
        if (v0 < v1 && s < p.nseg) {
            sd = p.segs[s];
            od = opt[s];
        }
        while (ok && v0 < v1 && s < p.nseg) {
            const int64_t seg_end = sd.vec_begin + sd.nvec;
            const int64_t lo = v0 - sd.vec_begin;
            const int64_t hi = (v1 < seg_end ? v1 : seg_end) - sd.vec_begin;
            // the next segment is fetched while this one streams; the run ends with its layer
            SegDev next;
            OptSegDev onext;
            const bool more = seg_end < v1 && s + 1 < p.nseg;
            if (more) {
                next = p.segs[s + 1];
                onext = opt[s + 1];
            }
            const bool run_ends = !more || next.layer != sd.layer;
            // vectors [kf0, kf1) lie inside w with their windows inside m, v and the gradient
            int64_t kf0 = sd.lead > 0 ? 1 : 0;
            int64_t kf1 = (int64_t(sd.lead) + sd.numel) / 4;
            window_bounds(od.m, sd, 16, kf0, kf1);
            window_bounds(od.v, sd, 16, kf0, kf1);
            window_bounds(od.grad, sd, od.grad_bf16 ? 8 : 16, kf0, kf1);
            if (kf1 < kf0) kf1 = kf0;
            if (lo < kf0) ok = post(kAJobScalar, s, slot, lo, (hi < kf0 ? hi : kf0));
            const int64_t e = hi < kf1 ? hi : kf1;
            for (int64_t x = lo > kf0 ? lo : kf0; ok && x < e; x += kAChunkVec)
                ok = post(kAJobChunk, s, slot, x, (x + kAChunkVec < e ? x + kAChunkVec : e));
            if (ok && hi > kf1) ok = post(kAJobScalar, s, slot, (lo > kf1 ? lo : kf1), hi);
            if (ok && run_ends) ok = post(kAJobFlush, s, slot++, 0, 0);
            ++s;
            v0 = sd.vec_begin + hi;
            sd = next;
            od = onext;
        }
    }
    if (ok) ok = post(kAJobEnd, 0, 0, 0, 0);
    if (!ok) {
        raise_fault(p.fault);
        const uint64_t first = k > uint64_t(kAStages) ? k - kAStages : 0;
        for (uint64_t c = first; c < k; ++c)
            mbar_wait_bounded(full_s + 8 * int(c % kAStages), uint32_t((c / kAStages) & 1), kDrainNs);
    }
}

__device__ __forceinline__ uint4 words4(const uint32_t* w) { return make_uint4(w[0], w[1], w[2], w[3]); }

// The updated vector q of m or v (first staged word at w, which is `off`
// bytes into its granule): the words stay where they were read, for the
// storer; those outside the chunk's whole granules go to global memory here.
__device__ __forceinline__ void put_words(uint32_t* w, uint8_t* global, uint32_t off, int q, int n,
                                          const float (&x)[4]) {
#pragma unroll
    for (int e = 0; e < 4; ++e) {
        w[e] = __float_as_uint(x[e]);
        if (off && ((q == 0 && off + 4 * e < 16) || (q == n - 1 && off + 4 * e >= 16)))
            *reinterpret_cast<float*>(global + 16 * int64_t(q) + 4 * e) = x[e];
    }
}

// The model copy's four bf16 at any 2-byte boundary.
__device__ __forceinline__ void put_model(uint8_t* to, uint32_t lo, uint32_t hi) {
    if ((uintptr_t(to) & 7) == 0) {
        st_u2(to, make_uint2(lo, hi));
    } else if ((uintptr_t(to) & 3) == 0) {
        reinterpret_cast<uint32_t*>(to)[0] = lo;
        reinterpret_cast<uint32_t*>(to)[1] = hi;
    } else {
        *reinterpret_cast<uint16_t*>(to) = uint16_t(lo);
        *reinterpret_cast<uint32_t*>(to + 2) = (lo >> 16) | (hi << 16);
        *reinterpret_cast<uint16_t*>(to + 6) = uint16_t(hi >> 16);
    }
}

// One staged chunk.  In kALined, m, v, the gradient and the model copy line
// up with w's vectors.  Otherwise the gradient (and in kALoose m and v) starts
// where it likes: its staged words are read, and m's and v's written back, one
// by one (four-way bank conflicts), and the Eq. 1 chains keep their rounding
// errors (CompSum): such segments used to be added element by element in fp64,
// and the sums are within fp64's last place of those.  With bf16 gradients off
// the vectors of 412 M parameters in 146 segments, a step and its decision took
// 4880 us element by element and takes 1811 (floor 1696 at 6.8 TB/s).
template <int FORM>
__device__ __forceinline__ void adam_chunk(const AJob& j, uint8_t* buf, int tid, const AdamConsts& c, double& dd,
                                           double& da, float& td, float& ta) {
    constexpr bool LINED = FORM == kALined, MOMENTS = FORM != kALoose;
    const int n = j.n;
    uint4* W = reinterpret_cast<uint4*>(buf);
    const uint32_t om = MOMENTS ? 0u : uint32_t(uintptr_t(j.m) & 15), ov = MOMENTS ? 0u : uint32_t(uintptr_t(j.v) & 15);
    const uint32_t og = uint32_t(j.grad_off);
    uint8_t* Mb = buf + kAPart + om;
    uint8_t* Vb = buf + 2 * kAPart + ov;
    const uint8_t* G = buf + 3 * kAPart + og;
    float ad[4] = {0.f, 0.f, 0.f, 0.f}, aa[4] = {0.f, 0.f, 0.f, 0.f};
    CompSum cd, ca;
    for (int q = tid; q < n; q += kAConsumers) {
        const uint4 pw = W[q];
        const uint4 mw = MOMENTS ? reinterpret_cast<const uint4*>(Mb)[q]
                                 : words4(reinterpret_cast<const uint32_t*>(Mb) + 4 * q);
        const uint4 vw = MOMENTS ? reinterpret_cast<const uint4*>(Vb)[q]
                                 : words4(reinterpret_cast<const uint32_t*>(Vb) + 4 * q);
        float g[4];
        if (j.grad_bf16) {
            uint2 g2;
            if (LINED) {
                g2 = reinterpret_cast<const uint2*>(G)[q];
            } else {
                const uint32_t* gw = reinterpret_cast<const uint32_t*>(G - (og & 2)) + 2 * q;
                g2 = make_uint2(gw[0], gw[1]);
                if (og & 2)
                    g2 = make_uint2(__funnelshift_r(gw[0], gw[1], 16), __funnelshift_r(gw[1], gw[2], 16));
            }
            g[0] = bf16_lo(g2.x); g[1] = bf16_hi(g2.x); g[2] = bf16_lo(g2.y); g[3] = bf16_hi(g2.y);
        } else {
            const uint4 g4 = LINED ? reinterpret_cast<const uint4*>(G)[q]
                                   : words4(reinterpret_cast<const uint32_t*>(G) + 4 * q);
            g[0] = __uint_as_float(g4.x); g[1] = __uint_as_float(g4.y);
            g[2] = __uint_as_float(g4.z); g[3] = __uint_as_float(g4.w);
        }
        float pv[4] = {__uint_as_float(pw.x), __uint_as_float(pw.y), __uint_as_float(pw.z), __uint_as_float(pw.w)};
        float m[4] = {__uint_as_float(mw.x), __uint_as_float(mw.y), __uint_as_float(mw.z), __uint_as_float(mw.w)};
        float v[4] = {__uint_as_float(vw.x), __uint_as_float(vw.y), __uint_as_float(vw.z), __uint_as_float(vw.w)};
        float pn[4];
#pragma unroll
        for (int e = 0; e < 4; ++e) adam_elem(pv[e], m[e], v[e], g[e], c, pn[e]);
        if (LINED) {
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                ad[e] += fabsf(pn[e] - pv[e]);
                aa[e] += fabsf(pv[e]);
            }
        } else {
            float big = 0.f;                // a NaN is added like any number
#pragma unroll
            for (int e = 0; e < 4; ++e) big = fmaxf(big, fmaxf(fabsf(pn[e] - pv[e]), fabsf(pv[e])));
            const bool fine = big < 1e37f;
#pragma unroll
            for (int e = 0; e < 4; e += 2) {
                cd.add(F2::of(fine ? fabsf(pn[e] - pv[e]) : 0.f, fine ? fabsf(pn[e + 1] - pv[e + 1]) : 0.f));
                ca.add(F2::of(fine ? fabsf(pv[e]) : 0.f, fine ? fabsf(pv[e + 1]) : 0.f));
            }
            if (!fine) {                    // near the end of fp32's range, or infinite
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    dd += double(fabsf(pn[e] - pv[e]));
                    da += double(fabsf(pv[e]));
                }
            }
        }
        const uint4 pnw = make_uint4(__float_as_uint(pn[0]), __float_as_uint(pn[1]), __float_as_uint(pn[2]),
                                     __float_as_uint(pn[3]));
        W[q] = pnw;
        if (MOMENTS) {
            reinterpret_cast<uint4*>(Mb)[q] = make_uint4(__float_as_uint(m[0]), __float_as_uint(m[1]),
                                                         __float_as_uint(m[2]), __float_as_uint(m[3]));
            reinterpret_cast<uint4*>(Vb)[q] = make_uint4(__float_as_uint(v[0]), __float_as_uint(v[1]),
                                                         __float_as_uint(v[2]), __float_as_uint(v[3]));
        } else {
            put_words(reinterpret_cast<uint32_t*>(Mb) + 4 * q, j.m, om, q, n, m);
            put_words(reinterpret_cast<uint32_t*>(Vb) + 4 * q, j.v, ov, q, n, v);
        }
        if (j.model) {
            const uint32_t lo = bf16_pair(pn[0], pn[1]), hi = bf16_pair(pn[2], pn[3]);
            if (LINED) st_u2(j.model + 8 * q, make_uint2(lo, hi));
            else put_model(j.model + 8 * q, lo, hi);
        }
    }
    if (LINED) {
        td = (ad[0] + ad[1]) + (ad[2] + ad[3]);
        ta = (aa[0] + aa[1]) + (aa[2] + aa[3]);
    } else {
        float ed, ea;
        cd.total(td, ed);
        ca.total(ta, ea);
        dd += double(ed);
        da += double(ea);
    }
}

__device__ void adam_consume(const MeasureParams& p, const OptSegDev* opt, const AdamConsts& c,
                             uint8_t* ring, ARing& r) {
    const uint32_t full_s = smem_addr(r.full), empty_s = smem_addr(r.empty);
    const uint32_t done_s = smem_addr(r.computed);
    const int tid = int(threadIdx.x) - 32 * kAFirstConsumerWarp;
    const int warp = tid >> 5, lane = tid & 31;
    double dd = 0.0, da = 0.0;
    for (uint64_t k = 0;; ++k) {
        const int st = int(k % kAStages);
        const uint32_t parity = uint32_t((k / kAStages) & 1);
        if (!mbar_wait_warp(full_s + 8 * st, parity)) {
            if (lane == 0) raise_fault(p.fault);
            break;
        }
        const AJob j = r.jobs[st];
        if (j.kind == kAJobEnd) {
            if (lane == 0) mbar_arrive(done_s + 8 * st);   // lets the storer see the end
            break;
        }
        float td = 0.f, ta = 0.f;   // the chunk's sums
        if (j.kind == kAJobChunk) {
            uint8_t* buf = ring + size_t(st) * kAStage;
            if (j.form == kALined) adam_chunk<kALined>(j, buf, tid, c, dd, da, td, ta);
            else if (j.form == kAMoments) adam_chunk<kAMoments>(j, buf, tid, c, dd, da, td, ta);
            else adam_chunk<kALoose>(j, buf, tid, c, dd, da, td, ta);
            // the storer's bulk copies read what this thread wrote to the buffer
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        } else if (j.kind == kAJobScalar) {
            const SegDev sd = p.segs[j.seg];
            const OptSegDev od = opt[j.seg];
            for (int64_t q = j.k0 + tid; q < j.k1; q += kAConsumers) adam_scalar_vector(sd, od, q, c, dd, da);
        } else {
            run_flush<kAConsumerWarps>(r.box, st, warp, lane, dd, da, p.partials + j.slot);
            dd = 0.0;
            da = 0.0;
        }
        mbar_arrive_warp(done_s + 8 * st, lane);
        after_handback(td, ta);
        dd += double(td);
        da += double(ta);
    }
}

// The whole granules of n vectors that start at `first`, staged from the
// granule below it on.
__device__ __forceinline__ void put_granules(uint8_t* first, uint32_t staged, uint32_t n) {
    const uint32_t off = uint32_t(uintptr_t(first) & 15);
    if (off == 0) bulk_s2g(first, staged, 16 * n);
    else if (n > 1) bulk_s2g(first - off + 16, staged + 16, 16 * (n - 1));
}

// Once every consumer warp is done with a buffer, write its
// updated w, m and v back with bulk stores, and hand the buffer to the
// producer when those stores have read it.
__device__ void adam_store(const MeasureParams& p, const uint8_t* ring, ARing& r) {
    const uint32_t done_s = smem_addr(r.computed), empty_s = smem_addr(r.empty);
    const uint32_t ring_s = smem_addr(ring);
    for (uint64_t k = 0;; ++k) {
        const int st = int(k % kAStages);
        if (!mbar_wait_bounded(done_s + 8 * st, uint32_t((k / kAStages) & 1), kWaitNs)) {
            raise_fault(p.fault);
            break;
        }
        const AJob j = r.jobs[st];
        if (j.kind == kAJobEnd) break;
        if (j.kind == kAJobChunk) {
            const uint32_t n = uint32_t(j.n);
            const uint32_t buf = ring_s + uint32_t(st) * kAStage;
            bulk_s2g(j.w, buf, 16 * n);
            put_granules(j.m, buf + kAPart, n);
            put_granules(j.v, buf + 2 * kAPart, n);
            asm volatile("cp.async.bulk.commit_group;" ::: "memory");
            asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory");
        }
        mbar_arrive(empty_s + 8 * st);
    }
    asm volatile("cp.async.bulk.wait_group 0;" ::: "memory");
}

__global__ void __launch_bounds__(kMeasureThreads, 1) adamw_bulk_kernel(const MeasureParams p,
                                                                         const OptSegDev* opt,
                                                                         const AdamConsts c) {
    extern __shared__ __align__(128) uint8_t ring[];
    __shared__ __align__(8) ARing r;
    __shared__ unsigned int s_ticket;
    __shared__ __align__(8) FinTables tables;
    if (threadIdx.x == 0) {
        for (int st = 0; st < kAStages; ++st) {
            mbar_init(smem_addr(&r.full[st]), 1);
            mbar_init(smem_addr(&r.computed[st]), kAConsumerWarps);
            mbar_init(smem_addr(&r.empty[st]), 1);
            r.box.count[st] = 0u;
        }
        mbar_init_fence();
    }
    fin_prefetch(p, tables);
    dependents_may_start();
    dependency_wait();
    __syncthreads();
    if (threadIdx.x == 0) {
        adam_produce(p, opt, ring, r);
    } else if (threadIdx.x < 64) {
        if (threadIdx.x == 32) adam_store(p, ring, r);
    } else if (threadIdx.x >= 32) {
        adam_consume(p, opt, c, ring, r);
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
    // every load and bulk store of the ring is complete: it stages the combine
    finalize(p, reinterpret_cast<double2*>(ring), int32_t(kAdamBulkSmem / sizeof(double2)), &tables);
}

}  // namespace

cudaError_t launch_adamw_measure(const MeasureParams& p, const OptSegDev* opt, const AdamConsts& c,
                                 int grid, cudaStream_t s) {
    cudaGetLastError();
    adamw_measure_kernel<<<grid, kMeasureThreads, 0, s>>>(p, opt, c);
    return cudaGetLastError();
}

cudaError_t launch_adamw_bulk(const MeasureParams& p, const OptSegDev* opt, const AdamConsts& c, int grid,
                              cudaStream_t s) {
    return launch_dependent(adamw_bulk_kernel, grid, kMeasureThreads, kAdamBulkSmem, s, p, opt, c);
}

cudaError_t adamw_bulk_prepare(int* blocks_per_sm) {
    const cudaError_t e = cudaFuncSetAttribute(adamw_bulk_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                               int(kAdamBulkSmem));
    if (e != cudaSuccess) return e;
    return cudaOccupancyMaxActiveBlocksPerMultiprocessor(blocks_per_sm, adamw_bulk_kernel, kMeasureThreads,
                                                         kAdamBulkSmem);
}

}  // namespace lc
