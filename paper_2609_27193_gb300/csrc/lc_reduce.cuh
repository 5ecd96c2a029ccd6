// lc_reduce.cuh -- device helpers shared by the kernels that reduce over
// the measure work space (lc_measure.cu: the Eq. 1 scan; lc_adamw.cu: the
// fused optimizer step): streaming loads and stores, bf16 decoding, the
// fixed-order CTA sum and the last-CTA fp64 combine per layer,
// and fp32 chains that keep their rounding errors.
#pragma once

#include "lc_internal.cuh"

namespace lc {
namespace {

#ifndef LC_LD_PREFETCH
#define LC_LD_PREFETCH 1
#endif

__device__ __forceinline__ uint4 ld_stream(const void* p) {
    uint4 v;
#if LC_LD_PREFETCH
    asm volatile("ld.global.nc.L1::no_allocate.L2::256B.v4.u32 {%0,%1,%2,%3}, [%4];"
                 : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w)
                 : "l"(p));
#else
    asm volatile("ld.global.nc.L1::no_allocate.v4.u32 {%0,%1,%2,%3}, [%4];"
                 : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w)
                 : "l"(p));
#endif
    return v;
}

// Coherent load for R when the kernel also writes R (accumulate mode).
__device__ __forceinline__ uint4 ld_coherent(const void* p) {
    uint4 v;
    asm volatile("ld.global.L1::no_allocate.v4.u32 {%0,%1,%2,%3}, [%4];"
                 : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w)
                 : "l"(p)
                 : "memory");
    return v;
}

__device__ __forceinline__ void st_vec(void* p, uint4 v) {
    asm volatile("st.global.v4.u32 [%0], {%1,%2,%3,%4};"
                 :
                 : "l"(p), "r"(v.x), "r"(v.y), "r"(v.z), "r"(v.w)
                 : "memory");
}

__device__ __forceinline__ float bf16_lo(uint32_t x) { return __uint_as_float(x << 16); }
__device__ __forceinline__ float bf16_hi(uint32_t x) { return __uint_as_float(x & 0xffff0000u); }

// a + b, its rounding error added to e: Knuth's TwoSum, which recovers the
// error exactly whichever operand is the larger.
__device__ __forceinline__ float two_sum(float a, float b, float& e) {
    const float s = a + b, t = s - a;
    e += (a - (s - t)) + (b - t);
    return s;
}

// Two fp32 values in one 64-bit register pair; an operation on both is one
// instruction.
struct F2 {
    uint64_t v;
    static __device__ __forceinline__ F2 of(float lo, float hi) {
        F2 r;
        asm("mov.b64 %0, {%1, %2};" : "=l"(r.v) : "f"(lo), "f"(hi));
        return r;
    }
    __device__ __forceinline__ void split(float& lo, float& hi) const {
        asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(v));
    }
    __device__ __forceinline__ F2 abs() const { return F2{v & 0x7fffffff7fffffffull}; }
};
__device__ __forceinline__ F2 operator+(F2 a, F2 b) {
    F2 r;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
    return r;
}
__device__ __forceinline__ F2 operator-(F2 a, F2 b) {
    F2 r;
    asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
    return r;
}

// A chunk's sum of one thread: two fp32 chains and the rounding errors of
// their additions, recovered exactly (two_sum) and added in fp32.  With
// non-negative terms, n of them in a chain, the error words are below
// n 2^-24 of the chain, so what they lose themselves is below n^2 2^-48 of it
// (and nothing for bf16 values no more than 2^35 below the chain).  One pair of
// chains: their latency is hidden by the other chain and warps, and the loops
// that hold it stay short (lc_measure.cu has the times).
struct CompSum {
    F2 s{0}, e{0};
    __device__ __forceinline__ void add(F2 x) {
        const F2 n = s + x, t = n - s;
        e = e + ((s - (n - t)) + (x - t));
        s = n;
    }
    __device__ __forceinline__ void total(float& sum, float& err) const {
        float a, b, c, d;
        s.split(a, b);
        e.split(c, d);
        err = c + d;
        sum = two_sum(a, b, err);
    }
};

// Sum over the CTA in a fixed order; the result is valid in thread 0.
__device__ __forceinline__ void block_sum(double& d, double& a, double* sd, double* sa) {
    constexpr int kWarps = kMeasureThreads / 32;
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) {
        d += __shfl_down_sync(0xffffffffu, d, off);
        a += __shfl_down_sync(0xffffffffu, a, off);
    }
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if (lane == 0) { sd[warp] = d; sa[warp] = a; }
    __syncthreads();
    if (threadIdx.x == 0) {
        double td = 0.0, ta = 0.0;
#pragma unroll
        for (int w = 0; w < kWarps; ++w) { td += sd[w]; ta += sa[w]; }
        d = td;
        a = ta;
    }
    __syncthreads();
}

// A run's partial from a bulk kernel's consumer warps.  Each warp leaves its
// reduced (d, a) in the run's box; the last of the N contributing warps to
// arrive adds them in warp order and writes the run's one partial slot.  No
// warp waits for another.  A box is used again only once every warp has
// arrived at it and gone on (the kernels say why).
//
// fp64 runs at a few operations per cycle per SM here and a warp-wide add
// costs the same with one lane busy or 32, so the reduction keeps both sums
// in one add: lanes 0..15 carry d and lanes 16..31 a from the first step on,
// five adds instead of ten, and a warp whose lanes all hold zero skips them.
template <int NBOXES, int MAXW>
struct RunBox {
    double v[NBOXES][2][MAXW];   // d, a
    unsigned int count[NBOXES];
};

template <int N, int NBOXES, int MAXW>
__device__ __forceinline__ void run_flush(RunBox<NBOXES, MAXW>& b, int box, int w, int lane, double d, double a,
                                          double2* slot) {
    static_assert(N <= MAXW, "run box too small");
    const int half = lane >> 4;
    double x = half ? a : d;
    if (__any_sync(0xffffffffu, d != 0.0 || a != 0.0)) {
        x += __shfl_xor_sync(0xffffffffu, half ? d : a, 16);
#pragma unroll
        for (int off = 8; off > 0; off >>= 1) x += __shfl_xor_sync(0xffffffffu, x, off);
    }
    volatile double* v = b.v[box][half];
    if ((lane & 15) == 0) {
        v[w] = x;
        __threadfence_block();
    }
    __syncwarp();
    int last = 0;
    if (lane == 0) last = atomicAdd(&b.count[box], 1u) == unsigned(N - 1) ? 1 : 0;
    last = __shfl_sync(0xffffffffu, last, 0);
    if (!last) return;
    __threadfence_block();
    if ((lane & 15) == 0) {
        double sum = 0.0;
        for (int i = 0; i < N; ++i) sum += v[i];
        reinterpret_cast<double*>(slot)[half] = sum;
    }
    __syncwarp();
    if (lane == 0) *reinterpret_cast<volatile unsigned int*>(&b.count[box]) = 0u;
    __syncwarp();
}

// The next pool range for the calling CTA (its producer thread), or -1 once
// the pool is empty.  Asked for only when the CTA's current range has been
// handed to its consumers, so a unit is claimed by whichever CTA is ready
// first.
__device__ __forceinline__ int next_pool_range(const MeasureParams& p) {
    if (p.units <= 0) return -1;
    const unsigned int u = atomicAdd(p.unit_next, 1u);
    return u < unsigned(p.units) ? int(gridDim.x) + int(u) : -1;
}

// Run by the last CTA: the partial slots of every layer, contiguous in
// `partials`, are added.  The order of every addition is fixed by the layout.
// The combine runs while the rest of the GPU is idle, so its latency is the
// kernel's tail, and that is the latency of dependent fp64 adds and of trips
// to global memory.  A layer of at most kFinLane slots is added by two
// threads, one for d and one for a, in slot order (16 layers per warp
// instruction); a larger one by a warp, lanes 0..15 for d and 16..31 for a,
// each lane every 16th slot, then a fixed tree.
//
// The bulk kernels give it `stage` (shared memory free for reuse, stage_slots
// slots of it: their rings), where the whole CTA first copies the slots with
// kFinLoads independent loads in flight per thread, and `tables`: every CTA
// fetches the combine's tables while its range streams (fin_prefetch,
// asynchronous copies; which CTA is the last shows at the end), so the slots
// are the combine's only trip.  Larger layouts go in tiles of kFinLayers
// layers, each with a trip for its tables and one for its slots: the measure
// of 20,000 parameters a layer takes 31 us with 724 layers and 120 with 4096
// (39 and 197 with slots and tables of all layers from global memory), of a
// million a layer 576 with 1024 (604).
// Without `stage` and `tables`, or with more slots in a tile than `stage`
// holds (other grids and pools could bring that), slots are read from global
// memory.
//
// Runs, and so slots, are per (range, layer): a flush costs the consumer warps
// about as much as a chunk, and a small model's CTA crosses several tensors of
// a layer.  For 6 M parameters in 38 tensors and 6 layers the last consumer is
// done 9.5 us after the launch and the combine takes 2.0 us (13.4 and 4.6 with
// runs per tensor and a combine by tensor, then layer): 8 us of a decision's
// 43, and 3.5 of 119.5 over 138 M parameters.
constexpr int kFinLoads = 8;
constexpr int kFinLane = 24;
constexpr int kFinLayers = 512;

struct FinTables {
    int32_t slot_begin[kFinLayers + 1];
    double layer_n[kFinLayers];
};

template <int BYTES>
__device__ __forceinline__ void fetch_async(void* smem, const void* global) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], %2;" ::"r"(
                     static_cast<uint32_t>(__cvta_generic_to_shared(smem))),
                 "l"(global), "n"(BYTES)
                 : "memory");
}

// The tables of the layers from l0 on, as many as fit.
__device__ __forceinline__ void fin_prefetch(const MeasureParams& p, FinTables& t, int l0 = 0) {
    const int n = p.nlayers - l0 < kFinLayers ? p.nlayers - l0 : kFinLayers;
    for (int i = threadIdx.x; i <= n; i += blockDim.x) fetch_async<4>(&t.slot_begin[i], p.layer_slot_begin + l0 + i);
    for (int i = threadIdx.x; i < n; i += blockDim.x) fetch_async<8>(&t.layer_n[i], p.layer_n + l0 + i);
}

// Every thread, before the CTA's last barrier.
__device__ __forceinline__ void fin_prefetch_wait() { asm volatile("cp.async.wait_all;" ::: "memory"); }

// Both sums of n layers from slot(j, component).
template <typename Slot>
__device__ __forceinline__ void fin_layers(double* sums, int n, const int32_t* slot_begin, const double* layer_n,
                                           const Slot& slot) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
    for (int i = threadIdx.x; i < 2 * n; i += blockDim.x) {
        const int l = i >> 1, c = i & 1;
        const int32_t b0 = slot_begin[l], b1 = slot_begin[l + 1];
        if (c == 0) sums[3 * l + 2] = layer_n[l];
        if (b1 - b0 > kFinLane) continue;
        double x = 0.0;
#pragma unroll 4
        for (int32_t j = b0; j < b1; ++j) x += slot(j, c);
        sums[3 * l + c] = x;
    }
    for (int l = warp; l < n; l += nw) {
        const int32_t b0 = slot_begin[l], b1 = slot_begin[l + 1];
        if (b1 - b0 <= kFinLane) continue;
        double x = 0.0;
#pragma unroll 4
        for (int32_t j = b0 + (lane & 15); j < b1; j += 16) x += slot(j, lane >> 4);
#pragma unroll
        for (int off = 8; off > 0; off >>= 1) x += __shfl_xor_sync(0xffffffffu, x, off);
        if ((lane & 15) == 0) sums[3 * l + (lane >> 4)] = x;
    }
}

__device__ void finalize(const MeasureParams& p, double2* stage = nullptr, int32_t stage_slots = 0,
                         FinTables* tables = nullptr) {
    if (threadIdx.x == 0) {
        *p.ticket = 0u;
        if (p.unit_next) *p.unit_next = 0u;   // every CTA has left the pool
    }
    const double* global = reinterpret_cast<const double*>(p.partials);
    auto global_slot = [&](int32_t j, int c) { return __ldcg(global + 2 * j + c); };
    if (!tables) {
        fin_layers(p.sums, p.nlayers, p.layer_slot_begin, p.layer_n, global_slot);
        return;
    }
    for (int l0 = 0; l0 < p.nlayers; l0 += kFinLayers) {
        if (l0 > 0) {
            __syncthreads();   // every thread is done with the tile before
            fin_prefetch(p, *tables, l0);
            fin_prefetch_wait();
            __syncthreads();
        }
        const int nl = p.nlayers - l0 < kFinLayers ? p.nlayers - l0 : kFinLayers;
        const int32_t first = tables->slot_begin[0], n = tables->slot_begin[nl] - first;
        double* sums = p.sums + 3 * l0;
        if (n > stage_slots) {
            fin_layers(sums, nl, tables->slot_begin, tables->layer_n, global_slot);
            continue;
        }
        for (int32_t i0 = 0; i0 < n; i0 += int32_t(blockDim.x) * kFinLoads) {
            double2 v[kFinLoads];
#pragma unroll
            for (int k = 0; k < kFinLoads; ++k) {
                const int32_t i = i0 + k * int32_t(blockDim.x) + int32_t(threadIdx.x);
                if (i < n) v[k] = __ldcg(&p.partials[first + i]);
            }
#pragma unroll
            for (int k = 0; k < kFinLoads; ++k) {
                const int32_t i = i0 + k * int32_t(blockDim.x) + int32_t(threadIdx.x);
                if (i < n) stage[i] = v[k];
            }
        }
        __syncthreads();
        const double* staged = reinterpret_cast<const double*>(stage);
        fin_layers(sums, nl, tables->slot_begin, tables->layer_n,
                   [&](int32_t j, int c) { return staged[2 * (j - first) + c]; });
    }
}

}  // namespace
}  // namespace lc
