// lc_select.cu -- §3.2 Eq. 2-4 and the §3.3 staleness guard on the device,
// plus the packed-stream layout of the persisted layers (one CTA).
//
// From the per-layer sums of Eq. 1 the kernel forms u_l, updates the
// accumulator Delta_l, persists a layer when Delta_l >= tau * tau_mult[l],
// when its staleness t - t_l has reached S_max, or when the drift is not
// finite; it resets Delta_l and sets t_l = t for persisted layers.  It then
// assigns each persisted layer its offset in the packed stream (layers
// ascending) and writes the copy lists of the pack and of the snapshot
// commit, so the host never builds them.  If the stream would not fit the
// destination, it persists nothing and restores every layer's state to the
// not-persisted update (the drift stays accumulated).  The step comes from
// the host, or from a device counter when the step runs as a CUDA graph.
#include "lc_internal.cuh"

namespace lc {
namespace {

constexpr int kSelWarps = kSelectThreads / 32;
constexpr uint64_t kExact = uint64_t(1) << 53;   // whole numbers below it add exactly in binary64

// Inclusive scan over the warp.
__device__ __forceinline__ uint64_t warp_scan(uint64_t x, int lane) {
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
        const uint64_t y = __shfl_up_sync(0xffffffffu, x, off);
        if (lane >= off) x += y;
    }
    return x;
}

__device__ __forceinline__ uint64_t warp_add(uint64_t x) {
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) x += __shfl_xor_sync(0xffffffffu, x, off);
    return x;
}

// The kernel's time is latency: one CTA, a few trips to memory that wait for
// one another.  Every input of a layer is loaded at once by the layer's
// thread, a tile of kSelectThreads layers at a time; the stream layout is a
// scan over the tile; and the decision goes straight to the pinned host block
// that the host polls, header word last, instead of to a device block and a
// copy and an event behind the kernel.  The decision over 6 M parameters in 6
// layers takes 22.1 us, of which this kernel is about 4 once the sums are
// there: 0.7 for the loads, 1.1 for Eq. 1's fp64 quotients (fp64 is slow here;
// whole numbers and the host do the rest), 0.9 for the scans, 0.3 for the
// lists and 0.7 for the host's block.  With one thread laying out the stream,
// a copy and an event the decision took 6 us longer (146 layers: 13).  256
// threads keep the CTA's registers at half an SM's, so that it finds room
// beside other work.
__global__ void __launch_bounds__(kSelectThreads, 2) select_kernel(const SelectParams p) {
    const ResultLayout L = result_layout(p.nlayers);
    uint8_t* const h_mask = p.host_block + L.mask_off;
    double* const h_u = reinterpret_cast<double*>(p.host_block + L.u_off);
    uint64_t* const h_off = reinterpret_cast<uint64_t*>(p.host_block + L.off_off);
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;

    // a persisted layer's place in the packed stream and in the copy lists:
    // shared memory holds it for up to a tile of layers
    __shared__ LayerPlace s_place[kSelectThreads];
    LayerPlace* const place = p.nlayers <= kSelectThreads ? s_place : p.layer_place;
    __shared__ uint64_t w_bytes[kSelWarps], w_work[kSelWarps], w_sec[kSelWarps], w_num[kSelWarps], w_den[kSelWarps];
    __shared__ int64_t w_mx[kSelWarps];
    __shared__ uint32_t w_cnt[kSelWarps], w_odd[kSelWarps];

    const int nsec_all = p.nsec;
    dependents_may_start();
    dependency_wait();
    const int64_t step = p.step_from_counter ? __ldcg(p.step_counter) + 1 : p.step;
    uint64_t run = 0, commit_work = 0, sec = 0, num = 0, den = 0;   // sec: sections | W sections << 32
    uint32_t cnt = 0, odd = 0;                                      // selected | nonfinite << 16; not exact in 2^53
    int64_t mx = 0;
    int nsel = 0, nnonfinite = 0;
    for (int base = 0; base < p.nlayers; base += kSelectThreads) {
        const int l = base + tid;
        const bool in = l < p.nlayers;
        uint64_t b = 0, work = 0, secs = 0, xn = 0, xd = 0;
        int64_t st = 0;
        bool persist = false, nonfinite = false, inexact = false;
        if (in) {
            const double d = p.sums[3 * l], a = p.sums[3 * l + 1], n = p.sums[3 * l + 2];
            const int64_t t_last = (p.again ? p.tl_save : p.t_last)[l], numel = p.layer_numel[l];
            const double mult = p.tau_mult[l], before = p.mode == 1 ? (p.again ? p.delta_save : p.delta)[l] : 0.0;
            const uint64_t lb = p.layer_bytes[l], lw = p.layer_commit_work[l];
            const int32_t s0 = p.layer_sec_begin[l], s1 = p.layer_sec_begin[l + 1], ws = p.layer_wsec_count[l];
            const double u = (d / n) / (a / n + p.eps_w);                 // Eq. 1
            const double acc = p.mode == 1 ? before + u : u;              // Eq. 2
            nonfinite = !isfinite(acc);
            persist = nonfinite || acc >= p.tau * mult                    // Eq. 3
                      || step - t_last >= int64_t(p.max_staleness);       // §3.3
            p.acc_save[l] = acc;
            p.tl_save[l] = t_last;
            p.delta_save[l] = before;
            p.delta[l] = persist ? 0.0 : acc;                             // Eq. 4
            if (persist || p.again) p.t_last[l] = persist ? step : t_last;
            h_mask[l] = persist ? 1 : 0;
            h_u[l] = u;
            st = persist ? 0 : step - t_last;
            if (persist) {
                b = lb;
                work = lw;
                secs = uint64_t(uint32_t(s1 - s0)) | uint64_t(uint32_t(ws)) << 32;
            }
            // the staleness sums in whole numbers; past 2^53 they are taken again below
            inexact = st < 0 || uint64_t(numel) >= kExact || __umul64hi(uint64_t(numel), uint64_t(st)) != 0 ||
                      uint64_t(numel) * uint64_t(st) >= kExact;
            xn = inexact ? 0 : uint64_t(numel) * uint64_t(st);
            xd = inexact ? 0 : uint64_t(numel);
        }
        // the layer's place: what the tile's layers before it take
        const uint64_t sb = warp_scan(b, lane), sw = warp_scan(work, lane), ss = warp_scan(secs, lane);
        const uint64_t an = warp_add(xn), ad = warp_add(xd);
        int64_t m = st;
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) {
            const int64_t o = __shfl_xor_sync(0xffffffffu, m, off);
            m = o > m ? o : m;
        }
        const uint32_t c = uint32_t(__popc(__ballot_sync(0xffffffffu, persist))) |
                           uint32_t(__popc(__ballot_sync(0xffffffffu, nonfinite))) << 16;
        const bool any_inexact = __any_sync(0xffffffffu, inexact);
        if (lane == 31) {
            w_bytes[warp] = sb;
            w_work[warp] = sw;
            w_sec[warp] = ss;
            w_num[warp] = an;
            w_den[warp] = ad;
            w_mx[warp] = m;
            w_cnt[warp] = c;
            w_odd[warp] = any_inexact ? 1u : 0u;
        }
        __syncthreads();
        uint64_t pb = run, pw = commit_work, ps = sec;
        cnt = 0;
        const int warps = (p.nlayers - base + 31) / 32 < kSelWarps ? (p.nlayers - base + 31) / 32 : kSelWarps;
        for (int w = 0; w < warps; ++w) {
            if (w < warp) {
                pb += w_bytes[w];
                pw += w_work[w];
                ps += w_sec[w];
            }
            run += w_bytes[w];
            commit_work += w_work[w];
            sec += w_sec[w];
            num += w_num[w];
            den += w_den[w];
            mx = w_mx[w] > mx ? w_mx[w] : mx;
            cnt += w_cnt[w];
            odd |= w_odd[w];
        }
        if (num >= kExact || den >= kExact) odd = 1;
        nsel += int(cnt & 0xffffu);
        nnonfinite += int(cnt >> 16);
        if (in) {
            LayerPlace q;
            q.off = pb + (sb - b);
            q.commit_off = pw + (sw - work);
            q.pack_idx = int32_t(uint32_t(ps + (ss - secs)));
            q.commit_idx = int32_t((ps + (ss - secs)) >> 32);
            q.selected = persist ? 1 : 0;
            q.nwsec = int32_t(secs >> 32);
            place[l] = q;
            h_off[l] = persist ? q.off : 0;
        }
        __syncthreads();
    }

    // a stream larger than the destination persists nothing this step
    const bool fits = run <= p.capacity;
    if (tid == 0) {
        ResultHeader h;
        h.step = step;
        h.n_selected = nsel;
        h.n_nonfinite = nnonfinite;
        h.bytes = run;
        h.n_pack_desc = fits ? int32_t(uint32_t(sec)) : 0;
        h.n_commit_desc = fits ? int32_t(sec >> 32) : 0;
        h.commit_work = fits ? commit_work : 0;
        h.max_staleness = mx;
        double wn = double(num), wd = double(den);
        if (odd) {
            // whole numbers past 2^53: the sums in binary64, layers ascending
            wn = wd = 0.0;
            for (int l = 0; l < p.nlayers; ++l) {
                const bool now = place[l].selected != 0;
                const int64_t st = now ? 0 : step - p.tl_save[l];
                wn = __dadd_rn(wn, __dmul_rn(double(p.layer_numel[l]), double(st)));
                wd = __dadd_rn(wd, double(p.layer_numel[l]));
            }
        }
        h.stale_num = wn;
        h.stale_den = wd;
        h.magic = 0;
        h.status = fits ? kStatusOk : kStatusCapacity;
        h.pack_bytes = fits ? run : 0;
        *reinterpret_cast<ResultHeader*>(p.result) = h;
        *reinterpret_cast<ResultHeader*>(p.host_block) = h;
        *p.step_counter = step;
    }
    if (fits) {
        // the copy lists, one section per thread: a persisted layer's sections
        // go to its pack entries (and its W sections to its commit entries)
        const bool fused = p.fuse_commit != 0 && p.mode == 0;
        for (int j = tid; j < nsec_all; j += kSelectThreads) {
            const SectionDev sc = p.secs[j];
            const LayerPlace q = place[sc.layer];
            if (!q.selected) continue;
            CopyDesc d;
            d.woff = q.off + sc.off_in_layer;
            d.nbytes = sc.nbytes;
            d.span = sc.span;
            d.src = sc.src;
            d.dst = nullptr;
            d.dst2 = (fused && sc.ref) ? sc.ref : nullptr;
            p.pack_desc[q.pack_idx + sc.idx] = d;
            if (sc.idx < q.nwsec) {
                CopyDesc c;
                c.woff = q.commit_off + sc.commit_off;
                c.nbytes = sc.nbytes;
                c.span = (sc.nbytes + 15) & ~uint64_t(15);
                c.src = sc.src;
                c.dst = sc.ref;
                c.dst2 = nullptr;
                p.commit_desc[q.commit_idx + sc.idx] = c;
            }
        }
    } else {
        // roll back to "nothing persisted": the drift stays accumulated
        for (int l = tid; l < p.nlayers; l += kSelectThreads) {
            p.delta[l] = p.acc_save[l];
            p.t_last[l] = p.tl_save[l];
        }
    }
    __threadfence_system();   // this thread's part of the host block, before the header's magic word
    __syncthreads();
    if (tid == 0)
        *reinterpret_cast<volatile uint32_t*>(&reinterpret_cast<ResultHeader*>(p.host_block)->magic) = p.magic;
}

}  // namespace

cudaError_t launch_select(const SelectParams& p, cudaStream_t s) {
    return launch_dependent(select_kernel, 1, kSelectThreads, 0, s, p);
}

}  // namespace lc
