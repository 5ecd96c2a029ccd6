// lc_noalloc.cu -- lc_measure_noalloc: the per-layer sums of lc_measure for
// callers that cannot allocate device memory.
//
// It launches the same measure kernels as lc_measure (the bulk-load one when
// every W and R is cudaMalloc memory), on the same partition, but every table
// and scratch buffer that they need (segment table, partition, partial sums,
// counters) lives in one file-scope static device array of
// LC_NOALLOC_SCRATCH_BYTES.  Host code never uses the array's name as an
// address: at set-up, once per device and with that device current, the
// array's device address is looked up with cudaGetSymbolAddress and cached.
// The tables are built on the host and reach the array as the kernel
// parameters of small upload kernels launched on the caller's stream ahead
// of the measure, so the driver copies them when each upload is launched and
// nothing reads host memory once the call has returned.  The counters and the
// fault word travel in the upload as zeros.  No cudaMalloc, cudaFree or other
// allocating routine is called.
#include "layercheck.h"
#include "lc_internal.cuh"
#include "lc_partition.cuh"

#include <cuda.h>

#include <cstdarg>
#include <cstdio>
#include <cstring>
#include <mutex>

using namespace lc;

namespace {

constexpr int kMaxSeg = LC_NOALLOC_MAX_SEGMENTS;
constexpr int kMaxLayers = LC_NOALLOC_MAX_LAYERS;
constexpr int kMaxRanges = 4096;
// Pool units a CTA on average: fewer than a context's, since every unit's table
// entries are built and uploaded with each call (1.2 G parameters: the same
// time, one upload instead of two, 20 us less on the host).
constexpr int kPoolUnits = 2;
constexpr int kMaxDevices = 64;

constexpr size_t al256(size_t x) { return (x + 255) & ~size_t(255); }

constexpr size_t al16(size_t x) { return (x + 15) & ~size_t(15); }

// Where each table of one call sits in the array: the tables are packed
// back to back (16-byte aligned) for the call's sizes, so the upload moves
// only the bytes the measure will read.
struct TableLayout {
    size_t segs, cta_vec, layer_n, cta_seg, cta_slot, layer_slot, counters, bytes;
};

constexpr TableLayout table_layout(size_t nseg, size_t nlayers, size_t R) {
    TableLayout t{};
    t.segs = 0;
    t.cta_vec = al16(t.segs + sizeof(SegDev) * nseg);
    t.layer_n = al16(t.cta_vec + sizeof(int64_t) * (R + 1));
    t.cta_seg = al16(t.layer_n + sizeof(double) * nlayers);
    t.cta_slot = al16(t.cta_seg + sizeof(int32_t) * R);
    t.layer_slot = al16(t.cta_slot + sizeof(int32_t) * R);
    t.counters = al16(t.layer_slot + sizeof(int32_t) * (nlayers + 1));   // completion, pool, fault word
    t.bytes = al16(t.counters + 3 * sizeof(unsigned int));
    return t;
}

// Scratch layout: the tables (at most kTableBytes), then the kernel scratch.
constexpr size_t kTableBytes = al256(table_layout(kMaxSeg, kMaxLayers, kMaxRanges).bytes);
constexpr size_t kOffPartials = kTableBytes;
constexpr size_t kScratchUsed = al256(kOffPartials + sizeof(double2) * (kMaxRanges + kMaxLayers));
static_assert(kScratchUsed <= LC_NOALLOC_SCRATCH_BYTES, "scratch layout exceeds its array");

}  // namespace

// The scratch of every lc_measure_noalloc call on a device.
static __device__ __align__(256) unsigned char g_noalloc_scratch[LC_NOALLOC_SCRATCH_BYTES];

namespace {

// One upload: `nbytes` (a multiple of 16) of the table image, to be written
// at byte `dst_off` of the scratch array.  Passed by value, so the launch
// itself carries the bytes.
// 31.75 KB of payload per launch, what kernel parameters hold: one launch for
// the tables of up to about 300 segments.
constexpr int kUploadVecs = 2032;
struct UploadChunk {
    uint32_t dst_off;
    uint32_t nbytes;
    uint4 data[kUploadVecs];
};
static_assert(sizeof(UploadChunk) <= 32764, "kernel parameters are limited to 32764 bytes");

// Parameters are constant memory, which serves one address a time and warp: the
// lanes' loads follow one another.  So the bytes are spread over many small
// CTAs: 31.75 KB take 2.6 us, in one CTA of 256 threads 9.7.
constexpr int kUploadThreads = 64;
__global__ void __launch_bounds__(kUploadThreads) noalloc_upload_kernel(const __grid_constant__ UploadChunk c) {
    uint4* dst = reinterpret_cast<uint4*>(g_noalloc_scratch + c.dst_off);
    const uint32_t nv = c.nbytes / 16, i = blockIdx.x * kUploadThreads + threadIdx.x;
    if (i < nv) dst[i] = c.data[i];
}

}  // namespace

namespace {

struct DeviceScratch {
    bool ready = false;
    unsigned char* addr = nullptr;   // device address of g_noalloc_scratch
    int max_grid = 0;                // resident CTAs of the thread kernel
    int bulk_grid = 0;               // and of the bulk-load kernel
    void* range_of = nullptr;        // the driver's cuMemGetAddressRange, or null
};
DeviceScratch g_scratch[kMaxDevices];
std::mutex g_scratch_mu;

// Table image built on the host; one per host thread, no heap.  The upload
// launches copy it into their parameters, so it may be rebuilt as soon as
// the call returns.
thread_local unsigned char t_image[kTableBytes] __attribute__((aligned(16)));
thread_local UploadChunk t_chunk;

lc_status err(lc_status st, const char* fmt, ...) __attribute__((format(printf, 2, 3)));
lc_status err(lc_status st, const char* fmt, ...) {
    char buf[512];
    va_list ap;
    va_start(ap, fmt);
    vsnprintf(buf, sizeof buf, fmt, ap);
    va_end(ap);
    set_last_error(buf);
    return st;
}

struct CurrentDevice {
    int prev = -1;
    bool ok = false;
    explicit CurrentDevice(int dev) {
        if (cudaGetDevice(&prev) != cudaSuccess) prev = -1;
        ok = (prev == dev) || cudaSetDevice(dev) == cudaSuccess;
    }
    ~CurrentDevice() {
        int cur = -1;
        if (prev >= 0 && cudaGetDevice(&cur) == cudaSuccess && cur != prev) cudaSetDevice(prev);
    }
};

// Once per device, with the device current: the array's device address.
lc_status setup_device(int device, DeviceScratch* out) {
    std::lock_guard<std::mutex> lk(g_scratch_mu);
    DeviceScratch& d = g_scratch[device];
    if (!d.ready) {
        void* addr = nullptr;
        cudaError_t e = cudaGetSymbolAddress(&addr, g_noalloc_scratch);
        if (e != cudaSuccess) {
            cudaGetLastError();
            return err(LC_ERR_CUDA, "lc_measure_noalloc: cudaGetSymbolAddress failed: %s",
                       cudaGetErrorString(e));
        }
        int sms = 0, occ = 0, bocc = 0;
        e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, device);
        if (e == cudaSuccess) e = measure_occupancy(&occ);
        if (e == cudaSuccess) e = measure_bulk_prepare(&bocc);
        if (e != cudaSuccess) {
            cudaGetLastError();
            return err(LC_ERR_CUDA, "lc_measure_noalloc: device query failed: %s", cudaGetErrorString(e));
        }
        d.addr = static_cast<unsigned char*>(addr);
        cudaDriverEntryPointQueryResult found;
        if (cudaGetDriverEntryPointByVersion("cuMemGetAddressRange", &d.range_of, 12000, cudaEnableDefault, &found) !=
                cudaSuccess ||
            found != cudaDriverEntryPointSuccess) {
            cudaGetLastError();
            d.range_of = nullptr;
        }
        d.max_grid = sms * (occ > 0 ? occ : 1);
        if (d.max_grid > kMaxRanges) d.max_grid = kMaxRanges;
        // room for the pool's ranges too
        d.bulk_grid = sms * (bocc > 0 ? bocc : 1) * LC_MEASURE_BULK_WAVES;
        if (d.bulk_grid > kMaxRanges / (1 + kPoolUnits)) d.bulk_grid = kMaxRanges / (1 + kPoolUnits);
        d.ready = true;
    }
    *out = d;
    return LC_OK;
}

// The allocations that this call's pointers were found in: tensors mostly
// share a few (a pool's blocks, flat buffers), and a pointer inside one of them
// needs no question of its own, which is what a call on a small model spends
// most of its time on (0.17 us each, two a segment).  Where they do not share,
// the ranges are no longer asked for after a while.
typedef CUresult (*AddressRangeFn)(CUdeviceptr*, size_t*, CUdeviceptr);
struct KnownMemory {
    static constexpr int kRanges = 8;
    AddressRangeFn range_of = nullptr;
    uintptr_t lo[kRanges], hi[kRanges];
    int n = 0, asked = 0, hits = 0;

    bool has(uintptr_t p) {
        for (int i = 0; i < n; ++i)
            if (p >= lo[i] && p < hi[i]) {
                ++hits;
                return true;
            }
        return false;
    }
    void add(uintptr_t p) {
        if (!range_of || (asked >= kRanges && hits < asked)) return;
        CUdeviceptr base = 0;
        size_t size = 0;
        ++asked;
        if (range_of(&base, &size, CUdeviceptr(p)) != CUDA_SUCCESS) return;
        const int i = n < kRanges ? n++ : asked % kRanges;
        lo[i] = uintptr_t(base);
        hi[i] = uintptr_t(base) + size;
    }
};

// `plain` becomes false for managed memory, which the bulk engine is not given.
bool is_device_memory(const void* p, int device, bool* plain, KnownMemory& known) {
    if (known.has(reinterpret_cast<uintptr_t>(p))) return true;
    cudaPointerAttributes a;
    if (cudaPointerGetAttributes(&a, p) != cudaSuccess) {
        cudaGetLastError();
        return false;
    }
    if (a.type == cudaMemoryTypeManaged) {
        *plain = false;
        return true;
    }
    if (a.type != cudaMemoryTypeDevice || a.device != device) return false;
    known.add(reinterpret_cast<uintptr_t>(p));   // cudaMalloc memory of this device, all of it
    return true;
}

lc_status measure_noalloc(int device, void* cuda_stream, const lc_segment* segs, int32_t nseg, int32_t nlayers,
                          double* sums_out, bool stall) {
    set_last_error("");
    if (!segs || nseg <= 0) return err(LC_ERR_INVALID_ARG, "lc_measure_noalloc: no segments");
    if (nlayers <= 0) return err(LC_ERR_INVALID_ARG, "lc_measure_noalloc: nlayers must be > 0");
    if (nseg > kMaxSeg)
        return err(LC_ERR_CAPACITY, "lc_measure_noalloc: %d segments exceed LC_NOALLOC_MAX_SEGMENTS (%d)",
                   nseg, kMaxSeg);
    if (nlayers > kMaxLayers)
        return err(LC_ERR_CAPACITY, "lc_measure_noalloc: %d layers exceed LC_NOALLOC_MAX_LAYERS (%d)",
                   nlayers, kMaxLayers);
    if (!sums_out || (reinterpret_cast<uintptr_t>(sums_out) & 7))
        return err(LC_ERR_INVALID_ARG, "lc_measure_noalloc: sums_out must be 8-byte aligned device memory");
    int ndev = 0;
    if (cudaGetDeviceCount(&ndev) != cudaSuccess) {
        cudaGetLastError();
        return err(LC_ERR_CUDA, "lc_measure_noalloc: no CUDA device");
    }
    if (device < 0 || device >= ndev || device >= kMaxDevices)
        return err(LC_ERR_INVALID_ARG, "lc_measure_noalloc: device %d out of range", device);
    CurrentDevice cur(device);
    if (!cur.ok) return err(LC_ERR_CUDA, "lc_measure_noalloc: cannot make device %d current", device);
    DeviceScratch ds;
    lc_status st = setup_device(device, &ds);
    if (st != LC_OK) return st;
    KnownMemory known;
    known.range_of = reinterpret_cast<AddressRangeFn>(ds.range_of);
    bool bulk = true;
    bool sums_plain = true;
    if (!is_device_memory(sums_out, device, &sums_plain, known))
        return err(LC_ERR_INVALID_ARG, "lc_measure_noalloc: sums_out is not device memory");

    // validate and order the segments: layers ascending, registration order within
    int32_t per_layer[kMaxLayers + 1];
    std::memset(per_layer, 0, sizeof per_layer);
    for (int32_t i = 0; i < nseg; ++i) {
        const lc_segment& s = segs[i];
        if (s.layer < 0 || s.layer >= nlayers)
            return err(LC_ERR_INVALID_ARG, "lc_measure_noalloc: segment %d layer %d outside [0, %d)", i,
                       s.layer, nlayers);
        if (s.w_dtype != LC_BF16 && s.w_dtype != LC_F32)
            return err(LC_ERR_INVALID_ARG, "lc_measure_noalloc: segment %d has unknown dtype", i);
        if (s.numel <= 0 || !s.w || !s.snap)
            return err(LC_ERR_INVALID_ARG, "lc_measure_noalloc: segment %d needs numel > 0, w and snap", i);
        if (s.snap == s.w)
            return err(LC_ERR_INVALID_ARG, "lc_measure_noalloc: segment %d: snap must not alias w", i);
        const uintptr_t esz = s.w_dtype == LC_BF16 ? 2 : 4;
        if ((reinterpret_cast<uintptr_t>(s.w) % esz) || (reinterpret_cast<uintptr_t>(s.snap) % esz))
            return err(LC_ERR_INVALID_ARG, "lc_measure_noalloc: segment %d not element-aligned", i);
        if (!is_device_memory(s.w, device, &bulk, known) || !is_device_memory(s.snap, device, &bulk, known))
            return err(LC_ERR_INVALID_ARG, "lc_measure_noalloc: segment %d is not device memory", i);
        per_layer[s.layer] += 1;
    }
    int32_t layer_begin[kMaxLayers + 1];
    layer_begin[0] = 0;
    for (int32_t l = 0; l < nlayers; ++l) {
        if (per_layer[l] == 0) return err(LC_ERR_INVALID_ARG, "lc_measure_noalloc: layer %d has no segment", l);
        layer_begin[l + 1] = layer_begin[l] + per_layer[l];
    }
    // the segment table sits at offset 0 whatever the grid; the rest of the
    // layout depends on the grid, known once the work space is measured
    SegDev* sd = reinterpret_cast<SegDev*>(t_image);
    int32_t fill[kMaxLayers];
    std::memcpy(fill, layer_begin, sizeof(int32_t) * nlayers);
    for (int32_t i = 0; i < nseg; ++i) {
        const lc_segment& s = segs[i];
        SegDev& d = sd[fill[s.layer]++];
        const int esz_log2 = s.w_dtype == LC_BF16 ? 1 : 2;
        const int ve = 16 >> esz_log2;
        d.w = static_cast<const uint8_t*>(s.w);
        d.r = static_cast<uint8_t*>(s.snap);
        d.numel = s.numel;
        d.lead = int32_t((reinterpret_cast<uintptr_t>(s.w) & 15) >> esz_log2);
        d.esz_log2 = esz_log2;
        d.rshift = int32_t((reinterpret_cast<uintptr_t>(s.snap) - reinterpret_cast<uintptr_t>(s.w)) & 15);
        d.layer = s.layer;
        d.nvec = (int64_t(d.lead) + s.numel + ve - 1) / ve;
    }
    int64_t V = 0;
    int64_t shifted = 0;   // vectors of segments whose R is shifted
    for (int32_t i = 0; i < nseg; ++i) {
        sd[i].vec_begin = V;
        V += sd[i].nvec;
        if (sd[i].rshift) shifted += sd[i].nvec;
    }
    const PartitionShape sh = partition_shape(V, bulk ? ds.bulk_grid : ds.max_grid, bulk ? kPoolUnits : 0, shifted);
    const TableLayout L = table_layout(size_t(nseg), size_t(nlayers), size_t(sh.ranges()));
    if (sh.ranges() > kMaxRanges || L.bytes > kTableBytes)
        return err(LC_ERR_CUDA, "lc_measure_noalloc: internal table overflow");
    double* layer_n = reinterpret_cast<double*>(t_image + L.layer_n);
    for (int32_t l = 0; l < nlayers; ++l) {
        int64_t n = 0;
        for (int32_t i = layer_begin[l]; i < layer_begin[l + 1]; ++i) n += sd[i].numel;
        layer_n[l] = double(n);
    }
    partition_fill(sh, sd, nseg, nlayers, reinterpret_cast<int64_t*>(t_image + L.cta_vec),
                   reinterpret_cast<int32_t*>(t_image + L.cta_seg), reinterpret_cast<int32_t*>(t_image + L.cta_slot),
                   reinterpret_cast<int32_t*>(t_image + L.layer_slot));
    std::memset(t_image + L.counters, 0, 3 * sizeof(unsigned int));

    cudaStream_t stream = static_cast<cudaStream_t>(cuda_stream);
    // the tables and a zero completion counter into the scratch array,
    // stream-ordered before the measure; each launch carries its bytes
    cudaGetLastError();
    for (size_t off = 0; off < L.bytes; off += sizeof t_chunk.data) {
        const size_t n = L.bytes - off < sizeof t_chunk.data ? L.bytes - off : sizeof t_chunk.data;
        t_chunk.dst_off = uint32_t(off);
        t_chunk.nbytes = uint32_t(n);
        std::memcpy(t_chunk.data, t_image + off, n);
        noalloc_upload_kernel<<<unsigned((n / 16 + kUploadThreads - 1) / kUploadThreads), kUploadThreads, 0, stream>>>(
            t_chunk);
        const cudaError_t e = cudaGetLastError();
        if (e != cudaSuccess)
            return err(LC_ERR_CUDA, "lc_measure_noalloc: table upload failed: %s", cudaGetErrorString(e));
    }
    MeasureParams p{};
    p.segs = reinterpret_cast<const SegDev*>(ds.addr + L.segs);
    p.cta_vec_begin = reinterpret_cast<const int64_t*>(ds.addr + L.cta_vec);
    p.cta_seg0 = reinterpret_cast<const int32_t*>(ds.addr + L.cta_seg);
    p.cta_slot0 = reinterpret_cast<const int32_t*>(ds.addr + L.cta_slot);
    p.layer_slot_begin = reinterpret_cast<const int32_t*>(ds.addr + L.layer_slot);
    p.layer_n = reinterpret_cast<const double*>(ds.addr + L.layer_n);
    p.partials = reinterpret_cast<double2*>(ds.addr + kOffPartials);
    p.sums = sums_out;
    unsigned int* counters = reinterpret_cast<unsigned int*>(ds.addr + L.counters);
    p.ticket = counters;
    p.unit_next = counters + 1;
    p.units = int32_t(sh.units);
    p.fault = counters + 2;
    p.nan_on_fault = 1;
    p.stall_first = stall ? 1 : 0;
    p.nseg = nseg;
    p.nlayers = nlayers;
    const cudaError_t e = bulk ? launch_measure_bulk(p, int(sh.G), false, stream)
                               : launch_measure(p, int(sh.G), false, stream);
    if (e != cudaSuccess) {
        cudaGetLastError();
        return err(LC_ERR_CUDA, "lc_measure_noalloc: launch failed: %s", cudaGetErrorString(e));
    }
    return LC_OK;
}

}  // namespace

extern "C" lc_status lc_measure_noalloc(int device, void* cuda_stream, const lc_segment* segs,
                                        int32_t nseg, int32_t nlayers, double* sums_out) {
    return measure_noalloc(device, cuda_stream, segs, nseg, nlayers, sums_out, false);
}

extern "C" lc_status lc_measure_noalloc_debug(int device, void* cuda_stream, const lc_segment* segs, int32_t nseg,
                                              int32_t nlayers, double* sums_out, int32_t debug_flags) {
    if (debug_flags & ~LC_DEBUG_MEASURE_STALL) {
        set_last_error("");
        return err(LC_ERR_INVALID_ARG, "lc_measure_noalloc_debug: unknown debug flags %d", debug_flags);
    }
    return measure_noalloc(device, cuda_stream, segs, nseg, nlayers, sums_out, debug_flags != 0);
}
