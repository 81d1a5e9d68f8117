// dsm_global_step_noalloc: the global step of dsm_global_step() on buffers
// the caller already owns, for callers that cannot allocate device memory
// (a host framework that owns all of HBM through its own pool and forbids
// outside allocations, or a latency-critical loop that must not block or
// synchronise in cudaMalloc/cudaFree).  The tile table and the per-tile
// statistics, which dsm_create() keeps in the caller's arena, live here in
// one static device array instead; this file allocates nothing.

#include <cstdio>
#include <string>

#include "dsm.h"
#include "dsm_device.cuh"

namespace dsm {
namespace {

constexpr uint64_t align256(uint64_t v) { return (v + 255) / 256 * 256; }

constexpr uint32_t kNaMaxTensors = DSM_NOALLOC_MAX_TENSORS;
constexpr uint32_t kNaMaxTiles = DSM_NOALLOC_MAX_TILES;
// Regions of the scratch array (byte offsets).
constexpr uint64_t kOffTensors = 0;
constexpr uint64_t kOffTiles = align256(kOffTensors + sizeof(TensorDesc) * kNaMaxTensors);
constexpr uint64_t kOffPartials = align256(kOffTiles + sizeof(TileDesc) * uint64_t(kNaMaxTiles));
constexpr uint64_t kOffStats = align256(kOffPartials + sizeof(StatPartial) * uint64_t(kNaMaxTiles));
constexpr uint64_t kScratchBytes = align256(kOffStats + sizeof(TensorStats) * kNaMaxTensors);
static_assert(kScratchBytes == DSM_NOALLOC_SCRATCH_BYTES, "scratch size in dsm.h is out of date");

// The scratch array: shared by every call on a device, kept until the process exits.
static __device__ __align__(256) unsigned char g_noalloc_scratch[kScratchBytes];

// Up to kListTensors consecutive tensors, passed to the kernel by value: where each starts (elements, tiles), with
// the end of the last, and whether weight decay applies.  The host, which checks the list anyway, adds up the sizes.
constexpr uint32_t kListTensors = 256;
struct TensorList {
    uint32_t first, count;                // tensors first .. first + count - 1
    float lam_global;
    uint32_t wd[kListTensors / 32];       // bit i: tensor first + i
    uint32_t tile[kListTensors + 1];
    uint64_t off[kListTensors + 1];
};

// The tensor and tile tables of the listed tensors: tile ti belongs to the last tensor whose first tile is <= ti.
// One launch for up to 256 tensors, with no copy before it.  (The list copied from the host, a prefix sum over it by
// one CTA and the tile table in a second kernel took 16 us of the 50 us of a call on 3.4 M parameters.)
__global__ void __launch_bounds__(kThreads) k_noalloc_tables(unsigned char* scratch, const __grid_constant__ TensorList l) {
    TensorDesc* tensors = reinterpret_cast<TensorDesc*>(scratch + kOffTensors);
    TileDesc* tiles = reinterpret_cast<TileDesc*>(scratch + kOffTiles);
    __shared__ uint32_t s_tile[kListTensors + 1];
    for (uint32_t i = threadIdx.x; i <= l.count; i += kThreads) s_tile[i] = l.tile[i];
    __syncthreads();
    wait_previous();  // the previous call's kernels read the tables
    const uint32_t id = blockIdx.x * kThreads + threadIdx.x, threads = gridDim.x * kThreads;
    for (uint32_t i = id; i < l.count; i += threads) {
        TensorDesc t{};
        t.off = l.off[i];
        t.numel = l.off[i + 1] - l.off[i];
        t.lam_global = (l.wd[i / 32] >> (i % 32) & 1u) ? l.lam_global : 0.0f;
        t.tile_begin = s_tile[i];
        t.tile_end = s_tile[i + 1];
        tensors[l.first + i] = t;
    }
    for (uint32_t ti = s_tile[0] + id; ti < s_tile[l.count]; ti += threads) {
        uint32_t lo = 0, hi = l.count;  // first tensor with a first tile beyond ti
        while (lo < hi) {
            const uint32_t mid = (lo + hi) / 2;
            if (s_tile[mid] <= ti) lo = mid + 1;
            else hi = mid;
        }
        const uint32_t i = lo - 1;
        tiles[ti] = make_tile(l.off[i], l.off[i + 1] - l.off[i], l.first + i, ti - s_tile[i]);
    }
}

// Launches k_noalloc_tables for every kListTensors tensors of the layout.
cudaError_t launch_tables(unsigned char* scratch, const dsm_layout* layout, float lam_global, cudaStream_t s) {
    uint64_t off = 0;
    uint32_t tile = 0;
    for (uint32_t first = 0; first < layout->count; first += kListTensors) {
        TensorList l{};
        l.first = first;
        l.count = layout->count - first < kListTensors ? layout->count - first : kListTensors;
        l.lam_global = lam_global;
        for (uint32_t i = 0; i < l.count; ++i) {
            const dsm_tensor& t = layout->tensors[first + i];
            l.off[i] = off;
            l.tile[i] = tile;
            if (t.wd) l.wd[i / 32] |= 1u << (i % 32);
            off += t.numel;
            tile += static_cast<uint32_t>((t.numel + kTile - 1) / kTile);
        }
        l.off[l.count] = off;
        l.tile[l.count] = tile;
        const uint32_t work = l.tile[l.count] - l.tile[0] > l.count ? l.tile[l.count] - l.tile[0] : l.count;
        const uint32_t blocks = (work + kThreads - 1) / kThreads;
        const cudaError_t err = launch(k_noalloc_tables, static_cast<int>(blocks < 1024 ? blocks : 1024), kThreads, 0, s,
                                       true, scratch, l);
        if (err != cudaSuccess) return err;
    }
    return cudaSuccess;
}

}  // namespace
}  // namespace dsm

using namespace dsm;

namespace {

// Failures are reported through dsm_last_error(), like every other call.
int na_fail(int code, const char* msg) {
    char buf[512];
    snprintf(buf, sizeof buf, "dsm_global_step_noalloc: %s", msg);
    set_last_error_message(buf);
    return code;
}

int na_cuda(cudaError_t e, const char* what) {
    cudaGetLastError();  // reported here: it must not be found again by a later call's check
    char buf[512];
    snprintf(buf, sizeof buf, "dsm_global_step_noalloc: %s: %s", what, cudaGetErrorString(e));
    set_last_error_message(buf);
    return DSM_ECUDA;
}

bool aligned16(const void* p) { return (reinterpret_cast<uintptr_t>(p) & 15u) == 0; }

// DSM_OK if p is device (or managed) memory of device `dev`; the name goes into the message otherwise.
int check_device_buffer(const void* p, int dev, const char* name) {
    cudaPointerAttributes attr;
    const cudaError_t err = cudaPointerGetAttributes(&attr, p);
    if (err != cudaSuccess) {
        char what[96];
        snprintf(what, sizeof what, "cudaPointerGetAttributes(%s)", name);
        return na_cuda(err, what);
    }
    if ((attr.type != cudaMemoryTypeDevice && attr.type != cudaMemoryTypeManaged) || attr.device != dev) {
        char msg[128];
        snprintf(msg, sizeof msg, "%s is not device memory of the current device", name);
        return na_fail(DSM_EINVAL, msg);
    }
    return DSM_OK;
}

}  // namespace

extern "C" int dsm_global_step_noalloc(const dsm_layout* layout, uint32_t n, const dsm_hparams* hp, float gamma,
                                       uint64_t round, float* x, float* m, float* replicas,
                                       uint64_t replica_stride, dsm_tensor_stats* stats, int stats_is_device,
                                       dsm_stream_t stream) {
    if (!layout || !hp || !x || !m || !replicas) return na_fail(DSM_EINVAL, "NULL argument");
    // the tensor list passes the same checks as in dsm_create()
    uint64_t d = 0, tiles = 0;
    if (const int rc = check_tensor_list(layout, &d, &tiles); rc != DSM_OK) {
        const std::string why = dsm_last_error();
        return na_fail(rc, why.c_str());
    }
    if (layout->count > kNaMaxTensors) return na_fail(DSM_ERANGE, "more than DSM_NOALLOC_MAX_TENSORS (4096) tensors");
    if (n == 0 || n > kMaxWorkers) return na_fail(n == 0 ? DSM_EINVAL : DSM_ERANGE, "n must lie in [1, 64]");
    if (!(gamma > 0.f && gamma < 3.0e38f)) return na_fail(DSM_EINVAL, "gamma must be finite and > 0");
    if (!(hp->g_b1 >= 0.f && hp->g_b1 <= 1.f) || !(hp->g_b2 >= 0.f && hp->g_b2 <= 1.f))
        return na_fail(DSM_EINVAL, "global betas must lie in [0, 1]");
    if (!(hp->g_eta >= 0.f && hp->g_eta < 3.0e38f) || !(hp->g_wd >= 0.f && hp->g_wd < 3.0e38f))
        return na_fail(DSM_EINVAL, "global eta and lambda must be finite and >= 0");
    if (hp->sign_mode < DSM_SIGN || hp->sign_mode > DSM_RSIGN_PM) return na_fail(DSM_EINVAL, "sign mode unknown");
    if (hp->global_mode < DSM_GLOBAL_SIGN_MOMENTUM || hp->global_mode > DSM_GLOBAL_LOOKAHEAD)
        return na_fail(DSM_EINVAL, "global step must be DSM_GLOBAL_SIGN_MOMENTUM, _SLOWMO, _SIGNED_SLOWMO or "
                                   "_LOOKAHEAD here (global AdamW needs a second-moment buffer)");
    if (hp->global_mode != DSM_GLOBAL_SIGN_MOMENTUM && hp->sign_mode != DSM_SIGN)
        return na_fail(DSM_EINVAL, "the randomized signs apply to the sign-momentum global step only");
    if (hp->sign_mode != DSM_SIGN && !(hp->rsign_B > 0.f && hp->rsign_B < 3.0e38f))
        return na_fail(DSM_EINVAL, "randomized sign needs a finite bound B > 0");
    if (tiles > kNaMaxTiles)
        return na_fail(DSM_ERANGE, "layout needs more than DSM_NOALLOC_MAX_TILES (524288) tiles of 1024 elements");
    if (replica_stride < d || replica_stride % 8 != 0)
        return na_fail(DSM_EINVAL, "replica_stride must be >= d and a multiple of 8");
    if (!aligned16(x) || !aligned16(m) || !aligned16(replicas))
        return na_fail(DSM_EALIGN, "x, m and replicas must be 16-byte aligned");

    int dev = 0;
    cudaError_t err = cudaGetDevice(&dev);
    if (err != cudaSuccess) return na_cuda(err, "cudaGetDevice");
    if (int rc = check_device_buffer(x, dev, "x"); rc != DSM_OK) return rc;
    if (int rc = check_device_buffer(m, dev, "m"); rc != DSM_OK) return rc;
    if (int rc = check_device_buffer(replicas, dev, "replicas"); rc != DSM_OK) return rc;
    if (stats && stats_is_device)
        if (int rc = check_device_buffer(stats, dev, "stats"); rc != DSM_OK) return rc;

    // The scratch array's device address on the current device, looked up by every call (a lookup,
    // no allocation), so that it is never stale: not after cudaDeviceReset, and not in another
    // context.  The first call on a device may load the library's device code there.
    void* scratch_v = nullptr;
    err = cudaGetSymbolAddress(&scratch_v, g_noalloc_scratch);
    if (err != cudaSuccess) return na_cuda(err, "cudaGetSymbolAddress(scratch)");
    unsigned char* scratch = static_cast<unsigned char*>(scratch_v);
    cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);

    // Tensor and tile tables, rebuilt in the scratch array by every call.
    if ((err = launch_tables(scratch, layout, hp->g_wd, s)) != cudaSuccess) return na_cuda(err, "launch the tables");

    Problem p{};
    p.tensors = reinterpret_cast<const TensorDesc*>(scratch + kOffTensors);
    p.tiles = reinterpret_cast<const TileDesc*>(scratch + kOffTiles);
    p.num_tensors = layout->count;
    p.num_tiles = static_cast<uint32_t>(tiles);
    p.n = n;
    p.d_stride = replica_stride;
    p.x = x;
    p.m = m;
    p.X = replicas;
    p.partials = reinterpret_cast<StatPartial*>(scratch + kOffPartials);
    // statistics in device memory are written there at once
    const bool in_place = stats && stats_is_device && reinterpret_cast<uintptr_t>(stats) % alignof(TensorStats) == 0;
    p.stats = in_place ? reinterpret_cast<TensorStats*>(stats) : reinterpret_cast<TensorStats*>(scratch + kOffStats);

    p.global_mode = hp->global_mode;
    p.early = true;
    p.fresh_tables = true;
    LaunchShape ls;
    if ((err = query_global_shape(p, &ls)) != cudaSuccess) return na_cuda(err, "occupancy query");
    GlobalScalars g{};
    g.b1 = hp->g_b1;
    g.b2 = hp->g_b2;
    g.c1 = float((1.0 - double(hp->g_b1)) / double(gamma));
    g.c2 = float((1.0 - double(hp->g_b2)) / double(gamma));
    g.eta_gamma = float(double(hp->g_eta) * double(gamma));
    g.inv_gamma = float(1.0 / double(gamma));
    g.eta = hp->g_eta;
    g.mode = hp->global_mode;
    g.B = hp->rsign_B;
    g.n_f = float(n);
    g.sign_mode = hp->sign_mode;
    g.philox_k0 = static_cast<uint32_t>(hp->seed & 0xFFFFFFFFull);
    g.philox_k1 = static_cast<uint32_t>(round & 0xFFFFFFFFull);
    g.philox_q0 = layout->first_element >> 2;
    uint32_t grid = 0;
    if ((err = launch_global(p, ls, g, s, &grid)) != cudaSuccess) return na_cuda(err, "launch global step");
    if ((err = launch_stats(p, grid, s)) != cudaSuccess) return na_cuda(err, "launch statistics");
    if (stats && !in_place) {
        err = cudaMemcpyAsync(stats, p.stats, sizeof(TensorStats) * layout->count,
                              stats_is_device ? cudaMemcpyDeviceToDevice : cudaMemcpyDeviceToHost, s);
        if (err != cudaSuccess) return na_cuda(err, "copy statistics");
        if (!stats_is_device && (err = cudaStreamSynchronize(s)) != cudaSuccess)
            return na_cuda(err, "synchronise after the global step");
    }
    return DSM_OK;
}
