// noalloc.cu -- tsu_grid_step_noalloc: one dimensionally split step of a
// uniform grid that lives in the caller's device memory, without allocating
// anything.
//
// Who needs this: applications whose device memory is owned end to end by
// their own allocator (a framework's caching allocator, or a service that
// reserves all of HBM up front and hands out slices) must not call cudaMalloc
// behind its back, and latency-critical loops cannot afford a cudaMalloc that
// may block or fail.  The context-based entry points allocate (the patch
// arena, tables, flags); this one keeps its few bytes of scratch -- patch
// descriptor, dt, the CTA count and the wave-speed accumulator --
// in one file-scope __device__ array instead.
//
// The scratch array is shared by every call in the process on a given GPU
// and keeps the contents of the last call; each call rewrites all of it (and
// clears the speed accumulator) before use.  Calls whose work overlaps on the
// GPU (different streams, or different host threads) race on it.
#include <cstdint>
#include <cstring>
#include <mutex>
#include <cuda_runtime.h>

#include "../../include/tsunami.h"
#include "amr_kernels.h"
#include "tile_rules.h"
#include "tsu_device.h"

namespace tsu {

namespace {

constexpr size_t kScratchBytes = 512;               // per GPU
constexpr size_t kDescOff = 0;                      // PatchDesc
constexpr size_t kDtOff = 256;                      // double dt
constexpr size_t kDtfOff = 264;                     // float dt
constexpr size_t kCountOff = 268;                   // unsigned, CTAs done
constexpr size_t kSmaxOff = 272;                    // unsigned long long smax[2]
static_assert(sizeof(PatchDesc) <= kDtOff, "the descriptor fits its slot");
constexpr int kMaxDevices = 64;

static __device__ __align__(256) unsigned char g_noalloc_scratch[kScratchBytes];

// Where the last CTA of a small grid's update leaves the two largest speeds: this
// page of the library's own, page-locked in place (a copy of 16 bytes to pageable
// memory costs 6 us of a 32 us call).  Calls are serialised by their caller, as for
// the scratch; each device has its own pair.
alignas(4096) double g_speeds[512];

struct DeviceState {
    void *scratch = nullptr;
    double *speeds = nullptr;   // the device's pointer to its pair in g_speeds; null: copied instead
};
std::mutex g_mu;
DeviceState g_state[kMaxDevices];
bool g_registered = false, g_tried = false;

// The scratch array's address on the current device (the host-side name of a
// __device__ array is not a device address) and its pair of speeds, looked up once
// per device.
cudaError_t state_of_device(DeviceState *out, double **host_speeds)
{
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 0 || dev >= kMaxDevices) return cudaErrorInvalidDevice;
    std::lock_guard<std::mutex> lk(g_mu);
    DeviceState &d = g_state[dev];
    if (!d.scratch) {
        void *p = nullptr;
        e = cudaGetSymbolAddress(&p, g_noalloc_scratch);
        if (e != cudaSuccess) return e;
        if (!g_tried) {
            g_tried = true;
            g_registered = cudaHostRegister(g_speeds, sizeof g_speeds, cudaHostRegisterPortable | cudaHostRegisterMapped) == cudaSuccess;
            if (!g_registered) cudaGetLastError();   // the copy serves as well
        }
        void *q = nullptr;
        if (g_registered && cudaHostGetDevicePointer(&q, g_speeds, 0) == cudaSuccess)
            d.speeds = static_cast<double *>(q) + 2 * dev;
        else cudaGetLastError();
        d.scratch = p;
    }
    *out = d;
    *host_speeds = g_speeds + 2 * dev;
    return cudaSuccess;
}

}  // namespace
}  // namespace tsu

using namespace tsu;

extern "C" int tsu_grid_step_noalloc(int precision, void *block, int nx, int ny, int pitch, long long field_stride,
                                     int cur, double dx, double dy, double dt, double g, double drytol, const int *bc,
                                     double *max_speeds, void *cuda_stream)
{
    if (precision != TSU_F64 && precision != TSU_F32P) return TSU_ERR_ARG;
    if (!block || !bc || !max_speeds) return TSU_ERR_ARG;
    if (nx < 1 || ny < 1 || nx > TSU_NOALLOC_MAX_SIDE || ny > TSU_NOALLOC_MAX_SIDE) return TSU_ERR_ARG;
    if (pitch < nx + 4 || field_stride < (long long)pitch * (ny + 4) || (cur != 0 && cur != 1)) return TSU_ERR_ARG;
    if (!(dx > 0) || !(dy > 0) || !(dt >= 0) || !(g > 0) || !(drytol > 0)) return TSU_ERR_ARG;
    for (int k = 0; k < 4; k++)
        if (bc[k] != TSU_BC_WALL && bc[k] != TSU_BC_EXTRAP) return TSU_ERR_ARG;
    const size_t esz = precision == TSU_F64 ? 8 : 4;
    if (((uintptr_t)block) % esz) return TSU_ERR_ARG;
    // tiles found from the CTA's index
    const int nt = precision == TSU_F64 ? step_threads_f64(0) : step_threads_f32p();
    const int W = precision == TSU_F64 ? step_strip_width_f64(nt, 0) : step_strip_width_f32p(nt, 0);
    const int rows = tile_cut(ny, work_rows(1, &nx, &ny, W, nt, true, precision == TSU_F64));
    const int nsx = (nx + W - 1) / W, nsy = (ny + rows - 1) / rows;

    cudaStream_t st = (cudaStream_t)cuda_stream;
    DeviceState ds;
    double *host_speeds = nullptr;
    if (state_of_device(&ds, &host_speeds) != cudaSuccess) return TSU_ERR_CUDA;
    unsigned char *scratch = reinterpret_cast<unsigned char *>(ds.scratch);

    PatchDesc d;
    std::memset(&d, 0, sizeof d);
    d.fs = field_stride;
    d.nx = nx; d.ny = ny; d.pitch = pitch;
    d.bcmask = 15;
    GridStart gs{};
    gs.desc = reinterpret_cast<PatchDesc *>(scratch + kDescOff);
    gs.dt = reinterpret_cast<double *>(scratch + kDtOff);
    gs.dtf = reinterpret_cast<float *>(scratch + kDtfOff);
    gs.smax = reinterpret_cast<unsigned long long *>(scratch + kSmaxOff);
    gs.count = reinterpret_cast<unsigned *>(scratch + kCountOff);
    gs.dt_value = dt;
    for (int k = 0; k < 4; k++) gs.bc[k] = bc[k];
    if (k_grid_start(precision, d, block, cur, gs, st) != 0) return TSU_ERR_CUDA;
    const PatchDesc *desc = gs.desc;

    StepArgs a{};
    a.descs = desc;
    a.tile_rows = rows;
    a.tile_nsx = nsx;
    a.arena = block;
    a.cur = cur;
    a.dt1 = reinterpret_cast<const double *>(scratch + kDtOff);
    a.smax = reinterpret_cast<unsigned long long *>(scratch + kSmaxOff);
    a.R = 1.0;
    a.dx = dx;
    a.dy = dy;
    a.g = g;
    a.drytol = drytol;
    a.dt1f = reinterpret_cast<const float *>(scratch + kDtfOff);
    set_f32_constants(a);
    const bool direct = ds.speeds != nullptr && nsx * nsy <= kTailMaxCtas;
    if (direct) {
        a.tail.count = gs.count;
        a.tail.speeds_out = ds.speeds;
    }
    int e = precision == TSU_F64 ? launch_step_f64(a, nsx * nsy, nt, st) : launch_step_f32p(a, nsx * nsy, nt, st);
    if (e != 0) return TSU_ERR_CUDA;

    if (direct) {
        if (cudaStreamSynchronize(st) != cudaSuccess) return TSU_ERR_CUDA;
        max_speeds[0] = host_speeds[0];
        max_speeds[1] = host_speeds[1];
        return TSU_OK;
    }
    unsigned long long bits[2] = {0ull, 0ull};
    if (cudaMemcpyAsync(bits, scratch + kSmaxOff, sizeof bits, cudaMemcpyDeviceToHost, st) != cudaSuccess)
        return TSU_ERR_CUDA;
    if (cudaStreamSynchronize(st) != cudaSuccess) return TSU_ERR_CUDA;
    for (int k = 0; k < 2; k++) {
        double v;
        std::memcpy(&v, &bits[k], sizeof v);
        max_speeds[k] = v;
    }
    return TSU_OK;
}
