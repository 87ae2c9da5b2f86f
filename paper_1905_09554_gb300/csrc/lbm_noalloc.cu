// Allocation-free ligament diagnostics (lbm_diag_noalloc in include/lbm_sc.h).
//
// Who needs it: callers that may not allocate device memory while they run.
// Examples are a host application whose device memory is handed out entirely
// by its own pool allocator (so a raw cudaMalloc would fail or fragment the
// pool), or a tight time-stepping loop where cudaMalloc/cudaFree would
// implicitly synchronise the device.  Such a caller owns its population array
// and its output arrays and calls this entry point, which uses only the
// fixed scratch array below.
//
// The scratch is a file-scope __device__ array: every GPU that loads the
// library holds LBM_NOALLOC_MAX_NZ * 8 doubles of it (512 KiB) until the
// process exits.  In host code its name is only a host-side stand-in, so its
// device address is looked up once per device with cudaGetSymbolAddress.
#include <cuda_runtime.h>

#include <cmath>
#include <mutex>

#include "../../include/lbm_sc.h"
#include "codec.cuh"
#include "diag_cell.cuh"
#include "lattice.cuh"

using namespace lbm;

namespace {

constexpr int kMaxNz = LBM_NOALLOC_MAX_NZ;
constexpr int kMaxDevices = 64;

// Per-slice sums, quantity-major: row k*kMaxNz with k = 0 mass,
// 1..3 momentum, 4 liquid area, 5 max rho, 6 bad cells (parts of slices and the
// slices' sums, see below); then the 4 totals
// (mass, momentum) and the total bad-cell count at 7*kMaxNz.
static __device__ __align__(256) double g_noalloc_scratch[8 * kMaxNz];

std::mutex g_setup_mutex;
double* g_scratch_ptr[kMaxDevices] = {nullptr};

// A z slice in the parts in which the context-based diagnostics sum it, one
// block each: part i of slice z at slot parts * z + i of the quantity-major
// scratch layout.
template <class Codec>
__global__ void __launch_bounds__(kDiagThreads)
slice_diag_noalloc_kernel(double* __restrict__ scratch, const typename Codec::S* __restrict__ f, int nx, int ny,
                          long long n, double rho_l, double rho_v, DevParams dev) {
    const int z = blockIdx.x, parts = gridDim.y;
    const long long plane = (long long)nx * ny;
    const double sum = diag_part<Codec>(f + z * plane, n, plane, dev, rho_l, rho_v, nullptr, blockIdx.y, parts);
    if (threadIdx.x < 7) scratch[threadIdx.x * kMaxNz + parts * z + blockIdx.y] = sum;
}

// Slices of several parts: their sums, in turn, to slot kJoined + z (both fit:
// several parts are kDiagMaxParts in all at most).
constexpr int kJoined = kDiagMaxParts;
static_assert(2 * kDiagMaxParts <= kMaxNz, "parts and joined slices in one scratch row");
__global__ void join_parts_noalloc_kernel(double* __restrict__ scratch, int nz, int parts) {
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < 7 * nz; i += gridDim.x * blockDim.x) {
        const int k = i / nz, z = i - k * nz;
        const double* const p = scratch + k * kMaxNz + parts * z;
        double v = p[0];
        for (int j = 1; j < parts; ++j) v = diag_join(k, v, p[j]);
        scratch[k * kMaxNz + kJoined + z] = v;
    }
}

// Totals over slices (slot z of `rows`), summed in z order by one thread (deterministic), into
// tot[0..4]; optionally copies the per-slice area / max rho and
// the totals to caller device arrays.
__global__ void totals_noalloc_kernel(const double* __restrict__ rows, double* __restrict__ tot, int nz, double* mass,
                                      double* mom, double* area_z, double* maxrho_z) {
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        double m = 0, jx = 0, jy = 0, jz = 0, bad = 0;
        for (int z = 0; z < nz; ++z) {
            m += rows[0 * kMaxNz + z];
            jx += rows[1 * kMaxNz + z];
            jy += rows[2 * kMaxNz + z];
            jz += rows[3 * kMaxNz + z];
            bad += rows[6 * kMaxNz + z];
        }
        tot[0] = m;
        tot[1] = jx;
        tot[2] = jy;
        tot[3] = jz;
        tot[4] = bad;
        if (mass) *mass = m;
        if (mom) {
            mom[0] = jx;
            mom[1] = jy;
            mom[2] = jz;
        }
    }
    for (int z = blockIdx.x * blockDim.x + threadIdx.x; z < nz; z += gridDim.x * blockDim.x) {
        if (area_z) area_z[z] = rows[4 * kMaxNz + z];
        if (maxrho_z) maxrho_z[z] = rows[5 * kMaxNz + z];
    }
}

// Device address of the scratch array on the current device, looked up once
// per device (the first call on each device does it).
cudaError_t scratch_address(double** out) {
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 0 || dev >= kMaxDevices) return cudaErrorInvalidDevice;
    std::lock_guard<std::mutex> lock(g_setup_mutex);
    if (!g_scratch_ptr[dev]) {
        void* p = nullptr;
        e = cudaGetSymbolAddress(&p, g_noalloc_scratch);
        if (e != cudaSuccess) return e;
        g_scratch_ptr[dev] = static_cast<double*>(p);
    }
    *out = g_scratch_ptr[dev];
    return cudaSuccess;
}

template <class Codec>
cudaError_t launch_slices(double* scratch, const void* f, int nx, int ny, int nz, double rho_l, double rho_v,
                          const DevParams& dev, int parts, cudaStream_t st) {
    slice_diag_noalloc_kernel<Codec><<<dim3(nz, parts), kDiagThreads, 0, st>>>(
        scratch, static_cast<const typename Codec::S*>(f), nx, ny, (long long)nx * ny * nz, rho_l, rho_v, dev);
    return cudaGetLastError();
}

}  // namespace

extern "C" lbm_status lbm_diag_noalloc(const void* f, int storage, int nx, int ny, int nz, double rho_ref,
                                       double dev_scale, double rho_l, double rho_v, double* mass, double mom[3],
                                       double* area_z, double* maxrho_z, int on_device, void* stream) {
    if (!f) return LBM_EINVAL;
    if (nx < 1 || ny < 1 || nz < 1) return LBM_EINVAL;
    if (nz > kMaxNz) return LBM_EUNSUPPORTED;  // beyond the static scratch capacity
    if (!(rho_l > rho_v)) return LBM_EINVAL;
    if (storage < LBM_F64 || storage > LBM_BF16_DEV) return LBM_EINVAL;
    if (storage >= LBM_F16_DEV && !(dev_scale > 0)) return LBM_EINVAL;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    double* scratch = nullptr;
    cudaError_t e = scratch_address(&scratch);
    if (e != cudaSuccess) return LBM_ECUDA;
    int device = 0, num_sms = 0;
    e = cudaGetDevice(&device);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&num_sms, cudaDevAttrMultiProcessorCount, device);
    if (e != cudaSuccess) return LBM_ECUDA;
    const int parts = diag_parts((long long)nx * ny, nz, num_sms);
    const DevParams dev = make_dev_params(rho_ref, dev_scale > 0 ? dev_scale : 1.0);
    switch (storage) {
        case LBM_F64: e = launch_slices<CodecF64>(scratch, f, nx, ny, nz, rho_l, rho_v, dev, parts, st); break;
        case LBM_F32: e = launch_slices<CodecF32>(scratch, f, nx, ny, nz, rho_l, rho_v, dev, parts, st); break;
        case LBM_F16_DEV: e = launch_slices<CodecF16Dev>(scratch, f, nx, ny, nz, rho_l, rho_v, dev, parts, st); break;
        default: e = launch_slices<CodecBF16Dev>(scratch, f, nx, ny, nz, rho_l, rho_v, dev, parts, st); break;
    }
    if (e != cudaSuccess) return LBM_ECUDA;
    const int tb = 256, tg = (nz + tb - 1) / tb, at = parts > 1 ? kJoined : 0;
    if (parts > 1) join_parts_noalloc_kernel<<<(7 * nz + tb - 1) / tb, tb, 0, st>>>(scratch, nz, parts);
    if (on_device) totals_noalloc_kernel<<<tg, tb, 0, st>>>(scratch + at, scratch + 7 * kMaxNz, nz, mass, mom, area_z, maxrho_z);
    else totals_noalloc_kernel<<<tg, tb, 0, st>>>(scratch + at, scratch + 7 * kMaxNz, nz, nullptr, nullptr, nullptr, nullptr);
    e = cudaGetLastError();
    if (e != cudaSuccess) return LBM_ECUDA;
    double tot[5];
    e = cudaMemcpyAsync(tot, scratch + 7 * kMaxNz, sizeof(tot), cudaMemcpyDeviceToHost, st);
    if (e == cudaSuccess && !on_device) {
        if (area_z) e = cudaMemcpyAsync(area_z, scratch + 4 * kMaxNz + at, sizeof(double) * nz, cudaMemcpyDeviceToHost, st);
        if (e == cudaSuccess && maxrho_z)
            e = cudaMemcpyAsync(maxrho_z, scratch + 5 * kMaxNz + at, sizeof(double) * nz, cudaMemcpyDeviceToHost, st);
    }
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    if (e != cudaSuccess) return LBM_ECUDA;
    if (!on_device) {
        if (mass) *mass = tot[0];
        if (mom) {
            mom[0] = tot[1];
            mom[1] = tot[2];
            mom[2] = tot[3];
        }
    }
    if (tot[4] > 0 || !std::isfinite(tot[0]))
        return LBM_ENONFINITE;
    return LBM_OK;
}
