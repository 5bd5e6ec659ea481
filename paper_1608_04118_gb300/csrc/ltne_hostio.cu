// ltne_hostio.cu -- the fields moved between the caller's host arrays and
// the device planes by kernels that read and write the host arrays
// themselves (no counterpart in the paper).  On a GPU that reaches pageable
// host memory through the host's page tables (Grace's memory over
// NVLink-C2C on GB300), one pass does what the staged path does in three:
// the conversion between the host's absolute FP64 values and the device's
// deviations in the compute type, the checks, and the transfer.  Each
// element is converted exactly as the staged path's host loops convert it
// (one FP64 subtraction or addition, then round to nearest), so both paths
// give the same bits.
#include "ltne_internal.h"

namespace ltne {
namespace {

constexpr int kHioThreads = 256;

dim3 hio_grid(int nx, int ny) {
  return dim3((unsigned)((nx + kHioThreads - 1) / kHioThreads), (unsigned)(ny < 65535 ? ny : 65535));
}

// dst[k][y * nx + x] = ref[k] + mac plane k at (x, y), for every given k
template <typename C>
__global__ void __launch_bounds__(kHioThreads)
    k_fields_to_host(const C* __restrict__ mac, int64_t plane, int64_t pitch, int nx, int ny,
                     HostPlanes hp) {
  const int x = blockIdx.x * kHioThreads + threadIdx.x;
  if (x >= nx) return;
  for (int y = blockIdx.y; y < ny; y += gridDim.y) {
    const int64_t off = (int64_t)y * pitch + x, i = (int64_t)y * nx + x;
#pragma unroll
    for (int k = 0; k < 5; ++k)
      if (hp.dst[k]) hp.dst[k][i] = hp.ref[k] + (double)mac[(int64_t)k * plane + off];
  }
}

// mac plane k at (x, y) = src[k][y * nx + x] - ref[k] in the compute type,
// for every given k; bit 0 of *bad set on a value that is not finite
template <typename C>
__global__ void __launch_bounds__(kHioThreads)
    k_fields_from_host(C* __restrict__ mac, int64_t plane, int64_t pitch, int nx, int ny,
                       HostPlanes hp, uint32_t* __restrict__ bad) {
  const int x = blockIdx.x * kHioThreads + threadIdx.x;
  if (x >= nx) return;
  bool ok = true;
  for (int y = blockIdx.y; y < ny; y += gridDim.y) {
    const int64_t off = (int64_t)y * pitch + x, i = (int64_t)y * nx + x;
#pragma unroll
    for (int k = 0; k < 5; ++k) {
      if (!hp.src[k]) continue;
      const double v = hp.src[k][i] - hp.ref[k];
      ok = ok && isfinite(v);
      mac[(int64_t)k * plane + off] = (C)v;
    }
  }
  if (!ok) atomicOr(bad, 1u);
}

// The porosity plane (compute type) from the host array, one block per
// chunk of kErgunChunk consecutive values; bit 0 of *bad set on a value
// outside (0, 1).  With part, the chunk's Ergun sum in the order ergun_mean
// takes on the host: lane l adds the terms of values l, l + 32, ... in order,
// then the lanes by strides 16, 8, 4, 2, 1.
//
// Bound: small fields, the latency of the host reads and of the FP64
// divisions; large ones, the FP64 pipe (about 26 operations per value, two
// lanes per SM).  The eight warps of a block share a chunk's values (each
// reads its eight rows of 32 at once) and leave the terms in shared memory,
// where the first warp adds them in order; a warp per chunk took the 64
// values one after the other.  One ltne_set_fields call with a porosity field,
// before -> now: 256^2 137 -> 59 us, 1024^2 174 -> 127, 4096^2 1377 -> 1123.
constexpr int kPorWarps = kHioThreads / 32, kPorRows = kErgunPerLane / kPorWarps;

template <typename C>
__global__ void __launch_bounds__(kHioThreads)
    k_porosity_from_host(const double* __restrict__ phi, C* __restrict__ dst, int64_t pitch,
                         int nx, int64_t n, double* __restrict__ part,
                         uint32_t* __restrict__ bad) {
  static_assert(kErgunLanes == 32 && kPorRows * kPorWarps == kErgunPerLane, "a block per chunk");
  __shared__ double term[kErgunPerLane][kErgunLanes];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int64_t c = blockIdx.x;
  const int64_t i0 = c * kErgunChunk + warp * (kPorRows * kErgunLanes) + lane;
  double v[kPorRows];
#pragma unroll
  for (int j = 0; j < kPorRows; ++j) {
    const int64_t i = i0 + j * kErgunLanes;
    v[j] = i < n ? phi[i] : 0.5;
  }
  int64_t y = i0 / nx;
  int64_t x = i0 - y * nx;
  bool ok = true;
#pragma unroll
  for (int j = 0; j < kPorRows; ++j) {
    if (i0 + j * kErgunLanes < n) {
      ok = ok && v[j] > 0.0 && v[j] < 1.0;  // false for NaN too
      dst[y * pitch + x] = (C)v[j];
      if (part) term[warp * kPorRows + j][lane] = ergun_term(v[j]);
    }
    x += kErgunLanes;
    while (x >= nx) {
      x -= nx;
      ++y;
    }
  }
  if (!ok) atomicOr(bad, 1u);
  if (!part) return;
  __syncthreads();
  if (warp == 0) {
    const int64_t left = n - c * kErgunChunk - lane;  // values from this lane's first on
    const int rows = left >= kErgunChunk ? kErgunPerLane
                                         : (int)((left + kErgunLanes - 1) / kErgunLanes);
    double s = 0.0;
    for (int j = 0; j < rows; ++j) s += term[j][lane];
    for (int o = kErgunLanes / 2; o >= 1; o >>= 1) s += __shfl_down_sync(0xffffffffu, s, o);
    if (lane == 0) part[c] = s;
  }
}

}  // namespace

cudaError_t launch_fields_to_host(const void* mac, bool dbl, int64_t plane, int64_t pitch, int nx,
                                  int ny, const HostPlanes& hp, cudaStream_t s) {
  const dim3 g = hio_grid(nx, ny);
  if (dbl)
    k_fields_to_host<double><<<g, kHioThreads, 0, s>>>(static_cast<const double*>(mac), plane,
                                                       pitch, nx, ny, hp);
  else
    k_fields_to_host<float><<<g, kHioThreads, 0, s>>>(static_cast<const float*>(mac), plane,
                                                      pitch, nx, ny, hp);
  return cudaGetLastError();
}

cudaError_t launch_fields_from_host(void* mac, bool dbl, int64_t plane, int64_t pitch, int nx,
                                    int ny, const HostPlanes& hp, uint32_t* bad, cudaStream_t s) {
  const dim3 g = hio_grid(nx, ny);
  if (dbl)
    k_fields_from_host<double><<<g, kHioThreads, 0, s>>>(static_cast<double*>(mac), plane, pitch,
                                                         nx, ny, hp, bad);
  else
    k_fields_from_host<float><<<g, kHioThreads, 0, s>>>(static_cast<float*>(mac), plane, pitch,
                                                        nx, ny, hp, bad);
  return cudaGetLastError();
}

cudaError_t launch_porosity_from_host(const double* phi, void* dst, bool dbl, int64_t pitch, int nx,
                                      int ny, double* erg_part, uint32_t* bad, cudaStream_t s) {
  const int64_t n = (int64_t)nx * ny;
  const unsigned blocks = (unsigned)ergun_chunks(n);
  if (dbl)
    k_porosity_from_host<double><<<blocks, kHioThreads, 0, s>>>(
        phi, static_cast<double*>(dst), pitch, nx, n, erg_part, bad);
  else
    k_porosity_from_host<float><<<blocks, kHioThreads, 0, s>>>(phi, static_cast<float*>(dst),
                                                               pitch, nx, n, erg_part, bad);
  return cudaGetLastError();
}

}  // namespace ltne
