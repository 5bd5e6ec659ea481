// ltne_tile.cuh -- several time steps per launch on small cavities, one node
// per thread, from tiles held in shared memory.
//
// A step of a lattice that fits one wave of blocks takes the latency of one
// node's chain (about 1 us, more at a wall, whose rebuild comes first) and as
// much again for the launch, the loads from L2 and the stores' way back.
// Here a block owns a tile and makes kTileSteps steps of it in one launch: the
// first from global memory on the tile widened by kTileSteps - 1 nodes, the
// others from shared memory on ever narrower regions, the last on the tile
// itself, to global memory.  The widened borders are computed by each
// neighbour for itself; blocks never wait on one another.  Bound: the chain's
// latency, about 0.95 us per step inside the tile (a warp issues every 4.7
// cycles: issue 1, fixed latency 0.7, MUFU and shared memory 0.9, waiting for the
// slower wall warps 1.3, instruction fetch 0.9).  Measured, us a step, one step
// per launch -> this:
//   64^2 FP32, uniform porosity          1.74 -> 1.22
//   131 x 97 FP32, per-node porosity     2.19 -> 1.71
//   192^2 FP32, per-node porosity        2.44 -> 2.24
// Eight steps per launch gain nothing over four (64^2: 1.35: the widened
// region grows to 2.6 times the tile), and a warp apart for the wall nodes
// loses 5 % at 64^2.
//
// The arithmetic of a node is update_node, as in the one-step kernel, and what
// passes from step to step is the stored value (16-bit storage: the same
// random words), so the results are the bits of single steps.
#pragma once

#include "ltne_step_impl.cuh"

namespace ltne {

constexpr int kTileSteps = 4;      // steps per launch
constexpr int kTileNodes = 512;    // nodes of the widest region a tile may have
constexpr int kTileThreads = 512;

template <typename S, typename C>
struct TileSmem {
  S pops[2][19][kTileNodes];  // the state before and after a step
  C um[2][kTileNodes];        // |u| (local h_v)
};

template <typename S, typename C, bool kHv>
__global__ void __launch_bounds__(kTileThreads) k_step_tile(
    const S* __restrict__ src, S* __restrict__ dst, const C* __restrict__ phi, C* __restrict__ mac,
    const __grid_constant__ NodeParams<C> P, const int nx, const int ny, const int64_t pitch,
    const int64_t plane, const C scale, const C inv_scale, const int write_macros,
    const uint32_t* __restrict__ tick_in, uint32_t* __restrict__ tick_out,
    const C* __restrict__ um_in, C* __restrict__ um_out, const int steps) {
  extern __shared__ __align__(16) char smem_raw[];
  TileSmem<S, C>& sm = *reinterpret_cast<TileSmem<S, C>*>(smem_raw);
  grid_dep_wait();
  uint32_t tick = 0;
  if constexpr (Codec<S, C>::kStochastic) {
    tick = *tick_in;
    if (blockIdx.x == 0 && blockIdx.y == 0 && threadIdx.x == 0) *tick_out = tick + steps;
  }
  // tiles of even size, at least 2 x 2 (plan_tiles): a wall node's rebuild
  // reaches two columns or rows inwards, which the region one step wider holds
  const int x0 = blockIdx.x * nx / gridDim.x, x1 = (blockIdx.x + 1) * nx / gridDim.x;
  const int y0 = blockIdx.y * ny / gridDim.y, y1 = (blockIdx.y + 1) * ny / gridDim.y;
  // the first step's region, which holds all others: origin and row length
  const int ox = max(x0 - steps + 1, 0), oy = max(y0 - steps + 1, 0);
  const int W = min(x1 + steps - 1, nx) - ox;
#pragma unroll 1
  for (int s = 0; s < steps; ++s) {
    const int e = steps - 1 - s;  // nodes this step goes beyond the tile
    const int ax = max(x0 - e, 0), ay = max(y0 - e, 0);
    const int w = min(x1 + e, nx) - ax, n = w * (min(y1 + e, ny) - ay);
    const int in = (s & 1) ^ 1, out = s & 1;
    const uint32_t magic = (65536u + w - 1) / w;  // i / w = (i magic) >> 16 for i < kTileNodes
#pragma unroll 1
    for (int i = threadIdx.x; i < n; i += blockDim.x) {
      const int ly = (int)(((uint32_t)i * magic) >> 16);
      const int y = ay + ly, x = ax + i - ly * w;
      int kind = -1;
      if (x == 0 || x == nx - 1) kind = x == 0 ? 0 : 1;
      else if (y == 0 || y == ny - 1) kind = 2;
      const int cx = min(max(x, 1), nx - 2), cy = min(max(y, 1), ny - 2);
      const uint32_t off = (uint32_t)y * (uint32_t)pitch + x;
      const uint32_t noff = (uint32_t)cy * (uint32_t)pitch + cx;
      const int q = (y - oy) * W + (x - ox);
      C f[9], gf[5], gs[5];
      const C *um = um_in + off, *umn = um_in + noff;
      if (s == 0) {
        Pops<S, C>::pull(src, pitch, plane, cx, cx - 1, cx + 1, cy, cy - 1, cy + 1, inv_scale, f,
                         gf, gs);
      } else {
        const int lx = cx - ox, lc = cy - oy;
        Pops<S, C>::pull(&sm.pops[in][0][0], W, kTileNodes, lx, lx - 1, lx + 1, lc, lc - 1, lc + 1,
                         inv_scale, f, gf, gs);
        um = &sm.um[in][q];
        umn = &sm.um[in][lc * W + lx];
      }
      Macro<C> m;
      update_node<C, BC_CAVITY>(P, phi, off, noff, kind, um, umn, 0, nullptr, f, gf, gs, m);
      if (e == 0) {
        if (kHv || P.hv_local) um_out[off] = kHv ? full_speed<C>(m.umag, m.ux, m.uy) : m.umag;
        if (write_macros) store_macros<C>(mac, plane, off, m);
        Pops<S, C>::store(dst, plane, off, scale, f, gf, gs, off, tick + s);
      } else {
        if (kHv || P.hv_local) sm.um[out][q] = kHv ? full_speed<C>(m.umag, m.ux, m.uy) : m.umag;
        Pops<S, C>::store(&sm.pops[out][0][0], kTileNodes, q, scale, f, gf, gs, off, tick + s);
      }
    }
    if (e) __syncthreads();
  }
}

// The tiles of an nx x ny cavity: at most one block per SM, as square as that
// allows (the smallest widened tile), none narrower than two nodes; an empty
// plan if the widened tile is too large.
inline TilePlan plan_tiles(int nx, int ny) {
  TilePlan p;
  const int h = 2 * (kTileSteps - 1);
  int best = kTileNodes + 1;
  for (int tx = 1; tx <= kSMs && 2 * tx <= nx; ++tx) {
    const int ty = 2 * (kSMs / tx) > ny ? ny / 2 : kSMs / tx;
    const int64_t n = (int64_t)((nx + tx - 1) / tx + h) * ((ny + ty - 1) / ty + h);
    if (n < best) {
      best = (int)n;
      p.ntx = tx;
      p.nty = ty;
      p.threads = (best + 31) / 32 * 32;
    }
  }
  return p;
}

template <typename S, typename C>
cudaError_t launch_step_tile_t(const LatticeArgs& a, const NodeParams<double>& Pd,
                               const StepShape& shape, cudaStream_t st) {
  const TilePlan& p = shape.tiles;
  if (shape.steps > kTileSteps || !p.ntx || a.bc != BC_CAVITY) return cudaErrorInvalidValue;
  const auto k = Pd.hv_local ? k_step_tile<S, C, true> : k_step_tile<S, C, false>;
  constexpr int bytes = (int)sizeof(TileSmem<S, C>);
  const cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
  if (e != cudaSuccess) return e;
  return launch_kernel(a.chained != 0, k, dim3(p.ntx, p.nty), dim3(p.threads), bytes, st,
                       static_cast<const S*>(a.src), static_cast<S*>(a.dst),
                       static_cast<const C*>(a.phi), static_cast<C*>(a.mac), cast_params<C>(Pd),
                       a.nx, a.ny, a.pitch, a.plane, C(a.enc_scale), C(1.0 / a.enc_scale),
                       a.write_macros, a.tick_in, a.tick_out, static_cast<const C*>(a.um_in),
                       static_cast<C*>(a.um_out), shape.steps);
}

}  // namespace ltne
