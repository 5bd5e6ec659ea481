// ltne_march.cuh -- two time steps in one pass over memory, two neighbouring
// nodes per thread (cavity walls, FP32 arithmetic).
//
// One step moves every population once in and once out, so on lattices
// beyond L2 the one-step kernels end at the HBM roofline (FP32 4096^2 with
// per-node porosity: 377 us a step, 101 % of the measured copy).  Here a
// warp owns a strip of 32 node pairs and walks up the rows of a segment.  At
// row r it makes the first step of row r from HBM, and with it the second
// step of row r - 1, whose 19 pulled values are then all at hand: those that
// stream down (e_y = -1) from row r itself, those that stay (e_y = 0) from
// row r - 1, those that stream up from row r - 2.  The values along x come
// from the neighbouring lanes by shuffles, and the rows' delay is a line of
// 9 + 2 x 5 slots per thread in shared memory that no other thread touches:
// no barrier, no block of warps in step, and 19 reads and 19 writes from HBM
// per two steps.
//
// What it pays: the first step of a strip's two outer pairs and of the rows
// below and above a segment is made twice, once by each neighbour (about
// (seg + 2) / seg * 32 / 30 of the first steps).  Bound: 16-bit storage, the
// FMA pipe (busy 70 % of the cycles at 4096^2: a paired instruction holds it
// for two), with 64 % of the issue slots taken; FP32, that (57 and 52 %) and the
// rows' loads (DRAM at 76 % of the copy).  Measured, us a step, one-step kernel -> this:
//   4096^2 FP32, per-node porosity   374 -> 279  (60.2 GLUPS)
//   2048^2 FP32, per-node porosity    96 -> 84
//   8192^2 FP16, uniform porosity   1000 -> 963  (69.7 GLUPS)
//   8192^2 FP16, per-node porosity  1206 -> 1075
//   8192^2 BF16, per-node porosity  1135 -> 996
// One warp per block: blocks of four warps keep the slots of finished warps
// (4096^2: 287).  20 blocks per SM, 96 registers: at 80 registers and 24
// blocks the spills cost more than the warps give (348).  The next row's
// values copied ahead into shared memory by cp.async take the load stalls
// away and gain little or lose: BF16 1041 -> 1015, FP32 278 -> 310 (its stages
// leave too little L1, or too few warps); prefetches into L2 lose 2 %.  The
// node's arithmetic stands once, in the loop over the passes of a row: with a
// copy per step the time depended on where the code fell (278 or 292).
//
// The results are the bits of two launches of k_step_pair: the same per-node
// functions in the same paired arithmetic, the values between the steps as
// the populations would have stored them (16-bit storage: rounded with the
// same random words), the odd last node of a row in the one-node arithmetic
// (MarchOdd).
#pragma once

#include "ltne_pair.cuh"

namespace ltne {

// A node pair as the population planes hold it.
template <typename S> struct PairPack;

template <> struct PairPack<float> {
  using T = float2;
  static __device__ __forceinline__ T enc(F2 v, float, uint32_t) { return v.v; }
  static __device__ __forceinline__ F2 dec(T w, float) { return F2(w); }
  static __device__ __forceinline__ T low(uint32_t bits) {
    return make_float2(__uint_as_float(bits), 0.0f);
  }
  // the pair (x0 - 1, x0) as it streams into (x0, x0 + 1), and (x0 + 1, x0 + 2)
  static __device__ __forceinline__ T from_left(T w) {
    return make_float2(__shfl_up_sync(0xffffffffu, w.y, 1), w.x);
  }
  static __device__ __forceinline__ T from_right(T w) {
    return make_float2(w.y, __shfl_down_sync(0xffffffffu, w.x, 1));
  }
};

struct PairPack16 {
  using T = uint32_t;
  static __device__ __forceinline__ T low(uint32_t bits) { return bits; }
  static __device__ __forceinline__ T from_left(T w) {
    return __byte_perm(__shfl_up_sync(0xffffffffu, w, 1), w, 0x5432);
  }
  static __device__ __forceinline__ T from_right(T w) {
    return __byte_perm(w, __shfl_down_sync(0xffffffffu, w, 1), 0x5432);
  }
};

template <> struct PairPack<__half> : PairPack16 {
  static __device__ __forceinline__ T enc(F2 v, float scale, uint32_t r) {
    return Codec<__half, float>::enc2(v.v.x, v.v.y, scale, r);
  }
  static __device__ __forceinline__ F2 dec(T w, float inv_scale) {
    const __half2 h = *reinterpret_cast<const __half2*>(&w);
    return F2(mul2_(__half22float2(h), make_float2(inv_scale, inv_scale)));
  }
};

template <> struct PairPack<__nv_bfloat16> : PairPack16 {
  static __device__ __forceinline__ T enc(F2 v, float scale, uint32_t r) {
    return Codec<__nv_bfloat16, float>::enc2(v.v.x, v.v.y, scale, r);
  }
  static __device__ __forceinline__ F2 dec(T w, float) {
    return F2(__uint_as_float(w << 16), __uint_as_float(w & 0xffff0000u));
  }
};

// e_x and e_y of value i of the 19 (f_0..f_8, g_f0..g_f4, g_s0..g_s4; Eq. 8).
__host__ __device__ constexpr int value_ex(int i) {
  return i < 9 ? (i == 1 || i == 5 || i == 8 ? 1 : (i == 3 || i == 6 || i == 7 ? -1 : 0))
               : ((i - 9) % 5 == 1 ? 1 : ((i - 9) % 5 == 3 ? -1 : 0));
}
__host__ __device__ constexpr int value_ey(int i) {
  return i < 9 ? (i == 2 || i == 5 || i == 6 ? 1 : (i == 4 || i == 7 || i == 8 ? -1 : 0))
               : ((i - 9) % 5 == 2 ? 1 : ((i - 9) % 5 == 4 ? -1 : 0));
}

// The pair's 19 values as one list.
__device__ __forceinline__ F2& pair_value(int i, F2 (&f)[9], F2 (&gf)[5], F2 (&gs)[5]) {
  return i < 9 ? f[i < 9 ? i : 0] : (i < 14 ? gf[(i - 9) % 5] : gs[(i - 9) % 5]);
}

struct PairSide {
  bool left, right;  // the pair holds the left / right wall node
};

// The wall rebuild of a pair from its 19 values v pulled around row cy (noff:
// the pair's offset there), in place: step_pair's rebuild of a bottom or top
// row and step_pair_side's of a pair holding a side wall node, whose other
// node is the one the wall node is rebuilt from.  Out of line with v in local
// memory, so that the wall code takes no registers from the interior path.
static __device__ __noinline__ void march_wall(const NodeParams<F2>& P,
                                               const float* __restrict__ phi, uint32_t noff,
                                               bool wall_row, PairSide sd, F2* v) {
  const bool side = sd.left || sd.right;
  F2 f[9], gf[5], gs[5];
  auto both = [&](F2 w) {  // side pairs: both lanes take the interior node's value
    const float s = sd.left ? w.v.y : w.v.x;
    return side ? F2(s, s) : w;
  };
#pragma unroll
  for (int i = 0; i < 9; ++i) f[i] = both(v[i]);
#pragma unroll
  for (int i = 0; i < 5; ++i) {
    gf[i] = both(v[9 + i]);
    gs[i] = both(v[14 + i]);
  }
  Medium<F2> mdn = phi ? medium_at<F2>(P, both(ld_f2(phi + noff))) : P.um;
  Macro<F2> mn;
  macros<F2>(P, mdn, f, gf, gs, mn);
  const float tw = sd.left ? P.dT_hot.v.x : P.dT_cold.v.x;
  F2 twf = mn.dTf, tws = mn.dTs;  // adiabatic rows: the neighbour's temperatures
  if (sd.left) twf.v.x = tws.v.x = tw;
  if (sd.right) twf.v.y = tws.v.y = tw;
#pragma unroll
  for (int i = 0; i < 9; ++i) v[i] = f[i];
#pragma unroll
  for (int i = 0; i < 5; ++i) {
    v[9 + i] = gf[i];
    v[14 + i] = gs[i];
  }
  nee<F2>(P, mn, twf, tws, f, gf, gs);
  const bool wx = sd.left || wall_row, wy = sd.right || wall_row;
  auto pick = [&](F2 r, F2 w) { return F2(wx ? r.v.x : w.v.x, wy ? r.v.y : w.v.y); };
#pragma unroll
  for (int i = 0; i < 9; ++i) v[i] = pick(f[i], v[i]);
#pragma unroll
  for (int i = 0; i < 5; ++i) {
    v[9 + i] = pick(gf[i], v[9 + i]);
    v[14 + i] = pick(gs[i], v[14 + i]);
  }
}

// The last node of an odd row (a wall node, x = nx - 1) in the one-node
// arithmetic of step_node, from the 19 values v pulled around the node it is
// rebuilt from (offset noff): e receives the stored elements' bits, mac5 the
// macroscopic values.
template <typename S>
static __device__ __noinline__ void march_odd(const NodeParams<float>& P,
                                              const float* __restrict__ phi, uint32_t off,
                                              uint32_t noff, float scale, uint32_t tick,
                                              const float* v, uint32_t* e, float* mac5) {
  float f[9], gf[5], gs[5];
#pragma unroll
  for (int i = 0; i < 9; ++i) f[i] = v[i];
#pragma unroll
  for (int i = 0; i < 5; ++i) {
    gf[i] = v[9 + i];
    gs[i] = v[14 + i];
  }
  const Medium<float> mdn = phi ? medium_at<float>(P, phi[noff]) : P.um;
  Macro<float> m;
  macros<float>(P, mdn, f, gf, gs, m);
  nee<float>(P, m, P.dT_cold, P.dT_cold, f, gf, gs);
  const Medium<float> md = phi ? medium_at<float>(P, phi[off]) : P.um;
  macros<float>(P, md, f, gf, gs, m);
  mac5[0] = m.drho;
  mac5[1] = m.ux;
  mac5[2] = m.uy;
  mac5[3] = m.dTf;
  mac5[4] = m.dTs;
  collide<float>(P, m, f, gf, gs);
  auto val = [&](int i) { return i < 9 ? f[i] : (i < 14 ? gf[i - 9] : gs[i - 14]); };
  if constexpr (Codec<S, float>::kStochastic) {  // the pairing of Pops::store
    RandomBits rb(off, tick);
#pragma unroll
    for (int i = 0; i < 19; i += 2) {
      const uint32_t d =
          Codec<S, float>::enc2(val(i), i + 1 < 19 ? val(i + 1) : 0.0f, scale, rb.next());
      e[i] = d & 0xffffu;
      if (i + 1 < 19) e[i + 1] = d >> 16;
    }
  } else {
#pragma unroll
    for (int i = 0; i < 19; ++i) e[i] = __float_as_uint(val(i));
  }
}

template <typename S> __device__ __forceinline__ S element(uint32_t bits) {
  return bits_to<S>((unsigned short)bits);
}
template <> __device__ __forceinline__ float element<float>(uint32_t bits) {
  return __uint_as_float(bits);
}

constexpr int kMarchBlocks = 20;  // one-warp blocks per SM (96 registers)
constexpr int kMarchRows = 24;    // rows of a segment at most (march_rows)

// The lone last node of an odd row runs in the one-node arithmetic, over which
// one lane takes a warp as long as all 32 would.  So the rows of a segment are
// spread over the lanes: the first step of the column's nodes is one pass before
// the walk (of its results the strip needs the five values with e_x = -1), the
// second step one pass after it, from the values pulled on the way.  With a pass
// per row, 513 x 32,804 FP16 took 470 us a step, 2049 x 8288 uniform 309, 129 x
// 32,713 FP32 188 (one step per launch: 413, 288, 185); this way 353, 282, 154.
template <bool kOdd> struct MarchOdd {
  uint32_t left[5][32];             // values 3, 6, 7, 12, 17 after the first step, by row
  float pulled[kMarchRows + 1][19];  // around the column beside, before the second
};
template <> struct MarchOdd<false> {};

template <typename S, bool kOdd>
__global__ void __launch_bounds__(32, kMarchBlocks) k_step2_pair(
    const S* __restrict__ src, S* __restrict__ dst, const float* __restrict__ phi,
    float* __restrict__ mac, const __grid_constant__ NodeParams<F2> P,
    const __grid_constant__ NodeParams<float> P1, const int nx, const int ny, const uint32_t pi,
    const uint32_t pl, const float scale, const float inv_scale, const int write_macros,
    const uint32_t* __restrict__ tick_in, uint32_t* __restrict__ tick_out, const int seg_rows) {
  using PP = PairPack<S>;
  using PT = typename PP::T;
  constexpr bool kRandom = Codec<S, float>::kStochastic;
  __shared__ PT line[19][32];  // slots 0-8: e_y = 0, one row; 9-18: e_y = +1, two rows
  [[maybe_unused]] __shared__ MarchOdd<kOdd> column;
  grid_dep_wait();
  uint32_t tick = 0;
  if constexpr (kRandom) {
    tick = *tick_in;
    if (blockIdx.x == 0 && blockIdx.y == 0 && threadIdx.x == 0) *tick_out = tick + 2u;
  }
  const int lane = threadIdx.x;
  const int npairs = (nx + 1) >> 1;
  int pr = blockIdx.x * kMarchLanes + lane;
  // the second step needs both neighbouring lanes, except at the lattice's sides
  const bool own = pr < npairs && (lane > 0 || pr == 0) && (lane < 31 || pr == npairs - 1);
  pr = min(pr, npairs - 1);  // lanes beyond the lattice repeat its last pair and store nothing
  const uint32_t x0 = 2 * pr;
  const bool last = pr == npairs - 1;
  const bool odd = kOdd && last;  // only the wall node x = nx - 1
  const PairSide sd{pr == 0, !kOdd && last};
  const bool odd_strip = kOdd && __any_sync(0xffffffffu, last);
  const int ya = blockIdx.y * seg_rows, yb = min(ny, ya + seg_rows);
  const int r0 = max(ya - 1, 0), r1 = min(yb, ny - 1);  // rows of the first step
  if constexpr (kOdd) {
    if (odd_strip) {  // first step of the column x = nx - 1, row r0 + lane
      const int y = min(r0 + lane, r1), cy = min(max(y, 1), ny - 2);
      float f[9], gf[5], gs[5], v[19], mac5[5];
      uint32_t e[19];
      Pops<S, float>::pull(src, pi, pl, nx - 2, nx - 3, nx - 1, cy, cy - 1, cy + 1, inv_scale, f,
                           gf, gs);
#pragma unroll
      for (int i = 0; i < 19; ++i) v[i] = i < 9 ? f[i] : (i < 14 ? gf[i - 9] : gs[i - 14]);
      march_odd<S>(P1, phi, (uint32_t)y * pi + (nx - 1), (uint32_t)cy * pi + (nx - 2), scale, tick,
                   v, e, mac5);
      const int from[5] = {3, 6, 7, 12, 17};
#pragma unroll
      for (int k = 0; k < 5; ++k) column.left[k][lane] = e[from[k]];
      __syncwarp();
    }
  }

  for (int r = r0; r <= r1; ++r) {
    // pass 0: first step of row r; pass 1: second step of row j = r - 1; pass 2:
    // the wall row beside row 1 or ny - 2, rebuilt from the same pulled values
    const int j = r - 1;
    const bool wall_next = j == 1 || j == ny - 2;
    int y = r, cy = r == 0 ? 1 : (r == ny - 1 ? ny - 2 : r);
    F2 f[9], gf[5], gs[5];
    PairPops<S>::pull(src, pl, pi, (int)x0, (int)x0 - 1, (int)x0 + 2, cy, cy - 1, cy + 1, inv_scale,
                      f, gf, gs);
    F2 t[19];  // pass 1's pulled values, kept for pass 2
#pragma unroll 1
    for (int pass = 0;; ++pass) {
      const uint32_t off = (uint32_t)y * pi + x0, noff = (uint32_t)cy * pi + x0;
      if (y != cy || sd.left || sd.right) {
        F2 u[19];
#pragma unroll
        for (int i = 0; i < 19; ++i) u[i] = pair_value(i, f, gf, gs);
        march_wall(P, phi, noff, y != cy, sd, u);
#pragma unroll
        for (int i = 0; i < 19; ++i) pair_value(i, f, gf, gs) = u[i];
      }
      const Medium<F2> md = phi ? medium_at<F2>(P, ld_f2(phi + off)) : P.um;
      Macro<F2> m;
      macros<F2>(P, md, f, gf, gs, m);
      if (pass && own && !odd && write_macros) {
        st_f2(mac + off, m.drho);
        st_f2(mac + pl + off, m.ux);
        st_f2(mac + 2u * pl + off, m.uy);
        st_f2(mac + 3u * pl + off, m.dTf);
        st_f2(mac + 4u * pl + off, m.dTs);
      }
      collide<F2>(P, m, f, gf, gs);
      if (pass == 0) {
        // the values as stored, streamed along x, and along y by their delay
        RandomBits rb(off, tick);
        const int par = r & 1;
#pragma unroll
        for (int i = 0; i < 19; ++i) {
          F2& v = pair_value(i, f, gf, gs);
          PT w = PP::enc(v, scale, kRandom ? rb.next() : 0u);
          if constexpr (kOdd) {
            const int k = i == 3 ? 0 : i == 6 ? 1 : i == 7 ? 2 : i == 12 ? 3 : 4;
            if (odd && value_ex(i) < 0) w = PP::low(column.left[k][r - r0]);
          }
          if (value_ex(i) > 0) w = PP::from_left(w);
          if (value_ex(i) < 0) w = PP::from_right(w);
          if (value_ey(i) >= 0) {
            constexpr int slot[19] = {0, 1, 9, 2, 0, 10, 11, 0, 0, 3, 4, 12, 5, 0, 6, 7, 13, 8, 0};
            PT& s = line[value_ey(i) > 0 && par ? slot[i] + 5 : slot[i]][lane];
            const PT o = s;
            s = w;
            w = o;
          }
          v = PP::dec(w, inv_scale);
        }
        if (r < r0 + 2) break;  // the line is not full yet
        if constexpr (kOdd) {
          if (pr == npairs - 2) {
#pragma unroll
            for (int i = 0; i < 19; ++i)
              column.pulled[r - r0 - 2][i] = pair_value(i, f, gf, gs).v.y;
          }
        }
        if (wall_next) {
#pragma unroll
          for (int i = 0; i < 19; ++i) t[i] = pair_value(i, f, gf, gs);
        }
        y = cy = j;
        continue;
      }
      if (own && !odd) PairPops<S>::store(dst, pl, off, scale, f, gf, gs, off, tick + 1u);
      if (!wall_next || pass == 2) break;
      y = j == 1 ? 0 : ny - 1;
#pragma unroll
      for (int i = 0; i < 19; ++i) pair_value(i, f, gf, gs) = t[i];
    }
  }
  if constexpr (kOdd) {
    const int j0 = r0 + 1, j1 = r1 - 1;  // rows of the second step, wall rows apart
    if (odd_strip && j0 <= j1) {
      __syncwarp();
      const int y = (j0 == 1 ? 0 : j0) + lane;
      if (y <= (j1 == ny - 2 ? ny - 1 : j1)) {
        const int cy = min(max(y, 1), ny - 2);
        const uint32_t off = (uint32_t)y * pi + (nx - 1);
        float v[19], mac5[5];
        uint32_t e[19];
#pragma unroll
        for (int i = 0; i < 19; ++i) v[i] = column.pulled[cy - j0][i];
        march_odd<S>(P1, phi, off, (uint32_t)cy * pi + (nx - 2), scale, tick + 1u, v, e, mac5);
        for (int i = 0; i < 19; ++i) dst[(uint32_t)i * pl + off] = element<S>(e[i]);
        if (write_macros)
          for (int k = 0; k < 5; ++k) mac[(uint32_t)k * pl + off] = mac5[k];
      }
    }
  }
}

// Rows per segment.  A segment of s rows costs 2 s + 2 row steps, its first
// row of waves fills up and its last drains in about 0.7 of a segment's
// time (fitted to sweeps of s: 6, 10, 14, 20 took 84, 88, 91, 106 us a step at
// 2048^2 FP32, 284, 277, 279, 285 at 4096^2 FP32, and 10, 14, 20, 24 took 1018,
// 996, 984, 982 at 8192^2 BF16).  Not above kMarchRows: the rows in work at one time
// then spread over more memory than L2 and the address translation hold
// (4096^2: 404 us with one wave of 98-row segments).
inline int march_rows(int strips, int ny, int warps) {
  int best = 6;
  double cost = 1e30;
  for (int s = 6; s <= kMarchRows; s += 2) {
    const double waves = (double)strips * ((ny + s - 1) / s) / warps;
    const double c = (waves + 0.7) * (2 * s + 2);
    if (c < cost) {
      cost = c;
      best = s;
    }
  }
  return best;
}

template <typename S>
cudaError_t launch_step2_pair_t(const LatticeArgs& a, const NodeParams<double>& Pd,
                                cudaStream_t st) {
  const NodeParams<F2> P = cast_params<F2>(Pd);
  const NodeParams<float> P1 = cast_params<float>(Pd);
  const int strips = march_strips((a.nx + 1) / 2);
  const int seg = march_rows(strips, a.ny, kSMs * kMarchBlocks);
  const dim3 grid(strips, (a.ny + seg - 1) / seg);
  if (grid.y > (unsigned)kMaxGridY) return cudaErrorInvalidValue;
  return launch_kernel(a.chained != 0, a.nx % 2 ? k_step2_pair<S, true> : k_step2_pair<S, false>,
                       grid, dim3(32), 0, st, static_cast<const S*>(a.src), static_cast<S*>(a.dst),
                       static_cast<const float*>(a.phi), static_cast<float*>(a.mac), P, P1, a.nx,
                       a.ny, (uint32_t)a.pitch, (uint32_t)a.plane, a.enc_scale,
                       1.0f / a.enc_scale, a.write_macros, a.tick_in, a.tick_out, seg);
}

// The same walk with one node per lane (FP32 storage), for lattices whose
// schedule has one node per thread: strips of 32 nodes, 30 of which take the
// second step, and segments of 8 rows (4, 6, 8, 12, 16 rows took 24.3, 24.9, 24.3,
// 24.6, 28.1 us a step at 1024^2, 82, 79, 78, 79, 79 at 2048 x 2047).  64 registers,
// 32 one-warp blocks per SM.  Bound: instruction issue, and at 1024^2 the last
// wave of segments.  Measured, us a step, one-step kernel -> this: 1024^2 FP32,
// per-node porosity, 25.7 -> 24.7, 1448^2 50.3 -> 43.1, 2048 x 2047 96.0 -> 78.5 (724^2
// 10.9 -> 13.6: too few segments).  The bits of two launches of k_step.
constexpr int kMarchNodeBlocks = 32;
constexpr int kMarchNodeRows = 8;

static __global__ void __launch_bounds__(32, kMarchNodeBlocks) k_step2_node(
    const float* __restrict__ src, float* __restrict__ dst, const float* __restrict__ phi,
    float* __restrict__ mac, const __grid_constant__ NodeParams<float> P, const int nx,
    const int ny, const int64_t pitch, const int64_t plane, const int write_macros,
    const int seg_rows) {
  __shared__ float line[19][32];  // the slots of k_step2_pair
  grid_dep_wait();
  const int lane = threadIdx.x;
  int x = blockIdx.x * kMarchLanes + lane;
  const bool own = x < nx && (lane > 0 || x == 0) && (lane < 31 || x == nx - 1);
  x = min(x, nx - 1);
  const int side = x == 0 ? 0 : (x == nx - 1 ? 1 : -1);
  const int cx = min(max(x, 1), nx - 2);
  const bool side_strip = __any_sync(0xffffffffu, side >= 0);
  // a side node's rebuild takes the values of the node it is rebuilt from
  const int from = side == 0 ? lane + 1 : (side == 1 ? lane - 1 : lane);
  const int ya = blockIdx.y * seg_rows, yb = min(ny, ya + seg_rows);
  const int r0 = max(ya - 1, 0), r1 = min(yb, ny - 1);
  const uint32_t pi = (uint32_t)pitch;
  for (int r = r0; r <= r1; ++r) {
    const int j = r - 1;
    const bool wall_next = j == 1 || j == ny - 2;
    int y = r, cy = r == 0 ? 1 : (r == ny - 1 ? ny - 2 : r);
    float f[9], gf[5], gs[5], t[19];
    Pops<float, float>::pull(src, pitch, plane, cx, cx - 1, cx + 1, cy, cy - 1, cy + 1, 1.0f, f, gf,
                             gs);
    auto value = [&](int i) -> float& {
      return i < 9 ? f[i < 9 ? i : 0] : (i < 14 ? gf[(i - 9) % 5] : gs[(i - 9) % 5]);
    };
#pragma unroll 1
    for (int pass = 0;; ++pass) {
      const uint32_t off = (uint32_t)y * pi + x, noff = (uint32_t)cy * pi + cx;
      Macro<float> m;
      update_node<float, BC_CAVITY>(P, phi, off, noff, side >= 0 ? side : (y != cy ? 2 : -1),
                                    nullptr, nullptr, plane, nullptr, f, gf, gs, m);
      if (pass == 0) {
        const int par = r & 1;
#pragma unroll
        for (int i = 0; i < 19; ++i) {
          float& v = value(i);
          if (value_ex(i) > 0) v = __shfl_up_sync(0xffffffffu, v, 1);
          if (value_ex(i) < 0) v = __shfl_down_sync(0xffffffffu, v, 1);
          if (value_ey(i) >= 0) {
            constexpr int slot[19] = {0, 1, 9, 2, 0, 10, 11, 0, 0, 3, 4, 12, 5, 0, 6, 7, 13, 8, 0};
            float& s = line[value_ey(i) > 0 && par ? slot[i] + 5 : slot[i]][lane];
            const float o = s;
            s = v;
            v = o;
          }
        }
        if (r < r0 + 2) break;  // the line is not full yet
        if (side_strip) {
#pragma unroll
          for (int i = 0; i < 19; ++i) value(i) = __shfl_sync(0xffffffffu, value(i), from);
        }
        if (wall_next) {
#pragma unroll
          for (int i = 0; i < 19; ++i) t[i] = value(i);
        }
        y = cy = j;
        continue;
      }
      if (own) {
        if (write_macros) store_macros<float>(mac, plane, off, m);
        Pops<float, float>::store(dst, plane, off, 1.0f, f, gf, gs, 0u, 0u);
      }
      if (!wall_next || pass == 2) break;
      y = j == 1 ? 0 : ny - 1;
#pragma unroll
      for (int i = 0; i < 19; ++i) value(i) = t[i];
    }
  }
}

inline cudaError_t launch_step2_node(const LatticeArgs& a, const NodeParams<double>& Pd,
                                     cudaStream_t st) {
  const int strips = march_strips(a.nx);
  const dim3 grid(strips, (a.ny + kMarchNodeRows - 1) / kMarchNodeRows);
  if (grid.y > (unsigned)kMaxGridY) return cudaErrorInvalidValue;
  return launch_kernel(a.chained != 0, k_step2_node, grid, dim3(32), 0, st,
                       static_cast<const float*>(a.src), static_cast<float*>(a.dst),
                       static_cast<const float*>(a.phi), static_cast<float*>(a.mac),
                       cast_params<float>(Pd), a.nx, a.ny, a.pitch, a.plane, a.write_macros,
                       kMarchNodeRows);
}

}  // namespace ltne
