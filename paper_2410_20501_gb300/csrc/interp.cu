// Force from the potential and its interpolation to the particles:
//  - g = -grad(Phi) with the central stencils of Table 1, where for f(R)
//    Phi = phi + alpha (2 eps + eps^2), alpha = -(c~^2/2) fbar, i.e. the
//    force F = F_N + (c~^2/2) grad f~_R of §3.10 (the constant background part
//    of f~_R = fbar (1 + eps)^2 has no gradient);
//  - inverse TSC (§3.4) at the cell-sorted particles, optionally fused with
//    the kick v += a dt_kick and the drift x += v dt_drift on uint32
//    fixed-point positions (exact periodic wrap).
#include "pm_device.cuh"
#include "pm_internal.cuh"

namespace pmgb {

namespace {

__device__ __forceinline__ int64_t idx3(int i, int j, int k, int log2n) {
  return ((int64_t)i << (2 * log2n)) | ((int64_t)j << log2n) | k;
}

// Table 1 coefficients c_1..c_3 of the antisymmetric central derivative
// (1/h) sum_k c_k (u_{i+k} - u_{i-k}).
template <int ORDER> struct Stencil;
template <> struct Stencil<3> { static constexpr int R = 1; __device__ static float c(int k) { return 0.5f; } };
template <> struct Stencil<5> {
  static constexpr int R = 2;
  __device__ static float c(int k) { return k == 1 ? 2.0f / 3.0f : -1.0f / 12.0f; }
};
template <> struct Stencil<7> {
  static constexpr int R = 3;
  __device__ static float c(int k) { return k == 1 ? 0.75f : (k == 2 ? -0.15f : 1.0f / 60.0f); }
};

// A thread owns four consecutive z cells of a row and marches over a chunk of
// x planes with the 2R + 1 potential runs around its plane in registers, so a
// plane step loads one new run, the 2R rows beside it and the runs on either
// side in z (16 bytes each, all in flight together; the CTA's rows share them
// through L1) and writes three runs.  Bound by HBM and L2: 16 bytes a cell.
// 256^3, order 7: 166 -> 65 us, 512^3 order 5: 0.92 -> 0.35 ms against planes staged in shared
// memory with two barriers each.
constexpr int GNT = 256;

template <int ORDER, bool FR>
__global__ void __launch_bounds__(GNT) k_gradient(const float* __restrict__ phi, const float* __restrict__ eps,
                                                  float alpha, float* __restrict__ g, int log2n, float inv_h, int chunk,
                                                  int nh) {
  pdl_entry();
  constexpr int R = Stencil<ORDER>::R, W = 2 * R + 1;
  const int m = (1 << log2n) - 1, lq = log2n - 2;
  const int64_t N = (int64_t)1 << (3 * log2n);
  const uint32_t t = blockIdx.x * GNT + threadIdx.x;          // run of the plane
  if (t >= 1u << (2 * log2n - 2)) return;
  phi += (int64_t)blockIdx.z * N;              // the box of a batched launch
  if (FR) eps += (int64_t)blockIdx.z * N;
  g += (int64_t)blockIdx.z * 3 * N;
  const int j = (int)(t >> lq), k = (int)(t & ((1 << lq) - 1)) << 2, x0 = blockIdx.y * chunk;
  auto run = [&](int x, int y, int z) -> float4 {
    const int64_t c = idx3(x & m, y & m, z & m, log2n);
    float4 v = __ldg(reinterpret_cast<const float4*>(phi + c));
    if (FR) {
      const float4 e = __ldg(reinterpret_cast<const float4*>(eps + c));
      auto both = [&](float p, float q) {
        return fmaf(alpha, nh == 2 ? q * fmaf(q, 3.0f + q, 3.0f) : q * (2.0f + q), p);
      };
      v = make_float4(both(v.x, e.x), both(v.y, e.y), both(v.z, e.z), both(v.w, e.w));
    }
    return v;
  };
  float4 P[W];   // planes x - R .. x + R
#pragma unroll
  for (int q = 0; q < W - 1; ++q) P[q + 1] = run(x0 - R + q, j, k);
  for (int x = x0; x < x0 + chunk; ++x) {
#pragma unroll
    for (int q = 0; q < W - 1; ++q) P[q] = P[q + 1];
    P[W - 1] = run(x + R, j, k);
    const float4 left = run(x, j, k - 4), right = run(x, j, k + 4);
    float4 yp[R], ym[R];
#pragma unroll
    for (int q = 0; q < R; ++q) {
      yp[q] = run(x, j + q + 1, k);
      ym[q] = run(x, j - q - 1, k);
    }
    const float zr[12] = {left.x, left.y, left.z, left.w, P[R].x, P[R].y, P[R].z, P[R].w,
                          right.x, right.y, right.z, right.w};
    auto at = [](const float4& v, int i) { return i == 0 ? v.x : i == 1 ? v.y : i == 2 ? v.z : v.w; };
    float o[3][4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      float gx = 0.0f, gy = 0.0f, gz = 0.0f;
#pragma unroll
      for (int q = R; q >= 1; --q) {
        const float w = Stencil<ORDER>::c(q);
        gx = fmaf(w, at(P[R + q], i) - at(P[R - q], i), gx);
        gy = fmaf(w, at(yp[q - 1], i) - at(ym[q - 1], i), gy);
        gz = fmaf(w, zr[4 + i + q] - zr[4 + i - q], gz);
      }
      o[0][i] = -gx * inv_h;
      o[1][i] = -gy * inv_h;
      o[2][i] = -gz * inv_h;
    }
#pragma unroll
    for (int d = 0; d < 3; ++d)
      *reinterpret_cast<float4*>(g + d * N + idx3(x, j, k, log2n)) = make_float4(o[d][0], o[d][1], o[d][2], o[d][3]);
  }
}

// Inverse TSC; mode 1 also kicks and drifts.  Particles are read in cell
// order (Xs, Vs) and written in the same order (Xo, Vo).
template <bool MAXES>
__global__ void __launch_bounds__(256) k_interp_kdk(const float* __restrict__ g, const uint32_t* __restrict__ Xs,
                                                    const float* __restrict__ Vs,
                                                    const uint32_t* __restrict__ ids_in, int64_t np, int log2n,
                                                    float* __restrict__ acc, uint32_t* __restrict__ Xo,
                                                    float* __restrict__ Vo, uint32_t* __restrict__ ids_out,
                                                    float dt_kick, float drift_scale, int mode, int64_t np_box,
                                                    const float* __restrict__ dtk_box,
                                                    const float* __restrict__ dtd_box,
                                                    float2* __restrict__ blockmax) {
  pdl_entry();
  const int m = (1 << log2n) - 1, sh = 32 - log2n;
  const int64_t N = (int64_t)1 << (3 * log2n);
  // the box of a batched launch: its grid and its particles p0 .. p0 + np_box
  // (np stays the plane stride of the particle arrays)
  const int64_t p0 = (int64_t)blockIdx.z * np_box, p1 = p0 + np_box;
  g += (int64_t)blockIdx.z * 3 * N;
  if (dtk_box) dt_kick = __ldg(dtk_box + blockIdx.z);
  if (dtd_box) drift_scale = __ldg(dtd_box + blockIdx.z) * 4294967296.0f;
  float amax = 0.0f, vmax = 0.0f;   // largest |a| and |v after the kick| of this thread
  for (int64_t p = p0 + blockIdx.x * (int64_t)blockDim.x + threadIdx.x; p < p1;
       p += (int64_t)gridDim.x * blockDim.x) {
    const uint32_t x = __ldg(Xs + p), y = __ldg(Xs + np + p), z = __ldg(Xs + 2 * np + p);
    float wx[3], wy[3], wz[3];
    tsc_weights(cell_offset(x, log2n), wx);
    tsc_weights(cell_offset(y, log2n), wy);
    tsc_weights(cell_offset(z, log2n), wz);
    const int ix = (int)(x >> sh), iy = (int)(y >> sh), iz = (int)(z >> sh);
    float ax = 0.0f, ay = 0.0f, az = 0.0f;
#pragma unroll
    for (int ox = 0; ox < 3; ++ox) {
      const int ci = (ix + ox - 1) & m;
#pragma unroll
      for (int oy = 0; oy < 3; ++oy) {
        const int cj = (iy + oy - 1) & m;
        const float wxy = wx[ox] * wy[oy];
#pragma unroll
        for (int oz = 0; oz < 3; ++oz) {
          const int64_t c = idx3(ci, cj, (iz + oz - 1) & m, log2n);
          const float w = wxy * wz[oz];
          ax = fmaf(w, __ldg(g + c), ax);
          ay = fmaf(w, __ldg(g + N + c), ay);
          az = fmaf(w, __ldg(g + 2 * N + c), az);
        }
      }
    }
    if (acc) {
      acc[p] = ax;
      acc[np + p] = ay;
      acc[2 * np + p] = az;
    }
    if (MAXES) amax = fmaxf(amax, sqrtf(fmaf(ax, ax, fmaf(ay, ay, az * az))));
    if (mode == 1) {
      const float vx = fmaf(ax, dt_kick, __ldg(Vs + p));
      const float vy = fmaf(ay, dt_kick, __ldg(Vs + np + p));
      const float vz = fmaf(az, dt_kick, __ldg(Vs + 2 * np + p));
      Vo[p] = vx;
      Vo[np + p] = vy;
      Vo[2 * np + p] = vz;
      if (MAXES) vmax = fmaxf(vmax, sqrtf(fmaf(vx, vx, fmaf(vy, vy, vz * vz))));
      Xo[p] = x + (uint32_t)__float2int_rn(vx * drift_scale);
      Xo[np + p] = y + (uint32_t)__float2int_rn(vy * drift_scale);
      Xo[2 * np + p] = z + (uint32_t)__float2int_rn(vz * drift_scale);
      if (ids_out) ids_out[p] = __ldg(ids_in + p);
    }
  }
  if (MAXES) {   // block maxima (non-negative floats order like their bit patterns)
    __shared__ unsigned wa[8], wv[8];
    const unsigned ua = __reduce_max_sync(0xffffffffu, __float_as_uint(amax));
    const unsigned uv = __reduce_max_sync(0xffffffffu, __float_as_uint(vmax));
    if ((threadIdx.x & 31) == 0) {
      wa[threadIdx.x >> 5] = ua;
      wv[threadIdx.x >> 5] = uv;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
      unsigned ma = 0, mv = 0;
      for (int w = 0; w < (int)(blockDim.x >> 5); ++w) {
        ma = max(ma, wa[w]);
        mv = max(mv, wv[w]);
      }
      blockmax[(int64_t)blockIdx.z * gridDim.x + blockIdx.x] = make_float2(__uint_as_float(ma), __uint_as_float(mv));
    }
  }
}

// How many blocks of 4 x 4 rows of cells (columns along z) the warp's particles with
// cells (ix, iy, .) touch: few in cell order and on a displaced lattice, whose particles
// change rows all the time but stay near each other, so that L1 holds what they look
// up; nearly 32 in random order.
__device__ __forceinline__ int row_blocks(uint32_t ix, uint32_t iy) {
  const unsigned same = __match_any_sync(0xffffffffu, (ix >> 2) << 16 | iy >> 2);
  return __popc(__ballot_sync(0xffffffffu, (same & ((1u << (threadIdx.x & 31)) - 1u)) == 0u));
}
// Up to this many, the particles of a warp look up their cells one by one: a lattice
// displaced by one cell (rms, each particle on its own; 3.6 blocks) is 1.4 to 1.7 times as
// fast so, one displaced by three (10.8) half as fast.
constexpr int kNearBlocks = 7;

// A particle's cell and weights.
struct PointWeights {
  float wx[3], wy[3], wz[3];
  int ix, iy, iz;
  __device__ __forceinline__ PointWeights(uint32_t x, uint32_t y, uint32_t z, int log2n) {
    tsc_weights(cell_offset(x, log2n), wx);
    tsc_weights(cell_offset(y, log2n), wy);
    tsc_weights(cell_offset(z, log2n), wz);
    const int sh = 32 - log2n;
    ix = (int)(x >> sh);
    iy = (int)(y >> sh);
    iz = (int)(z >> sh);
  }
};
__device__ __forceinline__ uint32_t box_cell(int i, int j, int k, int log2n) {   // offset inside one box (below 2^30)
  return (uint32_t)i << (2 * log2n) | (uint32_t)j << log2n | (uint32_t)k;
}
// The sums of k_interp_kdk from the three planes, cell by cell.
__device__ __forceinline__ void gather_cells(const float* __restrict__ g, const PointWeights& w, int log2n, float (&a)[3]) {
  const int m = (1 << log2n) - 1;
  const int64_t N = (int64_t)1 << (3 * log2n);
#pragma unroll
  for (int ox = 0; ox < 3; ++ox) {
#pragma unroll
    for (int oy = 0; oy < 3; ++oy) {
      const float wxy = w.wx[ox] * w.wy[oy];
#pragma unroll
      for (int oz = 0; oz < 3; ++oz) {
        const uint32_t c = box_cell((w.ix + ox - 1) & m, (w.iy + oy - 1) & m, (w.iz + oz - 1) & m, log2n);
        const float wc = wxy * w.wz[oz];
#pragma unroll
        for (int d = 0; d < 3; ++d) a[d] = fmaf(wc, __ldg(g + d * N + c), a[d]);
      }
    }
  }
}

// Inverse TSC at particles in any order: the sums of k_interp_kdk in the same order
// (bitwise the same).  A warp whose particles are near each other looks up cell by cell
// (its lanes share lines); one whose particles are scattered is bound by the line
// lookups of L1, one per load and lane, and takes the three z cells of a row and
// component in the aligned 16 bytes that hold the first and, where they go on, the
// next 8: 40 lookups a particle instead of 81.
//
// 48 registers (five CTAs an SM): at 64 dense cell-ordered particles are up to 6%
// slower, at 40 sparse ones up to 25%.  Against all warps cell by cell: 262144 particles
// in cell order on 128^3 13.4 -> 12.3 us, 10^7 on 256^3 232 -> 224; in random order 64 ->
// 34 and 3410 -> 3254; 256^3 on a lattice displaced by 0.3, 1 and 3 cells 429 -> 413, 983 ->
// 979, 3176 -> 1706 us.
__global__ void __launch_bounds__(256, 5) k_interp_points(const float* __restrict__ g, const uint32_t* __restrict__ Xs,
                                                          int64_t np, int log2n, float* __restrict__ acc) {
  pdl_entry();
  const int m = (1 << log2n) - 1;
  const int64_t N = (int64_t)1 << (3 * log2n);
  const int64_t p = blockIdx.x * (int64_t)256 + threadIdx.x;
  const bool live = p < np;
  const uint32_t x = live ? __ldg(Xs + p) : 0u, y = live ? __ldg(Xs + np + p) : 0u, z = live ? __ldg(Xs + 2 * np + p) : 0u;
  const PointWeights w(x, y, z, log2n);
  const bool near = row_blocks(w.ix, w.iy) <= kNearBlocks;   // the same for the whole warp
  if (!live) return;
  float a[3] = {0.0f, 0.0f, 0.0f};
  if (near) {
    gather_cells(g, w, log2n, a);
  } else {
    const int z0 = (w.iz - 1) & m, k0 = z0 & ~3, k1 = (k0 + 4) & m;
    const bool two = (z0 & 3) >= 2, odd = z0 & 1;   // the row's cells are z0 & 3 and the two after it
#pragma unroll
    for (int ox = 0; ox < 3; ++ox) {
#pragma unroll
      for (int oy = 0; oy < 3; ++oy) {
        const float wxy = w.wx[ox] * w.wy[oy];
        const float w0 = wxy * w.wz[0], w1 = wxy * w.wz[1], w2 = wxy * w.wz[2];
        const uint32_t row = box_cell((w.ix + ox - 1) & m, (w.iy + oy - 1) & m, 0, log2n);
#pragma unroll
        for (int d = 0; d < 3; ++d) {
          const float* r = g + d * N + row;
          const float4 u = __ldg(reinterpret_cast<const float4*>(r + k0));
          float2 v = make_float2(0.0f, 0.0f);
          if (two) v = __ldg(reinterpret_cast<const float2*>(r + k1));
          const float c0 = two ? u.z : u.x, c1 = two ? u.w : u.y, c2 = two ? v.x : u.z, c3 = two ? v.y : u.w;
          a[d] = fmaf(w0, odd ? c1 : c0, a[d]);
          a[d] = fmaf(w1, odd ? c2 : c1, a[d]);
          a[d] = fmaf(w2, odd ? c3 : c2, a[d]);
        }
      }
    }
  }
#pragma unroll
  for (int d = 0; d < 3; ++d) acc[d * np + p] = a[d];
}

// Group k of K of 32 neighbouring particles, spread evenly over the particles (np >= 32):
// this lane's x and y cells.
__device__ __forceinline__ uint2 sample_cells(const uint32_t* __restrict__ Xs, int64_t np, int log2n, int k, int K) {
  const int64_t p = (np - 32) * k / (K - 1) + (threadIdx.x & 31);
  return make_uint2(__ldg(Xs + p) >> (32 - log2n), __ldg(Xs + np + p) >> (32 - log2n));
}

// *flag = 1 if 32 neighbouring particles change their row of cells more than `rows`
// times (a sample's mean; one block).
__global__ void __launch_bounds__(1024) k_order_sample(const uint32_t* __restrict__ Xs, int64_t np, int log2n,
                                                       float rows, int* __restrict__ flag) {
  pdl_entry();
  __shared__ int total;
  constexpr int PER_WARP = 8, GROUPS = 32 * PER_WARP;
  const int lane = threadIdx.x & 31;
  if (threadIdx.x == 0) total = 0;
  __syncthreads();
  uint2 c[PER_WARP];
#pragma unroll
  for (int k = 0; k < PER_WARP; ++k) c[k] = sample_cells(Xs, np, log2n, (threadIdx.x >> 5) * PER_WARP + k, GROUPS);
  int sum = 0;
#pragma unroll
  for (int k = 0; k < PER_WARP; ++k) {
    const uint32_t row = (c[k].x << log2n) | c[k].y, prev = __shfl_up_sync(0xffffffffu, row, 1);
    sum += __popc(__ballot_sync(0xffffffffu, lane == 0 || row != prev));
  }
  if (lane == 0) atomicAdd(&total, sum);   // integers: any order
  __syncthreads();
  if (threadIdx.x == 0) *flag = (float)total / GROUPS > rows;
}

// Cells of the force field as float4 (g_x, g_y, g_z, 0), four at a time a thread, if 32
// neighbouring particles touch more than `blocks` blocks of rows (row_blocks, a
// sample's mean), which goes to *flag.  Every block takes the sample (8 loads a thread,
// one wave of blocks, all deciding the same): as a kernel before this one it costs the
// particles that need no packing a launch more.
constexpr int kPackBlocks = 4 * 152;
__global__ void __launch_bounds__(256, 4) k_pack_force(const float* __restrict__ g, float4* __restrict__ out, int64_t N,
                                                       const uint32_t* __restrict__ Xs, int64_t np, int log2n,
                                                       float blocks, int* __restrict__ flag) {
  pdl_entry();
  __shared__ int total;
  constexpr int PER_WARP = 4, GROUPS = 8 * PER_WARP;
  if (threadIdx.x == 0) total = 0;
  __syncthreads();
  uint2 cell[PER_WARP];
#pragma unroll
  for (int k = 0; k < PER_WARP; ++k) cell[k] = sample_cells(Xs, np, log2n, (threadIdx.x >> 5) * PER_WARP + k, GROUPS);
  int sum = 0;
#pragma unroll
  for (int k = 0; k < PER_WARP; ++k) sum += row_blocks(cell[k].x, cell[k].y);
  if ((threadIdx.x & 31) == 0) atomicAdd(&total, sum);   // integers: any order
  __syncthreads();
  const bool scattered = (float)total / GROUPS > blocks;
  if (blockIdx.x == 0 && threadIdx.x == 0) *flag = scattered;
  if (!scattered) return;
  for (int64_t c = 4 * (blockIdx.x * (int64_t)256 + threadIdx.x); c < N; c += 4 * (int64_t)gridDim.x * 256) {
    const float4 x = __ldg(reinterpret_cast<const float4*>(g + c));
    const float4 y = __ldg(reinterpret_cast<const float4*>(g + N + c));
    const float4 z = __ldg(reinterpret_cast<const float4*>(g + 2 * N + c));
    out[c] = make_float4(x.x, y.x, z.x, 0.0f);
    out[c + 1] = make_float4(x.y, y.y, z.y, 0.0f);
    out[c + 2] = make_float4(x.z, y.z, z.z, 0.0f);
    out[c + 3] = make_float4(x.w, y.w, z.w, 0.0f);
  }
}

// Two neighbouring packed cells (32 bytes, aligned) in one load.
struct CellPair {
  float4 a, b;
};
__device__ __forceinline__ CellPair load_pair(const float4* p) {
  CellPair v;
  asm("ld.global.nc.v8.f32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
      : "=f"(v.a.x), "=f"(v.a.y), "=f"(v.a.z), "=f"(v.a.w), "=f"(v.b.x), "=f"(v.b.y), "=f"(v.b.z), "=f"(v.b.w)
      : "l"(p));
  return v;
}

// Inverse TSC from the packed field if *flag, else from the three planes, cell by cell:
// the sums of k_interp_kdk in the same order (bitwise the same).  The three z cells of a
// row come in two aligned 32-byte loads: 18 lookups and sectors a particle against 40
// and 34 of k_interp_points.  Where the packed field is larger than L2 that is bound by
// HBM (10^7 random on 256^3: 9.8 GB read in 1.51 ms, 0.96 of the copy rate).
//
// 40 registers (six CTAs an SM), which cell-ordered particles gain by; with the rows in
// a loop that is not unrolled the packed form needs no more and is as fast as with 64
// (10^7 random on 256^3 1.51 ms, in cell order 206 us against 224).
__global__ void __launch_bounds__(256, 6) k_interp_packed(const float4* __restrict__ gp, const float* __restrict__ g,
                                                          const uint32_t* __restrict__ Xs, int64_t np, int log2n,
                                                          float* __restrict__ acc, const int* __restrict__ flag) {
  pdl_entry();
  const int m = (1 << log2n) - 1;
  const int64_t p = blockIdx.x * (int64_t)256 + threadIdx.x;
  if (p >= np) return;
  const bool packed = *flag != 0;
  const PointWeights w(__ldg(Xs + p), __ldg(Xs + np + p), __ldg(Xs + 2 * np + p), log2n);
  float a[3] = {0.0f, 0.0f, 0.0f};
  if (packed) {
    const int z0 = (w.iz - 1) & m, k0 = z0 & ~1, k1 = (k0 + 2) & m;
    const bool odd = z0 & 1;                     // the row's cells are b, a, b of two pairs, else a, b, a
#pragma unroll 1
    for (int o = 0; o < 9; ++o) {
      const int ox = o / 3, oy = o - 3 * ox;
      const float wx = ox == 0 ? w.wx[0] : ox == 1 ? w.wx[1] : w.wx[2];
      const float wy = oy == 0 ? w.wy[0] : oy == 1 ? w.wy[1] : w.wy[2];
      const float4* row = gp + box_cell((w.ix + ox - 1) & m, (w.iy + oy - 1) & m, 0, log2n);
      const CellPair u = load_pair(row + k0), v = load_pair(row + k1);
      const float wxy = wx * wy;
      const float w0 = wxy * w.wz[0], w1 = wxy * w.wz[1], w2 = wxy * w.wz[2];
      a[0] = fmaf(w0, odd ? u.b.x : u.a.x, a[0]);
      a[1] = fmaf(w0, odd ? u.b.y : u.a.y, a[1]);
      a[2] = fmaf(w0, odd ? u.b.z : u.a.z, a[2]);
      a[0] = fmaf(w1, odd ? v.a.x : u.b.x, a[0]);
      a[1] = fmaf(w1, odd ? v.a.y : u.b.y, a[1]);
      a[2] = fmaf(w1, odd ? v.a.z : u.b.z, a[2]);
      a[0] = fmaf(w2, odd ? v.b.x : v.a.x, a[0]);
      a[1] = fmaf(w2, odd ? v.b.y : v.a.y, a[1]);
      a[2] = fmaf(w2, odd ? v.b.z : v.a.z, a[2]);
    }
  } else {
    gather_cells(g, w, log2n, a);
  }
#pragma unroll
  for (int d = 0; d < 3; ++d) acc[d * np + p] = a[d];
}

// Force and inverse TSC + kick-drift-kick in one pass for cell-sorted
// particles (n >= 32): a CTA owns a IT_Y x IT_Z column of cells and a chunk
// of x planes and walks the planes in order.  The force planes around plane
// x (with a one-cell halo in y and z) are computed in shared memory from the
// potential (the gradient of k_gradient, same arithmetic), so the force field
// never goes through HBM; the particles of the column's cells on plane x are
// IT_Y contiguous runs of the sorted arrays (one per row), which the threads
// take in flat order.  Every particle then reads its 27 x 3 force values
// from shared memory at fixed offsets from its cell, in the same order and
// with the same operations as k_interp_kdk (bitwise the same result).
//
// Shared memory's wavefronts bound it (81 of the 150 a warp of particles takes
// are the force values themselves, 35 bank conflicts of scattered cells, 21 the
// planes; the pipe is 80% busy), and what is left is latency: the thread's next
// particle and the next plane's runs are in flight while the force plane is
// computed and the particles before it are summed.  With the f(R) potential's
// second field there are no registers for that at four CTAs an SM (the particle
// ahead and the paired sums took 460 us there against 443), so it loads each
// particle in turn.  256^3: 402 -> 386 us, clustered 445 -> 431, with maxima
// 454 -> 434; f(R) 512^3 3.09 -> 2.99 ms.
constexpr int IT_Y = 16, IT_Z = 32, IE_Y = IT_Y + 2, IE_Z = IT_Z + 2, I_PL = IE_Y * IE_Z, I_THREADS = 256;
// One warp: the runs of the column's rows on plane q (start of each row's
// particles, flat prefix of the run lengths) from the cell starts `v` that its
// lanes loaded (column_start).
__device__ __forceinline__ uint32_t column_start(const uint32_t* __restrict__ cellstart, int q, int y0, int z0,
                                                 int log2n) {
  const int lane = threadIdx.x & 31, m = (1 << log2n) - 1, j = lane & (IT_Y - 1);
  const int64_t row = ((int64_t)(q & m) << (2 * log2n)) | ((int64_t)(y0 + j) << log2n);
  return __ldg(cellstart + row + z0 + (lane < IT_Y ? 0 : IT_Z));
}
__device__ __forceinline__ void column_runs(uint32_t v, uint32_t* start, uint32_t* pre) {
  const int lane = threadIdx.x & 31, j = lane & (IT_Y - 1);
  const uint32_t end = __shfl_down_sync(0xffffffffu, v, IT_Y);
  uint32_t incl = lane < IT_Y ? end - v : 0u;
#pragma unroll
  for (int o = 1; o < IT_Y; o <<= 1) {
    const uint32_t y = __shfl_up_sync(0xffffffffu, incl, o);
    if (j >= o) incl += y;
  }
  if (lane < IT_Y) {
    start[j] = v;
    pre[j + 1] = incl;
    if (j == 0) pre[0] = 0;
  }
}

// A particle on its way to column_particle: its index, position and, for a
// step, velocity.
struct ColumnParticle {
  uint32_t p, x, y, z;
  float vx, vy, vz;
};
// Loads flat particle i of the plane whose runs are st, pre.
__device__ __forceinline__ void column_load(ColumnParticle& a, uint32_t i, const uint32_t* st, const uint32_t* pre,
                                            const uint32_t* __restrict__ Xs, const float* __restrict__ Vs, int64_t np,
                                            int mode) {
  int j = 0;   // the run holding flat index i
#pragma unroll
  for (int b = IT_Y / 2; b > 0; b >>= 1)
    if (pre[j + b] <= i) j += b;
  a.p = st[j] + (i - pre[j]);
  a.x = __ldg(Xs + a.p);
  a.y = __ldg(Xs + np + a.p);
  a.z = __ldg(Xs + 2 * np + a.p);
  if (mode == 1) {
    a.vx = __ldg(Vs + a.p);
    a.vy = __ldg(Vs + np + a.p);
    a.vz = __ldg(Vs + 2 * np + a.p);
  }
}

// Inverse TSC (+ kick and drift) of one particle of a plane of a column, force
// planes x-1, x, x+1 at S2[0..2] (g_x, g_y) and Sz[0..2] (g_z), each
// [IE_Y][IE_Z], in the operations and the order of k_interp_kdk.  PAIR: the x and
// y sums in the paired float instructions.
template <bool MAXES, bool PAIR>
__device__ __forceinline__ void column_particle(const ColumnParticle& a, const float2* const S2[3],
                                                const float* const Sz[3], int y0, int z0,
                                                const uint32_t* __restrict__ ids_in, int64_t np, int log2n,
                                                float* __restrict__ acc, uint32_t* __restrict__ Xo,
                                                float* __restrict__ Vo, uint32_t* __restrict__ ids_out, float dt_kick,
                                                float drift_scale, int mode, float& amax, float& vmax) {
  const int sh = 32 - log2n;
  float wx[3], wy[3], wz[3];
  tsc_weights(cell_offset(a.x, log2n), wx);
  tsc_weights(cell_offset(a.y, log2n), wy);
  tsc_weights(cell_offset(a.z, log2n), wz);
  const int c = ((int)(a.y >> sh) - y0 + 1) * IE_Z + ((int)(a.z >> sh) - z0 + 1);
  float2 axy = make_float2(0.0f, 0.0f);
  float az = 0.0f;
#pragma unroll
  for (int ox = 0; ox < 3; ++ox) {
#pragma unroll
    for (int oy = 0; oy < 3; ++oy) {
      const float wxy = wx[ox] * wy[oy];
      const float2* r2 = S2[ox] + c + (oy - 1) * IE_Z;
      const float* rz = Sz[ox] + c + (oy - 1) * IE_Z;
      const float2 wxy2 = __fmul2_rn(make_float2(wx[ox], wx[ox]), make_float2(wy[oy], wy[oy]));
#pragma unroll
      for (int oz = 0; oz < 3; ++oz) {
        const float2 fxy = r2[oz - 1];
        if (PAIR) {
          const float2 w = __fmul2_rn(wxy2, make_float2(wz[oz], wz[oz]));
          axy = __ffma2_rn(w, fxy, axy);
          az = fmaf(w.x, rz[oz - 1], az);
        } else {
          const float w = wxy * wz[oz];
          axy.x = fmaf(w, fxy.x, axy.x);
          axy.y = fmaf(w, fxy.y, axy.y);
          az = fmaf(w, rz[oz - 1], az);
        }
      }
    }
  }
  const float ax = axy.x, ay = axy.y;
  const int64_t p = a.p;
  if (acc) {
    acc[p] = ax;
    acc[np + p] = ay;
    acc[2 * np + p] = az;
  }
  if (MAXES) amax = fmaxf(amax, sqrtf(fmaf(ax, ax, fmaf(ay, ay, az * az))));
  if (mode == 1) {
    const float vx = fmaf(ax, dt_kick, a.vx);
    const float vy = fmaf(ay, dt_kick, a.vy);
    const float vz = fmaf(az, dt_kick, a.vz);
    Vo[p] = vx;
    Vo[np + p] = vy;
    Vo[2 * np + p] = vz;
    if (MAXES) vmax = fmaxf(vmax, sqrtf(fmaf(vx, vx, fmaf(vy, vy, vz * vz))));
    Xo[p] = a.x + (uint32_t)__float2int_rn(vx * drift_scale);
    Xo[np + p] = a.y + (uint32_t)__float2int_rn(vy * drift_scale);
    Xo[2 * np + p] = a.z + (uint32_t)__float2int_rn(vz * drift_scale);
    if (ids_out) ids_out[p] = __ldg(ids_in + p);
  }
}

// Block maxima of |a| and |v| (non-negative floats order like their bit
// patterns), one float2 per block.
__device__ __forceinline__ void block_maxima(float amax, float vmax, float2* __restrict__ blockmax) {
  __shared__ unsigned wa[I_THREADS / 32], wv[I_THREADS / 32];
  const int tid = threadIdx.x;
  const unsigned ua = __reduce_max_sync(0xffffffffu, __float_as_uint(amax));
  const unsigned uv = __reduce_max_sync(0xffffffffu, __float_as_uint(vmax));
  if ((tid & 31) == 0) {
    wa[tid >> 5] = ua;
    wv[tid >> 5] = uv;
  }
  __syncthreads();
  if (tid == 0) {
    unsigned ma = 0, mv = 0;
    for (int w = 0; w < I_THREADS / 32; ++w) {
      ma = max(ma, wa[w]);
      mv = max(mv, wv[w]);
    }
    blockmax[(int64_t)blockIdx.z * gridDim.x + blockIdx.x] = make_float2(__uint_as_float(ma), __uint_as_float(mv));
  }
}

// The force planes from the potential in shared memory, then the particles.
// Per plane step u: the potential plane u (with a halo of R + 1 in y and z;
// loaded into registers one step ahead, combined with eps for f(R)) goes to a
// ring of 2R + 2 slots; after the step's one barrier the force plane u - R
// (with a one-cell halo) is computed into a ring of 4 slots while the
// particles of plane u - R - 2 are interpolated from the three force planes
// computed in the steps before.
template <int ORDER, bool FR, bool MAXES>
__global__ void __launch_bounds__(I_THREADS, 4) k_force_interp_stream(
    const float* __restrict__ phi, const float* __restrict__ eps, float alpha, int nh, float inv_h,
    const uint32_t* __restrict__ cellstart, const uint32_t* __restrict__ Xs, const float* __restrict__ Vs,
    const uint32_t* __restrict__ ids_in, int64_t np, int log2n, int chunk, int nitems, float* __restrict__ acc,
    uint32_t* __restrict__ Xo, float* __restrict__ Vo, uint32_t* __restrict__ ids_out, float dt_kick,
    float drift_scale, int mode, const float* __restrict__ dtk_box, const float* __restrict__ dtd_box,
    float2* __restrict__ blockmax) {
  pdl_entry();
  constexpr int R = Stencil<ORDER>::R, H = R + 1, PEY = IT_Y + 2 * H, PEZ = IT_Z + 2 * H, PPL = PEY * PEZ,
                PS = 2 * R + 2, PL_T = (PPL + I_THREADS - 1) / I_THREADS;
  extern __shared__ float fsm[];
  float2* Gxy = reinterpret_cast<float2*>(fsm);   // [4][IE_Y][IE_Z] (g_x, g_y)
  float* Gz = fsm + 4 * 2 * I_PL;                  // [4][IE_Y][IE_Z] g_z
  float* Ps = fsm + 4 * 3 * I_PL;                  // [PS][PEY][PEZ]
  __shared__ uint32_t s_start[2][IT_Y], s_pre[2][IT_Y + 1];
  const int n = 1 << log2n, m = n - 1;
  const int64_t N = (int64_t)1 << (3 * log2n);
  phi += (int64_t)blockIdx.z * N;   // the box of a batched launch
  if (FR) eps += (int64_t)blockIdx.z * N;
  cellstart += (int64_t)blockIdx.z * N;
  if (dtk_box) dt_kick = __ldg(dtk_box + blockIdx.z);
  if (dtd_box) drift_scale = __ldg(dtd_box + blockIdx.z) * 4294967296.0f;
  const int tiles_z = n / IT_Z, tiles = (n / IT_Y) * tiles_z;
  const int tid = threadIdx.x;
  float amax = 0.0f, vmax = 0.0f;
  for (int item = blockIdx.x; item < nitems; item += gridDim.x) {
    const int tile = item % tiles, xc = item / tiles;
    const int y0 = (tile / tiles_z) * IT_Y, z0 = (tile % tiles_z) * IT_Z;
    const int x0 = xc * chunk, x1 = x0 + chunk;
    // raw potential (and eps) of plane q at this thread's positions
    float rp[PL_T], re[PL_T];
    auto fetch = [&](int q) {
      const int64_t pb = (int64_t)(q & m) << (2 * log2n);
#pragma unroll
      for (int k = 0; k < PL_T; ++k) {
        const int e = tid + k * I_THREADS;
        if (e < PPL) {
          const int ly = e / PEZ, lz = e - ly * PEZ;
          const int64_t c = pb | ((int64_t)((y0 - H + ly) & m) << log2n) | ((z0 - H + lz) & m);
          rp[k] = __ldg(phi + c);
          if (FR) re[k] = __ldg(eps + c);
        }
      }
    };
    auto store = [&](int q) {
      float* P = Ps + (((q % PS) + PS) % PS) * PPL;
#pragma unroll
      for (int k = 0; k < PL_T; ++k) {
        const int e = tid + k * I_THREADS;
        if (e < PPL) {
          float v = rp[k];
          if (FR) {
            const float ev = re[k];
            v = fmaf(alpha, nh == 2 ? ev * fmaf(ev, 3.0f + ev, 3.0f) : ev * (2.0f + ev), v);
          }
          P[e] = v;
        }
      }
    };
    // step u: potential plane u stored, force plane u - R computed, particles
    // of plane u - R - 2 interpolated (their force planes were computed in
    // the three steps before): one barrier per step
    const int u0 = x0 - 1 - R, ulast = x1 + R + 1;
    fetch(u0);
    for (int u = u0; u <= ulast; ++u) {
      if (u <= x1 + R) store(u);
      if (u < x1 + R) fetch(u + 1);
      __syncthreads();
      const int qg = u - R;
      const int t = qg - 2;   // particle plane of this step
      // in flight while the force plane is computed: this thread's first particle
      // and, on the last warp (which gets the fewest), the next plane's runs
      const uint32_t *st = s_start[t & 1], *pre = s_pre[t & 1];
      const uint32_t total = t >= x0 && t < x1 ? pre[IT_Y] : 0u;
      ColumnParticle next;
      if (!FR && tid < total) column_load(next, tid, st, pre, Xs, Vs, np, mode);
      const bool runs = t + 1 >= x0 && t + 1 < x1 && tid >= I_THREADS - 32;
      uint32_t cs = 0;
      if (runs) cs = column_start(cellstart, t + 1, y0, z0, log2n);
      if (qg >= x0 - 1 && qg <= x1) {
        float2* G2 = Gxy + (qg & 3) * I_PL;
        float* G1 = Gz + (qg & 3) * I_PL;
        const float* Pc = Ps + (((qg % PS) + PS) % PS) * PPL;
        for (int e = tid; e < I_PL; e += I_THREADS) {
          const int ly = e / IE_Z, lz = e - ly * IE_Z;
          const int c = (ly + R) * PEZ + lz + R;   // potential position of force cell (ly - 1, lz - 1)
          float gx = 0.0f, gy = 0.0f, gz = 0.0f;
#pragma unroll
          for (int q = R; q >= 1; --q) {
            const float w = Stencil<ORDER>::c(q);
            const float* Pp = Ps + ((((qg + q) % PS) + PS) % PS) * PPL;
            const float* Pm = Ps + ((((qg - q) % PS) + PS) % PS) * PPL;
            gx = fmaf(w, Pp[c] - Pm[c], gx);
            gy = fmaf(w, Pc[c + q * PEZ] - Pc[c - q * PEZ], gy);
            gz = fmaf(w, Pc[c + q] - Pc[c - q], gz);
          }
          G2[e] = make_float2(-gx * inv_h, -gy * inv_h);
          G1[e] = -gz * inv_h;
        }
      }
      if (runs) column_runs(cs, s_start[(t + 1) & 1], s_pre[(t + 1) & 1]);
      if (total) {
        const float2* S2[3];
        const float* Sz[3];
#pragma unroll
        for (int ox = 0; ox < 3; ++ox) {
          S2[ox] = Gxy + ((t + ox - 1) & 3) * I_PL;
          Sz[ox] = Gz + ((t + ox - 1) & 3) * I_PL;
        }
        for (uint32_t i = tid; i < total; i += I_THREADS) {
          ColumnParticle cur;
          if (FR) {
            column_load(cur, i, st, pre, Xs, Vs, np, mode);
          } else {
            cur = next;
            if (i + I_THREADS < total) column_load(next, i + I_THREADS, st, pre, Xs, Vs, np, mode);
          }
          column_particle<MAXES, !FR>(cur, S2, Sz, y0, z0, ids_in, np, log2n, acc, Xo, Vo, ids_out, dt_kick, drift_scale,
                                 mode, amax, vmax);
        }
      }
    }
    __syncthreads();   // the rings and run buffers are reused by the next item
  }
  if (MAXES) block_maxima(amax, vmax, blockmax);
}

template <int ORDER>
constexpr size_t force_interp_smem() {
  return sizeof(float) * (4 * 3 * I_PL + (2 * Stencil<ORDER>::R + 2) * (IT_Y + 2 * Stencil<ORDER>::R + 2) *
                                             (IT_Z + 2 * Stencil<ORDER>::R + 2));
}

// Largest |v| of the velocity planes V [3][np]: one float2 (0, max) per block
// (float bits of non-negative values order like unsigned integers).
__global__ void __launch_bounds__(256) k_speed_max(const float* __restrict__ V, int64_t np,
                                                   float2* __restrict__ blockmax) {
  pdl_entry();
  __shared__ unsigned wv[8];
  unsigned mv = 0;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < np; i += (int64_t)gridDim.x * blockDim.x) {
    const float vx = __ldg(V + i), vy = __ldg(V + np + i), vz = __ldg(V + 2 * np + i);
    mv = max(mv, __float_as_uint(sqrtf(vx * vx + vy * vy + vz * vz)));
  }
  mv = __reduce_max_sync(0xffffffffu, mv);
  if ((threadIdx.x & 31) == 0) wv[threadIdx.x >> 5] = mv;
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int w = 0; w < 8; ++w) mv = max(mv, wv[w]);
    blockmax[blockIdx.x] = make_float2(0.0f, __uint_as_float(mv));
  }
}

// Maximum over count float2 pairs, per component, into out[0], out[1]
// (float64); one block.
__global__ void __launch_bounds__(1024) k_max_pairs(const float2* __restrict__ v, int64_t count,
                                                    double* __restrict__ out) {
  pdl_entry();
  __shared__ unsigned wa[32], wv[32];
  unsigned ma = 0, mv = 0;
  for (int64_t i = threadIdx.x; i < count; i += blockDim.x) {
    const float2 x = v[i];
    ma = max(ma, __float_as_uint(x.x));
    mv = max(mv, __float_as_uint(x.y));
  }
  ma = __reduce_max_sync(0xffffffffu, ma);
  mv = __reduce_max_sync(0xffffffffu, mv);
  if ((threadIdx.x & 31) == 0) {
    wa[threadIdx.x >> 5] = ma;
    wv[threadIdx.x >> 5] = mv;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int w = 0; w < (int)(blockDim.x >> 5); ++w) {
      ma = max(ma, wa[w]);
      mv = max(mv, wv[w]);
    }
    out[0] = __uint_as_float(ma);
    out[1] = __uint_as_float(mv);
  }
}

template <int ORDER>
pm_status launch_grad(const float* phi, const float* eps, float alpha, float* g, int n, cudaStream_t s, int B, int nh) {
  const int64_t N = (int64_t)n * n * n;
  const double bytes = ((eps ? 8.0 : 4.0) * N + 12.0 * N) * B;
  const unsigned gx = grid_for((int64_t)n * n / 4, GNT);
  int chunk = n < 16 ? n : 16;   // planes a thread marches over, as many as leave four CTAs per SM
  while (chunk > 1 && (int64_t)gx * (n / chunk) * B < 4 * 152) chunk >>= 1;
  const dim3 grid(gx, (unsigned)(n / chunk), (unsigned)B);
  if (eps)
    PM_LAUNCH(K_GRADIENT, bytes, (k_gradient<ORDER, true>), grid, GNT, 0, s, phi, eps, alpha, g, ilog2(n), (float)n,
              chunk, nh);
  else
    PM_LAUNCH(K_GRADIENT, bytes, (k_gradient<ORDER, false>), grid, GNT, 0, s, phi, eps, alpha, g, ilog2(n), (float)n,
              chunk, nh);
  return launch_status();
}

}  // namespace

pm_status gradient_launch(const float* phi, const float* eps, float alpha, float* g, int n, int order, cudaStream_t s,
                          int batch, int nh) {
  if (order == 3) return launch_grad<3>(phi, eps, alpha, g, n, s, batch, nh);
  if (order == 5) return launch_grad<5>(phi, eps, alpha, g, n, s, batch, nh);
  if (order == 7) return launch_grad<7>(phi, eps, alpha, g, n, s, batch, nh);
  return PM_EINVAL;
}

pm_status order_sample(const uint32_t* X, int64_t np, int n, float rows, int* flag, cudaStream_t s) {
  if (np < 32) return PM_EINVAL;
  PM_LAUNCH_EARLY(K_INTERP, 0.0, k_order_sample, 1, 1024, 0, s, X, np, ilog2(n), rows, flag);
  return launch_status();
}

// The field is packed where that pays: from 5 blocks of rows in 32 neighbouring
// particles on, more where the particles are few for the cells to be packed.  256^3 on a
// lattice displaced by d cells (rms), planes / packed: d = 0.3 (1.9 blocks) 415 / 590 us, 1
// (3.6) 960 / 990, 2 (7) 1960 / 1048; 128^3 56 / 84, 108 / 126, 199 / 140.
pm_status interp_packed_launch(const float* g, const uint32_t* X, int64_t np, int n, float* acc, int* flag,
                               float4* packed, cudaStream_t s) {
  if (np < 32) return PM_EINVAL;
  const int64_t N = (int64_t)n * n * n;
  const float blocks = 5.0f + (float)N / (float)np;
  PM_LAUNCH_EARLY(K_INTERP, 0.0, k_pack_force, grid_for(N / 4, 256, kPackBlocks), 256, 0, s, g, packed, N, X, np,
                  ilog2(n), blocks, flag);
  PM_LAUNCH(K_INTERP, 12.0 * N + 24.0 * np, k_interp_packed, grid_for(np, 256), 256, 0, s, packed, g, X, np, ilog2(n),
            acc, flag);
  return launch_status();
}

template <int ORDER>
pm_status launch_force_interp(const float* phi, const float* eps, float alpha, int nh, const uint32_t* cellstart,
                              const uint32_t* Xs, const float* Vs, const uint32_t* ids_in, int64_t np, int n,
                              float* acc, uint32_t* Xo, float* Vo, uint32_t* ids_out, float dt_kick,
                              float drift_scale, int mode, cudaStream_t s, const Batch& bt, float2* blockmax,
                              int64_t* nblocks) {
  constexpr size_t smem = force_interp_smem<ORDER>();
  PM_TRY(smem_attr(k_force_interp_stream<ORDER, false, false>, smem));
  PM_TRY(smem_attr(k_force_interp_stream<ORDER, false, true>, smem));
  PM_TRY(smem_attr(k_force_interp_stream<ORDER, true, false>, smem));
  PM_TRY(smem_attr(k_force_interp_stream<ORDER, true, true>, smem));
  const int tiles = (n / IT_Y) * (n / IT_Z);
  // A chunk repeats 2 R + 2 planes of run-up, so the longest that gives every SM
  // four times its four resident CTAs, down to 16 planes; a grid that then still
  // leaves CTA slots empty takes shorter ones, since a column marched by one CTA
  // is a chain of plane latencies.  Force pass at 16 -> 2 planes: 32^3 53 -> 14 us,
  // 64^3 59 -> 18; 16 -> 4: 128^3 84 -> 66 (2: 73); 256^3 400 at 32, 16 and 8, 425 at 4.
  int chunk = n;
  while (chunk > 16 && (int64_t)tiles * (n / chunk) * bt.B < 16 * 152) chunk >>= 1;
  while (bt.B == 1 && chunk > 2 && (int64_t)tiles * (n / chunk) < 4 * 152) chunk >>= 1;
  if (bt.B > 1) {   // batches: the x chunk is tuned (each particle's force is chunk-independent)
    int cand[3], nc = 0;
    for (int c = 16; c <= 64 && c <= n; c *= 2) cand[nc++] = c;
    chunk = tune_begin(TUNE_FORCE_CHUNK, n, bt.B, ORDER, cand, nc, chunk, s);
  }
  const int nitems = tiles * (n / chunk);
  const dim3 grid((unsigned)nitems, 1, (unsigned)bt.B);
  *nblocks = (int64_t)grid.x * grid.z;
  const double N = (double)n * n * n * bt.B;
  const double bytes = (eps ? 8.0 : 4.0) * N + np * (12.0 + (mode ? 36.0 : 0.0) + (acc ? 12.0 : 0.0) +
                                                      (ids_out ? 8.0 : 0.0));
#define PM_FI(FRB, MX)                                                                                          \
  PM_LAUNCH(K_INTERP, bytes, (k_force_interp_stream<ORDER, FRB, MX>), grid, I_THREADS, smem, s, phi, eps, alpha, nh, \
            (float)n, cellstart, Xs, Vs, ids_in, np, ilog2(n), chunk, nitems, acc, Xo, Vo, ids_out, dt_kick,       \
            drift_scale, mode, bt.dt_kick, bt.dt_drift, blockmax)
  if (eps) {
    if (blockmax) PM_FI(true, true); else PM_FI(true, false);
  } else {
    if (blockmax) PM_FI(false, true); else PM_FI(false, false);
  }
#undef PM_FI
  if (bt.B > 1) tune_end(s);
  return launch_status();
}

pm_status max_speed_launch(const float* V, int64_t np, float2* blockmax, double* max_out, cudaStream_t s) {
  const unsigned nb = grid_for(np, 256, 152 * 16);
  PM_LAUNCH(K_REDUCE, 12.0 * np, k_speed_max, nb, 256, 0, s, V, np, blockmax);
  PM_LAUNCH(K_REDUCE, 8.0 * nb, k_max_pairs, 1, 1024, 0, s, blockmax, (int64_t)nb, max_out);
  return launch_status();
}

pm_status force_interp_launch(const float* phi, const float* eps, float alpha, int nh, int order,
                              const uint32_t* cellstart, const uint32_t* Xs, const float* Vs, const uint32_t* ids_in,
                              int64_t np, int n, float* acc, uint32_t* Xo, float* Vo, uint32_t* ids_out,
                              float dt_kick, float dt_drift, int mode, cudaStream_t s, const Batch& bt,
                              float2* blockmax, double* max_out) {
  if (np == 0) return PM_OK;
  if (n < 32 || !cellstart) return PM_EINVAL;
  const float drift_scale = (float)((double)dt_drift * 4294967296.0);
  if (!max_out) blockmax = nullptr;
  int64_t nblocks = 0;
  pm_status r = PM_EINVAL;
  if (order == 3)
    r = launch_force_interp<3>(phi, eps, alpha, nh, cellstart, Xs, Vs, ids_in, np, n, acc, Xo, Vo, ids_out, dt_kick,
                               drift_scale, mode, s, bt, blockmax, &nblocks);
  else if (order == 5)
    r = launch_force_interp<5>(phi, eps, alpha, nh, cellstart, Xs, Vs, ids_in, np, n, acc, Xo, Vo, ids_out, dt_kick,
                               drift_scale, mode, s, bt, blockmax, &nblocks);
  else if (order == 7)
    r = launch_force_interp<7>(phi, eps, alpha, nh, cellstart, Xs, Vs, ids_in, np, n, acc, Xo, Vo, ids_out, dt_kick,
                               drift_scale, mode, s, bt, blockmax, &nblocks);
  if (r != PM_OK) return r;
  if (blockmax) PM_LAUNCH(K_REDUCE, 8.0 * nblocks, k_max_pairs, 1, 1024, 0, s, blockmax, nblocks, max_out);
  return launch_status();
}

pm_status interp_launch(const float* g, const uint32_t* Xs, const float* Vs, const uint32_t* ids_in, int64_t np,
                        int n, float* acc, uint32_t* Xo, float* Vo, uint32_t* ids_out, float dt_kick,
                        float dt_drift, int mode, cudaStream_t s, const Batch& bt,
                        float2* blockmax, double* max_out) {
  if (np == 0) return PM_OK;
  const float drift_scale = (float)((double)dt_drift * 4294967296.0);
  const double bytes = 12.0 * n * n * (double)n * bt.B +
                       np * (12.0 + (mode ? 36.0 : 0.0) + (acc ? 12.0 : 0.0) + (ids_out ? 8.0 : 0.0));
  const int64_t np_box = bt.B > 1 ? bt.np_box : np;
  const dim3 grid(grid_for(np_box, 256), 1, (unsigned)bt.B);
  if (!max_out) blockmax = nullptr;
  if (mode == 0 && bt.B == 1 && !blockmax) {
    PM_LAUNCH(K_INTERP, bytes, k_interp_points, grid.x, 256, 0, s, g, Xs, np, ilog2(n), acc);
    return launch_status();
  }
#define PM_INTERP(MX)                                                                                               \
  PM_LAUNCH(K_INTERP, bytes, k_interp_kdk<MX>, grid, 256, 0, s, g, Xs, Vs, ids_in, np, ilog2(n), acc, Xo, Vo, ids_out, \
            dt_kick, drift_scale, mode, np_box, bt.dt_kick, bt.dt_drift, blockmax)
  if (blockmax) PM_INTERP(true); else PM_INTERP(false);
#undef PM_INTERP
  if (blockmax) {
    const int64_t nb = (int64_t)grid.x * grid.z;
    PM_LAUNCH(K_REDUCE, 8.0 * nb, k_max_pairs, 1, 1024, 0, s, blockmax, nb, max_out);
  }
  return launch_status();
}

}  // namespace pmgb
