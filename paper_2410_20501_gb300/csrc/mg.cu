// Linear multigrid for the periodic 7-point Poisson problem (§3.5, §3.6.1):
// red-black SOR smoothing (Eq. jacobi_sweep_laplacian with over-relaxation),
// residual + 8-child-average restriction, 27/9/3/1 prolongation and
// correction, a single-CTA coarsest-level solve, V-cycles.
//
// Precision: smoothing and transfers in float32.  The finest-level residual is
// formed from sums that carry their rounding (TwoSum), so the float32-stored
// iterate is tested against f with float64-class accuracy; norms are accumulated
// in float64.
#include <math.h>

#include "pm_device.cuh"
#include "pm_internal.cuh"
#include "rb_march.cuh"

namespace pmgb {

namespace {

constexpr float kSixth = 1.0f / 6.0f;

__device__ __forceinline__ float load_mean(const Src& f) { return f.mean ? (float)*f.mean : 0.0f; }

// Offset of cell (i, j, k) inside one box (n <= 1024: below 2^30).
__device__ __forceinline__ uint32_t idx3(int i, int j, int k, int log2n) {
  return ((uint32_t)i << (2 * log2n)) | ((uint32_t)j << log2n) | (uint32_t)k;
}

// u = -h^2 f / 6 (Eq. multigrid_initial_guess), four cells a thread.
__global__ void k_jacobi_guess(float* __restrict__ u, Src f, int64_t count, float h2) {
  pdl_entry();
  const int64_t c = 4 * (blockIdx.x * (int64_t)blockDim.x + threadIdx.x);
  if (c >= count) return;
  u += (int64_t)blockIdx.z * count;
  f = box_src(f, count);
  const float mean = load_mean(f);
  const float4 v = __ldg(reinterpret_cast<const float4*>(f.p + c));
  auto guess = [&](float x) { return -h2 * (f.s * (x - mean)) * kSixth; };
  *reinterpret_cast<float4*>(u + c) = make_float4(guess(v.x), guess(v.y), guess(v.z), guess(v.w));
}

// u *= a (per box: ab[box] if ab is set).
__global__ void k_scale(float* __restrict__ u, int64_t count, float a, const float* __restrict__ ab) {
  pdl_entry();
  u += (int64_t)blockIdx.z * count;
  if (ab) a = __ldg(ab + blockIdx.z);
  for (int64_t c = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; c < count;
       c += (int64_t)gridDim.x * blockDim.x)
    u[c] *= a;
}

// The linear update rule: (old value, 6 neighbours in the order x+, x-, y+, y-,
// z+, z-, source value, neighbours-never-updated, own-never-updated) -> new value.
struct PoissonUpdate {
  float h2, omega;
  float gscale;        // warm-start rescale applied to never-updated values
  const float* gbox;   // per-box gscale of a batched launch (replaces gscale), or NULL
  __device__ __forceinline__ PoissonUpdate box(int b) const {
    PoissonUpdate u = *this;
    if (gbox) u.gscale = __ldg(gbox + b);
    return u;
  }
  // Explicit rounding intrinsics (no other contraction) so that the fused and
  // the colour-by-colour kernels produce bitwise identical updates.
  __device__ __forceinline__ float operator()(float old, const float nb[6], float fv, bool nb_old, bool own_old) const {
    float s = __fadd_rn(nb[0], nb[1]);
    s = __fadd_rn(s, nb[2]);
    s = __fadd_rn(s, nb[3]);
    s = __fadd_rn(s, nb[4]);
    s = __fadd_rn(s, nb[5]);
    if (nb_old) s = __fmul_rn(gscale, s);
    const float ugs = __fmul_rn(__fsub_rn(s, __fmul_rn(h2, fv)), 1.0f / 6.0f);
    if (omega == 1.0f) return ugs;
    const float o = own_old ? __fmul_rn(gscale, old) : old;
    return __fmaf_rn(omega, ugs, __fmul_rn(1.0f - omega, o));
  }
};

// One colour of a red-black SOR sweep.  zero: the values of this level are
// taken as 0 (the coarse-level error starts from zero): the red pass reads
// nothing, the black pass ignores its own old value.
//
// These levels live in L2 and a pass is over in a few microseconds, so what
// bounds it is the latency of its loads: a thread takes four consecutive z
// cells (two of the colour) and has its five 16-byte row loads, the z
// neighbour beyond the run and the sources in flight together.
constexpr int kSweepThreads = 128;
__global__ void __launch_bounds__(kSweepThreads) k_rb_sweep(float* __restrict__ u, Src f, int log2n, int colour,
                                                            PoissonUpdate upd, int nb_old, int own_old, int zero) {
  pdl_entry();
  const uint32_t t = blockIdx.x * kSweepThreads + threadIdx.x;
  if (t >= 1u << (3 * log2n - 2)) return;
  u += (int64_t)blockIdx.z << (3 * log2n);
  f = box_src(f, (int64_t)1 << (3 * log2n));
  upd = upd.box(blockIdx.z);
  const int m = (1 << log2n) - 1;
  const int k0 = (int)(t << 2) & m, j = (int)(t >> (log2n - 2)) & m, i = (int)(t >> (2 * log2n - 2));
  const bool odd = ((colour + i + j) & 1) != 0;   // cells k0 + odd and k0 + odd + 2
  const uint32_t c = idx3(i, j, k0, log2n);
  float4 XP = make_float4(0.0f, 0.0f, 0.0f, 0.0f), XM = XP, YP = XP, YM = XP, C = XP;
  float ze = 0.0f;
  auto row4 = [&](int ii, int jj) { return *reinterpret_cast<const float4*>(u + idx3(ii & m, jj & m, k0, log2n)); };
  if (!(zero && colour == 0)) {
    XP = row4(i + 1, j);
    XM = row4(i - 1, j);
    YP = row4(i, j + 1);
    YM = row4(i, j - 1);
    C = row4(i, j);
    ze = u[idx3(i, j, (odd ? k0 + 4 : k0 - 1) & m, log2n)];
  }
  const float4 F = __ldg(reinterpret_cast<const float4*>(f.p + c));
  const float mean = load_mean(f);
  const float nb0[6] = {odd ? XP.y : XP.x, odd ? XM.y : XM.x, odd ? YP.y : YP.x, odd ? YM.y : YM.x,
                        odd ? C.z : C.y, odd ? C.x : ze};
  const float nb1[6] = {odd ? XP.w : XP.z, odd ? XM.w : XM.z, odd ? YP.w : YP.z, odd ? YM.w : YM.z,
                        odd ? ze : C.w, odd ? C.z : C.y};
  const float o0 = zero ? 0.0f : odd ? C.y : C.x, o1 = zero ? 0.0f : odd ? C.w : C.z;
  const float f0 = f.s * ((odd ? F.y : F.x) - mean), f1 = f.s * ((odd ? F.w : F.z) - mean);
  u[c + odd] = upd(o0, nb0, f0, nb_old != 0, own_old != 0);
  u[c + odd + 2] = upd(o1, nb1, f1, nb_old != 0, own_old != 0);
}

// A pair of floats with what rounding took from it: s + e is exact after every
// add (TwoSum per component; e itself is a float sum).
struct PairSum {
  float2 s, e;
  __device__ __forceinline__ explicit PairSum(float2 v) : s(v), e(both(0.0f)) {}
  __device__ __forceinline__ void add(float2 v) {
    const float2 m = both(-1.0f);
    const float2 t = add2(s, v), vp = fma2(s, m, t);               // t - s
    const float2 se = fma2(fma2(vp, m, t), m, s), ve = fma2(vp, m, v);   // s - (t - vp), v - vp
    e = add2(e, add2(se, ve));
    s = t;
  }
  // subtracts k times another sum (k v split exactly by a fused multiply-add)
  __device__ __forceinline__ void sub_times(float k, const PairSum& v) {
    const float2 p = mul2(v.s, both(-k)), pe = fma2(v.s, both(-k), mul2(p, both(-1.0f)));
    add(p);
    e = add2(e, fma2(v.e, both(-k), pe));
  }
};

// The right-hand sides of two coarse cells next to each other in z from their
// children's rows (core [x][y], four cells along z), the rows beyond them in x
// (xf [side][y]) and y (yf [x][side]), the cells before (zl) and after (zr) the
// rows and the sources' rows (fr [x][y]; source fs (fr - mean)).
template <bool COMP>
__device__ __forceinline__ float2 restrict_pair(const float4 (&core)[2][2], const float4 (&xf)[2][2],
                                                const float4 (&yf)[2][2], const float4 (&fr)[2][2],
                                                const float (&zl)[2][2], const float (&zr)[2][2], float fs, float mean,
                                                float inv_h2) {
  // (first coarse cell, second coarse cell): even fine cells, odd fine cells
  auto ev = [](const float4& v) { return make_float2(v.x, v.z); };
  auto od = [](const float4& v) { return make_float2(v.y, v.w); };
  auto source = [&](float2 v) { return mul2(both(fs), add2(v, both(-mean))); };
  float2 d;
  if (COMP) {
    PairSum S(ev(xf[0][0])), C(ev(core[0][0])), F(source(ev(fr[0][0])));
#pragma unroll
    for (int a = 0; a < 2; ++a)
#pragma unroll
      for (int b = 0; b < 2; ++b) {
        if (a + b) {
          S.add(ev(xf[a][b]));
          C.add(ev(core[a][b]));
          F.add(source(ev(fr[a][b])));
        }
        S.add(od(xf[a][b]));
        S.add(ev(yf[a][b]));
        S.add(od(yf[a][b]));
        S.add(make_float2(zl[a][b], core[a][b].y));
        S.add(make_float2(core[a][b].z, zr[a][b]));
        C.add(od(core[a][b]));
        F.add(source(od(fr[a][b])));
      }
    S.sub_times(3.0f, C);
    d = add2(fma2(both(-inv_h2), S.s, F.s), fma2(both(-inv_h2), S.e, F.e));
  } else {
    // per row, so that what cancels is subtracted early: neighbours minus three times the children
    float2 L = both(0.0f), F = both(0.0f);
#pragma unroll
    for (int a = 0; a < 2; ++a)
#pragma unroll
      for (int b = 0; b < 2; ++b) {
        const float2 ce = mul2(ev(core[a][b]), both(-1.0f)), co = mul2(od(core[a][b]), both(-1.0f));
        const float2 fe = add2(ev(xf[a][b]), ce), fo = add2(od(xf[a][b]), co);
        const float2 ge = add2(ev(yf[a][b]), ce), go = add2(od(yf[a][b]), co);
        const float2 lo = add2(make_float2(zl[a][b], core[a][b].y), ce), hi = add2(make_float2(core[a][b].z, zr[a][b]), co);
        L = add2(L, add2(add2(add2(fe, fo), add2(ge, go)), add2(lo, hi)));
        F = add2(F, add2(source(ev(fr[a][b])), source(od(fr[a][b]))));
      }
    d = fma2(both(-inv_h2), L, F);
  }
  return mul2(d, both(0.125f));
}

// Coarse right-hand side fc = R(f - L u): residual of the 8 children,
// averaged.  Summed over the 2x2x2 block the Laplacian fluxes through the 12
// inner faces cancel pairwise, so  h^2 sum_c L u_c  is the sum of the 24 outer
// neighbours minus three times that of the 8 children.  With COMP both sums
// carry their rounding (PairSum), as does the sum of the sources, and the one
// cancelling subtraction is a single rounding (fused multiply-add).
//
// The compensated sums' arithmetic and the number of loads in flight bound it:
// a thread takes two coarse cells along z, so its fine rows come in 16-byte
// loads and the two cells go through the paired float instructions.  512^3:
// 0.314 -> 0.231 ms against one cell a thread with the 24 differences
// summed one by one; 256^3 42 -> 32 us.
template <bool COMP>
__global__ void __launch_bounds__(128) k_resid_restrict(const float* __restrict__ u, Src f, int log2n, float inv_h2,
                                                        float* __restrict__ fc) {
  pdl_entry();
  const int lc = log2n - 1, mc = (1 << lc) - 1, m = (1 << log2n) - 1, lg = lc - 1;
  u += (int64_t)blockIdx.z << (3 * log2n);
  f = box_src(f, (int64_t)1 << (3 * log2n));
  fc += (int64_t)blockIdx.z << (3 * lc);
  const uint32_t t = blockIdx.x * blockDim.x + threadIdx.x;   // two coarse cells, K = 2 G and 2 G + 1
  if (t >= 1u << (3 * lc - 1)) return;
  const int G = (int)(t & ((1u << lg) - 1u)), J = (int)(t >> lg) & mc, I = (int)(t >> (lg + lc));
  const int z0 = 4 * G;
  auto row = [&](const float* p, int x, int y) {
    return __ldg(reinterpret_cast<const float4*>(p + idx3(x & m, y & m, z0, log2n)));
  };
  float4 core[2][2], xf[2][2], yf[2][2], fr[2][2];   // [x][y], [side][y], [x][side]
  float zl[2][2], zr[2][2];
#pragma unroll
  for (int a = 0; a < 2; ++a)
#pragma unroll
    for (int b = 0; b < 2; ++b) {
      core[a][b] = row(u, 2 * I + a, 2 * J + b);
      zl[a][b] = __ldg(u + idx3(2 * I + a, 2 * J + b, (z0 - 1) & m, log2n));
      zr[a][b] = __ldg(u + idx3(2 * I + a, 2 * J + b, (z0 + 4) & m, log2n));
      xf[a][b] = row(u, a ? 2 * I + 2 : 2 * I - 1, 2 * J + b);
      yf[a][b] = row(u, 2 * I + a, b ? 2 * J + 2 : 2 * J - 1);
      fr[a][b] = row(f.p, 2 * I + a, 2 * J + b);
    }
  *reinterpret_cast<float2*>(fc + 2 * t) =
      restrict_pair<COMP>(core, xf, yf, fr, zl, zr, f.s, load_mean(f), inv_h2);
}

// Residual norm^2 and source norm^2 partials (finest level, compensated
// residual): partial[blockIdx] and partial[gridDim + blockIdx].  A thread takes
// four z cells at a time: 16-byte loads, and the neighbour sum minus 6 u with its
// rounding (PairSum) in the paired float instructions, which is what it spends
// its time on.  256^3: 100 -> 45 us against one cell a time with the six
// differences summed one by one.
__global__ void __launch_bounds__(256) k_resid_norm(const float* __restrict__ u, Src f, int log2n,
                                                    float inv_h2, double* __restrict__ partial) {
  pdl_entry();
  __shared__ double scratch[32];
  const float mean = load_mean(f);
  const int m = (1 << log2n) - 1;
  const uint32_t runs = 1u << (3 * log2n - 2);
  float sd[2] = {0.0f, 0.0f}, cd[2] = {0.0f, 0.0f}, sf[2] = {0.0f, 0.0f}, cf[2] = {0.0f, 0.0f};
  for (uint32_t t = blockIdx.x * blockDim.x + threadIdx.x; t < runs; t += gridDim.x * blockDim.x) {
    const int k = (int)(t << 2) & m, j = (int)(t >> (log2n - 2)) & m, i = (int)(t >> (2 * log2n - 2));
    auto row = [&](int x, int y) { return __ldg(reinterpret_cast<const float4*>(u + idx3(x & m, y & m, k, log2n))); };
    const float4 c = row(i, j), xp = row(i + 1, j), xm = row(i - 1, j), yp = row(i, j + 1), ym = row(i, j - 1);
    const float zl = __ldg(u + idx3(i, j, (k - 1) & m, log2n)), zr = __ldg(u + idx3(i, j, (k + 4) & m, log2n));
    const float4 fr = __ldg(reinterpret_cast<const float4*>(f.p + 4 * (int64_t)t));
#pragma unroll
    for (int h = 0; h < 2; ++h) {   // cells 0, 1, then 2, 3
      auto two = [&](const float4& v) { return h ? make_float2(v.z, v.w) : make_float2(v.x, v.y); };
      PairSum S(two(xp));
      S.add(two(xm));
      S.add(two(yp));
      S.add(two(ym));
      S.add(h ? make_float2(c.w, zr) : make_float2(c.y, c.z));
      S.add(h ? make_float2(c.y, c.z) : make_float2(zl, c.x));
      S.sub_times(6.0f, PairSum(two(c)));
      const float2 fv = mul2(both(f.s), add2(two(fr), both(-mean)));
      const float2 d = add2(fma2(both(-inv_h2), S.s, fv), mul2(both(-inv_h2), S.e));
      kahan_add(sd[0], cd[0], d.x * d.x);
      kahan_add(sd[1], cd[1], d.y * d.y);
      kahan_add(sf[0], cf[0], fv.x * fv.x);
      kahan_add(sf[1], cf[1], fv.y * fv.y);
    }
  }
  kahan_add(sd[0], cd[0], sd[1] - cd[1]);
  kahan_add(sf[0], cf[0], sf[1] - cf[1]);
  block_sum_to(partial + blockIdx.x, sd[0], cd[0], scratch);
  block_sum_to(partial + gridDim.x + blockIdx.x, sf[0], cf[0], scratch);
}

// Block sum of per-thread float64 values, written by thread 0 to *out (a
// fixed order: shuffles, then the warps in order).
__device__ __forceinline__ void block_sum_f64(double* out, double v, double* scratch32) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
  if ((threadIdx.x & 31) == 0) scratch32[threadIdx.x >> 5] = v;
  __syncthreads();
  if (threadIdx.x == 0) {
    double t = 0.0;
    for (int i = 0; i < (int)(blockDim.x >> 5); ++i) t += scratch32[i];
    *out = t;
  }
  __syncthreads();
}

// Residual of a float64 iterate in float64: r = (f - <f>) - (L(u) - 6u)/h^2,
// with L(u) - 6u as the neighbour sum minus 6u (the float64 pipe bounds this
// kernel on GB300, so it spends 12 float64 operations per cell; the six
// differences u_nb - u would take five more).  r is stored rounded to float32
// (the source of the correction solve); the squares of r and of f - <f> are
// summed per block in float64.
__global__ void __launch_bounds__(256) k_resid_f64(const double* __restrict__ u, const float* __restrict__ f,
                                                   const double* __restrict__ fmean, int log2n, double inv_h2,
                                                   float* __restrict__ r, double* __restrict__ partial) {
  pdl_entry();
  __shared__ double scratch[32];
  const double mean = *fmean;
  const int m = (1 << log2n) - 1;
  const int64_t total = (int64_t)1 << (3 * log2n);
  double sr = 0.0, sf = 0.0;
  for (int64_t c = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; c < total; c += (int64_t)gridDim.x * blockDim.x) {
    const int k = (int)(c & m), j = (int)((c >> log2n) & m), i = (int)(c >> (2 * log2n));
    const double uc = u[c];
    const double nsum = ((u[idx3((i + 1) & m, j, k, log2n)] + u[idx3((i - 1) & m, j, k, log2n)]) +
                         (u[idx3(i, (j + 1) & m, k, log2n)] + u[idx3(i, (j - 1) & m, k, log2n)])) +
                        (u[idx3(i, j, (k + 1) & m, log2n)] + u[idx3(i, j, (k - 1) & m, log2n)]);
    const double L = fma(-6.0, uc, nsum);
    const double fv = (double)__ldg(f + c) - mean;
    const double d = fma(-inv_h2, L, fv);
    r[c] = (float)d;
    sr = fma(d, d, sr);
    sf = fma(fv, fv, sf);
  }
  block_sum_f64(partial + blockIdx.x, sr, scratch);
  block_sum_f64(partial + gridDim.x + blockIdx.x, sf, scratch);
}

// u += e (float64 iterate, float32 correction).
__global__ void k_add_correction_f64(double* __restrict__ u, const float* __restrict__ e, int64_t count) {
  pdl_entry();
  for (int64_t c = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; c < count; c += (int64_t)gridDim.x * blockDim.x)
    u[c] += (double)__ldg(e + c);
}

// P(uc - uc2) at the 16 children of the coarse cells (I, J, K) and (I, J, K + 1), K
// even: put(x, y, the four along z).  Interpolated along z, then y, then x.
template <class Put>
__device__ __forceinline__ void prolong_pair(const float* __restrict__ uc, const float* __restrict__ uc2, int I, int J,
                                             int K, int lc, const Put& put) {
  const int mc = (1 << lc) - 1;
  float c[3][3][4];   // [x][y][z]: x, y = I-1 .. I+1, J-1 .. J+1; z = K-1 .. K+2
#pragma unroll
  for (int a = 0; a < 3; ++a)
#pragma unroll
    for (int b = 0; b < 3; ++b) {
      const int64_t base = idx3((I + a - 1) & mc, (J + b - 1) & mc, 0, lc);
      const float2 mid = __ldg(reinterpret_cast<const float2*>(uc + base + K));
      float v[4] = {__ldg(uc + base + ((K - 1) & mc)), mid.x, mid.y, __ldg(uc + base + ((K + 2) & mc))};
      if (uc2) {
        const float2 m2 = __ldg(reinterpret_cast<const float2*>(uc2 + base + K));
        v[0] -= __ldg(uc2 + base + ((K - 1) & mc));
        v[1] -= m2.x;
        v[2] -= m2.y;
        v[3] -= __ldg(uc2 + base + ((K + 2) & mc));
      }
#pragma unroll
      for (int z = 0; z < 4; ++z) c[a][b][z] = v[z];
    }
#pragma unroll
  for (int b = 0; b < 2; ++b) {
    const int jn = b ? 2 : 0;
    // z then y contractions: vy[x][q] for the fine z offsets q = 0..3 (coarse
    // cell q / 2 at column q / 2 + 1, child q & 1)
    float vy[3][4];
#pragma unroll
    for (int a = 0; a < 3; ++a)
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const int kc = (q >> 1) + 1, kn = (q & 1) ? kc + 1 : kc - 1;
        const float vz0 = fmaf(0.25f, c[a][1][kn], fmaf(0.75f, c[a][1][kc], 0.0f));
        const float vz1 = fmaf(0.25f, c[a][jn][kn], fmaf(0.75f, c[a][jn][kc], 0.0f));
        vy[a][q] = fmaf(0.25f, vz1, fmaf(0.75f, vz0, 0.0f));
      }
#pragma unroll
    for (int ax = 0; ax < 2; ++ax) {
      const int in = ax ? 2 : 0;
      put(ax, b, make_float4(fmaf(0.25f, vy[in][0], fmaf(0.75f, vy[1][0], 0.0f)),
                             fmaf(0.25f, vy[in][1], fmaf(0.75f, vy[1][1], 0.0f)),
                             fmaf(0.25f, vy[in][2], fmaf(0.75f, vy[1][2], 0.0f)),
                             fmaf(0.25f, vy[in][3], fmaf(0.75f, vy[1][3], 0.0f))));
    }
  }
}

// u += P(uc - uc2): cell-centred trilinear prolongation, weights 27/9/3/1 over
// 64 (§3.6.1); uc2 may be NULL.  One thread per two coarse cells along z
// (K = 2G, 2G + 1): it reads their 3x3x4 coarse neighbourhood once (a float2
// and two scalars per coarse row) and corrects their 16 children (runs of
// four along z as float4).  Per child the interpolation runs z, then y, then
// x, parent (weight 3/4) before neighbour (1/4), in fused multiply-adds.
//
// The latency of its loads bounds it, so the children's rows are loaded ahead of
// the coarse rows, all in flight together: 512^3 222 -> 171 us (the copy rate) against a
// row at a time behind each other's stores, 256^3 26 -> 19; with uc2 230 -> 212.
template <bool FAS>
__global__ void __launch_bounds__(128, 7) k_prolong_correct(float* __restrict__ u, const float* __restrict__ uc,
                                                            const float* __restrict__ uc2, int log2n) {
  pdl_entry();
  const int lc = log2n - 1, mc = (1 << lc) - 1;
  u += (int64_t)blockIdx.z << (3 * log2n);
  uc += (int64_t)blockIdx.z << (3 * lc);
  if (FAS) uc2 += (int64_t)blockIdx.z << (3 * lc);
  const int hz = lc - 1;   // log2 of the pairs per coarse row
  const uint32_t t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= 1u << (3 * lc - 1)) return;
  const int K = 2 * (int)(t & ((1u << hz) - 1u)), J = (int)(t >> hz) & mc, I = (int)(t >> (hz + lc));
  auto row = [&](int ax, int b) { return reinterpret_cast<float4*>(u + idx3(2 * I + ax, 2 * J + b, 2 * K, log2n)); };
  float4 w[2][2];
#pragma unroll
  for (int ax = 0; ax < 2; ++ax)
#pragma unroll
    for (int b = 0; b < 2; ++b) w[ax][b] = *row(ax, b);
  prolong_pair(uc, FAS ? uc2 : nullptr, I, J, K, lc, [&](int ax, int b, float4 e) {
    const float4 v = w[ax][b];
    *row(ax, b) = make_float4(v.x + e.x, v.y + e.y, v.z + e.z, v.w + e.w);
  });
}

// One side of a V-cycle on a level of up to 32^3 in one launch: the red-black
// sweeps before the coarse correction and the restriction after them (PRE), or
// the prolongation and the sweeps after it.  Such a level is a megabyte at most
// and a colour pass over it is all latency (2.3 us a launch, ten launches a
// cycle), so the sweeps are repeated instead of synchronised: a CTA takes TX x TY
// rows of full length with a halo of as many rows as the passes (and the
// residual) reach, every pass updates a row less on each side, and CTAs never
// exchange anything.  Rows are kept by colour (a thread's two cells of one colour
// are one 8-byte word, as are the neighbours' that it reads), so a pass reads one
// colour and writes the other.  The updates, the restriction and the
// prolongation are those of the kernels above, cell by cell: bitwise the same.
//
// Rows of 4 x 4 while one CTA an SM takes them all, of 8 x 8, which repeat less,
// beyond (16 boxes 52 us a V-cycle against 46; 4 boxes 31 against 34).  V-cycle from
// 32^3 against colour passes and the transfers' own launches, coarsest solve
// included: one box 33 -> 26 us, 16 boxes 70 -> 46, 64 boxes 111 -> 105.
//
// uin: the iterate (NULL: zeros), uout: not uin.  n >= 8.
constexpr int kTileN = 32;
template <int TX, int TY, bool PRE> struct TileGeom {
  static constexpr int H = PRE ? 5 : 4, EX = TX + 2 * H, EY = TY + 2 * H, ROWS = EX * EY;
  static constexpr int ITEMS = 4, THREADS = (ROWS * (kTileN / 4) / ITEMS + 31) / 32 * 32;   // items: four cells of a row
  static constexpr size_t smem = 2 * sizeof(float2) * ROWS * (kTileN / 4);
};
template <int TX, int TY, bool PRE, bool COMP>
__global__ void __launch_bounds__(TileGeom<TX, TY, PRE>::THREADS)
    k_rb_tile(const float* __restrict__ uin, float* __restrict__ uout, Src f, const float* __restrict__ uc,
              float* __restrict__ fc, int log2n, int sweeps, PoissonUpdate u0, PoissonUpdate u1) {
  pdl_entry();
  using T = TileGeom<TX, TY, PRE>;
  constexpr int H = T::H, EX = T::EX, EY = T::EY;
  extern __shared__ float4 tile_sm[];
  const int n = 1 << log2n, m = n - 1, lq = log2n - 2, Q = 1 << lq, items = T::ROWS << lq;
  float2* U = reinterpret_cast<float2*>(tile_sm);   // [colour][item]
  const int64_t box = (int64_t)blockIdx.z << (3 * log2n);
  f = box_src(f, (int64_t)1 << (3 * log2n));
  u0 = u0.box(blockIdx.z);
  const int x0 = (int)(blockIdx.x / (unsigned)(n / TY)) * TX - H, y0 = (int)(blockIdx.x % (unsigned)(n / TY)) * TY - H;
  const int tid = threadIdx.x;
  auto cell = [&](int x, int y, int q) { return idx3((x0 + x) & m, (y0 + y) & m, 4 * q, log2n); };
  auto put = [&](int x, int y, int q, const float4& v) {
    const int o = (x0 + x + y0 + y) & 1, i = ((x * EY + y) << lq) + q;
    U[o * items + i] = make_float2(v.x, v.z);
    U[(o ^ 1) * items + i] = make_float2(v.y, v.w);
  };
  auto get = [&](int x, int y, int q) {
    const int o = (x0 + x + y0 + y) & 1, i = ((x * EY + y) << lq) + q;
    const float2 e = U[o * items + i], d = U[(o ^ 1) * items + i];
    return make_float4(e.x, d.x, e.y, d.y);
  };
  const float mean = load_mean(f);
  float4 F[T::ITEMS];
#pragma unroll
  for (int k = 0; k < T::ITEMS; ++k) {
    const int i = tid + k * T::THREADS;
    if (i >= items) break;
    const int q = i & (Q - 1), row = i >> lq, x = row / EY, y = row - x * EY;
    const float4 v = __ldg(reinterpret_cast<const float4*>(f.p + cell(x, y, q)));
    F[k] = make_float4(f.s * (v.x - mean), f.s * (v.y - mean), f.s * (v.z - mean), f.s * (v.w - mean));
    if (PRE)
      put(x, y, q, uin ? *reinterpret_cast<const float4*>(uin + box + cell(x, y, q)) : make_float4(0.0f, 0.0f, 0.0f, 0.0f));
  }
  if (!PRE) {
    const int lc = log2n - 1, mc = (1 << lc) - 1;
    const float* ucb = uc + ((int64_t)blockIdx.z << (3 * lc));
    for (int i = tid; i < (EX / 2) * (EY / 2) << lq; i += T::THREADS) {
      const int q = i & (Q - 1), blk = i >> lq, bx = blk / (EY / 2), by = blk - bx * (EY / 2);
      prolong_pair(ucb, nullptr, ((x0 >> 1) + bx) & mc, ((y0 >> 1) + by) & mc, 2 * q, lc, [&](int ax, int ay, float4 e) {
        const int x = 2 * bx + ax, y = 2 * by + ay;
        const float4 w = *reinterpret_cast<const float4*>(uin + box + cell(x, y, q));
        put(x, y, q, make_float4(w.x + e.x, w.y + e.y, w.z + e.z, w.w + e.w));
      });
    }
  }
  for (int p = 0; p < 2 * sweeps; ++p) {
    __syncthreads();
    const int colour = p & 1;
    const PoissonUpdate upd = p < 2 ? u0 : u1;
    float2* own = U + colour * items;
    const float2* opp = U + (colour ^ 1) * items;
#pragma unroll
    for (int k = 0; k < T::ITEMS; ++k) {
      const int i = tid + k * T::THREADS;
      if (i >= items) break;
      const int q = i & (Q - 1), row = i >> lq, x = row / EY, y = row - x * EY;
      if (x <= p || x >= EX - 1 - p || y <= p || y >= EY - 1 - p) continue;
      const bool odd = ((colour + x0 + x + y0 + y) & 1) != 0;   // cells 4 q + odd and 4 q + odd + 2
      const float2 xp = opp[i + (EY << lq)], xm = opp[i - (EY << lq)], yp = opp[i + Q], ym = opp[i - Q], c = opp[i];
      const float2 side = opp[i - q + ((odd ? q + 1 : q - 1) & (Q - 1))], o = own[i];
      const float nb0[6] = {xp.x, xm.x, yp.x, ym.x, odd ? c.y : c.x, odd ? c.x : side.y};
      const float nb1[6] = {xp.y, xm.y, yp.y, ym.y, odd ? side.x : c.y, odd ? c.y : c.x};
      own[i] = make_float2(upd(o.x, nb0, odd ? F[k].y : F[k].x, p == 0, p < 2),
                           upd(o.y, nb1, odd ? F[k].w : F[k].z, p == 0, p < 2));
    }
  }
  __syncthreads();
  for (int i = tid; i < TX * TY << lq; i += T::THREADS) {
    const int q = i & (Q - 1), row = i >> lq, x = H + row / TY, y = H + row % TY;
    *reinterpret_cast<float4*>(uout + box + cell(x, y, q)) = get(x, y, q);
  }
  if (PRE) {
    const float inv_h2 = (float)n * (float)n;
    for (int i = tid; i < (TX / 2) * (TY / 2) << lq; i += T::THREADS) {
      const int q = i & (Q - 1), row = i >> lq, x = H + 2 * (row / (TY / 2)), y = H + 2 * (row % (TY / 2));
      float4 core[2][2], xf[2][2], yf[2][2], fr[2][2];
      float zl[2][2], zr[2][2];
#pragma unroll
      for (int a = 0; a < 2; ++a)
#pragma unroll
        for (int b = 0; b < 2; ++b) {
          core[a][b] = get(x + a, y + b, q);
          zl[a][b] = get(x + a, y + b, (q - 1) & (Q - 1)).w;
          zr[a][b] = get(x + a, y + b, (q + 1) & (Q - 1)).x;
          xf[a][b] = get(a ? x + 2 : x - 1, y + b, q);
          yf[a][b] = get(x + a, b ? y + 2 : y - 1, q);
          fr[a][b] = __ldg(reinterpret_cast<const float4*>(f.p + cell(x + a, y + b, q)));
        }
      const int lc = log2n - 1;
      const int64_t at = ((int64_t)blockIdx.z << (3 * lc)) + idx3(((x0 + x) & m) >> 1, ((y0 + y) & m) >> 1, 2 * q, lc);
      *reinterpret_cast<float2*>(fc + at) = restrict_pair<COMP>(core, xf, yf, fr, zl, zr, f.s, mean, inv_h2);
    }
  }
}

// Coarsest level (n = 4, 8 or 16) in one CTA: red-black SOR sweeps (factor
// omega) until the residual norm dropped by `drop`, its running minimum stalls
// for 5 sweeps (float32 floor), or `max_sweeps` sweeps.
//
// What bounds it is the chain of sweeps on one SM (about 25 of them at 16^3),
// so the sweep is kept short.  A thread owns a whole row (i, j): its n / 2 red
// and n / 2 black values stay in registers, the z neighbours with them, and
// only the four x and y neighbour rows come from shared memory, where the
// cells of one colour of a row lie together in 16-byte groups: a red cell and
// its x and y neighbours have the same index kk in their colour's row
// (z = 2 kk + o, o the parity of row and colour), z + 1 is at kk + o, z - 1
// at kk + o - 1.  The residual of a black cell comes from its own update (its
// neighbours do not move in the black pass), that of a red cell from the next
// sweep's neighbour sums, so a sweep is two passes and two barriers; its norm
// is summed over the block while the next sweep's red cells are already
// computed (kept apart until the norm has decided whether there is a next
// sweep).  16^3: 66 -> 29 us a solve against a thread per two pairs of cells
// in natural order with four barriers a sweep.
template <int VW> struct alignas(4 * VW) RowVec { float v[VW]; };
template <int LOG>
__global__ void __launch_bounds__(LOG == 2 ? 32 : 1 << (2 * LOG)) k_mg_coarse(float* __restrict__ u, Src f, float h2,
                                                                              float omega, int max_sweeps, float drop,
                                                                              int zero_guess) {
  pdl_entry();
  constexpr int n = 1 << LOG, m = n - 1, ROWS = n * n, H = n / 2, VW = H < 4 ? H : 4, NV = H / VW;
  constexpr int NW = ROWS < 32 ? 1 : ROWS / 32;   // warps
  using Vec = RowVec<VW>;
  __shared__ Vec S[2][NV][ROWS];   // [colour][group of kk][row]
  __shared__ float2 part[NW];
  u += (int64_t)blockIdx.z * ROWS * n;   // one CTA per box
  f = box_src(f, ROWS * n);
  const float mean = load_mean(f);
  const float inv_h2 = 1.0f / h2;
  const bool act = threadIdx.x < ROWS;
  const int row = act ? threadIdx.x : 0, i = row >> LOG, j = row & m, par = (i + j) & 1;
  const int rxp = (((i + 1) & m) << LOG) | j, rxm = (((i - 1) & m) << LOG) | j;
  const int ryp = (i << LOG) | ((j + 1) & m), rym = (i << LOG) | ((j - 1) & m);
  float v[2][H], fv[2][H];   // [colour][kk]
  {
    float t[n];
    auto split = [&](float dst[2][H]) {   // natural order -> colours (red first)
#pragma unroll
      for (int kk = 0; kk < H; ++kk) {
        dst[0][kk] = par ? t[2 * kk + 1] : t[2 * kk];
        dst[1][kk] = par ? t[2 * kk] : t[2 * kk + 1];
      }
    };
#pragma unroll
    for (int k = 0; k < n; k += 4) {
      const float4 q = __ldg(reinterpret_cast<const float4*>(f.p + row * n + k));
      t[k] = f.s * (q.x - mean); t[k + 1] = f.s * (q.y - mean);
      t[k + 2] = f.s * (q.z - mean); t[k + 3] = f.s * (q.w - mean);
    }
    split(fv);
#pragma unroll
    for (int k = 0; k < n; k += 4) {
      const float4 q = zero_guess ? make_float4(0.0f, 0.0f, 0.0f, 0.0f)
                                  : *reinterpret_cast<const float4*>(u + row * n + k);
      t[k] = q.x; t[k + 1] = q.y; t[k + 2] = q.z; t[k + 3] = q.w;
    }
    split(v);
  }
  auto put = [&](int c, const float w[H]) {
    if (!act) return;
#pragma unroll
    for (int g = 0; g < NV; ++g) {
      Vec x;
#pragma unroll
      for (int q = 0; q < VW; ++q) x.v[q] = w[g * VW + q];
      S[c][g][row] = x;
    }
  };
  // neighbour sums of the row's cells of colour c (order x+, x-, y+, y-, z+, z-)
  auto nbsum = [&](int c, float nb[H]) {
    const bool o = ((c + par) & 1) != 0;
    const float* w = v[1 - c];
#pragma unroll
    for (int g = 0; g < NV; ++g) {
      const Vec a = S[1 - c][g][rxp], b = S[1 - c][g][rxm], d = S[1 - c][g][ryp], e = S[1 - c][g][rym];
#pragma unroll
      for (int q = 0; q < VW; ++q) {
        const int kk = g * VW + q;
        const float zp = o ? w[(kk + 1) % H] : w[kk], zm = o ? w[kk] : w[(kk + H - 1) % H];
        nb[kk] = a.v[q] + b.v[q] + d.v[q] + e.v[q] + zp + zm;
      }
    }
  };
  auto sor = [&](float old, float nb, float fc) -> float {
    const float ugs = (nb - h2 * fc) * kSixth;
    return (omega == 1.0f) ? ugs : omega * ugs + (1.0f - omega) * old;
  };
  float sum[2], cmp[2];   // compensated sums of squared residuals, two chains
  auto clear = [&]() { sum[0] = sum[1] = cmp[0] = cmp[1] = 0.0f; };
  auto residuals = [&](int c, const float val[H], const float nb[H]) {
#pragma unroll
    for (int kk = 0; kk < H; ++kk) {
      const float d = fv[c][kk] - (nb[kk] - 6.0f * val[kk]) * inv_h2;
      kahan_add(sum[kk & 1], cmp[kk & 1], d * d);
    }
  };
  auto pair_add = [](float& s, float& c, float os, float oc) {
    float t, e;
    two_sum(s, os, t, e);
    s = t;
    c = c + oc + e;
  };
  // this warp's sum over its rows into part[] (idle threads add nothing)
  auto warp_part = [&]() {
    float s = act ? sum[0] - cmp[0] : 0.0f, c = 0.0f;
    pair_add(s, c, act ? sum[1] - cmp[1] : 0.0f, 0.0f);
#pragma unroll
    for (int d = 16; d > 0; d >>= 1) {
      const float os = __shfl_xor_sync(0xffffffffu, s, d), oc = __shfl_xor_sync(0xffffffffu, c, d);
      pair_add(s, c, os, oc);
    }
    if ((threadIdx.x & 31) == 0) part[threadIdx.x >> 5] = make_float2(s, c);
  };
  // the block's sum from part[], the same in every thread
  auto block_total = [&]() -> float {
    float2 t = part[0];
#pragma unroll
    for (int w = 1; w < NW; ++w) pair_add(t.x, t.y, part[w].x, part[w].y);
    return t.x + t.y;
  };

  put(0, v[0]);
  put(1, v[1]);
  __syncthreads();
  float nb[H];
  clear();
  nbsum(1, nb);
  residuals(1, v[1], nb);
  nbsum(0, nb);
  residuals(0, v[0], nb);
  warp_part();
  __syncthreads();
  float best = block_total();
  const float target = drop * drop * best;
  int stale = 0;
  for (int sweep = 0; sweep < max_sweeps; ++sweep) {
    // v, the shared rows: the values after `sweep` sweeps; nb: sums around the
    // red cells
    float red[H];
    if (sweep > 0) {
      nbsum(0, nb);
      residuals(0, v[0], nb);
      warp_part();
    }
#pragma unroll
    for (int kk = 0; kk < H; ++kk) red[kk] = sor(v[0][kk], nb[kk], fv[0][kk]);
    put(0, red);
    __syncthreads();
    if (sweep > 0) {   // the norm after `sweep` sweeps
      const float r = block_total();
      if (r <= target) break;
      if (r < 0.998f * best) {   // squared norms: a 0.1% improvement of the norm
        best = r;
        stale = 0;
      } else if (++stale >= 5) {
        break;                  // no progress for 5 sweeps: the float32 floor
      }
    }
#pragma unroll
    for (int kk = 0; kk < H; ++kk) v[0][kk] = red[kk];
    nbsum(1, nb);
    clear();
#pragma unroll
    for (int kk = 0; kk < H; ++kk) v[1][kk] = sor(v[1][kk], nb[kk], fv[1][kk]);
    residuals(1, v[1], nb);
    put(1, v[1]);
    __syncthreads();
  }
  if (act) {
    float t[n];
#pragma unroll
    for (int kk = 0; kk < H; ++kk) {
      t[2 * kk] = par ? v[1][kk] : v[0][kk];
      t[2 * kk + 1] = par ? v[0][kk] : v[1][kk];
    }
#pragma unroll
    for (int k = 0; k < n; k += 4)
      *reinterpret_cast<float4*>(u + row * n + k) = make_float4(t[k], t[k + 1], t[k + 2], t[k + 3]);
  }
}

// SOR factor of the coarsest level: the caller's, else Young's optimum
// 2 / (1 + sqrt(1 - mu^2)) for red-black ordering of the periodic 7-point
// Laplacian on n^3 cells, mu = (2 + cos(2 pi / n)) / 3 the largest Jacobi
// eigenvalue below 1 (the constant mode is absent from a zero-mean problem).
float coarse_omega(const mg_params& p, int n) {
  if (p.coarse_omega > 0.0f) return p.coarse_omega;
  const double mu = (2.0 + cos(2.0 * M_PI / n)) / 3.0;
  return (float)(2.0 / (1.0 + sqrt(1.0 - mu * mu)));
}

struct MG {
  int n0;
  const mg_params* p;
  cudaStream_t s;
  float* u[12];     // current iterate of each level
  float* alt[12];   // ping-pong partner of the fused sweeps (or NULL)
  Src f[12];
  bool first_cycle;
  float gscale;
  int B = 1;                    // boxes of a batched solve (blockIdx.z of every launch)
  const float* gbox = nullptr;  // per-box warm-start factors (batched MG_GUESS_SCALED)
  dim3 grid(unsigned gx) const { return dim3(gx, 1, (unsigned)B); }
};

pm_status march_attributes() {
  PM_TRY((march_attribute<LinearSweeps<true, true>, 1, kMarchTY, kMarchTZ>()));
  PM_TRY((march_attribute<LinearSweeps<false, false>, 1, kMarchTY, kMarchTZ>()));
  PM_TRY((march_attribute<LinearSweeps<true, true>, 2, kMarchTY, kMarchTZ>()));
  PM_TRY((march_attribute<LinearSweeps<true, false>, 2, kMarchTY, kMarchTZ>()));
  PM_TRY((march_attribute<LinearSweeps<false, true>, 2, kMarchTY, kMarchTZ>()));
  PM_TRY((march_attribute<LinearSweeps<false, false>, 2, kMarchTY, kMarchTZ>()));
  return PM_OK;
}

// SOR factor of sweep si of the `count` before (pre) or after the coarse
// correction: 1 for the first before and the last after it, omega for the others.
float sweep_factor(const mg_params& p, bool pre, int si, int count) {
  return si == (pre ? 0 : count - 1) ? 1.0f : p.omega;
}

// `count` smoothing sweeps on level l, before (pre) or after the coarse
// correction.  zero: the level's values start at 0; scale (sbox: per box):
// warm-start factor applied to the values present before the first sweep.
pm_status smooth(MG& g, int l, int count, bool pre, bool zero, float scale, const float* sbox = nullptr) {
  const int n = g.n0 >> l, log2n = ilog2(n);
  const float h2 = 1.0f / ((float)n * (float)n);
  const int64_t N = (int64_t)n * n * n;
  auto factor = [&](int si) { return sweep_factor(*g.p, pre, si, count); };
  int done = 0;
  // fused sweeps (two per pass over memory) or colour passes (two per sweep),
  // bitwise the same result.  Two sweeps: 512^3 0.83 -> 0.40 ms, 256^3 130 -> 63
  // us against one fused sweep a pass, 128^3 28 -> 18 us against the colour
  // passes; at 64^3 the two forms are even (a V-cycle from there 56 against 55
  // us), so one launch is taken instead of four.  On 64^3 levels of a batch the
  // form is tuned.
  const bool fused_valid = g.p->smoother != 1 && n >= 64 && g.alt[l] && march_aligned(g.u[l], g.alt[l], g.f[l].p);
  bool fused = fused_valid;
  const bool tune_form = fused_valid && g.B > 1 && n < 128;
  if (tune_form) {
    static const int forms[2] = {0, 1};
    fused = tune_begin(TUNE_MG_SMOOTHER, n, g.B, count << 2 | (zero ? 2 : 0) | (pre ? 1 : 0), forms, 2, 1, g.s) == 1;
  }
  const bool form_timed = tune_form && tune_active();
  if (fused) {
    while (done < count) {
      const int S = count - done >= 2 ? 2 : 1;
      const int z = (done == 0 && zero) ? 1 : 0;
      const float w0 = factor(done), w1 = S == 2 ? factor(done + 1) : 1.0f;
      const bool one0 = w0 == 1.0f, one1 = S == 2 && w1 == 1.0f;
      const int chunks = S == 2 ? march_chunks<2, kMarchTY, kMarchTZ>(n, g.B) : march_chunks<1, kMarchTY, kMarchTZ>(n, g.B);
      const dim3 grid = g.grid((unsigned)((n / kMarchTY) * (n / kMarchTZ) * chunks));
#define PM_MARCH(SW, ONE0, ONE1)                                                                                   \
  do {                                                                                                             \
    const LinearSweeps<ONE0, ONE1> sweeps{h2, done == 0 ? scale : 1.0f, w0, w1, done == 0 ? sbox : nullptr};        \
    PM_LAUNCH(l == 0 ? K_MG_SMOOTH0 : K_MG_SMOOTH, (z ? 8.0 : 12.0) * N * g.B,                                     \
              (k_rb_march<LinearSweeps<ONE0, ONE1>, SW, kMarchTY, kMarchTZ>), grid,                                \
              (MarchGeom<SW, kMarchTY, kMarchTZ>::THREADS), (MarchGeom<SW, kMarchTY, kMarchTZ>::smem), g.s, g.u[l], \
              g.alt[l], g.f[l], log2n, chunks, z, sweeps);                                                         \
  } while (0)
      if (S == 1) {
        if (one0) PM_MARCH(1, true, true); else PM_MARCH(1, false, false);
      } else if (one0) {
        if (one1) PM_MARCH(2, true, true); else PM_MARCH(2, true, false);
      } else {
        if (one1) PM_MARCH(2, false, true); else PM_MARCH(2, false, false);
      }
#undef PM_MARCH
      float* t = g.u[l];
      g.u[l] = g.alt[l];
      g.alt[l] = t;
      done += S;
    }
  } else {
    const unsigned grid = grid_for(N / 4, kSweepThreads);
    for (; done < count; ++done) {
      const PoissonUpdate upd{h2, factor(done), done == 0 ? scale : 1.0f, done == 0 ? sbox : nullptr};
      const int z = (done == 0 && zero) ? 1 : 0;
      const int first = done == 0 ? 1 : 0;
      PM_LAUNCH(l == 0 ? K_MG_SMOOTH0 : K_MG_SMOOTH, (z ? 4.0 : 6.0) * N * g.B, k_rb_sweep, g.grid(grid), kSweepThreads, 0,
                g.s, g.u[l], g.f[l], log2n, 0, upd, first, first, z);
      PM_LAUNCH(l == 0 ? K_MG_SMOOTH0 : K_MG_SMOOTH, (z ? 4.0 : 6.0) * N * g.B, k_rb_sweep, g.grid(grid), kSweepThreads, 0,
                g.s, g.u[l], g.f[l], log2n, 1, upd, 0, first, z);
    }
  }
  if (form_timed) tune_end(g.s);
  return PM_OK;
}

// One side of the V-cycle on a small level (k_rb_tile); zero: from zeros.
template <bool PRE>
pm_status tile_side(MG& g, int l, int count, bool zero, float scale, const float* sbox) {
  const int n = g.n0 >> l, log2n = ilog2(n);
  const float h2 = 1.0f / ((float)n * (float)n);
  const double N = (double)n * n * n;
  const PoissonUpdate u0{h2, sweep_factor(*g.p, PRE, 0, count), scale, sbox};
  const PoissonUpdate u1{h2, count > 1 ? sweep_factor(*g.p, PRE, 1, count) : 1.0f, 1.0f, nullptr};
  float* out = zero ? g.u[l] : g.alt[l];
  const float* in = zero ? nullptr : g.u[l];
  const float* uc = PRE ? nullptr : g.u[l + 1];
  float* fc = PRE ? const_cast<float*>(g.f[l + 1].p) : nullptr;
  const bool large = (n / 4) * (n / 4) * (int64_t)g.B > 152;
#define PM_TILE(TX, TY, COMP)                                                                                     \
  PM_LAUNCH(l == 0 ? K_MG_SMOOTH0 : K_MG_SMOOTH, (zero ? 8.0 : 12.0) * N * g.B, (k_rb_tile<TX, TY, PRE, PRE && COMP>), \
            g.grid((unsigned)((n / TX) * (n / TY))), (TileGeom<TX, TY, PRE>::THREADS), (TileGeom<TX, TY, PRE>::smem), \
            g.s, in, out, g.f[l], uc, fc, log2n, count, u0, u1)
  if (l == 0 && PRE) {
    if (large) PM_TILE(8, 8, true); else PM_TILE(4, 4, true);
  } else {
    if (large) PM_TILE(8, 8, false); else PM_TILE(4, 4, false);
  }
#undef PM_TILE
  if (!zero) {
    g.alt[l] = g.u[l];
    g.u[l] = out;
  }
  return PM_OK;
}

pm_status v_cycle(MG& g, int l, bool zero_guess) {
  const int n = g.n0 >> l, log2n = ilog2(n);
  const mg_params& p = *g.p;
  const float h2 = 1.0f / ((float)n * (float)n);
  const bool scaled = (l == 0 && g.first_cycle && (g.gbox || g.gscale != 1.0f));
  const float* sbox = scaled ? g.gbox : nullptr;
  if (n <= p.coarsest || n <= 4) {
    float* u = g.u[l];
    if (!zero_guess && scaled) {
      const int64_t N = (int64_t)n * n * n;
      PM_LAUNCH(K_MG_GUESS, 8.0 * N * g.B, k_scale, g.grid(grid_for(N, 256)), 256, 0, g.s, u, N, g.gscale, sbox);
    }
#define PM_COARSE(LOG, threads)                                                                                 \
  PM_LAUNCH(K_MG_COARSE, 12.0 * n * n * n * g.B, k_mg_coarse<LOG>, g.grid(1), threads, 0, g.s, u, g.f[l], h2, \
            coarse_omega(p, n), p.coarse_max_sweeps, p.coarse_drop, zero_guess ? 1 : 0)
    if (n == 16) PM_COARSE(4, 256);
    else if (n == 8) PM_COARSE(3, 64);
    else PM_COARSE(2, 32);
#undef PM_COARSE
    return PM_OK;
  }
  if (p.smoother != 1 && n <= kTileN && p.npre >= 1 && p.npre <= 2 && p.npost >= 1 && p.npost <= 2 && g.alt[l] &&
      march_aligned(g.u[l], g.alt[l], g.f[l].p)) {
    PM_TRY(tile_side<true>(g, l, p.npre, zero_guess, scaled ? g.gscale : 1.0f, sbox));
    PM_TRY(v_cycle(g, l + 1, true));
    return tile_side<false>(g, l, p.npost, false, 1.0f, nullptr);
  }
  if (p.npre == 0) {
    const int64_t N = (int64_t)n * n * n;
    if (zero_guess) PM_TRY(cuda_status(cudaMemsetAsync(g.u[l], 0, N * g.B * sizeof(float), g.s)));
    else if (scaled)
      PM_LAUNCH(K_MG_GUESS, 8.0 * N * g.B, k_scale, g.grid(grid_for(N, 256)), 256, 0, g.s, g.u[l], N, g.gscale, sbox);
  } else {
    PM_TRY(smooth(g, l, p.npre, true, zero_guess, scaled ? g.gscale : 1.0f, sbox));
  }
  const int64_t nc = ((int64_t)n * n * n) / 8;
  const unsigned grid = grid_for(nc / 2, 128);
  if (l == 0)
    PM_LAUNCH(K_MG_RESTRICT, 68.0 * nc * g.B, k_resid_restrict<true>, g.grid(grid), 128, 0, g.s, g.u[l], g.f[l],
              log2n, (float)n * (float)n, const_cast<float*>(g.f[l + 1].p));
  else
    PM_LAUNCH(K_MG_RESTRICT, 68.0 * nc * g.B, k_resid_restrict<false>, g.grid(grid), 128, 0, g.s, g.u[l], g.f[l],
              log2n, (float)n * (float)n, const_cast<float*>(g.f[l + 1].p));
  PM_TRY(v_cycle(g, l + 1, true));
  PM_LAUNCH(K_MG_PROLONG, 68.0 * nc * g.B, k_prolong_correct<false>, g.grid(grid_for(nc / 2, 128)), 128, 0, g.s, g.u[l],
            g.u[l + 1], (const float*)nullptr, log2n);
  if (p.npost > 0) PM_TRY(smooth(g, l, p.npost, false, false, 1.0f));
  return PM_OK;
}

}  // namespace

pm_status prolong_correct_launch(float* u, const float* uc, const float* uc2, int n_fine, int cls,
                                 cudaStream_t s, int B) {
  const int64_t N = (int64_t)n_fine * n_fine * n_fine;
  const double bytes = (8.0 * N + (uc2 ? 1.0 : 0.5) * N) * B;
  const dim3 grid(grid_for(N / 16, 128), 1, (unsigned)B);
  if (uc2)
    PM_LAUNCH(cls, bytes, k_prolong_correct<true>, grid, 128, 0, s, u, uc, uc2, ilog2(n_fine));
  else
    PM_LAUNCH(cls, bytes, k_prolong_correct<false>, grid, 128, 0, s, u, uc, uc2, ilog2(n_fine));
  return PM_OK;
}

pm_status fetch_scalars(const double* dev, double* host, int count, cudaStream_t s) {
  static double* pinned = nullptr;
  if (!pinned) PM_TRY(cuda_status(cudaHostAlloc((void**)&pinned, 64 * sizeof(double), cudaHostAllocPortable)));
  PM_TRY(cuda_status(cudaMemcpyAsync(pinned, dev, count * sizeof(double), cudaMemcpyDeviceToHost, s)));
  PM_TRY(cuda_status(cudaStreamSynchronize(s)));
  for (int i = 0; i < count; ++i) host[i] = pinned[i];
  return PM_OK;
}

pm_status mg_solve_batch_src(Src f, float* phi, int n, int B, const mg_params& prm, const float* gbox, Workspace& w,
                         cudaStream_t s) {
  if (B < 1 || prm.fixed_cycles < 1) return PM_EINVAL;
  MG g;
  g.n0 = n;
  g.p = &prm;
  g.s = s;
  g.B = B;
  g.u[0] = phi;
  g.f[0] = f;
  for (int l = 0; l < 12; ++l) {
    if (l > 0) {
      g.u[l] = w.mg_u[l];
      g.f[l] = Src{w.mg_f[l], 1.0f, nullptr};
    }
    g.alt[l] = w.mg_alt[l];
  }
  PM_TRY(march_attributes());
  g.first_cycle = true;
  g.gscale = 1.0f;
  g.gbox = prm.first_guess == MG_GUESS_SCALED ? gbox : nullptr;
  const int64_t N = (int64_t)n * n * n;
  const float h2 = 1.0f / ((float)n * (float)n);
  if (prm.first_guess == MG_GUESS_JACOBI)
    PM_LAUNCH(K_MG_GUESS, 8.0 * N * B, k_jacobi_guess, g.grid(grid_for(N / 4, 256)), 256, 0, s, phi, f, N, h2);
  for (int c = 0; c < prm.fixed_cycles; ++c) {
    PM_TRY(v_cycle(g, 0, false));
    g.first_cycle = false;
    if (g.u[0] != phi) {   // the iterate ended in the ping-pong partner: bring it home
      PM_TRY(cuda_status(cudaMemcpyAsync(phi, g.u[0], N * B * sizeof(float), cudaMemcpyDeviceToDevice, s)));
      g.alt[0] = g.u[0];
      g.u[0] = phi;
    }
  }
  return launch_status();
}

pm_status mg_solve_src(Src f, float* phi, int n, const mg_params& prm, mg_stats* st, Workspace& w,
                       cudaStream_t s) {
  MG g;
  g.n0 = n;
  g.p = &prm;
  g.s = s;
  g.u[0] = phi;
  g.f[0] = f;
  for (int l = 0; l < 12; ++l) {
    if (l > 0) {
      g.u[l] = w.mg_u[l];
      g.f[l] = Src{w.mg_f[l], 1.0f, nullptr};
    }
    g.alt[l] = w.mg_alt[l];
  }
  PM_TRY(march_attributes());
  g.first_cycle = true;
  g.gscale = prm.first_guess == MG_GUESS_SCALED ? prm.guess_scale : 1.0f;
  const int64_t N = (int64_t)n * n * n;
  const float h2 = 1.0f / ((float)n * (float)n);
  if (prm.first_guess == MG_GUESS_JACOBI)
    PM_LAUNCH(K_MG_GUESS, 8.0 * N, k_jacobi_guess, grid_for(N / 4, 256), 256, 0, s, phi, f, N, h2);
  mg_stats local{PM_OK, 0, -1.0, -1.0, -1.0};
  auto cycle = [&]() -> pm_status {
    PM_TRY(v_cycle(g, 0, false));
    g.first_cycle = false;
    if (g.u[0] != phi) {   // the iterate ended in the ping-pong partner: bring it home
      PM_TRY(cuda_status(cudaMemcpyAsync(phi, g.u[0], N * sizeof(float), cudaMemcpyDeviceToDevice, s)));
      g.alt[0] = g.u[0];
      g.u[0] = phi;
    }
    return PM_OK;
  };
  if (prm.fixed_cycles > 0) {
    for (int c = 0; c < prm.fixed_cycles; ++c) PM_TRY(cycle());
    local.cycles = prm.fixed_cycles;
    if (st) *st = local;
    return launch_status();
  }
  const int log2n = ilog2(n);
  const unsigned nb = grid_for(N, 256, 152 * 8);
  double prev = -1.0;
  pm_status status = PM_ENOCONV;
  for (int c = 0; c < prm.max_cycles; ++c) {
    PM_TRY(cycle());
    local.cycles = c + 1;
    PM_LAUNCH(K_MG_NORM, 8.0 * N, k_resid_norm, nb, 256, 0, s, phi, f, log2n, (float)n * (float)n, w.partials);
    PM_TRY(reduce_partials(w.partials, nb, nb, 2, 1.0, w.scalars + 4, s));
    double h[2];
    PM_TRY(fetch_scalars(w.scalars + 4, h, 2, s));
    const double res = sqrt(h[0]), nf = sqrt(h[1]);
    local.res = res;
    local.norm_f = nf;
    if (!isfinite(res)) { status = PM_ENAN; break; }
    if (res <= prm.tol * nf) { status = PM_OK; break; }
    // a cycle that gained less than 1/stall ends the solve only near the
    // float32 floor of the stored iterate (residual below 1e-3 of the source)
    if (prev > 0.0 && prm.stall > 0.0 && res > prm.stall * prev && res <= 1e-3 * nf) { status = PM_OK; break; }
    prev = res;
  }
  local.status = status;
  if (st) *st = local;
  PM_TRY(launch_status());
  return status;
}

pm_status mg_solve_refine_src(const float* f, const double* fmean, double* phi, int n, int outer,
                              const mg_params& prm, mg_stats* st, Workspace& w, cudaStream_t s) {
  const int64_t N = (int64_t)n * n * n;
  const int log2n = ilog2(n);
  const unsigned nb = grid_for(N, 256, 152 * 8);
  const double inv_h2 = (double)n * (double)n;
  mg_params cp = prm;
  cp.first_guess = MG_GUESS_INPUT;   // the correction starts from zero
  mg_stats local{PM_OK, 0, -1.0, -1.0, -1.0};
  // float64 residual of the current iterate into w.ref_r; its norm and ||f - <f>||
  auto residual = [&](double* res, double* nf) -> pm_status {
    PM_LAUNCH(K_MG_NORM, 16.0 * N, k_resid_f64, nb, 256, 0, s, phi, f, fmean, log2n, inv_h2, w.ref_r, w.partials);
    PM_TRY(reduce_partials(w.partials, nb, nb, 2, 1.0, w.scalars + 20, s));
    double h[2];
    PM_TRY(fetch_scalars(w.scalars + 20, h, 2, s));
    *res = sqrt(h[0]);
    *nf = sqrt(h[1]);
    return PM_OK;
  };
  pm_status status = PM_OK;
  for (int it = 0; it <= outer; ++it) {
    double res, nf;
    PM_TRY(residual(&res, &nf));
    if (it == 0) local.res0 = res;
    local.res = res;
    local.norm_f = nf;
    if (!isfinite(res)) { status = PM_ENAN; break; }
    if (it == outer || res == 0.0) break;
    // correction: (L(e) - 6e)/h^2 = r - <r>, float32 multigrid from e = 0
    PM_TRY(grid_mean(w.ref_r, N, w.partials, w.scalars + 22, s));
    PM_TRY(cuda_status(cudaMemsetAsync(w.ref_e, 0, N * sizeof(float), s)));
    mg_stats cst;
    const pm_status r = mg_solve_src(Src{w.ref_r, 1.0f, w.scalars + 22, nullptr}, w.ref_e, n, cp, &cst, w, s);
    if (r != PM_OK && r != PM_ENOCONV) return r;
    local.cycles += cst.cycles;
    PM_LAUNCH(K_MISC, 20.0 * N, k_add_correction_f64, grid_for(N, 256), 256, 0, s, phi, w.ref_e, N);
  }
  local.status = status;
  if (st) *st = local;
  PM_TRY(launch_status());
  return status;
}

}  // namespace pmgb
