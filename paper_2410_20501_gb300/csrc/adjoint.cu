// Adjoint (reverse-mode) kernels of the Newtonian PM step (§3.4-§3.7 forward
// operators, transposed):
//  - gradient: g = -G phi with the antisymmetric Table 1 stencil, so the
//    cotangent is phi_bar = G g_bar summed over axes (G^T = -G);
//  - Poisson: phi = A^+ s (rho - <rho>) with the self-adjoint 7-point
//    Laplacian, so rho_bar = s A^+ phi_bar (the same multigrid solve);
//  - inverse TSC a_p = sum_c W_pc g_c: g_bar = sum_p W_pc a_bar_p (a TSC
//    deposit of a_bar) and x_bar_p += n sum_c dW_pc (g_c . a_bar_p);
//  - TSC deposit rho_c = (n^3/N) sum_p W_pc: x_bar_p += (n^3/N) n sum_c dW_pc rho_bar_c;
//  - kick-drift: v' = v + a dt_kick, x' = x + v' dt_drift.
// dW is the derivative of the product of per-axis TSC weights with respect to
// the particle's offset along one axis (W_TSC is C1, so it is continuous).
#include "pm_device.cuh"
#include "pm_internal.cuh"

namespace pmgb {

namespace {

__device__ __forceinline__ void tsc_dweights(float d, float w[3]) {
  w[0] = d - 0.5f;          // d/dd of (1/2)(1/2 - d)^2
  w[1] = -2.0f * d;         // d/dd of 3/4 - d^2
  w[2] = 0.5f + d;          // d/dd of (1/2)(1/2 + d)^2
}

// a_bar = dt_kick (v_bar' + dt_drift x_bar'), the cotangent reaching the
// acceleration through the kick (x' = x + dt_drift v').
__global__ void k_adj_accel(const float* __restrict__ xbar_out, const float* __restrict__ vbar_out, int64_t np,
                            float dt_kick, float dt_drift, float* __restrict__ abar) {
  pdl_entry();
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < 3 * np;
       i += (int64_t)gridDim.x * blockDim.x)
    abar[i] = dt_kick * fmaf(dt_drift, __ldg(xbar_out + i), __ldg(vbar_out + i));
}

template <int ORDER> struct DStencil;
template <> struct DStencil<3> { static constexpr int R = 1; __device__ static float c(int) { return 0.5f; } };
template <> struct DStencil<5> {
  static constexpr int R = 2;
  __device__ static float c(int k) { return k == 1 ? 2.0f / 3.0f : -1.0f / 12.0f; }
};
template <> struct DStencil<7> {
  static constexpr int R = 3;
  __device__ static float c(int k) { return k == 1 ? 0.75f : (k == 2 ? -0.15f : 1.0f / 60.0f); }
};

// phi_bar = sum_d (1/h) sum_q c_q (g_bar_d(+q) - g_bar_d(-q)).
template <int ORDER>
__global__ void k_divergence(const float* __restrict__ gbar, float* __restrict__ phibar, int log2n, float inv_h) {
  pdl_entry();
  const int64_t N = (int64_t)1 << (3 * log2n);
  const int m = (1 << log2n) - 1;
  for (int64_t c = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; c < N; c += (int64_t)gridDim.x * blockDim.x) {
    const int k = (int)(c & m), j = (int)((c >> log2n) & m), i = (int)(c >> (2 * log2n));
    auto at = [&](int x, int y, int z) -> int64_t {
      return ((int64_t)(x & m) << (2 * log2n)) | ((int64_t)(y & m) << log2n) | (z & m);
    };
    float sx = 0.0f, sy = 0.0f, sz = 0.0f;
#pragma unroll
    for (int q = DStencil<ORDER>::R; q >= 1; --q) {
      const float w = DStencil<ORDER>::c(q);
      sx = fmaf(w, __ldg(gbar + at(i + q, j, k)) - __ldg(gbar + at(i - q, j, k)), sx);
      sy = fmaf(w, __ldg(gbar + N + at(i, j + q, k)) - __ldg(gbar + N + at(i, j - q, k)), sy);
      sz = fmaf(w, __ldg(gbar + 2 * N + at(i, j, k + q)) - __ldg(gbar + 2 * N + at(i, j, k - q)), sz);
    }
    phibar[c] = (sx + sy + sz) * inv_h;
  }
}

// Position (and velocity) cotangents of particle p (in the order of X):
//   x_bar = x_bar' + n sum_c dW q_c,  q_c = a_bar . g_c (with G) + s_rho psi_c
//   (with PSI),   v_bar = v_bar' + dt_drift x_bar'.
// xbar_out/vbar_out may be NULL (term absent).  With perm the results go to
// position perm[p] (back to the step's input order).
//
// The latency of the gathers bounds it: 27 (G: 81) scattered reads a particle,
// L1 holding most of them.  So what counts is how many are in flight, and the
// terms are kept few: the cells' values are contracted with a_bar first, then
// along z, y and x, which leaves three sums instead of a 3 x 3 matrix and three
// more (100 -> 48 registers).  128^3 particles on 128^3: G 156 -> 80 us, PSI 156 -> 33.
template <bool G, bool PSI>
__global__ void __launch_bounds__(256) k_pos_grad(const uint32_t* __restrict__ X, int64_t np, int log2n,
                                                  const float* __restrict__ g, const float* __restrict__ abar,
                                                  const float* __restrict__ psi, float s_rho,
                                                  const float* __restrict__ xbar_out,
                                                  const float* __restrict__ vbar_out, float dt_drift,
                                                  const uint32_t* __restrict__ perm, float* __restrict__ xbar_in,
                                                  float* __restrict__ vbar_in) {
  pdl_entry();
  const int m = (1 << log2n) - 1, sh = 32 - log2n;
  const int64_t N = (int64_t)1 << (3 * log2n);
  const float nf = (float)(1 << log2n);
  const int64_t p = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (p >= np) return;
  const uint32_t x = __ldg(X + p), y = __ldg(X + np + p), z = __ldg(X + 2 * np + p);
  float a[3] = {0.0f, 0.0f, 0.0f};
  if (G) {
#pragma unroll
    for (int d = 0; d < 3; ++d) a[d] = __ldg(abar + d * np + p);
  }
  float wx[3], wy[3], wz[3], vx[3], vy[3], vz[3];   // weights and their derivatives
  const float dx = cell_offset(x, log2n), dy = cell_offset(y, log2n), dz = cell_offset(z, log2n);
  tsc_weights(dx, wx); tsc_weights(dy, wy); tsc_weights(dz, wz);
  tsc_dweights(dx, vx); tsc_dweights(dy, vy); tsc_dweights(dz, vz);
  const int ix = (int)(x >> sh), iy = (int)(y >> sh), iz = (int)(z >> sh);
  float t[3] = {0.0f, 0.0f, 0.0f};
#pragma unroll
  for (int ox = 0; ox < 3; ++ox) {
    float ux = 0.0f, uy = 0.0f, uz = 0.0f;   // this plane's sums: plain, d/dy, d/dz
#pragma unroll
    for (int oy = 0; oy < 3; ++oy) {
      float r = 0.0f, rz = 0.0f;   // this row's sums: plain, d/dz
      const uint32_t row = ((uint32_t)((ix + ox - 1) & m) << (2 * log2n)) | ((uint32_t)((iy + oy - 1) & m) << log2n);
#pragma unroll
      for (int oz = 0; oz < 3; ++oz) {
        const uint32_t c = row | (uint32_t)((iz + oz - 1) & m);
        float q = 0.0f;
        if (G) q = fmaf(a[2], __ldg(g + 2 * N + c), fmaf(a[1], __ldg(g + N + c), a[0] * __ldg(g + c)));
        if (PSI) q = fmaf(s_rho, __ldg(psi + c), q);
        r = fmaf(wz[oz], q, r);
        rz = fmaf(vz[oz], q, rz);
      }
      ux = fmaf(wy[oy], r, ux);
      uy = fmaf(vy[oy], r, uy);
      uz = fmaf(wy[oy], rz, uz);
    }
    t[0] = fmaf(vx[ox], ux, t[0]);
    t[1] = fmaf(wx[ox], uy, t[1]);
    t[2] = fmaf(wx[ox], uz, t[2]);
  }
  const int64_t dst = perm ? (int64_t)__ldg(perm + p) : p;
#pragma unroll
  for (int d = 0; d < 3; ++d) {
    const float xo = xbar_out ? __ldg(xbar_out + d * np + p) : 0.0f;
    xbar_in[d * np + dst] = fmaf(nf, t[d], xo);
    if (vbar_in) {
      const float vo = vbar_out ? __ldg(vbar_out + d * np + p) : 0.0f;
      vbar_in[d * np + dst] = fmaf(dt_drift, xo, vo);
    }
  }
}

template <int ORDER>
void launch_div(const float* gbar, float* phibar, int n, cudaStream_t s) {
  const int64_t N = (int64_t)n * n * n;
  PM_LAUNCH(K_ADJOINT, 16.0 * N, k_divergence<ORDER>, grid_for(N, 256), 256, 0, s, gbar, phibar, ilog2(n), (float)n);
}

}  // namespace

pm_status divergence_launch(const float* gbar, float* phibar, int n, int order, cudaStream_t s) {
  if (order == 3) launch_div<3>(gbar, phibar, n, s);
  else if (order == 5) launch_div<5>(gbar, phibar, n, s);
  else if (order == 7) launch_div<7>(gbar, phibar, n, s);
  else return PM_EINVAL;
  return launch_status();
}

pm_status adj_accel_launch(const float* xbar_out, const float* vbar_out, int64_t np, float dt_kick, float dt_drift,
                           float* abar, cudaStream_t s) {
  if (np == 0) return PM_OK;
  PM_LAUNCH(K_ADJOINT, 36.0 * np, k_adj_accel, grid_for(3 * np, 256), 256, 0, s, xbar_out, vbar_out, np, dt_kick,
            dt_drift, abar);
  return launch_status();
}

pm_status pos_grad_launch(const uint32_t* X, int64_t np, int n, const float* g, const float* abar, const float* psi,
                          float s_rho, const float* xbar_out, const float* vbar_out, float dt_drift,
                          const uint32_t* perm, float* xbar_in, float* vbar_in, cudaStream_t s) {
  if (np == 0) return PM_OK;
  const double N = (double)n * n * n;
  const double bytes = (g ? 12.0 * N : 0.0) + (psi ? 4.0 * N : 0.0) +
                       np * (12.0 + (abar ? 12.0 : 0.0) + (perm ? 4.0 : 0.0) + (xbar_out ? 12.0 : 0.0) +
                             (vbar_out ? 12.0 : 0.0) + 12.0 + (vbar_in ? 12.0 : 0.0));
#define PM_POS_GRAD(G, PSI)                                                                                          \
  PM_LAUNCH(K_ADJOINT, bytes, (k_pos_grad<G, PSI>), grid_for(np, 256), 256, 0, s, X, np, ilog2(n), g, abar, psi, s_rho, \
            xbar_out, vbar_out, dt_drift, perm, xbar_in, vbar_in)
  if (g && psi) PM_POS_GRAD(true, true);
  else if (g) PM_POS_GRAD(true, false);
  else PM_POS_GRAD(false, true);
#undef PM_POS_GRAD
  return launch_status();
}

}  // namespace pmgb
