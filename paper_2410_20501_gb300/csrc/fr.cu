// Hu-Sawicki f(R) scalaron (n = 1 and n = 2) by non-linear FAS multigrid
// (§3.6.2, §3.10).  The kernels are templates on the exponent NH; the text
// below is for n = 1, and n = 2 follows the same pattern with u^3:
//   N_h(eps) = (fbar/h^2) sum_nb (eps_nb - eps)(3 + 3 eps_nb + 3 eps + eps_nb^2
//              + eps_nb eps + eps^2) + kappa eps/(1 + eps),
//   eps^4 + 4 eps^3 + 6 eps^2 + c1 eps + c0 = 0, c1 = 3 + beta (b - kappa) - T/6,
//   c0 = beta b - T/6, T = sum_nb eps_nb (3 + 3 eps_nb + eps_nb^2)
// (u^4 + p u + q = 0, the quartic of §3.10, with u = 1 + eps).
//
// Unknown: eps = u - 1 with u = (f~_R / fbar)^(1/2).  Discrete operator
//   N_h(eps) = (fbar/h^2) sum_nb (eps_nb - eps)(2 + eps_nb + eps) + kappa eps/(1 + eps)
// (= (fbar/h^2)(L(u^2) - 6u^2) - kappa (1/u - 1) written in differences, so the
// O(1) background cancels analytically), equation N_h(eps) = b.
// Gauss-Seidel: with the neighbours fixed, u solves the depressed cubic
// u^3 + p u + q = 0 of Eq. fr_depressed_equation; in eps it reads
//   eps^3 + 3 eps^2 + c1 eps + c0 = 0,
//   c1 = 2 + beta (b - kappa) - S/6,  c0 = beta b - S/6,
//   S = sum_nb eps_nb (2 + eps_nb),   beta = h^2 / (6 fbar),  q = beta kappa < 0,
// whose unique root eps > -1 is found in float32 by safeguarded Newton (the
// paper evaluates the closed-form root in float64, which the eps form makes
// unnecessary: no term of size 1 is ever subtracted).
#include <math.h>

#include "pm_device.cuh"
#include "pm_internal.cuh"
#include "rb_march.cuh"

namespace pmgb {

namespace {

__device__ __forceinline__ float load_mean(const Src& f) { return f.mean ? (float)*f.mean : 0.0f; }
__device__ __forceinline__ float src_at(const Src& f, int64_t i, float mean) {
  return f.s * (__ldg(f.p + i) - mean);
}
// Offset of cell (i, j, k) inside one box (n <= 1024: below 2^30).
__device__ __forceinline__ uint32_t idx3(int i, int j, int k, int log2n) {
  return ((uint32_t)i << (2 * log2n)) | ((uint32_t)j << log2n) | (uint32_t)k;
}

// Root eps > -1 of g(e) = e^3 + 3e^2 + c1 e + c0 (g(-1) = q < 0, g convex on
// e > -1, so the root is unique).  One step of root_step from the current value
// reaches float32 resolution in a warm sweep (the value moved little since the
// last one); what is left goes to Newton inside a shrinking bracket [lo, hi]
// (fr_root): when a step leaves the bracket (or g' <= 0) the upper end is set
// from the bound u* <= sqrt(max(-p, 0)) + (-q)^(1/3), p = c1 - 3, and the step
// falls back to bisection.  It stops when g is at its float32 rounding level or
// the step is below 2e-7 relative.
// g(e) of the cell equation in eps = u - 1 (NH = 1: cubic, NH = 2: quartic),
// its derivative, the
// float32 rounding level of its evaluation, and an upper bound of the root
// (from u* <= sqrt(max(-p, 0)) + (-q)^(1/3) for the cubic,
// u* <= max(1, (|p| + |q|)^(1/3)) for the quartic).
template <int NH> struct CellPoly;
template <> struct CellPoly<1> {
  __device__ static float g(float e, float c1, float c0) { return ((e + 3.0f) * e + c1) * e + c0; }
  __device__ static float gp(float e, float c1) { return (3.0f * e + 6.0f) * e + c1; }
  __device__ static float noise(float e, float c1, float c0) {
    const float e2 = e * e;
    return 1.5e-7f * (fabsf(c0) + fabsf(c1 * e) + 3.0f * e2 + fabsf(e2 * e));
  }
  __device__ static float upper(float c1, float q, float lo) {
    return fmaxf(sqrtf(fmaxf(3.0f - c1, 0.0f)) + cbrtf(-q) - 1.0f, lo);
  }
};
template <> struct CellPoly<2> {
  __device__ static float g(float e, float c1, float c0) { return (((e + 4.0f) * e + 6.0f) * e + c1) * e + c0; }
  __device__ static float gp(float e, float c1) { return ((4.0f * e + 12.0f) * e + 12.0f) * e + c1; }
  __device__ static float noise(float e, float c1, float c0) {
    const float e2 = e * e;
    return 1.5e-7f * (fabsf(c0) + fabsf(c1 * e) + 6.0f * e2 + 4.0f * fabsf(e2 * e) + e2 * e2);
  }
  __device__ static float upper(float c1, float q, float lo) {
    return fmaxf(fmaxf(cbrtf(fabsf(c1 - 4.0f) + fabsf(q)), 1.0f) - 1.0f, lo);
  }
};

template <int NH>
__device__ __forceinline__ float fr_root(float e, float c1, float c0, float q) {
  using P = CellPoly<NH>;
  float lo = -1.0f, hi = __int_as_float(0x7f800000);  // +inf until needed
  if (!(e > lo)) e = 0.0f;
  for (int it = 0; it < 30; ++it) {
    const float g = P::g(e, c1, c0);
    const float gp = P::gp(e, c1);
    if (g > 0.0f) hi = fminf(hi, e);
    else if (g < 0.0f) lo = fmaxf(lo, e);
    else return e;
    if (fabsf(g) <= P::noise(e, c1, c0)) return e;
    float en = gp > 0.0f ? e - __fdividef(g, gp) : lo;
    if (!(en > lo && en < hi)) {
      if (isinf(hi)) hi = P::upper(c1, q, lo);
      en = 0.5f * (lo + hi);
    }
    if (fabsf(en - e) <= 2e-7f * fabsf(en) + 1e-12f) return en;
    e = en;
  }
  return e;
}

__device__ __forceinline__ void load_nb(const float* u, int i, int j, int k, int log2n, float nb[6]) {
  const int m = (1 << log2n) - 1;
  nb[0] = u[idx3((i + 1) & m, j, k, log2n)];
  nb[1] = u[idx3((i - 1) & m, j, k, log2n)];
  nb[2] = u[idx3(i, (j + 1) & m, k, log2n)];
  nb[3] = u[idx3(i, (j - 1) & m, k, log2n)];
  nb[4] = u[idx3(i, j, (k + 1) & m, log2n)];
  nb[5] = u[idx3(i, j, (k - 1) & m, log2n)];
}

// N_h(eps) at one cell: (fbar/h^2) sum_nb (u_nb^(n+1) - u^(n+1)) written in
// differences, plus kappa eps/(1 + eps).
template <int NH>
__device__ __forceinline__ float fr_op(float ec, const float nb[6], float alpha, float kappa) {
  float L = 0.0f;
#pragma unroll
  for (int q = 0; q < 6; ++q) {
    if (NH == 1) {
      L = fmaf(nb[q] - ec, 2.0f + nb[q] + ec, L);
    } else {   // u_nb^3 - u^3 = (e_nb - e)(3 + 3 (e_nb + e) + e_nb^2 + e_nb e + e^2)
      const float s = nb[q] + ec;
      L = fmaf(nb[q] - ec, fmaf(3.0f, s, 3.0f) + fmaf(nb[q], s, ec * ec), L);
    }
  }
  return alpha * L + kappa * ec / (1.0f + ec);
}

// Approximate reciprocal (one instruction; a denormal argument gives infinity).
__device__ __forceinline__ float rcp_approx(float x) {
  float r;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
  return r;
}

// Cells in pairs (the paired float instructions halve the arithmetic of the
// root, which is most of a sweep).  Accumulates a neighbour's term of S:
// nb (2 + nb), for NH = 2 nb (3 + 3 nb + nb^2).
template <int NH>
__device__ __forceinline__ float2 add_term(float2 s, float2 nb) {
  return NH == 1 ? fma2(nb, add2(nb, both(2.0f)), s) : fma2(nb, fma2(nb, add2(nb, both(3.0f)), both(3.0f)), s);
}

// One step of a pair: Halley's, and from its point a Newton step with the slope
// g' + g'' d/2 that Halley's denominator holds; the value of g there is its
// (finite) Taylor sum.  With x = g g'' / (2 g'^2) (about g'' d / (2 g')) and
// s = d^2 times a sixth of the third derivative over g' the remaining error is about (x^3 + x s) d, so the step
// counts as done (ok) for |x| <= 0.006 and s < 1e-5, when that is below 3e-7 d.
// Written with few constants and signs (a pair instruction takes neither
// immediates nor, cheaply, a negated operand) and a test of five instructions a
// cell: the arithmetic is what a sweep takes.
template <int NH>
__device__ __forceinline__ float2 root_step(float2 e, float2 c1, float2 c0, bool& okx, bool& oky) {
  float2 g, gp, hg, sixth;   // g, its derivative, half its second and (NH = 2) a sixth of its third
  if (NH == 1) {
    const float2 t = mul2(e, add2(e, both(2.0f)));   // e^2 + 2 e
    g = fma2(add2(add2(t, e), c1), e, c0);
    gp = fma2(t, both(3.0f), c1);
    hg = fma2(e, both(3.0f), both(3.0f));
  } else {
    const float2 u = add2(e, both(1.0f));
    g = fma2(fma2(fma2(add2(e, both(4.0f)), e, both(6.0f)), e, c1), e, c0);
    gp = fma2(fma2(fma2(e, both(4.0f), both(12.0f)), e, both(12.0f)), e, c1);
    hg = mul2(mul2(u, u), both(6.0f));
    sixth = mul2(u, both(4.0f));
  }
  const float2 n = mul2(g, hg), gp2 = mul2(gp, gp);
  const float2 slope = make_float2(-gp.x * rcp_approx(gp2.x - n.x), -gp.y * rcp_approx(gp2.y - n.y));
  const float2 d = mul2(g, slope), e1 = add2(e, d);
  const float2 g1 = NH == 1 ? fma2(fma2(add2(hg, d), d, gp), d, g)
                            : fma2(fma2(fma2(add2(sixth, d), d, hg), d, gp), d, g);
  const float2 e2 = fma2(g1, slope, e1);
  const float2 s = NH == 1 ? mul2(d, d) : mul2(mul2(d, d), sixth);
  okx = fmaf(0.006f, gp2.x, -fabsf(n.x)) >= 0.0f && fmaf(1e-5f, gp.x, -s.x) > 0.0f && e2.x > -1.0f;
  oky = fmaf(0.006f, gp2.y, -fabsf(n.y)) >= 0.0f && fmaf(1e-5f, gp.y, -s.y) > 0.0f && e2.y > -1.0f;
  return e2;
}

// Roots of NP pairs of cell equations from the current values e: one step for
// all, which settles nearly every warm cell, and for those of the cells `need`
// (two bits a pair) that it does not a second one and then fr_root, one by one
// (selected, not indexed or called: the pairs stay in registers).
template <int NH, int NP>
__device__ __forceinline__ void fr_roots(float2 (&e)[NP], const float2 (&c1)[NP], const float2 (&c0)[NP], float q,
                                         unsigned need) {
  static_assert(NP == 1 || NP == 2, "one or two pairs");
  unsigned fail = 0;
  float2 n[NP];
#pragma unroll
  for (int i = 0; i < NP; ++i) {
    bool okx, oky;
    n[i] = root_step<NH>(e[i], c1[i], c0[i], okx, oky);
    if (!okx) fail |= 1u << (2 * i);
    if (!oky) fail |= 2u << (2 * i);
  }
  fail &= need;
  if (fail) {
#pragma unroll
    for (int i = 0; i < NP; ++i) {
      // from the step's point, or where it left the admissible range from its start
      const float2 f = make_float2(n[i].x > -1.0f && n[i].x < 1e3f ? n[i].x : e[i].x,
                                   n[i].y > -1.0f && n[i].y < 1e3f ? n[i].y : e[i].y);
      bool okx, oky;
      const float2 r = root_step<NH>(f, c1[i], c0[i], okx, oky);
      if (fail & (1u << (2 * i))) n[i].x = okx ? r.x : f.x;
      if (fail & (2u << (2 * i))) n[i].y = oky ? r.y : f.y;
      if (okx) fail &= ~(1u << (2 * i));
      if (oky) fail &= ~(2u << (2 * i));
    }
    for (; fail; fail &= fail - 1u) {
      const bool hi = NP == 2 && (fail & 3u) == 0u, y = ((hi ? fail >> 2 : fail) & 1u) == 0u;
      const float2 pe = hi ? n[NP - 1] : n[0], p1 = hi ? c1[NP - 1] : c1[0], p0 = hi ? c0[NP - 1] : c0[0];
      const float r = fr_root<NH>(y ? pe.y : pe.x, y ? p1.y : p1.x, y ? p0.y : p0.x, q);
      if (!hi && !y) n[0].x = r;
      if (!hi && y) n[0].y = r;
      if (hi && !y) n[NP - 1].x = r;
      if (hi && y) n[NP - 1].y = r;
    }
  }
#pragma unroll
  for (int i = 0; i < NP; ++i) e[i] = n[i];
}

// The cell equations of NP pairs with neighbour terms S and sources b (as
// beta b): c0 = beta b - S/6, c1 = c0 + k1, k1 = 2 - beta kappa (3 for NH = 2).
template <int NH, int NP>
__device__ __forceinline__ void fr_updates(float2 (&e)[NP], const float2 (&S)[NP], const float2 (&bb)[NP], float k1,
                                           float q, unsigned need = ~0u) {
  float2 c0[NP], c1[NP];
#pragma unroll
  for (int i = 0; i < NP; ++i) {
    c0[i] = fma2(S[i], both(-1.0f / 6.0f), bb[i]);
    c1[i] = add2(c0[i], both(k1));
  }
  fr_roots<NH, NP>(e, c1, c0, q, need);
}

// The sweeps of a level as the policy of k_rb_march; sources enter as beta b.
template <int NH>
struct CellSweeps {
  float beta, k1, q;
  __device__ __forceinline__ void box(int) {}
  __device__ __forceinline__ float2 source(float2 b) const { return mul2(both(beta), b); }
  __device__ __forceinline__ static float2 first(float2 a, float2 b) {
    return add_term<NH>(add_term<NH>(both(0.0f), a), b);
  }
  __device__ __forceinline__ static float2 add(float2 s, float2 nb) { return add_term<NH>(s, nb); }
  __device__ __forceinline__ static float2 add(float2 s, float x, float y) {
    return add_term<NH>(s, make_float2(x, y));
  }
  template <int ST>
  __device__ __forceinline__ void update(float2 (&v)[2], const float2 (&s)[2], const float2 (&bb)[2],
                                         unsigned need) const {
    fr_updates<NH, 2>(v, s, bb, k1, q, need);
  }
};

// One colour of a sweep, four z cells (one pair of the colour) a thread with
// 16-byte row loads, as the linear k_rb_sweep: these levels live in L2, and the
// latency of the loads and of the root is what a pass takes.
constexpr int kSweepThreads = 128;
template <int NH>
__global__ void __launch_bounds__(kSweepThreads) k_fr_sweep(float* __restrict__ e, Src b, int log2n, int colour,
                                                            float beta, float k1, float q) {
  pdl_entry();
  const uint32_t t = blockIdx.x * kSweepThreads + threadIdx.x;
  if (t >= 1u << (3 * log2n - 2)) return;
  {   // the box of a batched launch
    const int64_t N = (int64_t)1 << (3 * log2n);
    e += (int64_t)blockIdx.z * N;
    b = box_src(b, N);
  }
  const int m = (1 << log2n) - 1;
  const int k0 = (int)(t << 2) & m, j = (int)(t >> (log2n - 2)) & m, i = (int)(t >> (2 * log2n - 2));
  const bool odd = ((colour + i + j) & 1) != 0;   // cells k0 + odd and k0 + odd + 2
  const uint32_t c = idx3(i, j, k0, log2n);
  auto row4 = [&](int ii, int jj) { return *reinterpret_cast<const float4*>(e + idx3(ii & m, jj & m, k0, log2n)); };
  const float4 XP = row4(i + 1, j), XM = row4(i - 1, j), YP = row4(i, j + 1), YM = row4(i, j - 1), C = row4(i, j);
  const float ze = e[idx3(i, j, (odd ? k0 + 4 : k0 - 1) & m, log2n)];
  const float4 F = __ldg(reinterpret_cast<const float4*>(b.p + c));
  const float mean = load_mean(b);
  auto mine = [&](const float4& v) { return odd ? make_float2(v.y, v.w) : make_float2(v.x, v.z); };
  float2 S[1] = {add_term<NH>(both(0.0f), mine(XP))};
  S[0] = add_term<NH>(S[0], mine(XM));
  S[0] = add_term<NH>(S[0], mine(YP));
  S[0] = add_term<NH>(S[0], mine(YM));
  S[0] = add_term<NH>(S[0], odd ? make_float2(C.z, ze) : make_float2(C.y, C.w));
  S[0] = add_term<NH>(S[0], odd ? make_float2(C.x, C.z) : make_float2(ze, C.y));
  const float2 bb[1] = {mul2(both(beta), mul2(both(b.s), add2(mine(F), both(-mean))))};
  float2 v[1] = {mine(C)};
  fr_updates<NH, 1>(v, S, bb, k1, q);
  e[c + odd] = v[0].x;
  e[c + odd + 2] = v[0].y;
}

// L + the non-linear fluxes of N_h through two faces, (u_nb^(n+1) - u^(n+1)) in
// eps differences; a flux changes sign with its face's orientation.
template <int NH>
__device__ __forceinline__ float2 add_flux(float2 L, float2 enb, float2 ec) {
  const float2 d = fma2(ec, both(-1.0f), enb);
  if (NH == 1) return fma2(d, add2(add2(both(2.0f), enb), ec), L);
  const float2 s = add2(enb, ec);
  return fma2(d, add2(fma2(both(3.0f), s, both(3.0f)), fma2(enb, s, mul2(ec, ec))), L);
}

// eH = rH = R eps, bH = R(b - N_h eps).  Summed over the 2x2x2 block the
// fluxes through the 12 inner faces cancel pairwise, so only the 24 outer
// faces enter the restricted operator.  BOXES: a batched launch (box =
// blockIdx.z); the single-box form keeps its own register allocation.
//
// A thread takes two coarse cells along z: their fine rows come in 16-byte loads
// and the fluxes of the two go through the paired float instructions, which with
// the eight divisions a cell it is bound by.  512^3: 353 -> 242 us against one cell
// a thread, 256^3 47 -> 34.
template <int NH, bool BOXES>
__global__ void __launch_bounds__(128) k_fr_restrict(const float* __restrict__ e, Src b, int log2n, float alpha,
                                                     float kappa, float* __restrict__ eH, float* __restrict__ rH,
                                                     float* __restrict__ bH) {
  pdl_entry();
  const int lc = log2n - 1, mc = (1 << lc) - 1, m = (1 << log2n) - 1, lg = lc - 1;
  if (BOXES) {   // the box of a batched launch
    e += (int64_t)blockIdx.z << (3 * log2n);
    b = box_src(b, (int64_t)1 << (3 * log2n));
    const int64_t offc = (int64_t)blockIdx.z << (3 * lc);
    eH += offc;
    rH += offc;
    bH += offc;
  }
  const uint32_t t = blockIdx.x * blockDim.x + threadIdx.x;   // two coarse cells, K = 2 G and 2 G + 1
  if (t >= 1u << (3 * lc - 1)) return;
  const int G = (int)(t & ((1u << lg) - 1u)), J = (int)(t >> lg) & mc, I = (int)(t >> (lg + lc));
  const int z0 = 4 * G;
  auto row = [&](const float* p, int x, int y) {
    return __ldg(reinterpret_cast<const float4*>(p + idx3(x & m, y & m, z0, log2n)));
  };
  float4 core[2][2], xf[2][2], yf[2][2], br[2][2];   // [x][y], [side][y], [x][side], [x][y]
  float zl[2][2], zr[2][2];
#pragma unroll
  for (int a = 0; a < 2; ++a)
#pragma unroll
    for (int c = 0; c < 2; ++c) {
      core[a][c] = row(e, 2 * I + a, 2 * J + c);
      zl[a][c] = __ldg(e + idx3(2 * I + a, 2 * J + c, (z0 - 1) & m, log2n));
      zr[a][c] = __ldg(e + idx3(2 * I + a, 2 * J + c, (z0 + 4) & m, log2n));
      xf[a][c] = row(e, a ? 2 * I + 2 : 2 * I - 1, 2 * J + c);
      yf[a][c] = row(e, 2 * I + a, c ? 2 * J + 2 : 2 * J - 1);
      br[a][c] = row(b.p, 2 * I + a, 2 * J + c);
    }
  const float mean = load_mean(b);
  // (first coarse cell, second coarse cell): even fine cells, odd fine cells
  auto ev = [](const float4& v) { return make_float2(v.x, v.z); };
  auto od = [](const float4& v) { return make_float2(v.y, v.w); };
  auto source = [&](float2 v) { return mul2(both(b.s), add2(v, both(-mean))); };
  auto fraction = [](float2 v) { return make_float2(v.x / (1.0f + v.x), v.y / (1.0f + v.y)); };
  float2 se = both(0.0f), sb = se, sk = se, Lx = se, Ly = se, Lz = se;
#pragma unroll
  for (int a = 0; a < 2; ++a)
#pragma unroll
    for (int c = 0; c < 2; ++c) {
      const float2 c0 = ev(core[a][c]), c1 = od(core[a][c]);
      sb = add2(sb, add2(source(ev(br[a][c])), source(od(br[a][c]))));
      se = add2(add2(se, c0), c1);
      sk = add2(add2(sk, fraction(c0)), fraction(c1));
      Lx = add_flux<NH>(add_flux<NH>(Lx, ev(xf[a][c]), c0), od(xf[a][c]), c1);
      Ly = add_flux<NH>(add_flux<NH>(Ly, ev(yf[a][c]), c0), od(yf[a][c]), c1);
      Lz = add_flux<NH>(add_flux<NH>(Lz, make_float2(zl[a][c], core[a][c].y), c0), make_float2(core[a][c].z, zr[a][c]), c1);
    }
  const float2 ops = fma2(both(alpha), add2(add2(Lx, Ly), Lz), mul2(both(kappa), sk));
  const float2 mean_e = mul2(both(0.125f), se);
  reinterpret_cast<float2*>(eH)[t] = mean_e;
  reinterpret_cast<float2*>(rH)[t] = mean_e;
  reinterpret_cast<float2*>(bH)[t] = mul2(both(0.125f), fma2(ops, both(-1.0f), sb));
}

// bH += N_H(eH).  A thread takes four consecutive z cells of a row (n >= 4):
// the rows at x +- 1, y +- 1 and its own in 16-byte loads, plus the two z
// neighbours beyond the run; each cell sees its neighbours in the order
// x+, x-, y+, y-, z+, z- as everywhere else.
template <int NH>
__global__ void k_fr_coarse_op(const float* __restrict__ eH, float* __restrict__ bH, int log2n, float alpha,
                               float kappa) {
  pdl_entry();
  const uint32_t m = (1u << log2n) - 1;
  const uint32_t quads = 1u << (3 * log2n - 2);
  {   // the box of a batched launch
    const int64_t off = (int64_t)blockIdx.z << (3 * log2n);
    eH += off;
    bH += off;
  }
  for (uint32_t t = blockIdx.x * blockDim.x + threadIdx.x; t < quads; t += gridDim.x * blockDim.x) {
    const uint32_t c0 = t << 2;
    const uint32_t k0 = c0 & m, j = (c0 >> log2n) & m, i = c0 >> (2 * log2n);
    auto rowp = [&](uint32_t ii, uint32_t jj) -> const float* {
      return eH + (((ii & m) << (2 * log2n)) | ((jj & m) << log2n));
    };
    const float* rc = rowp(i, j);
    const float4 C = __ldg(reinterpret_cast<const float4*>(rc + k0));
    const float4 XP = __ldg(reinterpret_cast<const float4*>(rowp(i + 1, j) + k0));
    const float4 XM = __ldg(reinterpret_cast<const float4*>(rowp(i - 1, j) + k0));
    const float4 YP = __ldg(reinterpret_cast<const float4*>(rowp(i, j + 1) + k0));
    const float4 YM = __ldg(reinterpret_cast<const float4*>(rowp(i, j - 1) + k0));
    const float zl = __ldg(rc + ((k0 - 1) & m)), zr = __ldg(rc + ((k0 + 4) & m));
    float4* bp = reinterpret_cast<float4*>(bH + c0);
    float4 B = *bp;
    const float e[4] = {C.x, C.y, C.z, C.w}, xp[4] = {XP.x, XP.y, XP.z, XP.w}, xm[4] = {XM.x, XM.y, XM.z, XM.w},
                yp[4] = {YP.x, YP.y, YP.z, YP.w}, ym[4] = {YM.x, YM.y, YM.z, YM.w};
    float r[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const float nb[6] = {xp[q], xm[q], yp[q], ym[q], q < 3 ? e[q + 1] : zr, q > 0 ? e[q - 1] : zl};
      r[q] = fr_op<NH>(e[q], nb, alpha, kappa);
    }
    B.x += r[0];
    B.y += r[1];
    B.z += r[2];
    B.w += r[3];
    *bp = B;
  }
}

template <int NH>
__global__ void __launch_bounds__(256) k_fr_norm(const float* __restrict__ e, Src b, int log2n, float alpha,
                                                 float kappa, double* __restrict__ partial) {
  pdl_entry();
  __shared__ double scratch[32];
  const float mean = load_mean(b);
  const int m = (1 << log2n) - 1;
  const int64_t total = (int64_t)1 << (3 * log2n);
  float sd = 0.0f, cd = 0.0f, sb = 0.0f, cb = 0.0f;
  for (uint32_t c = blockIdx.x * blockDim.x + threadIdx.x; c < total; c += gridDim.x * blockDim.x) {
    const int k = (int)(c & m), j = (int)((c >> log2n) & m), i = (int)(c >> (2 * log2n));
    float nb[6];
    load_nb(e, i, j, k, log2n, nb);
    const float bv = src_at(b, c, mean);
    const float d = bv - fr_op<NH>(e[c], nb, alpha, kappa);
    kahan_add(sd, cd, d * d);
    kahan_add(sb, cb, bv * bv);
  }
  block_sum_to(partial + blockIdx.x, sd, cd, scratch);
  block_sum_to(partial + gridDim.x + blockIdx.x, sb, cb, scratch);
}

// Coarsest level (n = 4, 8 or 16) in one CTA: non-linear sweeps until the
// residual dropped by `drop`, its running minimum stalls for 5 sweeps (float32
// floor), or `max_sweeps` sweeps.
//
// One SM's arithmetic bounds it (a root for each of 4096 cells a sweep), and the
// barriers.  A thread owns up to eight z cells of a row, two pairs of either
// colour, in registers; shared memory holds the colours of a row apart (as in
// k_mg_coarse), so its x and y neighbours come in 16-byte loads.  The residual
// of a black pair is taken when it has been updated, that of a red pair when the
// next sweep updates it, from the neighbours that are at hand; the block's norm
// is summed by one warp beside the black pass, and a sweep too many is undone
// from the values kept: two barriers a sweep.  16^3: 46 -> 25 us a
// solve against separate passes for the norm and a cell at a time.
template <int NH, int LOG>
struct FrCoarse {
  static constexpr int n = 1 << LOG, H = n / 2, NP = H >= 4 ? 2 : 1, PARTS = H / (2 * NP);   // threads per row
  static constexpr int RUNS = n * n * PARTS, THREADS = RUNS < 32 ? 32 : RUNS;
};
template <int NH, int LOG>
__global__ void __launch_bounds__(FrCoarse<NH, LOG>::THREADS) k_fr_coarse(float* __restrict__ e, Src b, float alpha,
                                                                          float beta, float kappa, float k1, float q,
                                                                          int max_sweeps, float drop) {
  pdl_entry();
  using C = FrCoarse<NH, LOG>;
  constexpr int n = C::n, m = n - 1, H = C::H, NP = C::NP, HK = 2 * NP, N = n * n * n, NW = C::THREADS / 32;
  __shared__ alignas(16) float S[2][N / 2];   // [colour][row][kk]: cell z = 2 kk + parity of (row, colour)
  __shared__ float2 part[NW];
  __shared__ float total;
  e += (int64_t)blockIdx.z * N;   // one CTA per box of a batched launch
  b = box_src(b, N);
  const float mean = load_mean(b);
  const bool act = threadIdx.x < C::RUNS;
  const int t = act ? threadIdx.x : 0, row = t / C::PARTS, kk0 = (t - row * C::PARTS) * HK;
  const int i = row >> LOG, j = row & m, par = (i + j) & 1;
  const int own = row * H + kk0;
  const int xp = ((((i + 1) & m) << LOG) | j) * H + kk0, xm = ((((i - 1) & m) << LOG) | j) * H + kk0;
  const int yp = ((i << LOG) | ((j + 1) & m)) * H + kk0, ym = ((i << LOG) | ((j - 1) & m)) * H + kk0;
  float2 v[2][NP], src[2][NP];   // [colour]: values and sources
#pragma unroll
  for (int p = 0; p < NP; ++p) {   // natural order -> colours (red: z = 2 kk + par)
    const int z = row * n + 2 * kk0 + 4 * p;
    const float4 u = *reinterpret_cast<const float4*>(e + z), f = __ldg(reinterpret_cast<const float4*>(b.p + z));
    const float fs[4] = {b.s * (f.x - mean), b.s * (f.y - mean), b.s * (f.z - mean), b.s * (f.w - mean)};
    v[0][p] = par ? make_float2(u.y, u.w) : make_float2(u.x, u.z);
    v[1][p] = par ? make_float2(u.x, u.z) : make_float2(u.y, u.w);
    src[0][p] = par ? make_float2(fs[1], fs[3]) : make_float2(fs[0], fs[2]);
    src[1][p] = par ? make_float2(fs[0], fs[2]) : make_float2(fs[1], fs[3]);
  }
  auto put = [&](int c, const float2 (&w)[NP]) {
    if (!act) return;
#pragma unroll
    for (int p = 0; p < NP; ++p) *reinterpret_cast<float2*>(&S[c][own + 2 * p]) = w[p];
  };
  // the six neighbours of the thread's pairs of colour c, x+ .. z-
  auto neighbours = [&](int c, float2 (&nb)[6][NP]) {
    const float* w = S[1 - c];
    const int at[4] = {xp, xm, yp, ym};
#pragma unroll
    for (int d = 0; d < 4; ++d)
#pragma unroll
      for (int p = 0; p < NP; ++p) nb[d][p] = *reinterpret_cast<const float2*>(w + at[d] + 2 * p);
    const bool o = ((c + par) & 1) != 0;
    const float ze = w[row * H + (o ? (kk0 + HK) & (H - 1) : (kk0 + H - 1) & (H - 1))];
#pragma unroll
    for (int p = 0; p < NP; ++p) {
      const float2 x = v[1 - c][p];
      const float before = p > 0 ? v[1 - c][p > 0 ? p - 1 : 0].y : ze, after = p < NP - 1 ? v[1 - c][p < NP - 1 ? p + 1 : p].x : ze;
      nb[4][p] = o ? make_float2(x.y, after) : x;
      nb[5][p] = o ? x : make_float2(before, x.x);
    }
  };
  float sum = 0.0f, cmp = 0.0f;   // compensated sum of squared residuals
  auto residuals = [&](int c, const float2 (&nb)[6][NP]) {
#pragma unroll
    for (int p = 0; p < NP; ++p) {
      const float2 x = v[c][p], nx = mul2(x, both(-1.0f));
      float2 L = both(0.0f);
#pragma unroll
      for (int d = 0; d < 6; ++d) {
        const float2 s = add2(nb[d][p], x), df = add2(nb[d][p], nx);
        const float2 w = NH == 1 ? add2(s, both(2.0f)) : add2(fma2(s, both(3.0f), both(3.0f)), fma2(nb[d][p], s, mul2(x, x)));
        L = fma2(df, w, L);
      }
      const float d0 = src[c][p].x - fmaf(alpha, L.x, kappa * x.x / (1.0f + x.x));
      const float d1 = src[c][p].y - fmaf(alpha, L.y, kappa * x.y / (1.0f + x.y));
      kahan_add(sum, cmp, d0 * d0);
      kahan_add(sum, cmp, d1 * d1);
    }
  };
  auto update = [&](int c, const float2 (&nb)[6][NP], float2 (&out)[NP]) {
    float2 T[NP], bb[NP];
#pragma unroll
    for (int p = 0; p < NP; ++p) {
      T[p] = both(0.0f);
#pragma unroll
      for (int d = 0; d < 6; ++d) T[p] = add_term<NH>(T[p], nb[d][p]);
      bb[p] = mul2(both(beta), src[c][p]);
      out[p] = v[c][p];
    }
    fr_updates<NH, NP>(out, T, bb, k1, q);
  };
  auto pair_add = [](float& s, float& c, float os, float oc) {
    float r, err;
    two_sum(s, os, r, err);
    s = r;
    c = c + oc + err;
  };
  auto lanes_sum = [&](float& s, float& c) {
#pragma unroll
    for (int d = 16; d > 0; d >>= 1) {
      const float os = __shfl_xor_sync(0xffffffffu, s, d), oc = __shfl_xor_sync(0xffffffffu, c, d);
      pair_add(s, c, os, oc);
    }
  };
  auto warp_part = [&]() {   // this warp's sum into part[] (idle threads add nothing)
    float s = act ? sum - cmp : 0.0f, c = 0.0f;
    lanes_sum(s, c);
    if ((threadIdx.x & 31) == 0) part[threadIdx.x >> 5] = make_float2(s, c);
    sum = cmp = 0.0f;
  };
  auto block_total = [&]() {   // warp 0: the block's sum into total
    if (threadIdx.x >= 32) return;
    float2 x = threadIdx.x < NW ? part[threadIdx.x < NW ? threadIdx.x : 0] : make_float2(0.0f, 0.0f);
    lanes_sum(x.x, x.y);
    if (threadIdx.x == 0) total = x.x + x.y;
  };

  put(0, v[0]);
  put(1, v[1]);
  __syncthreads();
  float2 nb[6][NP];
  neighbours(1, nb);
  residuals(1, nb);
  neighbours(0, nb);
  residuals(0, nb);
  warp_part();
  __syncthreads();
  block_total();
  __syncthreads();
  float best = total;
  const float target = drop * drop * best;
  int stale = 0;
  float2 before[2][NP];   // the values one sweep earlier
  for (int sweep = 0; sweep < max_sweeps; ++sweep) {
    // v, the shared rows: the values after `sweep` sweeps
    neighbours(0, nb);
    if (sweep > 0) {
      residuals(0, nb);
      warp_part();
    }
    float2 next[NP];
    update(0, nb, next);
#pragma unroll
    for (int p = 0; p < NP; ++p) {
      before[0][p] = v[0][p];
      before[1][p] = v[1][p];
      v[0][p] = next[p];
    }
    put(0, v[0]);
    __syncthreads();
    if (sweep > 0) block_total();   // the norm after `sweep` sweeps
    neighbours(1, nb);
    update(1, nb, next);
#pragma unroll
    for (int p = 0; p < NP; ++p) v[1][p] = next[p];
    residuals(1, nb);
    put(1, v[1]);
    __syncthreads();
    if (sweep > 0) {
      const float r = total;
      bool stop = r <= target;
      if (!stop) {
        if (r < 0.998f * best) {   // squared norms: a 0.1% improvement of the norm
          best = r;
          stale = 0;
        } else {
          stop = ++stale >= 5;     // no progress for 5 sweeps: the float32 floor
        }
      }
      if (stop) {                  // it was the sweep before this one
#pragma unroll
        for (int p = 0; p < NP; ++p) {
          v[0][p] = before[0][p];
          v[1][p] = before[1][p];
        }
        break;
      }
    }
  }
  if (act) {
#pragma unroll
    for (int p = 0; p < NP; ++p) {
      const float2 ev = par ? v[1][p] : v[0][p], od = par ? v[0][p] : v[1][p];
      *reinterpret_cast<float4*>(e + row * n + 2 * kk0 + 4 * p) = make_float4(ev.x, od.x, ev.y, od.y);
    }
  }
}

struct FR {
  int n0;
  const fr_params* p;
  cudaStream_t s;
  float* e[12];
  float* alt[12];   // ping-pong partner of the fused sweeps (or NULL)
  float* r[12];
  Src b[12];
  double fbar, kappa;
  int nh;           // Hu-Sawicki exponent (1 or 2)
  int B = 1;        // boxes of a batched solve (blockIdx.z of every launch)
  dim3 grid(unsigned gx) const { return dim3(gx, 1, (unsigned)B); }
};

// Runs the statement with the compile-time exponent NH of f.
#define FR_NH(f, ...)                      \
  do {                                     \
    if ((f).nh == 2) {                     \
      constexpr int NH = 2;                \
      __VA_ARGS__;                         \
    } else {                               \
      constexpr int NH = 1;                \
      __VA_ARGS__;                         \
    }                                      \
  } while (0)

struct LevelConst {
  int n, log2n;
  float alpha, beta, kappa, q;
  float k1;   // 2 - beta kappa (3 - beta kappa for n = 2)
};

LevelConst level_const(const FR& f, int l) {
  LevelConst c;
  c.n = f.n0 >> l;
  c.log2n = ilog2(c.n);
  const double h = 1.0 / c.n, h2 = h * h;
  c.alpha = (float)(f.fbar / h2);
  c.beta = (float)(h2 / (6.0 * f.fbar));
  c.kappa = (float)f.kappa;
  c.q = (float)(h2 * f.kappa / (6.0 * f.fbar));
  c.k1 = (float)((f.nh == 2 ? 3.0 : 2.0) - h2 * f.kappa / (6.0 * f.fbar));
  return c;
}

// The fused sweeps' column tile.  Two rows of 64 x 32 cells a thread need 160
// registers, so a CTA of 352 threads has an SM to itself; 64 x 64 (96 registers,
// spilling) is slower: 0.49 against 0.47 ms at 512^3.  Against one cell at a time
// in shared memory (three CTAs per SM) a warm sweep went 0.57 -> 0.47 ms, 256^3
// 86 -> 73 us, 128^3 25 -> 17 us, a cold one at 512^3 0.73 -> 0.50 ms.  The colour
// passes take 2 x 0.27 ms there; below 128^3 they are the faster form (an F-cycle
// from 128^3 0.417 against 0.433 ms with fused sweeps at 64^3 too).
constexpr int kFrTY = 32, kFrTZ = 64;

template <int NH>
pm_status fr_smooth_nh(FR& f, int l, int count) {
  const LevelConst c = level_const(f, l);
  const double N = (double)c.n * c.n * c.n * f.B;
  // a box of a batch takes the kernels it would take alone, so every box
  // evolves bitwise as in a batch of one
  if (f.p->smoother != 1 && c.n >= 128 && f.alt[l] && march_aligned(f.e[l], f.alt[l], f.b[l].p)) {
    using G = MarchGeom<1, kFrTY, kFrTZ>;
    PM_TRY((march_attribute<CellSweeps<NH>, 1, kFrTY, kFrTZ>()));
    const int chunks = march_chunks<1, kFrTY, kFrTZ>(c.n, 1);
    const dim3 grid = f.grid((unsigned)((c.n / kFrTY) * (c.n / kFrTZ) * chunks));
    const CellSweeps<NH> sweeps{c.beta, c.k1, c.q};
    for (int it = 0; it < count; ++it) {
      PM_LAUNCH(l == 0 ? K_FR_SMOOTH0 : K_FR_SMOOTH, 12.0 * N, (k_rb_march<CellSweeps<NH>, 1, kFrTY, kFrTZ>), grid,
                G::THREADS, G::smem, f.s, f.e[l], f.alt[l], f.b[l], c.log2n, chunks, 0, sweeps);
      float* t = f.e[l];
      f.e[l] = f.alt[l];
      f.alt[l] = t;
    }
    return PM_OK;
  }
  const dim3 grid = f.grid(grid_for(((int64_t)c.n * c.n * c.n) / 4, kSweepThreads));
  for (int it = 0; it < count; ++it)
    for (int colour = 0; colour < 2; ++colour)
      PM_LAUNCH(l == 0 ? K_FR_SMOOTH0 : K_FR_SMOOTH, 6.0 * N, k_fr_sweep<NH>, grid, kSweepThreads, 0, f.s, f.e[l],
                f.b[l], c.log2n, colour, c.beta, c.k1, c.q);
  return PM_OK;
}

pm_status fr_smooth(FR& f, int l, int count) {
  return f.nh == 2 ? fr_smooth_nh<2>(f, l, count) : fr_smooth_nh<1>(f, l, count);
}

bool is_coarsest(const FR& f, int l) {
  const int n = f.n0 >> l;
  return n <= f.p->coarsest || n <= 4;
}

pm_status fr_coarse(FR& f, int l) {
  const LevelConst c = level_const(f, l);
#define PM_FR_COARSE(LOG)                                                                                             \
  FR_NH(f, PM_LAUNCH(K_FR_COARSE, 12.0 * c.n * c.n * (double)c.n * f.B, (k_fr_coarse<NH, LOG>), f.grid(1),           \
                     (FrCoarse<NH, LOG>::THREADS), 0, f.s, f.e[l], f.b[l], c.alpha, c.beta, c.kappa, c.k1, c.q,       \
                     f.p->coarse_max_sweeps, f.p->coarse_drop))
  if (c.n == 16) PM_FR_COARSE(4);
  else if (c.n == 8) PM_FR_COARSE(3);
  else PM_FR_COARSE(2);
#undef PM_FR_COARSE
  return PM_OK;
}

// Pre-smooth level l, then build the FAS coarse problem on level l + 1.
pm_status fr_to_coarse(FR& f, int l) {
  PM_TRY(fr_smooth(f, l, f.p->npre));
  const LevelConst c = level_const(f, l), cH = level_const(f, l + 1);
  const int64_t nc = (int64_t)cH.n * cH.n * cH.n;
  if (f.B == 1)
    FR_NH(f, PM_LAUNCH(K_FR_RESTRICT, 76.0 * nc, (k_fr_restrict<NH, false>), grid_for(nc / 2, 128), 128, 0, f.s, f.e[l],
                       f.b[l], c.log2n, c.alpha, c.kappa, f.e[l + 1], f.r[l + 1], const_cast<float*>(f.b[l + 1].p)));
  else
    FR_NH(f, PM_LAUNCH(K_FR_RESTRICT, 76.0 * nc * f.B, (k_fr_restrict<NH, true>), f.grid(grid_for(nc / 2, 128)), 128, 0,
                       f.s, f.e[l], f.b[l], c.log2n, c.alpha, c.kappa, f.e[l + 1], f.r[l + 1],
                       const_cast<float*>(f.b[l + 1].p)));
  FR_NH(f, PM_LAUNCH(K_FR_COARSEOP, 12.0 * nc * f.B, k_fr_coarse_op<NH>, f.grid(grid_for(nc / 4, 256)), 256, 0, f.s,
                     f.e[l + 1], const_cast<float*>(f.b[l + 1].p), cH.log2n, cH.alpha, cH.kappa));
  return PM_OK;
}

pm_status fr_v(FR& f, int l) {
  if (is_coarsest(f, l)) return fr_coarse(f, l);
  PM_TRY(fr_to_coarse(f, l));
  PM_TRY(fr_v(f, l + 1));
  PM_TRY(prolong_correct_launch(f.e[l], f.e[l + 1], f.r[l + 1], f.n0 >> l, K_FR_PROLONG, f.s, f.B));
  return fr_smooth(f, l, f.p->npost);
}

pm_status fr_f(FR& f, int l) {
  if (is_coarsest(f, l)) return fr_coarse(f, l);
  PM_TRY(fr_to_coarse(f, l));
  PM_TRY(fr_f(f, l + 1));
  PM_TRY(prolong_correct_launch(f.e[l], f.e[l + 1], f.r[l + 1], f.n0 >> l, K_FR_PROLONG, f.s, f.B));
  return fr_v(f, l);
}

}  // namespace

void fr_background(const fr_params& p, double* fbar, double* kappa, double* c2) {
  const double a = p.a;
  const double Rbar = 3.0 * p.Om * (1.0 / (a * a * a) + 4.0 * p.OL / p.Om);
  const double Rbar0 = 3.0 * p.Om * (1.0 + 4.0 * p.OL / p.Om);
  const double ratio = Rbar0 / Rbar;
  *fbar = a * a * p.fR0 * (p.nhs == 2 ? ratio * ratio * ratio : ratio * ratio);   // (R0/R)^(n+1)
  const double ct = 299792.458 / (100.0 * p.boxsize);
  *c2 = ct * ct;
  *kappa = a * a * a * a * Rbar / (3.0 * *c2);
}

pm_status fr_solve_src(Src b, float* eps, int n, const fr_params& prm, mg_stats* st, Workspace& w,
                       cudaStream_t s, int B) {
  FR f;
  f.n0 = n;
  f.B = B;
  f.p = &prm;
  f.s = s;
  f.e[0] = eps;
  f.r[0] = nullptr;
  f.b[0] = b;
  for (int l = 0; l < 12; ++l) {
    if (l > 0) {
      f.e[l] = w.fr_e[l];
      f.r[l] = w.fr_r[l];
      f.b[l] = Src{w.fr_b[l], 1.0f, nullptr};
    }
    f.alt[l] = w.fr_alt[l];
  }
  f.nh = prm.nhs == 2 ? 2 : 1;
  double c2;
  fr_background(prm, &f.fbar, &f.kappa, &c2);
  mg_stats local{PM_OK, 0, -1.0, -1.0, -1.0};
  const int64_t N0 = (int64_t)n * n * n * B;
  auto one = [&]() -> pm_status {
    PM_TRY(prm.cycle == 1 ? fr_f(f, 0) : fr_v(f, 0));
    if (f.e[0] != eps) {   // the iterate ended in the ping-pong partner: bring it home
      PM_TRY(cuda_status(cudaMemcpyAsync(eps, f.e[0], N0 * sizeof(float), cudaMemcpyDeviceToDevice, s)));
      f.alt[0] = f.e[0];
      f.e[0] = eps;
    }
    return PM_OK;
  };
  if (prm.tol <= 0.0 || B > 1) {
    for (int c = 0; c < prm.cycles; ++c) PM_TRY(one());
    local.cycles = prm.cycles;
    if (st) *st = local;
    return launch_status();
  }
  const LevelConst c0 = level_const(f, 0);
  const int64_t N = (int64_t)n * n * n;
  const unsigned nb = grid_for(N, 256, 152 * 8);
  pm_status status = PM_ENOCONV;
  for (int c = 0; c < prm.max_cycles; ++c) {
    PM_TRY(one());
    local.cycles = c + 1;
    FR_NH(f, PM_LAUNCH(K_FR_NORM, 8.0 * N, k_fr_norm<NH>, nb, 256, 0, s, eps, b, c0.log2n, c0.alpha, c0.kappa,
                       w.partials));
    PM_TRY(reduce_partials(w.partials, nb, nb, 2, 1.0, w.scalars + 8, s));
    double h[2];
    PM_TRY(fetch_scalars(w.scalars + 8, h, 2, s));
    local.res = sqrt(h[0]);
    local.norm_f = sqrt(h[1]);
    if (!isfinite(local.res)) { status = PM_ENAN; break; }
    if (local.res <= prm.tol * local.norm_f) { status = PM_OK; break; }
  }
  local.status = status;
  if (st) *st = local;
  PM_TRY(launch_status());
  return status;
}

}  // namespace pmgb
