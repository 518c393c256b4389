// S full red-black sweeps (S = 1 or 2) of a level in one pass over memory; the
// update is a policy: linear SOR (LinearSweeps, below) or the f(R) cell equation.
//
// A CTA owns a TY x TZ column of (y, z) cells and a chunk of x planes and
// marches along x.  Every thread keeps two rows (the even one first) of four z
// cells, on the column or in its halo of 2S rows and one run on either side,
// in registers for the whole march.  In step t stage s = 1 .. 2S updates the
// cells of one colour (red first) of plane t - s + 1: the x neighbours are the
// thread's own registers (the plane ahead was updated by the stage before in
// this step, the plane behind in an earlier step), so is one y neighbour of
// either row; the other y neighbour and the one z neighbour outside the run
// come from shared memory, where the stage before put the plane's cells of the
// other colour in the step before.  Each stage is valid on one ring less of
// the halo than the one before, so the last is valid on the column; plane
// t - 2S + 1 is then final and written.  Every update sees the neighbour
// values of the plain colour passes in the order x+, x-, y+, y-, z+, z-; the
// linear one rounds as PoissonUpdate does, so its result is bitwise theirs.  Old
// values come from `uin`, the result goes to `uout`.
//
// What bounds it: the shared-memory and load wavefronts and the instructions
// per update, as memory moves 12 bytes a cell for S sweeps.  Therefore two
// sweeps a pass although the halo then makes 40 x 72 cells of 32 x 64; the
// register march; the two cells of a run that have one colour as one pair
// for the paired float instructions (rounded as the single ones); rows in
// pairs and x chunks from an even plane, so that which cells of a run are red
// is known at compile time; and shared memory by place in the pair, so that
// every access is conflict-free.  Two buffers per stage make one barrier a
// step enough; old values and sources arrive by asynchronous copies four planes
// ahead.  Measured at 512^3: 0.40 ms for two sweeps (4.0 TB/s of the 12 bytes a
// cell), against 0.83 ms with one sweep a pass in shared memory; ncu at 256^3: 47
// us of 63 at the shared-memory pipe's half rate, 0.37 instructions a cycle and
// scheduler, the 12 warps waiting for it and each other.  One row a thread (23
// warps) takes 0.42 ms: more instructions, as many wavefronts.
#pragma once

#include "pm_internal.cuh"

namespace pmgb {

__device__ __forceinline__ void cp_async16(void* smem_dst, const void* gsrc) {
  const uint32_t d = (uint32_t)__cvta_generic_to_shared(smem_dst);
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(d), "l"(gsrc) : "memory");
}
__device__ __forceinline__ void cp_async_commit_group() { asm volatile("cp.async.commit_group;\n" ::: "memory"); }
template <int PENDING>
__device__ __forceinline__ void cp_async_wait_group() {
  asm volatile("cp.async.wait_group %0;\n" ::"n"(PENDING) : "memory");
}

// Runs of four cells move in 16-byte accesses (workspace levels are aligned;
// caller arrays are checked on entry).
inline bool march_aligned(const float* u, const float* alt, const float* f) {
  return (((uintptr_t)u | (uintptr_t)alt | (uintptr_t)f) & 15) == 0;
}

template <int S, int TY, int TZ>
struct MarchGeom {
  static constexpr int W = 2 * S + 2;                // planes held in registers (t + 1 .. t - 2S)
  static constexpr int HY = 2 * S;                   // halo rows on either side
  static constexpr int EP = TY / 2 + HY;             // row pairs held
  static constexpr int ER = TZ / 4 + 2;              // runs per row held (one halo run on either side: 2S <= 4 cells)
  static constexpr int RUNS = EP * ER;
  static constexpr int THREADS = (RUNS + 31) / 32 * 32;
  static constexpr int PL = RUNS + 2;                // floats of one place of one row of the row pairs, padded for z +- 1
  static constexpr int BUF = 4 * PL;                 // one colour of a plane: [row][place in the pair][PL]
  static constexpr int BUFS = 2 * 2 * S;             // two buffers for what each stage reads
  static constexpr int AHEAD = W - 2;                // planes t + 2 .. t + AHEAD are in flight during step t
  static constexpr int STAGED = 4 * RUNS;            // 16-byte runs of a plane in flight: [value, source][row][RUNS]
  static constexpr size_t smem = sizeof(float) * BUFS * BUF + sizeof(float4) * W * STAGED;
  static_assert(smem <= 227 * 1024, "one CTA per SM");
};

// Pairs of floats, each component rounded as the single operation.
__device__ __forceinline__ float2 add2(float2 a, float2 b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ float2 mul2(float2 a, float2 b) { return __fmul2_rn(a, b); }
__device__ __forceinline__ float2 fma2(float2 a, float2 b, float2 c) { return __ffma2_rn(a, b, c); }
__device__ __forceinline__ float2 both(float v) { return make_float2(v, v); }

// Linear SOR sweeps with factors om0, om1 (ONE0, ONE1: the factor is 1), as
// PoissonUpdate rounds them; gscale multiplies the values present before the
// first sweep (gbox: per box of a batched launch).  Sources enter as -h^2 f.
template <bool ONE0, bool ONE1>
struct LinearSweeps {
  float h2, gscale, om0, om1;
  const float* gbox;
  __device__ __forceinline__ void box(int b) { if (gbox) gscale = __ldg(gbox + b); }
  __device__ __forceinline__ float2 source(float2 f) const { return mul2(both(-h2), f); }
  __device__ __forceinline__ static float2 first(float2 a, float2 b) { return add2(a, b); }
  __device__ __forceinline__ static float2 add(float2 s, float2 nb) { return add2(s, nb); }
  __device__ __forceinline__ static float2 add(float2 s, float x, float y) {   // a pair from two places
    return make_float2(__fadd_rn(s.x, x), __fadd_rn(s.y, y));
  }
  // the rows' values v after stage ST (1 .. 2S) from their neighbour sums s (need:
  // the cells, two bits a row, that have to be right)
  template <int ST>
  __device__ __forceinline__ void update(float2 (&v)[2], float2 (&s)[2], const float2 (&nhf)[2], unsigned) const {
    constexpr bool ONE = ST <= 2 ? ONE0 : ONE1;
    const float om = ST <= 2 ? om0 : om1;
#pragma unroll
    for (int j = 0; j < 2; ++j) {
      if (ST == 1) s[j] = make_float2(__fmul_rn(gscale, s[j].x), __fmul_rn(gscale, s[j].y));   // rounded before the next sum
      const float2 g = mul2(add2(s[j], nhf[j]), both(1.0f / 6.0f));
      if (ONE) {
        v[j] = g;
      } else {
        if (ST <= 2) v[j] = mul2(both(gscale), v[j]);
        v[j] = fma2(both(om), g, mul2(both(1.0f - om), v[j]));
      }
    }
  }
};

// The registers of one thread's runs and its part of a step.
template <class P, int S, int TY, int TZ>
struct MarchRun {
  using G = MarchGeom<S, TY, TZ>;
  static constexpr int W = G::W;                // plane t in slot K of step<K>
  float2 R[W][2], B[W][2], FR[W][2], FB[W][2];  // [slot][row]: red and black pairs and sources of the planes held
  float4* in;                                   // this run's place in the planes in flight
  const float *uin, *fp;
  float* uout;
  float* buf;
  P pol;
  float fs, mean;
  uint32_t base, m;
  int log2n, up, dn, x0, x1;
  unsigned need[2];   // S = 1: the red cells (two bits a row) with all neighbours at hand, by the step's parity
  bool useful, zero;

  __device__ __forceinline__ uint32_t plane(int p) const { return ((uint32_t)p & m) << (2 * log2n); }
  // puts plane p in flight into slot K (read back by this thread only)
  template <int K>
  __device__ __forceinline__ void fetch(int p) const {
    if (p <= x1 + 2 * S - 1) {
      const uint32_t o = plane(p) | base;
      float4* d = in + K * G::STAGED;
#pragma unroll
      for (int j = 0; j < 2; ++j) {
        const uint32_t g = o + ((uint32_t)j << log2n);
        if (!zero) cp_async16(d + j * G::RUNS, uin + g);
        cp_async16(d + (2 + j) * G::RUNS, fp + g);
      }
    }
    cp_async_commit_group();
  }
  __device__ __forceinline__ float2 source(float a, float b) const {
    return pol.source(mul2(both(fs), add2(make_float2(a, b), both(-mean))));
  }
  __device__ __forceinline__ float* buffer(int stage, int p) const { return buf + (2 * stage + (p & 1)) * G::BUF; }
  __device__ __forceinline__ void put(int stage, int p, const float2 (&v)[2]) const {
    float* b = buffer(stage, p);
    b[0] = v[0].x;
    b[G::PL] = v[0].y;
    b[2 * G::PL] = v[1].x;
    b[3 * G::PL] = v[1].y;
  }
  // The plane that has arrived for slot K enters the registers; ODD: its parity
  // (x chunks start at even planes): row j's red cells are z + 1, z + 3 if
  // ODD + j is odd.
  template <int K, int ODD>
  __device__ __forceinline__ void split() {
#pragma unroll
    for (int j = 0; j < 2; ++j) {
      const float4* d = in + K * G::STAGED + j * G::RUNS;
      const float4 u = zero ? make_float4(0.0f, 0.0f, 0.0f, 0.0f) : d[0], s = d[2 * G::RUNS];
      if ((ODD + j) & 1) {
        R[K][j] = make_float2(u.y, u.w);
        B[K][j] = make_float2(u.x, u.z);
        FR[K][j] = source(s.y, s.w);
        FB[K][j] = source(s.x, s.z);
      } else {
        R[K][j] = make_float2(u.x, u.z);
        B[K][j] = make_float2(u.y, u.w);
        FR[K][j] = source(s.x, s.z);
        FB[K][j] = source(s.y, s.w);
      }
    }
  }
  // Stage ST of a step on plane p in slot K: the pairs v[K] of one colour from
  // those of the other, w[.], and the sources fv; ODD: the step's parity (row
  // j's cells of the stage's colour are z + 1, z + 3 if ODD + j is odd, in every
  // stage of a step).  From other threads come row 1 of the row pair below, row
  // 0 of the one above and either row's z neighbour outside the run.
  template <int K, int ST, int ODD>
  __device__ __forceinline__ void stage(int p, float2 (&v)[W][2], const float2 (&w)[W][2],
                                        const float2 (&fv)[W][2]) const {
    constexpr int KP = (K + 1) % W, KM = (K + W - 1) % W, PL = G::PL;
    const float* b = buffer(ST - 1, p);
    const float2 below = make_float2(b[2 * PL + dn], b[3 * PL + dn]), above = make_float2(b[up], b[PL + up]);
    const float ze[2] = {ODD ? b[1] : b[PL - 1], ODD ? b[3 * PL - 1] : b[2 * PL + 1]};
    float2 s[2];
#pragma unroll
    for (int j = 0; j < 2; ++j) {
      s[j] = P::first(w[KP][j], w[KM][j]);
      s[j] = P::add(s[j], j == 0 ? w[K][1] : above);
      s[j] = P::add(s[j], j == 0 ? below : w[K][0]);
      if ((ODD + j) & 1) {
        s[j] = P::add(s[j], w[K][j].y, ze[j]);
        s[j] = P::add(s[j], w[K][j]);
      } else {
        s[j] = P::add(s[j], w[K][j]);
        s[j] = P::add(s[j], ze[j], w[K][j].x);
      }
    }
    // cells whose value is used or has all its neighbours (S = 1; of S = 2 the policy does not ask)
    pol.template update<ST>(v[K], s, fv[K], ST == 1 ? need[ODD] : useful ? 15u : 0u);
    if (ST < 2 * S) put(ST, p, v[K]);
  }
  // One step with plane t, of parity ODD, in slot K: plane t + 1 enters, every
  // stage runs on its plane if a later one needs it, the last plane leaves.
  template <int K>
  __device__ __forceinline__ void step(int t) {
    constexpr int K1 = (K + 1) % W, ODD = (K + 1) & 1;
    fetch<(K + G::AHEAD) % W>(t + G::AHEAD);
    cp_async_wait_group<G::AHEAD - 1>();
    split<K1, 1 - ODD>();
    __syncthreads();
    put(0, t + 1, B[K1]);
    stage<K, 1, ODD>(t, R, B, FR);
    if (t - 1 >= x0 - (2 * S - 2) && t - 1 < x1 + 2 * S - 2) stage<(K + W - 1) % W, 2, ODD>(t - 1, B, R, FB);
    if constexpr (S == 2) {
      if (t - 2 >= x0 - 1 && t - 2 < x1 + 1) stage<(K + W - 2) % W, 3, ODD>(t - 2, R, B, FR);
      if (t - 3 >= x0) stage<(K + W - 3) % W, 4, ODD>(t - 3, B, R, FB);
    }
    const int p = t - 2 * S + 1;
    if (p >= x0 && useful) {
      constexpr int KO = (K + W - (2 * S - 1)) % W;   // of parity 1 - ODD
#pragma unroll
      for (int j = 0; j < 2; ++j) {
        const bool odd = ((1 - ODD + j) & 1) != 0;
        const float2 e = odd ? B[KO][j] : R[KO][j], o = odd ? R[KO][j] : B[KO][j];
        *reinterpret_cast<float4*>(uout + ((plane(p) | base) + ((uint32_t)j << log2n))) = make_float4(e.x, o.x, e.y, o.y);
      }
    }
  }
};

// zero: the level's values are taken as 0.  chunks: at most n / 2.
template <class P, int S, int TY, int TZ>
__global__ void __launch_bounds__(MarchGeom<S, TY, TZ>::THREADS, 1)
    k_rb_march(const float* __restrict__ uin, float* __restrict__ uout, Src f, int log2n, int chunks, int zero, P pol) {
  pdl_entry();
  using G = MarchGeom<S, TY, TZ>;
  constexpr int W = G::W;
  extern __shared__ float4 march_sm4[];
  MarchRun<P, S, TY, TZ> r;
  const uint32_t n = 1u << log2n;
  const int64_t off = (int64_t)blockIdx.z << (3 * log2n);   // the box of a batched launch
  f = box_src(f, (int64_t)1 << (3 * log2n));
  r.pol = pol;
  r.pol.box(blockIdx.z);
  r.uin = uin + off;
  r.uout = uout + off;
  r.fp = f.p;
  r.fs = f.s;
  r.mean = f.mean ? (float)*f.mean : 0.0f;
  r.m = n - 1;
  r.log2n = log2n;
  r.zero = zero != 0;
  const uint32_t tiles_z = n / TZ, tiles = (n / TY) * tiles_z;
  const uint32_t tile = blockIdx.x % tiles, xc = blockIdx.x / tiles;
  r.x0 = 2 * (int)((xc << (log2n - 1)) / (uint32_t)chunks);
  r.x1 = 2 * (int)(((xc + 1) << (log2n - 1)) / (uint32_t)chunks);
  const int y0 = (int)(tile / tiles_z) * TY, z0 = (int)(tile % tiles_z) * TZ;
  // threads beyond the last run repeat run 0 (the same values to the same places)
  const int run = (int)threadIdx.x < G::RUNS ? (int)threadIdx.x : 0;
  const int pair = run / G::ER, q = run - pair * G::ER;
  r.base = (((uint32_t)(y0 - G::HY + 2 * pair) & r.m) << log2n) | ((uint32_t)(z0 - 4 + 4 * q) & r.m);
  r.useful = pair >= S && pair < S + TY / 2 && q >= 1 && q <= TZ / 4;
  r.in = march_sm4 + run;
  r.buf = reinterpret_cast<float*>(march_sm4 + W * G::STAGED) + 1 + run;   // this run's place in every buffer
  r.up = pair < G::EP - 1 ? G::ER : 0;
  r.dn = pair > 0 ? -G::ER : 0;
#pragma unroll
  for (int odd = 0; odd < 2; ++odd) {   // not the outermost rows, nor a halo run's outermost cell
    unsigned k = (pair > 0 ? 3u : 0u) | (pair < G::EP - 1 ? 12u : 0u);
    if (q == 0) k &= odd ? ~4u : ~1u;                // z is red in the row of even parity
    if (q == G::ER - 1) k &= odd ? ~2u : ~8u;        // z + 3 in the other
    r.need[odd] = k;
  }
#pragma unroll
  for (int k = 0; k < W; ++k)
#pragma unroll
    for (int j = 0; j < 2; ++j) r.R[k][j] = r.B[k][j] = r.FR[k][j] = r.FB[k][j] = make_float2(0.0f, 0.0f);
  const int t0 = r.x0 - (2 * S - 1), tend = r.x1 + 2 * S - 1;   // steps t0 (odd) .. tend - 1
  // planes t0 - 1 (last slot), t0 (slot 0) and the AHEAD - 1 after it in flight
  r.template fetch<W - 1>(t0 - 1);
  r.template fetch<0>(t0);
  r.template fetch<1>(t0 + 1);
  if constexpr (W == 6) {
    r.template fetch<2>(t0 + 2);
    r.template fetch<3>(t0 + 3);
  }
  cp_async_wait_group<G::AHEAD - 1>();
  r.template split<W - 1, 0>();
  r.template split<0, 1>();
  r.put(0, t0, r.B[0]);
  for (int t = t0; t < tend; t += W) {
    r.template step<0>(t);
    if (t + 1 < tend) r.template step<1>(t + 1);
    if (t + 2 < tend) r.template step<2>(t + 2);
    if (t + 3 < tend) r.template step<3>(t + 3);
    if constexpr (W == 6) {
      if (t + 4 < tend) r.template step<4>(t + 4);
      if (t + 5 < tend) r.template step<5>(t + 5);
    }
  }
}

// Into how many x chunks (of nearly equal, even length) a level is cut: the
// count with the fewest plane steps in sequence, waves of one CTA per SM times
// the longest chunk and its 2S steps of run-up.
template <int S, int TY, int TZ>
inline int march_chunks(int n, int B) {
  const int64_t columns = (int64_t)(n / TY) * (n / TZ) * B;
  int best = 1;
  int64_t least = INT64_MAX;
  for (int c = 1; c <= n / 2; ++c) {
    const int64_t steps = ((columns * c + 151) / 152) * (2 * ((n / 2 + c - 1) / c) + 2 * S);
    if (steps < least) {
      least = steps;
      best = c;
    }
  }
  return best;
}

template <class P, int S, int TY, int TZ>
inline pm_status march_attribute() {
  return smem_attr(k_rb_march<P, S, TY, TZ>, MarchGeom<S, TY, TZ>::smem);
}

// The linear sweeps' column tile.
constexpr int kMarchTY = 32, kMarchTZ = 64;

}  // namespace pmgb
