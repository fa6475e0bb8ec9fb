// dg_lines32.cuh -- FP32-bulk kernels with one element line per thread (2D; GB300, sm_103a): the scheme,
// the reduced energy and the increments of dg_kernels_fp32.cuh, whose header comment states them.
//
// Work split.  A thread owns one x-line of an element (P + 1 nodes), a warp owns whole elements
// (EPW of them, a "tile"), and no block barrier is needed.
//   * x-derivatives are taken in the thread's registers, the derivative matrix being constant
//     operands: no shared-memory traffic.
//   * y-derivatives read the element's lines from shared memory in vector loads that the lanes of an
//     element share (a line of 4 is one 128-bit load), against the thread's own row of D.
//   * the four faces a thread works on -- west and east at its line's ends, south and north at its
//     column -- are known at compile time, so face signs and directions cost nothing at run time; its
//     west and east results stay in registers, the south and north ones reach the element's lines
//     through shared memory.
//   * node arrays and face records are stored by tile and lane (LineGeom), so that every access of a
//     warp is one run of consecutive 128-, 64- or 32-bit words, and padding lanes have slots of
//     their own.
//   * the face records and the volume part are all requested before the first flux is formed.
// It executes half of the thread instructions per node of the one-node-per-thread kernels (p = 4,
// viscous, surface tension: 780 instead of 1,560; no index arithmetic or divisions per face node, no
// shared load per term), which is what bounds those on grids of many waves, but a thread's chain is
// P + 1 times as long and a warp holds four to six times the nodes, so a mesh that does not fill the
// GPU, and a call too short for its ends, is left to the one-node-per-thread kernels (use_lines32).
// Measured, 10 steps of a viscous Rayleigh-Taylor problem with surface tension, 256 x 256, p = 4: 3089 us one
// node per thread, 2820 to 2840 here.  What bounds them is instruction issue with exposed load latency, at 12
// warps an SM.
//
// The terms are grouped as in the one-node-per-thread kernels; how the compiler contracts them differs in
// places.  On periodic meshes (p = 1 to 5, with and without each term) the right-hand side's rows of phi and
// psi came out the same bits in both, the others within 4e-7 of a row's largest value (7e-6 where its terms
// cancel: FP32 rounding of them), the state after four steps within 7e-9.  Grouping the
// momentum and energy terms for fewer operations brings 1.12 instead of 1.10 times
// on the problem above (1.09 instead of 1.04 on a batch of 32), but turns last bits of the FP32-rounded phase
// field, 9e-8 at single nodes after four steps.
// Batches keep one node per thread: on these kernels the mixed ensembles measured 7 to 15% slower, and
// small ones up to twice as slow.
#pragma once

#include "dg_kernels_fp32.cuh"

namespace dgpf {

// Division of an unsigned number below 2^31 by a constant d >= 1 as a multiplication: with
// 2^(s-1) < d <= 2^s and m = ceil(2^(31+s) / d), n m / 2^(31+s) exceeds n / d by less than
// n / 2^(31+s) <= 1/d, so its integer part is floor(n / d).
struct FastDiv {
  unsigned m, s;  // m < 2^32
};
__host__ inline FastDiv fast_div(unsigned d) {
  unsigned s = 0;
  while ((1ull << s) < d) ++s;
  return FastDiv{(unsigned)(((1ull << (31 + s)) + d - 1) / d), s};
}
__host__ __device__ inline unsigned div_by(unsigned n, FastDiv f) {
  return (unsigned)(((unsigned long long)n * f.m) >> (31 + f.s));
}

// What the line kernels need about one problem: geometry, boundaries, a single-precision copy of the
// closure constants (the two FP64 constants of the reduced energy besides) and the x-derivative
// matrix (2/hx) D, whose entries are constant operands of the unrolled contractions.
struct LineParams {
  int nx, ny, E, N;
  FastDiv by_nx;
  int bc[4];
  float p_bc[4];
  float eta_x, eta_y;
  float C2, dC, g2, dg, Bp;
  float rho01, rho02, drho0, mu1, mu2, sigma, gx, gy, Gamma, eps;
  int gravity, check_finite;
  double C2d, dCd;
  unsigned *status;
  const float *opsf;  // FP32 operator table (OpsLayout)
  float D[36];
};

// opsf: the host copy of the FP32 operator table; d_opsf: its device address.
__host__ inline LineParams line_params(const Params &p, int P1, const float *opsf, const float *d_opsf) {
  LineParams f{};
  f.nx = p.nx;
  f.ny = p.ny;
  f.E = p.E;
  f.N = p.N;
  f.by_nx = fast_div((unsigned)p.nx);
  for (int k = 0; k < 4; ++k) {
    f.bc[k] = p.bc[k];
    f.p_bc[k] = (float)p.p_bc[k];
  }
  f.eta_x = (float)p.eta_x;
  f.eta_y = (float)p.eta_y;
  f.C2 = (float)p.C2;
  f.dC = (float)p.dC;
  f.g2 = (float)p.g2;
  f.dg = (float)p.g1 - (float)p.g2;
  f.Bp = (float)p.Bp;
  f.rho01 = (float)p.rho01;
  f.rho02 = (float)p.rho02;
  f.drho0 = (float)p.drho0;
  f.mu1 = (float)p.mu1;
  f.mu2 = (float)p.mu2;
  f.sigma = (float)p.sigma;
  f.gx = (float)p.gx;
  f.gy = (float)p.gy;
  f.Gamma = (float)p.Gamma;
  f.eps = (float)p.eps;
  f.gravity = p.gravity;
  f.check_finite = p.check_finite;
  f.C2d = p.C2;
  f.dCd = p.dC;
  f.status = p.status;
  f.opsf = d_opsf;
  for (int k = 0; k < P1 * P1; ++k) f.D[k] = opsf[k];
  return f;
}

// phi_1 mu_1 + phi_2 mu_2: either phase's own viscosity where the other is absent, whatever their ratio
// (mu_2 + phi (mu_1 - mu_2) loses the smaller one in the difference's rounding).
__device__ __forceinline__ float mixture_mu(const LineParams &pf, float phi) {
  return pf.mu1 * phi + pf.mu2 * (1.f - phi);
}

// Geometry.  NL lines (threads) per element, EPW elements per warp.  Shared memory: a line is padded
// to RS floats (vector accesses); element starts are ES floats apart, which puts the lines that the
// elements of a warp read together into different banks.
// Global memory, per tile: node arrays [7][P1 * 32] (a field's lines, by lane: the first words of a
// line as one vector per lane, then the rest, each a run over the lanes), face records
// [4][3][32] float4.
template <int P>
struct LineGeom {
  static constexpr int P1 = P + 1;
  static constexpr int NP = P1 * P1;
  static constexpr int EPW = 32 / P1;
  static constexpr int RS = P1 == 2 ? 2 : (P1 <= 4 ? 4 : 8);
  static constexpr int ES = P1 * RS + (P1 >= 4 ? 4 : 0);
  static constexpr int SF = EPW * ES;               // one shared field of a warp
  static constexpr int NR = NV + 6;                 // y-face results per side: integrand, lifting coefficients
  static constexpr int FS = 2 * NR * RS + (P1 >= 4 ? 4 : 0);  // of one element
  static constexpr int TN = NV * P1 * 32;           // floats of a tile's node array
  static constexpr int TT = 4 * 3 * 32;             // float4 of a tile's face records
};
inline int line_tiles(int P1, int E) { return (E + 32 / P1 - 1) / (32 / P1); }
// Floats of a node array and of the face records of a context.
inline size_t line_node_floats(int P1, int E) { return (size_t)line_tiles(P1, E) * NV * P1 * 32; }
inline size_t line_trace_floats(int P1, int E) { return (size_t)line_tiles(P1, E) * 4 * 3 * 32 * 4; }

// Which calls of a single problem run the line kernels: dg_rhs, and captured sequences of at least `steps`
// steps (0: none).
//
// A thread's chain is P + 1 times as long here and a warp holds as many times the nodes, so the line kernels
// need enough warps on every SM, and they lose where the one-node kernels' grid still fits on the GPU at once
// (their time jumps by half when it no longer does) and where their own grid ends in a thin second wave.  The
// kernels at the FP64 ends of a call stage the state through shared memory, at fewer warps per SM: they cost
// what the stages between them win back only over several steps, and a right-hand side, which is nothing but
// ends, pays while they fit on the GPU at once (inviscid up to p = 4: a little longer).  Times on one line per thread over times on one node per
// thread, periodic in x, at w line warps per SM (right-hand side, sequences of 1, 2, 4 and 8 steps):
//   p = 1        w 1.5: 1.13 1.13 1.15 1.05 0.89    2.6: 1.01 1.25 1.07 0.90 0.77    4.1: 0.69 1.00 0.89 0.81 0.75
//   p = 1 visc.  w 1.5: 1.16 0.83 0.95 0.87 0.84    2.1: 0.80 0.90 0.86 0.81 0.72    26.9: 0.86 0.80 0.73 0.68 0.65
//   p = 2        w 5.6: 0.84 1.11 1.13 1.11 1.08    6.1: 0.76 0.85 0.78 0.74 0.71   (one node: all resident up to 5.6)
//   p = 2 visc.  w 1.8: 1.07 1.30 1.21 1.08 0.86    3.4: 0.95 1.06 0.93 0.76 0.65    5.6: 0.91 0.97 0.78 0.67 0.62
//   p = 3        w 4.8: 1.22 1.48 1.50 1.42 1.40    5.3: 0.88 1.00 0.97 0.92 0.89   12.6: 1.00 1.15 1.21 1.13 1.09
//                w 17.1: 1.11 1.12 1.04 0.97 0.93   30.3: 1.00 0.97 0.95 0.89 0.87
//   p = 3 visc.  w 7.0: 0.90 1.20 1.23 1.26 1.24    8.2: 0.85 1.00 0.95 0.92 0.89   25.5: 1.25 1.15 1.09 1.03 1.00
//   p = 4        w 5.7: 0.93 1.14 1.15 1.12 1.11    7.0: 0.90 1.00 0.94 0.89 0.86   18.0: 1.09 1.06 0.99 0.93 0.89
//   p = 4 tens.  w 8.5: 0.91 0.91 0.93 0.88 0.85   11.9: 0.85 0.89 0.86 0.80 0.76   18.0: 1.09 1.08 1.02 0.95 0.92
//   p = 4 visc.  w 8.5: 1.13 1.00 0.95 0.88 0.84   18.0: 1.28 1.10 1.05 0.96 0.92   71.9: 1.19 1.07 1.00 0.93 0.90
//   p = 5        w 7.6: 0.80 0.98 1.00 0.96 0.94    8.4: 1.15 1.15 1.15 1.01 0.93   27.3: 1.27 1.15 1.10 1.01 0.97
//   p = 5 full   w 6.8: 0.83 0.96 0.99 0.92 0.89    8.4: 1.47 1.39 1.47 1.30 1.22   33.7: 1.29 1.25 1.16 1.07 1.02
// (surface tension alone as inviscid, except at p = 5, where any term takes the registers.)
struct LineUse {
  bool rhs;
  int steps;
};
inline LineUse use_lines32(int P1, bool viscous, bool tension, int E, const KernelSet32 &one, const KernelSet32 &line) {
  static const int sms = [] {
    int dev = 0, n = 0;
    if (cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || n < 1)
      n = 152;
    return n;
  }();
  const long long tiles = line_tiles(P1, E), w = 10 * tiles / sms;  // line warps per SM, in tenths
  if (P1 == 2) {
    if (w < 15) return {false, 0};
    return {w >= (viscous ? 20 : 28), viscous || w >= 40 ? 1 : w >= 30 ? 2 : w >= 20 ? 3 : 5};
  }
  if (P1 == 3) {
    if (w < 15) return {false, 0};
    const bool rhs = w >= 24;
    if (!viscous) return {rhs, E > one.resident_stage() ? 1 : 0};
    return {rhs, w >= 50 ? 1 : w >= 30 ? 2 : w >= 24 ? 3 : w >= 21 ? 4 : 6};
  }
  if (w < 50) return {false, 0};
  const bool full5 = P1 == 6 && (viscous || tension), few5 = P1 == 6 && w < 60;
  const long long wave = line.resident_stage();
  LineUse u{!few5 && tiles <= (viscous || P1 == 6 ? line.resident_ends() : wave), 0};
  if (E <= one.resident_stage()) return u;
  if (tiles <= wave) {
    u.steps = P1 < 6 || (full5 && !few5) ? 1 : few5 && !full5 ? 0 : 4;
    return u;
  }
  // percent of the second wave that has to be there; in later ones it matters no more
  const int least = P1 == 4 && (viscous || tension) ? 60 : 35;
  if (full5 || (tiles <= 2 * wave && 100 * (tiles - wave) < least * wave)) return u;
  u.steps = P1 == 6 ? 4 : !viscous ? 2 : P1 == 4 ? 5 : 3;
  return u;
}

template <int P1>
__device__ __forceinline__ void ld_row(const float *p, float *v) {
  if constexpr (P1 == 2) {
    const float2 a = *reinterpret_cast<const float2 *>(p);
    v[0] = a.x; v[1] = a.y;
  } else {
    const float4 a = *reinterpret_cast<const float4 *>(p);
    v[0] = a.x; v[1] = a.y; v[2] = a.z;
    if constexpr (P1 >= 4) v[3] = a.w;
    if constexpr (P1 == 5) v[4] = p[4];
    if constexpr (P1 == 6) {
      const float2 b = *reinterpret_cast<const float2 *>(p + 4);
      v[4] = b.x; v[5] = b.y;
    }
  }
}
template <int P1>
__device__ __forceinline__ void st_row(float *p, const float *v) {
  if constexpr (P1 == 2) {
    *reinterpret_cast<float2 *>(p) = make_float2(v[0], v[1]);
  } else {
    *reinterpret_cast<float4 *>(p) = make_float4(v[0], v[1], v[2], P1 >= 4 ? v[3 % P1] : 0.f);
    if constexpr (P1 == 5) p[4] = v[4];
    if constexpr (P1 == 6) *reinterpret_cast<float2 *>(p + 4) = make_float2(v[4], v[5]);
  }
}

// A tile's line of one field in global memory, by lane.
template <int P1, bool COH>
__device__ __forceinline__ void ld_line(const float *__restrict__ field, int lane, float *v) {
  if constexpr (P1 == 2 || P1 == 3) {
    const float2 a = ld_in<COH>(reinterpret_cast<const float2 *>(field) + lane);
    v[0] = a.x; v[1] = a.y;
    if constexpr (P1 == 3) v[2] = ld_in<COH>(field + 64 + lane);
  } else {
    const float4 a = ld_in<COH>(reinterpret_cast<const float4 *>(field) + lane);
    v[0] = a.x; v[1] = a.y; v[2] = a.z; v[3] = a.w;
    if constexpr (P1 == 5) v[4] = ld_in<COH>(field + 128 + lane);
    if constexpr (P1 == 6) {
      const float2 b = ld_in<COH>(reinterpret_cast<const float2 *>(field + 128) + lane);
      v[4] = b.x; v[5] = b.y;
    }
  }
}
template <int P1>
__device__ __forceinline__ void st_line(float *field, int lane, const float *v) {
  if constexpr (P1 == 2 || P1 == 3) {
    reinterpret_cast<float2 *>(field)[lane] = make_float2(v[0], v[1]);
    if constexpr (P1 == 3) field[64 + lane] = v[2 % P1];
  } else {
    reinterpret_cast<float4 *>(field)[lane] = make_float4(v[0], v[1], v[2 % P1], v[3 % P1]);
    if constexpr (P1 == 5) field[128 + lane] = v[4 % P1];
    if constexpr (P1 == 6) reinterpret_cast<float2 *>(field + 128)[lane] = make_float2(v[4 % P1], v[5 % P1]);
  }
}
template <int P, bool COH>
__device__ __forceinline__ void ld_lines(const float *__restrict__ arr, int tile, float (*q)[P + 1]) {
  using G = LineGeom<P>;
  const float *f = arr + (size_t)tile * G::TN;
#pragma unroll
  for (int v = 0; v < NV; ++v) ld_line<G::P1, COH>(f + v * G::P1 * 32, threadIdx.x & 31, q[v]);
}
template <int P>
__device__ __forceinline__ void st_lines(float *arr, int tile, const float (*q)[P + 1]) {
  using G = LineGeom<P>;
  float *f = arr + (size_t)tile * G::TN;
#pragma unroll
  for (int v = 0; v < NV; ++v) st_line<G::P1>(f + v * G::P1 * 32, threadIdx.x & 31, q[v]);
}

// Derivative of a line in registers along x, over differences: out[i] = sum_c D[i][c] (f[c] - f[i]).
template <int P1>
__device__ __forceinline__ void ddx(const float *D, const float *f, float *out) {
#pragma unroll
  for (int i = 0; i < P1; ++i) {
    float a = 0.f;
    bool first = true;
#pragma unroll
    for (int c = 0; c < P1; ++c)
      if (c != i) {
        const float d = f[c] - f[i];
        a = first ? D[i * P1 + c] * d : fmaf(D[i * P1 + c], d, a);
        first = false;
      }
    out[i] = a;
  }
}

// A thread's place: its tile, its element (clamped to a valid one for padding threads, which compute
// on it and write to slots of their own), its line j and its element slot in the warp.
template <int P>
struct LinePlace {
  int tile, e, j, le;
  bool act;
  __device__ __forceinline__ LinePlace(int E, int tile_) {
    using G = LineGeom<P>;
    const int lane = threadIdx.x & 31, l = lane / G::P1;
    tile = tile_;
    le = l < G::EPW ? l : G::EPW - 1;
    j = lane - l * G::P1;
    const int e0 = tile * G::EPW + le;
    e = e0 < E ? e0 : E - 1;
    act = l < G::EPW && e0 < E;
  }
};

// Face-trace record: the seven state values, d(phi)/d(axis normal to the face), the level-set normal
// on that axis and what the reader would have to recompute -- inviscid: pressure, sound speed and
// 1/rho; viscous: the stress components tau . e_axis and the reciprocal of the mixture 1/(gamma-1).
enum LineTrace { LT_GPHI = 7, LT_N = 8, LT_P = 9, LT_C = 10, LT_IR = 11, LT_TX = 9, LT_TY = 10, LT_IG = 11 };

// The record of face f, face node k of element e (bounds-checked build: its tile's index).
template <int P, bool COH>
__device__ __forceinline__ void ld_trace(const float4 *__restrict__ tr, int E, unsigned *status, int e, int f, int k,
                                         float *T) {
  using G = LineGeom<P>;
  if (!in_bounds(status, e, E)) {
#pragma unroll
    for (int v = 0; v < 12; ++v) T[v] = 1.f;
    return;
  }
  const int tile = (unsigned)e / (unsigned)G::EPW, lane = (e - tile * G::EPW) * G::P1 + k;
  const float4 *r = tr + (size_t)tile * G::TT + f * 96 + lane;
#pragma unroll
  for (int p = 0; p < 3; ++p) {
    const float4 x = ld_in<COH>(r + 32 * p);
    T[4 * p] = x.x; T[4 * p + 1] = x.y; T[4 * p + 2] = x.z; T[4 * p + 3] = x.w;
  }
}

// ---------------------------------------------------------------------------
// Face flux
// ---------------------------------------------------------------------------

// One side of a face as the flux needs it.
struct Side32 {
  float u, v, P, c, B;
};
template <bool VISC>
__device__ __forceinline__ Side32 side_of(const LineParams &pf, const float *T) {
  Side32 s;
  const float rho = T[M1] + T[M2], ir = VISC ? rcp32(rho) : T[LT_IR];
  s.u = T[RU] * ir;
  s.v = T[RV] * ir;
  const float k = 0.5f * (s.u * s.u + s.v * s.v);
  s.P = VISC ? (T[RE] - rho * k) * T[LT_IG] : T[LT_P];
  s.c = VISC ? sqrtf((s.P + (s.P + fmaf(pf.dC, T[PHI], pf.C2)) * T[LT_IG]) * ir) : T[LT_C];
  s.B = s.P * pf.Bp;
  return s;
}

// Strong-form surface integrand F- - F^ of the seven equations at one face node (outward normal sign
// SG along x, XF, or y) and the lifting coefficients of the symmetric SIP term.  wf: the face weight.
// tm, tp: own and neighbour records; wall: the ghost side is formed here.
// The terms keep the one-node-per-thread kernels' grouping: the right-hand side reads the phase field
// rounded to FP32, where another grouping turns single nodes' last bit within a few steps, and the
// faces amplify that to several units.
template <bool VISC, bool XF, int SGI>
__device__ __forceinline__ void face_flux32(const LineParams &pf, const float *tm, float *tp, bool wall, float wf,
                                            float *S, float *lift) {
  constexpr float sg = (float)SGI;
  constexpr int f = XF ? (SGI > 0 ? 1 : 0) : (SGI > 0 ? 3 : 2);
  const Side32 m = side_of<VISC>(pf, tm);
  Side32 p;
  if (!wall) {
    p = side_of<VISC>(pf, tp);
  } else {
#pragma unroll
    for (int q = 0; q < 12; ++q) tp[q] = tm[q];
    p = m;
    const int bc = pf.bc[f];
    if (bc == BC_PRESSURE) {
      // exterior state at rest at p_bc: the reduced energy is p_bc times the mixture 1/(gamma-1)
      const float den = fmaf(tm[PHI], pf.dg, pf.g2), iG = rcp32(den);
      tp[RU] = tp[RV] = 0.f;
      tp[RE] = pf.p_bc[f] * den;
      p.u = p.v = 0.f;
      p.P = tp[RE] * iG;
      p.c = sqrtf((p.P + (p.P + fmaf(pf.dC, tm[PHI], pf.C2)) * iG) * rcp32(tm[M1] + tm[M2]));
      p.B = p.P * pf.Bp;
    } else {
      if (bc != BC_SLIP || XF) { tp[RU] = -tm[RU]; p.u = -m.u; }
      if (bc != BC_SLIP || !XF) { tp[RV] = -tm[RV]; p.v = -m.v; }
    }
  }
  const float unm = sg * (XF ? m.u : m.v), unp = sg * (XF ? p.u : p.v);
  const float lam = fmaxf(fabsf(unm) + m.c, fabsf(unp) + p.c);
  const float eta = XF ? pf.eta_x : pf.eta_y;
  {
    const float pm = sg * m.P, pp = sg * p.P;
    const float Fm[5] = {tm[M1] * unm, tm[M2] * unm, XF ? fmaf(tm[RU], unm, pm) : tm[RU] * unm,
                         XF ? tm[RV] * unm : fmaf(tm[RV], unm, pm), (tm[RE] + m.P) * unm};
    const float Fp[5] = {tp[M1] * unp, tp[M2] * unp, XF ? fmaf(tp[RU], unp, pp) : tp[RU] * unp,
                         XF ? tp[RV] * unp : fmaf(tp[RV], unp, pp), (tp[RE] + p.P) * unp};
#pragma unroll
    for (int c = 0; c < 5; ++c) {  // F- - F^ = (F- - F+)/2 + lambda [[w]]
      const int v = M1 + c;
      const float dF = (XF ? c == 2 : c == 3) ? Fm[c] - Fp[c]
                       : c == 4               ? fmaf(tm[RE] + m.P, unm, -Fp[4])
                                              : fmaf(tm[v], unm, -Fp[c]);
      S[v] = wf * fmaf(lam * 0.5f, tp[v] - tm[v], 0.5f * dF);
    }
  }
  // compression term on the face: -1/2 Cmix(phi+) (u+ - u-) . m
  S[RE] = fmaf(-(wf * 0.5f * fmaf(pf.dC, tp[PHI], pf.C2)), unp - unm, S[RE]);
  const float jump = tp[PHI] - tm[PHI];
  S[PHI] = wf * (lam - unm) * 0.5f * jump;
  S[PSI] = wf * (lam - unm) * 0.5f * (tp[PSI] - tm[PSI]);

  // SIP flux minus the own trace of the a_1 flux, for every a_1-derived term: C^ a^.m - C- a-.m
  // (at a wall no a_1 flux crosses: a^ = 0)
  const float km = 0.5f * (m.u * m.u + m.v * m.v), kp = 0.5f * (p.u * p.u + p.v * p.v);
  const float a1m = pf.Gamma * (pf.eps * tm[LT_GPHI] - tm[PHI] * (1.f - tm[PHI]) * tm[LT_N]) * sg;
  const float Co[6] = {1.f, pf.rho01, -pf.rho02, pf.drho0 * m.u, pf.drho0 * m.v, m.B + pf.drho0 * km};
  const int slot[6] = {PHI, M1, M2, RU, RV, RE};
  if (!wall) {
    const float gn = 0.5f * (tp[LT_GPHI] + tm[LT_GPHI]) * sg;
    const float sharp =
        0.5f * (tp[PHI] * (1.f - tp[PHI]) * tp[LT_N] + tm[PHI] * (1.f - tm[PHI]) * tm[LT_N]) * sg;
    const float ahat = pf.Gamma * (pf.eps * (gn + eta * jump) - sharp);
    const float Cq[6] = {1.f, pf.rho01, -pf.rho02, pf.drho0 * 0.5f * (p.u + m.u), pf.drho0 * 0.5f * (p.v + m.v),
                         0.5f * (p.B + m.B) + pf.drho0 * 0.5f * (kp + km)};
    const float sym = -wf * 0.5f * pf.Gamma * pf.eps * jump;
#pragma unroll
    for (int c = 0; c < 6; ++c) {
      S[slot[c]] += wf * (Cq[c] * ahat - Co[c] * a1m);
      lift[c] = Cq[c] * sym;
    }
  } else {
#pragma unroll
    for (int c = 0; c < 6; ++c) {
      S[slot[c]] -= wf * Co[c] * a1m;
      lift[c] = 0.f;
    }
  }
  if (VISC) {
    const float mua = 0.5f * (mixture_mu(pf, tp[PHI]) + mixture_mu(pf, tm[PHI]));
    const float tmx = tm[LT_TX] * sg, tmy = tm[LT_TY] * sg, tpx = tp[LT_TX] * sg, tpy = tp[LT_TY] * sg;
    // tau^ . m - tau- . m
    S[RU] += wf * (0.5f * (tpx - tmx) + eta * mua * (p.u - m.u));
    S[RV] += wf * (0.5f * (tpy - tmy) + eta * mua * (p.v - m.v));
    const float tum = tmx * m.u + tmy * m.v, tup = tpx * p.u + tpy * p.v;
    S[RE] += wf * (0.5f * (tup - tum) + eta * mua * (kp - km));
  }
}

// Neighbour of element e across face f, or -1 at a wall; ex, ey its coordinates.
__device__ __forceinline__ int neighbour32(const LineParams &p, int e, int ex, int ey, int f) {
  switch (f) {
    case 0: return ex > 0 ? e - 1 : (p.bc[0] == BC_PERIODIC ? e + p.nx - 1 : -1);
    case 1: return ex < p.nx - 1 ? e + 1 : (p.bc[1] == BC_PERIODIC ? e - p.nx + 1 : -1);
    case 2: return ey > 0 ? e - p.nx : (p.bc[2] == BC_PERIODIC ? e + p.nx * (p.ny - 1) : -1);
    default: return ey < p.ny - 1 ? e + p.nx : (p.bc[3] == BC_PERIODIC ? e - p.nx * (p.ny - 1) : -1);
  }
}

// ---------------------------------------------------------------------------
// Volume part
// ---------------------------------------------------------------------------

// Volume part of the thread's line on the state q: writes the volume lines and the face records.
// sm: the warp's shared memory (at least 6 fields of LineGeom::SF floats).
template <int P, bool VISC, bool ST>
__device__ __forceinline__ void vol32_line(const LineParams &pf, float *sm, const LinePlace<P> &pl,
                                           const float (*q)[P + 1], float *__restrict__ rvol,
                                           float4 *__restrict__ tr) {
  using G = LineGeom<P>;
  constexpr int P1 = G::P1, SF = G::SF;
  const float *opsf = pf.opsf, *D = pf.D;
  const int row = pl.le * G::ES + pl.j * G::RS, blk = pl.le * G::ES;
  float u[P1], v[P1], Pr[P1], iG[P1], ir[P1];
  bool bad = false;
#pragma unroll
  for (int i = 0; i < P1; ++i) {
    const float rho = q[M1][i] + q[M2][i];
    ir[i] = rcp32(rho);
    u[i] = q[RU][i] * ir[i];
    v[i] = q[RV][i] * ir[i];
    const float k = 0.5f * (u[i] * u[i] + v[i] * v[i]);
    iG[i] = rcp32(fmaf(q[PHI][i], pf.dg, pf.g2));
    Pr[i] = (q[RE][i] - rho * k) * iG[i];
    // Non-physical state: rho <= 0, a mixture 1/(gamma - 1) <= 0, or P + Pinf_mix <= 0, i.e.
    // rho c^2 = P + (P + Cm) / den <= 0 (Sec. 2 mixture rules).
    const float X = Pr[i] + (Pr[i] + fmaf(pf.dC, q[PHI][i], pf.C2)) * iG[i];
    bad |= rho <= 0.f || iG[i] <= 0.f || X <= 0.f;
  }
  if (pf.check_finite && pl.act && bad) atomicOr(pf.status, STATUS_NONPHYSICAL);
  float dy[P1];  // the thread's row of D along y
  st_row<P1>(sm + 0 * SF + row, q[PHI]);
  st_row<P1>(sm + 1 * SF + row, q[PSI]);
  st_row<P1>(sm + 2 * SF + row, v);
  if (VISC) st_row<P1>(sm + 3 * SF + row, u);
#pragma unroll
  for (int c = 0; c < P1; ++c) dy[c] = __ldg(opsf + P1 * P1 + pl.j * P1 + c);

  // gradients along x in registers
  float gpx[P1], gsx[P1], gpy[P1], gsy[P1], comp[P1];
  float gux[P1], gvx[P1], guy[P1], gvy[P1];
  ddx<P1>(D, q[PHI], gpx);
  ddx<P1>(D, q[PSI], gsx);
  float Cm[P1];
#pragma unroll
  for (int i = 0; i < P1; ++i) Cm[i] = fmaf(pf.dC, q[PHI][i], pf.C2);
  {
#pragma unroll
    for (int i = 0; i < P1; ++i) {
      comp[i] = gux[i] = 0.f;
#pragma unroll
      for (int c = 0; c < P1; ++c)
        if (c != i) {
          comp[i] = fmaf(D[i * P1 + c] * Cm[c], u[c] - u[i], comp[i]);
          if (VISC) gux[i] = fmaf(D[i * P1 + c], u[c] - u[i], gux[i]);
        }
      gpy[i] = gsy[i] = guy[i] = gvy[i] = gvx[i] = 0.f;
    }
  }
  if (VISC) ddx<P1>(D, v, gvx);
  {
    __syncwarp();
#pragma unroll
    for (int c = 0; c < P1; ++c) {
      float fp[P1], fs[P1], fv[P1], fu[P1];
      const float *r = sm + blk + c * G::RS;
      ld_row<P1>(r, fp);
      ld_row<P1>(r + SF, fs);
      ld_row<P1>(r + 2 * SF, fv);
      if (VISC) ld_row<P1>(r + 3 * SF, fu);
#pragma unroll
      for (int i = 0; i < P1; ++i) {
        gpy[i] = fmaf(dy[c], fp[i] - q[PHI][i], gpy[i]);
        gsy[i] = fmaf(dy[c], fs[i] - q[PSI][i], gsy[i]);
        comp[i] = fmaf(dy[c] * fmaf(pf.dC, fp[i], pf.C2), fv[i] - v[i], comp[i]);
        if (VISC) {
          gvy[i] = fmaf(dy[c], fv[i] - v[i], gvy[i]);
          guy[i] = fmaf(dy[c], fu[i] - u[i], guy[i]);
        }
      }
    }
    __syncwarp();
  }

  // level-set normal, a_1, stress, and the terms that need the gradients
  float ax[P1], ay[P1], txx[P1], txy[P1], tyy[P1], R[NV][P1], nc[P1], nx[P1], ny[P1];
#pragma unroll
  for (int i = 0; i < P1; ++i) {
    // n = 0 where |grad psi| cannot be told from zero: FP32 storage of a
    // distance-like psi leaves ~1e-6 of noise in its gradient (the FP64 path
    // uses 1e-12), so below 1e-4 the direction is noise.
    const float g2 = gsx[i] * gsx[i] + gsy[i] * gsy[i];
    const float r = g2 >= 1e-8f ? rsqrtf(g2) : 0.f;
    nx[i] = gsx[i] * r;
    ny[i] = gsy[i] * r;
    const float sphi = q[PHI][i] * (1.f - q[PHI][i]);
    ax[i] = pf.Gamma * (pf.eps * gpx[i] - sphi * nx[i]);
    ay[i] = pf.Gamma * (pf.eps * gpy[i] - sphi * ny[i]);
    nc[i] = u[i] * gpx[i] + v[i] * gpy[i];
    R[PSI][i] = -(u[i] * gsx[i] + v[i] * gsy[i]);
    if (VISC) {
      const float mu = mixture_mu(pf, q[PHI][i]);
      const float div3 = (gux[i] + gvy[i]) * (1.f / 3.f);
      txx[i] = 2.f * mu * (gux[i] - div3);
      tyy[i] = 2.f * mu * (gvy[i] - div3);
      txy[i] = mu * (guy[i] + gvx[i]);
    }
  }
  float cs[P1];  // CSF: sigma kappa |grad phi|, kappa = -div n
  if (ST) {
    float dv[P1];
    st_row<P1>(sm + row, ny);
    ddx<P1>(D, nx, dv);
    {
      __syncwarp();
#pragma unroll
      for (int c = 0; c < P1; ++c) {
        float fn[P1];
        ld_row<P1>(sm + blk + c * G::RS, fn);
#pragma unroll
        for (int i = 0; i < P1; ++i) dv[i] = fmaf(dy[c], fn[i] - ny[i], dv[i]);
      }
      __syncwarp();
    }
#pragma unroll
    for (int i = 0; i < P1; ++i) cs[i] = -pf.sigma * dv[i] * sqrtf(gpx[i] * gpx[i] + gpy[i] * gpy[i]);
  }

  // Fluxes, contracted over differences: along x at once, along y from shared memory.
  float Fy[6][P1];
#pragma unroll
  for (int eq = 0; eq < 6; ++eq) {
    const int vv = eq == 0 ? PHI : eq + 1;
    float fx[P1];
#pragma unroll
    for (int i = 0; i < P1; ++i) {
      switch (eq) {
        case 0:
          fx[i] = -ax[i];
          Fy[0][i] = -ay[i];
          break;
        case 1:
          fx[i] = q[M1][i] * u[i] - pf.rho01 * ax[i];
          Fy[1][i] = q[M1][i] * v[i] - pf.rho01 * ay[i];
          break;
        case 2:
          fx[i] = q[M2][i] * u[i] + pf.rho02 * ax[i];
          Fy[2][i] = q[M2][i] * v[i] + pf.rho02 * ay[i];
          break;
        case 3:
          fx[i] = q[RU][i] * u[i] + Pr[i] - pf.drho0 * ax[i] * u[i];
          Fy[3][i] = q[RU][i] * v[i] - pf.drho0 * ay[i] * u[i];
          if (VISC) {
            fx[i] -= txx[i];
            Fy[3][i] -= txy[i];
          }
          break;
        case 4:
          fx[i] = q[RV][i] * u[i] - pf.drho0 * ax[i] * v[i];
          Fy[4][i] = q[RV][i] * v[i] + Pr[i] - pf.drho0 * ay[i] * v[i];
          if (VISC) {
            fx[i] -= txy[i];
            Fy[4][i] -= tyy[i];
          }
          break;
        default: {
          const float k = 0.5f * (u[i] * u[i] + v[i] * v[i]), cE = pf.drho0 * k + Pr[i] * pf.Bp;
          fx[i] = (q[RE][i] + Pr[i]) * u[i] - cE * ax[i];
          Fy[5][i] = (q[RE][i] + Pr[i]) * v[i] - cE * ay[i];
          if (VISC) {
            fx[i] -= txx[i] * u[i] + txy[i] * v[i];
            Fy[5][i] -= txy[i] * u[i] + tyy[i] * v[i];
          }
        }
      }
    }
    st_row<P1>(sm + eq * SF + row, Fy[eq]);
    ddx<P1>(D, fx, R[vv]);
  }
  __syncwarp();
#pragma unroll
  for (int eq = 0; eq < 6; ++eq) {
    const int vv = eq == 0 ? PHI : eq + 1;
#pragma unroll
    for (int c = 0; c < P1; ++c) {
      float f[P1];
      ld_row<P1>(sm + eq * SF + blk + c * G::RS, f);
#pragma unroll
      for (int i = 0; i < P1; ++i) R[vv][i] = fmaf(dy[c], f[i] - Fy[eq][i], R[vv][i]);
    }
  }
  __syncwarp();
#pragma unroll
  for (int i = 0; i < P1; ++i) {  // -div F and the terms outside the divergence
    R[PHI][i] = -R[PHI][i] - nc[i];
    R[M1][i] = -R[M1][i];
    R[M2][i] = -R[M2][i];
    R[RU][i] = -R[RU][i];
    R[RV][i] = -R[RV][i];
    R[RE][i] = -R[RE][i] - comp[i];
    if (pf.gravity) {
      const float rho = q[M1][i] + q[M2][i];
      R[RU][i] += rho * pf.gx;
      R[RV][i] += rho * pf.gy;
      R[RE][i] += rho * (pf.gx * u[i] + pf.gy * v[i]);
    }
    if (ST) {
      R[RU][i] += cs[i] * nx[i];
      R[RV][i] += cs[i] * ny[i];
      R[RE][i] += cs[i] * (u[i] * nx[i] + v[i] * ny[i]);
    }
  }
  st_lines<P>(rvol, pl.tile, R);

  // Face records, to the slots of the threads that read them as their own.
  float4 *t0 = tr + (size_t)pl.tile * G::TT + pl.le * P1;
  auto put = [&](int i, int f, int k, float gn, float nn, float t1, float t2) {
    float4 *r = t0 + f * 96 + k;
    r[0] = make_float4(q[0][i], q[1][i], q[2][i], q[3][i]);
    r[32] = make_float4(q[4][i], q[5][i], q[6][i], gn);
    if (VISC) r[64] = make_float4(nn, t1, t2, iG[i]);
    else r[64] = make_float4(nn, Pr[i], sqrtf((Pr[i] + (Pr[i] + Cm[i]) * iG[i]) * ir[i]), ir[i]);
  };
  if (pl.act && in_bounds(pf.status, pl.e, pf.E)) {
    put(0, 0, pl.j, gpx[0], nx[0], VISC ? txx[0] : 0.f, VISC ? txy[0] : 0.f);
    put(P, 1, pl.j, gpx[P], nx[P], VISC ? txx[P] : 0.f, VISC ? txy[P] : 0.f);
    if (pl.j == 0 || pl.j == P) {
      const int f = pl.j == 0 ? 2 : 3;
#pragma unroll
      for (int i = 0; i < P1; ++i) put(i, f, i, gpy[i], ny[i], VISC ? txy[i] : 0.f, VISC ? tyy[i] : 0.f);
    }
  }
}

// ---------------------------------------------------------------------------
// Surface part
// ---------------------------------------------------------------------------

// M^-1 R of the thread's line: the volume lines plus the surface terms.  L[v][i] on return.
template <int P, bool VISC, bool PDL>
__device__ __forceinline__ void surf32_line(const LineParams &pf, float *sm, const LinePlace<P> &pl,
                                            const float *__restrict__ rvol, const float4 *__restrict__ tr,
                                            float (*L)[P + 1]) {
  using G = LineGeom<P>;
  constexpr int P1 = G::P1, NP = G::NP;
  const OpsLayout O{P1, NP};
  const int ey = (int)div_by((unsigned)pl.e, pf.by_nx), ex = pl.e - ey * pf.nx;
  int e2[4];
  float tm[4][12], tp[4][12];
#pragma unroll
  for (int f = 3; f >= 0; --f) {
    e2[f] = neighbour32(pf, pl.e, ex, ey, f);
    ld_trace<P, PDL>(tr, pf.E, pf.status, pl.e, f, pl.j, tm[f]);
    ld_trace<P, PDL>(tr, pf.E, pf.status, e2[f] < 0 ? pl.e : e2[f], f ^ 1, pl.j, tp[f]);
  }
  ld_lines<P, PDL>(rvol, pl.tile, L);
  const float wfx = __ldg(pf.opsf + O.wfx() + pl.j), wfy = __ldg(pf.opsf + O.wfy() + pl.j);
  float im[P1];
#pragma unroll
  for (int i = 0; i < P1; ++i) im[i] = __ldg(pf.opsf + O.invM() + pl.j * P1 + i);
  const float *Dy = pf.opsf + P1 * P1;
  const float lws = -__ldg(Dy + pl.j), lwn = __ldg(Dy + P * P1 + pl.j);

  // south and north faces at the thread's column, into shared memory
  float *fy = sm + pl.le * G::FS;
  float S[NV], lf[6];
  face_flux32<VISC, false, -1>(pf, tm[2], tp[2], e2[2] < 0, wfy, S, lf);
#pragma unroll
  for (int v = 0; v < NV; ++v) fy[v * G::RS + pl.j] = S[v];
#pragma unroll
  for (int c = 0; c < 6; ++c) fy[(NV + c) * G::RS + pl.j] = lf[c];
  face_flux32<VISC, false, 1>(pf, tm[3], tp[3], e2[3] < 0, wfy, S, lf);
#pragma unroll
  for (int v = 0; v < NV; ++v) fy[(G::NR + v) * G::RS + pl.j] = S[v];
#pragma unroll
  for (int c = 0; c < 6; ++c) fy[(G::NR + NV + c) * G::RS + pl.j] = lf[c];

  // west and east faces at the line's ends, then per equation the face terms, the symmetric SIP term
  // of the four faces, weighted by the boundary row of D, and M^-1
  float SW[NV], lw[6];
  face_flux32<VISC, true, -1>(pf, tm[0], tp[0], e2[0] < 0, wfx, SW, lw);
  face_flux32<VISC, true, 1>(pf, tm[1], tp[1], e2[1] < 0, wfx, S, lf);
  __syncwarp();
  const bool ends = pl.j == 0 || pl.j == P;
  const float *b = fy + (pl.j == 0 ? 0 : G::NR) * G::RS;
#pragma unroll
  for (int v = 0; v < NV; ++v) {
    float acc[P1];
#pragma unroll
    for (int i = 0; i < P1; ++i) acc[i] = i == 0 ? SW[v] : i == P ? S[v] : 0.f;
    if (ends) {
      float s[P1];
      ld_row<P1>(b + v * G::RS, s);
#pragma unroll
      for (int i = 0; i < P1; ++i) acc[i] += s[i];
    }
    if (v != PSI) {
      const int c = v == PHI ? 0 : v - 1;
      float s[P1], t[P1];
      ld_row<P1>(fy + (NV + c) * G::RS, s);
      ld_row<P1>(fy + (G::NR + NV + c) * G::RS, t);
#pragma unroll
      for (int i = 0; i < P1; ++i)
        acc[i] = fmaf(t[i], lwn, fmaf(s[i], lws, fmaf(lf[c], pf.D[P * P1 + i], fmaf(lw[c], -pf.D[i], acc[i]))));
    }
#pragma unroll
    for (int i = 0; i < P1; ++i) L[v][i] = fmaf(acc[i], im[i], L[v][i]);
  }
  __syncwarp();
}

// The stage update of the thread's line on L = M^-1 R (modes MODE_S1..MODE_S3 with hi_out / lo_out):
// writes the increment or the new step start, leaves the stage state (step start plus increment, in
// FP32; for MODE_S3 the new step start's hi part) in L.  Field by field: a field's lines of the step
// start and the increments are one run each.
template <int P, bool PDL>
__device__ __forceinline__ void update32_line(const LineParams &pf, const LinePlace<P> &pl, int mode, float dt,
                                              const StageIO &io, float (*L)[P + 1]) {
  using G = LineGeom<P>;
  constexpr int P1 = G::P1;
  const size_t base = (size_t)pl.tile * G::TN;
  const int lane = threadIdx.x & 31;
  float w0[NV][P1], dn[NV][P1];
  ld_lines<P, PDL>(io.w0, pl.tile, w0);
  if (mode != MODE_S1) {
    ld_lines<P, PDL>(io.din, pl.tile, dn);
  } else {
#pragma unroll
    for (int v = 0; v < NV; ++v)
#pragma unroll
      for (int i = 0; i < P1; ++i) dn[v][i] = 0.f;
  }
  float chk = 0.f;
  // d1 = dt L,  d2 = (d1 + dt L) / 4; the stage state is w0 + d;
  // w_{n+1} = (hi, lo) + 2 (d2 + dt L) / 3, in float-float
  const float cs = mode == MODE_S1 ? 1.f : mode == MODE_S2 ? 0.25f : 2.f / 3.f;
#pragma unroll
  for (int v = 0; v < NV; ++v) {
    const size_t o = base + v * P1 * 32;
    float d[P1];
#pragma unroll
    for (int i = 0; i < P1; ++i) d[i] = cs * fmaf(dt, L[v][i], dn[v][i]);
    if (mode == MODE_S3) {
      float lo[P1];
      ld_line<P1, PDL>(io.lo + o, lane, lo);
#pragma unroll
      for (int i = 0; i < P1; ++i) {
        L[v][i] = w0[v][i];
        ff_add(L[v][i], lo[i], d[i]);
      }
      st_line<P1>(io.hi_out + o, lane, L[v]);
      st_line<P1>(io.lo_out + o, lane, lo);
    } else {
#pragma unroll
      for (int i = 0; i < P1; ++i) L[v][i] = w0[v][i] + d[i];
      st_line<P1>(io.dout + o, lane, d);
    }
#pragma unroll
    for (int i = 0; i < P1; ++i) chk = fmaf(L[v][i], 0.f, chk);  // 0, or a NaN when a value is not finite
  }
  if (pf.check_finite && pl.act && !(chk == 0.f)) atomicOr(pf.status, STATUS_NONFINITE);
}

// The FP64 ends of a call pass through shared memory, so that the FP64 arrays are read and written
// in consecutive nodes: the warp's first node and number of nodes.
template <int P>
struct WarpNodes {
  int n0, count;
  __device__ __forceinline__ WarpNodes(int E, int tile) {
    using G = LineGeom<P>;
    const int e0 = tile * G::EPW, ne = E - e0 < G::EPW ? E - e0 : G::EPW;
    n0 = e0 * G::NP;
    count = ne > 0 ? ne * G::NP : 0;
  }
  // position of node t of the warp in a staged field
  __device__ __forceinline__ int at(int t) const {
    using G = LineGeom<P>;
    const int le = t / G::NP, a = t - le * G::NP, row = a / G::P1;
    return le * G::ES + row * G::RS + (a - row * G::P1);
  }
};

// The FP64 state of the warp's elements into the FP32 internal state: hi (w32out, and the thread's
// line in q) and, when lo_out is given, lo; the FP64 values as read into w64copy when given.
// sm: fourteen fields.
template <int P, bool PDL>
__device__ __forceinline__ void load_state64(const LineParams &pf, float *sm, const LinePlace<P> &pl,
                                             const double *__restrict__ w64, float *__restrict__ w32out,
                                             float *__restrict__ lo_out, double *__restrict__ w64copy,
                                             float (*q)[P + 1]) {
  using G = LineGeom<P>;
  const WarpNodes<P> wn(pf.E, pl.tile);
  constexpr int NI = (G::EPW * G::NP + 31) / 32;
#pragma unroll
  for (int k = 0; k < NI; ++k) {
    const int t = (threadIdx.x & 31) + 32 * k;
    const int n = wn.n0 + t;
    if (t >= wn.count || !in_bounds(pf.status, n, pf.N)) continue;
    double d[NV];
#pragma unroll
    for (int v = 0; v < NV; ++v) d[v] = ld_in<PDL>(w64 + (size_t)v * pf.N + n);
    if (w64copy) {
      // a device copy of a state in host memory, for the last stage to add to (one read over the
      // host link per call instead of two)
#pragma unroll
      for (int v = 0; v < NV; ++v) w64copy[(size_t)v * pf.N + n] = d[v];
    }
    // the stiffened-gas constant leaves rho E in FP64 first
    d[RE] = d[RE] - fma(pf.dCd, d[PHI], pf.C2d);
    const int p = wn.at(t);
#pragma unroll
    for (int v = 0; v < NV; ++v) {
      if (lo_out) {  // a call of several steps carries the step start as hi + lo
        float h, lo;
        split_ff(d[v], h, lo);
        sm[v * G::SF + p] = h;
        sm[(NV + v) * G::SF + p] = lo;
      } else {  // a single step adds its last increment to the FP64 state itself: hi alone
        sm[v * G::SF + p] = __double2float_rn(d[v]);
      }
    }
  }
  __syncwarp();
  // (a tile past the mesh has no elements: its lines hold a state at rest)
  const int row = pl.le * G::ES + pl.j * G::RS;
  const bool have = wn.count > pl.le * G::NP;
#pragma unroll
  for (int v = 0; v < NV; ++v) {
    if (have) {
      ld_row<G::P1>(sm + v * G::SF + row, q[v]);
    } else {
#pragma unroll
      for (int i = 0; i < G::P1; ++i) q[v][i] = v == M1 || v == M2 ? 1.f : 0.f;
    }
  }
  st_lines<P>(w32out, pl.tile, q);
  if (lo_out) {
#pragma unroll
    for (int v = 0; v < NV; ++v) {
      float lo[G::P1];
#pragma unroll
      for (int i = 0; i < G::P1; ++i) lo[i] = 0.f;
      if (have) ld_row<G::P1>(sm + (NV + v) * G::SF + row, lo);
      st_line<G::P1>(lo_out + (size_t)pl.tile * G::TN + v * G::P1 * 32, threadIdx.x & 31, lo);
    }
  }
  __syncwarp();
}

// Shared floats per warp: `fields` staged fields, or the y-face results.
template <int P>
__host__ __device__ constexpr int line_smem(int fields) {
  using G = LineGeom<P>;
  const int a = fields * G::SF, b = G::EPW * G::FS;
  return ((a > b ? a : b) + 3) / 4 * 4;
}

// Whether a tile's last node lies below the node count, and with it the tile's slots in the node arrays
// (the bounds-checked build; else constant true).  The whole warp agrees.
template <int P>
__device__ __forceinline__ bool tile_in_bounds(const LineParams &pf, int tile) {
  using G = LineGeom<P>;
  const long long end = (long long)(tile + 1) * G::EPW;
  return in_bounds(pf.status, (end < pf.E ? end : pf.E) * G::NP - 1, pf.N);
}

// Bodies of the three kernels for one tile (tiles past the mesh are skipped by the whole warp).
template <int P, bool VISC, bool ST, bool PDL>
__device__ __forceinline__ void volume32_tile(const LineParams &pf, float *sm, int tile, const float *__restrict__ w,
                                              float *__restrict__ rvol, float4 *__restrict__ tr,
                                              const double *__restrict__ w64, float *__restrict__ w32out,
                                              float *__restrict__ lo_out, double *__restrict__ w64copy) {
  using G = LineGeom<P>;
  if (tile * G::EPW >= pf.E || !tile_in_bounds<P>(pf, tile)) return;
  const LinePlace<P> pl(pf.E, tile);
  float q[NV][G::P1];
  if (w64) load_state64<P, PDL>(pf, sm, pl, w64, w32out, lo_out, w64copy, q);
  else ld_lines<P, PDL>(w, tile, q);
  vol32_line<P, VISC, ST>(pf, sm, pl, q, rvol, tr);
}

template <int P, bool VISC, bool ST, bool PDL>
__device__ __forceinline__ void surfvol32_tile(const LineParams &pf, float *sm, int tile, int mode, float dt,
                                               const StageIO &io, const float *__restrict__ rvol_in,
                                               const float4 *__restrict__ tr_in, float *__restrict__ rvol_out,
                                               float4 *__restrict__ tr_out) {
  if (tile * LineGeom<P>::EPW >= pf.E || !tile_in_bounds<P>(pf, tile)) return;
  const LinePlace<P> pl(pf.E, tile);
  float L[NV][P + 1];
  surf32_line<P, VISC, PDL>(pf, sm, pl, rvol_in, tr_in, L);
  update32_line<P, PDL>(pf, pl, mode, dt, io, L);
  vol32_line<P, VISC, ST>(pf, sm, pl, L, rvol_out, tr_out);
}

// The surface part alone: MODE_RHS (L in FP64), a stage's increment, or a call's last stage, which
// writes the FP64 state (io.out64).  sm: fourteen fields (seven when io.w64in is given).
template <int P, bool VISC, bool PDL>
__device__ __forceinline__ void surface32_tile(const LineParams &pf, float *sm, int tile, int mode, float dt,
                                               const StageIO &io, const float *__restrict__ rvol,
                                               const float4 *__restrict__ tr) {
  using G = LineGeom<P>;
  constexpr int P1 = G::P1;
  if (tile * G::EPW >= pf.E || !tile_in_bounds<P>(pf, tile)) return;
  const LinePlace<P> pl(pf.E, tile);
  float L[NV][P1];
  surf32_line<P, VISC, PDL>(pf, sm, pl, rvol, tr, L);
  if (!io.out64) {
    update32_line<P, PDL>(pf, pl, mode, dt, io, L);
    return;
  }
  const size_t base = (size_t)tile * G::TN;
  const int lane = threadIdx.x & 31, row = pl.le * G::ES + pl.j * G::RS;
  const bool from64 = mode == MODE_S3 && io.w64in != nullptr;
  float chk = 0.f;
#pragma unroll
  for (int v = 0; v < NV; ++v) {
    if (mode == MODE_S3) {
      // L becomes the increment 2 (d2 + dt L) / 3 (from64), or the new step start's hi part, with its
      // lo part in the second seven fields
      float dn[P1];
      ld_line<P1, PDL>(io.din + base + v * P1 * 32, lane, dn);
#pragma unroll
      for (int i = 0; i < P1; ++i) L[v][i] = (2.f / 3.f) * fmaf(dt, L[v][i], dn[i]);
      if (!from64) {
        float w0[P1], lo[P1];
        ld_line<P1, PDL>(io.w0 + base + v * P1 * 32, lane, w0);
        ld_line<P1, PDL>(io.lo + base + v * P1 * 32, lane, lo);
#pragma unroll
        for (int i = 0; i < P1; ++i) {
          ff_add(w0[i], lo[i], L[v][i]);
          L[v][i] = w0[i];
        }
        if (pl.act) st_row<P1>(sm + (NV + v) * G::SF + row, lo);
      }
    }
#pragma unroll
    for (int i = 0; i < P1; ++i) chk = fmaf(L[v][i], 0.f, chk);
    if (pl.act) st_row<P1>(sm + v * G::SF + row, L[v]);
  }
  if (pf.check_finite && pl.act && !(chk == 0.f)) atomicOr(pf.status, STATUS_NONFINITE);
  __syncwarp();
  const WarpNodes<P> wn(pf.E, tile);
  constexpr int NI = (G::EPW * G::NP + 31) / 32;
#pragma unroll
  for (int k = 0; k < NI; ++k) {
    const int t = lane + 32 * k;
    const int n = wn.n0 + t;
    if (t >= wn.count || !in_bounds(pf.status, n, pf.N)) continue;
    const int p = wn.at(t);
    float d[NV];
#pragma unroll
    for (int v = 0; v < NV; ++v) d[v] = sm[v * G::SF + p];
    double *o = io.out64 + n;
    if (mode == MODE_RHS) {
      const double lphi = f2d(d[PHI]);
#pragma unroll
      for (int v = 0; v < RE; ++v) o[(size_t)v * pf.N] = v == PHI ? lphi : f2d(d[v]);
      o[(size_t)RE * pf.N] = fma(pf.dCd, lphi, f2d(d[RE]));
    } else if (from64) {
      // w_{n+1} = w_n + 2 (d2 + dt L) / 3 in FP64 on the caller's state; the increment of the
      // reduced energy becomes one of rho E by adding (C_1 - C_2) times that of phi
      double w[NV];
#pragma unroll
      for (int v = 0; v < NV; ++v) w[v] = __ldca(io.w64in + (size_t)v * pf.N + n);
      const double dphi = f2d(d[PHI]);
#pragma unroll
      for (int v = 0; v < RE; ++v) o[(size_t)v * pf.N] = w[v] + (v == PHI ? dphi : f2d(d[v]));
      o[(size_t)RE * pf.N] = w[RE] + fma(pf.dCd, dphi, f2d(d[RE]));
    } else {
      // last stage of a call: hand back the FP64 state hi + lo, restoring the stiffened-gas
      // constant with the carried phi
      float lo[NV];
#pragma unroll
      for (int v = 0; v < NV; ++v) lo[v] = sm[(NV + v) * G::SF + p];
      const double phi64 = ff_to_double(d[PHI], lo[PHI]);
#pragma unroll
      for (int v = 0; v < RE; ++v) o[(size_t)v * pf.N] = v == PHI ? phi64 : ff_to_double(d[v], lo[v]);
      o[(size_t)RE * pf.N] = ff_to_double(d[RE], lo[RE]) + fma(pf.dCd, phi64, pf.C2d);
    }
  }
}

// ---------------------------------------------------------------------------
// Kernels of one problem
// ---------------------------------------------------------------------------
constexpr int WPB32 = 2;  // warps per block
// Blocks per SM asked of the compiler for the stage kernel.  An SM's four schedulers hold 16,384 registers
// each, so the caps are 128 a thread at p <= 2 (spilling up to 80 bytes), 168 at p = 3 and 4 (p = 4 spills 44
// bytes with viscous stress and surface tension, 36 with surface tension, 24 with viscous stress, none without),
// 168 at p = 5 (ten warps are three on one scheduler; 136 bytes spilled) and 255 there with any term (254 used).
// Microseconds a step when these were chosen: p = 3 at 160 x 160, 168 registers 51, 144 57, 128 59; p = 4 with
// all terms at 256 x 256, uncapped (207) 301, 168 271, 144 313; p = 5 at 128 x 128, five blocks asked 83, four
// (255) 96, and with all terms at 96 x 96 75 and 69.
template <int P, bool FULL>
constexpr int LINE_MINB = P <= 2 ? 8 : P <= 4 ? 6 : FULL ? 4 : 5;

// PDL: launched as a programmatic dependent of the kernel before (launch_dependent).
template <int P, bool VISC, bool ST, bool PDL>
__global__ void __launch_bounds__(32 * WPB32)
k_volume32_lines(const __grid_constant__ LineParams pf, const float *__restrict__ w, float *__restrict__ rvol,
                 float4 *__restrict__ tr, const double *__restrict__ w64, float *__restrict__ w32out,
                 float *__restrict__ lo_out, double *__restrict__ w64copy) {
  __shared__ __align__(16) float sm[WPB32][line_smem<P>(14)];
  if (PDL) grid_dependency_wait();
  const int wi = threadIdx.x / 32;
  volume32_tile<P, VISC, ST, PDL>(pf, sm[wi], blockIdx.x * WPB32 + wi, w, rvol, tr, w64, w32out, lo_out, w64copy);
}

template <int P, bool VISC, bool PDL>
__global__ void __launch_bounds__(32 * WPB32)
k_surface32_lines(const __grid_constant__ LineParams pf, int mode, float dt, const StageIO io,
                  const float *__restrict__ rvol, const float4 *__restrict__ tr) {
  __shared__ __align__(16) float sm[WPB32][line_smem<P>(14)];
  if (PDL) grid_dependency_wait();
  if (io.dt_dev) dt = (float)ld_in<PDL>(io.dt_dev);
  const int wi = threadIdx.x / 32;
  surface32_tile<P, VISC, PDL>(pf, sm[wi], blockIdx.x * WPB32 + wi, mode, dt, io, rvol, tr);
}

// The fused stage kernel (see k_surfvol32): the stage state is handed from the surface part to the
// volume part in registers.
template <int P, bool VISC, bool ST, bool PDL>
__global__ void __launch_bounds__(32 * WPB32, LINE_MINB<P, VISC || ST>)
k_surfvol32_lines(const __grid_constant__ LineParams pf, int mode, float dt, const StageIO io,
                  const float *__restrict__ rvol_in, const float4 *__restrict__ tr_in, float *__restrict__ rvol_out,
                  float4 *__restrict__ tr_out) {
  __shared__ __align__(16) float sm[WPB32][line_smem<P>(6)];
  if (PDL) grid_dependency_wait();
  if (io.dt_dev) dt = (float)ld_in<PDL>(io.dt_dev);
  const int wi = threadIdx.x / 32;
  surfvol32_tile<P, VISC, ST, PDL>(pf, sm[wi], blockIdx.x * WPB32 + wi, mode, dt, io, rvol_in, tr_in, rvol_out, tr_out);
}

template <int P>
inline int line_blocks(int E) {
  return (line_tiles(P + 1, E) + WPB32 - 1) / WPB32;
}

// A grid that the GPU holds at once is launched as a programmatic dependent, a larger one plainly, as
// in dg_kernels_fp32.cuh.
template <int P, bool VISC, bool ST>
cudaError_t launch_volume32_lines(const Params &, const ParamsF &, const LineParams &lp, const float *, const float *w,
                                  float *rvol, float *trace, const double *w64, float *w32out, float *lo_out,
                                  double *w64copy, cudaStream_t s) {
  constexpr int T = 32 * WPB32;
  const int blocks = line_blocks<P>(lp.E);
  float4 *tr = reinterpret_cast<float4 *>(trace);
  static const int resident = resident_blocks(k_volume32_lines<P, VISC, ST, true>, T);
  if (blocks <= resident)
    return launch_dependent(k_volume32_lines<P, VISC, ST, true>, blocks, T, 0, s, lp, w, rvol, tr, w64, w32out, lo_out,
                            w64copy);
  k_volume32_lines<P, VISC, ST, false><<<blocks, T, 0, s>>>(lp, w, rvol, tr, w64, w32out, lo_out, w64copy);
  return cudaGetLastError();
}

template <int P, bool VISC, bool ST>
cudaError_t launch_surface32_lines(const Params &, const ParamsF &, const LineParams &lp, const float *, int mode,
                                   float dt, const StageIO &io, const float *rvol, const float *trace,
                                   cudaStream_t s) {
  constexpr int T = 32 * WPB32;
  const int blocks = line_blocks<P>(lp.E);
  const float4 *tr = reinterpret_cast<const float4 *>(trace);
  static const int resident = resident_blocks(k_surface32_lines<P, VISC, true>, T);
  if (blocks <= resident)
    return launch_dependent(k_surface32_lines<P, VISC, true>, blocks, T, 0, s, lp, mode, dt, io, rvol, tr);
  k_surface32_lines<P, VISC, false><<<blocks, T, 0, s>>>(lp, mode, dt, io, rvol, tr);
  return cudaGetLastError();
}

template <int P, bool VISC, bool ST>
cudaError_t launch_surfvol32_lines(const Params &, const ParamsF &, const LineParams &lp, const float *, int mode,
                                   float dt, const StageIO &io, const float *rvol_in, const float *tr_in,
                                   float *rvol_out, float *tr_out, cudaStream_t s) {
  constexpr int T = 32 * WPB32;
  const int blocks = line_blocks<P>(lp.E);
  const float4 *ti = reinterpret_cast<const float4 *>(tr_in);
  float4 *to = reinterpret_cast<float4 *>(tr_out);
  static const int resident = resident_blocks(k_surfvol32_lines<P, VISC, ST, true>, T);
  if (blocks <= resident)
    return launch_dependent(k_surfvol32_lines<P, VISC, ST, true>, blocks, T, 0, s, lp, mode, dt, io, rvol_in, ti,
                            rvol_out, to);
  k_surfvol32_lines<P, VISC, ST, false><<<blocks, T, 0, s>>>(lp, mode, dt, io, rvol_in, ti, rvol_out, to);
  return cudaGetLastError();
}

template <int P, bool VISC, bool ST>
KernelSet32 make_lines32() {
  return KernelSet32{&launch_volume32_lines<P, VISC, ST>, &launch_surface32_lines<P, VISC, ST>,
                     &launch_surfvol32_lines<P, VISC, ST>,
                     [] { return WPB32 * resident_blocks(k_surfvol32_lines<P, VISC, ST, true>, 32 * WPB32); },
                     [] {
                       return WPB32 * std::min(resident_blocks(k_volume32_lines<P, VISC, ST, true>, 32 * WPB32),
                                               resident_blocks(k_surface32_lines<P, VISC, true>, 32 * WPB32));
                     }};
}

// Line kernels of order P (2D).
template <int P>
KernelSet32 lines_fp32_p(bool viscous, bool st) {
  if (!viscous && !st) return make_lines32<P, false, false>();
  if (viscous && !st) return make_lines32<P, true, false>();
  if (!viscous) return make_lines32<P, false, true>();
  return make_lines32<P, true, true>();
}

}  // namespace dgpf
