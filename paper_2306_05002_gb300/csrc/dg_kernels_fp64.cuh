// dg_kernels_fp64.cuh -- FP64 kernels of the DG right-hand side (GB300, sm_103a).
//
// Two kernels per right-hand side evaluation, both element-blocked (one CTA
// holds EPB whole elements, one thread per node):
//
//   k_volume   closure (stiffened gas, Sec. 2), broken gradients of phi and
//              psi (and u, v when viscous) by sum-factorised 1D contractions,
//              level-set normal n = grad psi/|grad psi|, a_1, curvature,
//              conservative fluxes, the weak-form volume term (tensor-product
//              Dhat contractions, Sec. 3 eq. "weakDG"), the non-conservative
//              transport -u.grad(phi) of Sec. 3 and the sources of Sec. 2.
//              Writes the volume part of M^-1 R and one trace record per face
//              node.
//   k_surface  per face node: Lax-Friedrichs flux, quasi-conservative
//              transport flux, SIP flux of a_1 and its derived terms, viscous
//              penalty flux (Sec. 3); lifts the SIP symmetric term along the
//              normal line; applies M^-1; adds the volume part; and writes
//              either L or one SSP-RK3 stage (fused update).
//
// On GB300 the FP64 pipe (two operations per clock and SM) bounds this path, so the kernels spend
// FP64 instructions only on the scheme's arithmetic: operator tables are premultiplied by 2/h, signs,
// comparisons, selections and index work are integer, divisions by one denominator share its
// reciprocal (dg_math64.cuh), and a node adds one face value per axis.
//
// These kernels serve the contexts that have a discrete adjoint, whose gradient of
// max(|u-.m| + c-, |u+.m| + c+) jumps with the last bits of the state where the two speeds tie and
// the traces do not (a rounding changed in one kernel moved the gradient of a 20-step 128 x 128,
// p = 3 trajectory by 5e-8).  They therefore hold to one order of rounded operations: every
// statement below gives the bits of the scheme's formula as written in its comment, with
// multiplications by powers of two, signs and zero terms folded.  Variants with viscous stress or
// surface tension, which have no adjoint, regroup the operations (dg_kernels_full64.cuh).
#pragma once

#include "dg_common.cuh"
#include "dg_math64.cuh"
#include "dg_pdl.cuh"

namespace dgpf {

// Block geometry of one kernel family.  EPBX > 0 overrides the number of
// elements per block (the batched kernels' tuned tile).
template <int P, int DIM, bool VISC, bool ST, int EPBX = 0>
struct Geom {
  static constexpr int P1 = P + 1;
  static constexpr int NP = DIM == 2 ? P1 * P1 : P1;
  static constexpr int NF = 2 * DIM;                 // faces per element
  static constexpr int NK = DIM == 2 ? P1 : 1;       // nodes per face
  static constexpr int NFK = NF * NK;                // face nodes per element
  // Elements per block of the FP32-bulk kernels with one node per thread and of
  // k_ri_sign (the other FP64 kernels choose at launch, pick_epb64; the batched
  // kernels give EPBX): the smallest count that fills at least 60 threads with
  // under 7% of the last warp idle.  Small blocks spread a grid evenly over the SMs.
  static constexpr int pick_epb() {
    for (int e = 1; e <= 64; ++e) {
      const int t = e * NP, tp = ((t + 31) / 32) * 32;
      if (t >= 60 && (tp - t) * 100 < 7 * tp) return e;
    }
    return (128 + NP - 1) / NP;
  }
  static constexpr int EPB = EPBX > 0 ? EPBX : pick_epb();
  static constexpr int THREADS = ((EPB * NP + 31) / 32) * 32;
  static constexpr int NSTAGE = 12;                  // staged fields per node
  static constexpr int OPS = 4 * P1 * P1 + 3 * P1 + NP;  // operator table (OpsLayout) up to cf()
};

// Neighbour of element e across face f (0 W, 1 E, 2 S, 3 N), or -1 at a wall.
__device__ __forceinline__ int neighbour(const ParamsCore &p, int e, int f) {
  const int ex = e % p.nx, ey = e / p.nx;
  switch (f) {
    case 0: return ex > 0 ? e - 1 : (p.bc[0] == BC_PERIODIC ? e + p.nx - 1 : -1);
    case 1: return ex < p.nx - 1 ? e + 1 : (p.bc[1] == BC_PERIODIC ? e - p.nx + 1 : -1);
    case 2: return ey > 0 ? e - p.nx : (p.bc[2] == BC_PERIODIC ? e + p.nx * (p.ny - 1) : -1);
    default: return ey < p.ny - 1 ? e + p.nx : (p.bc[3] == BC_PERIODIC ? e - p.nx * (p.ny - 1) : -1);
  }
}

// phi_1 C_1 + phi_2 C_2, in the formula's own operation order.
__device__ __forceinline__ double mixture_constant(const Params &p, double phi) {
  return __dadd_rn(__dmul_rn(phi, p.C1), __dmul_rn(__dsub_rn(1.0, phi), p.C2));
}

// Stiffened-gas pressure (Sec. 2), in the formula's own operation order:
//   rho e = rho E - (|rho u|^2 / 2) / rho
//   P = (rho e - (phi_1 C_1 + phi_2 C_2)) / (phi_1 g_1 + phi_2 g_2)
__device__ __forceinline__ double sg_pressure(const Params &p, double phi, double rho, double ru, double rv,
                                              double rE, double *Cm, double *den) {
  const double phi2 = __dsub_rn(1.0, phi);
  const double rhok = __ddiv_rn(__dmul_rn(0.5, __dadd_rn(__dmul_rn(ru, ru), __dmul_rn(rv, rv))), rho);
  const double rhoe = __dsub_rn(rE, rhok);
  *Cm = __dadd_rn(__dmul_rn(phi, p.C1), __dmul_rn(phi2, p.C2));
  *den = __dadd_rn(__dmul_rn(phi, p.g1), __dmul_rn(phi2, p.g2));
  return __ddiv_rn(__dsub_rn(rhoe, *Cm), *den);
}

// Elements per block of an FP64 kernel, chosen at launch.  The FP64 pipe of the fullest SM sets the
// time: ceil(blocks / SMs) blocks of cn instructions per node warp and cf per face-node warp.  So
// a mesh of a few blocks per SM takes the count that spreads it best over the SMs (800 elements of
// p = 4: one 25-lane warp per element, 6 to an SM, instead of 5 elements in 4 warps, 8 to an SM), a
// large one the count that leaves the fewest idle lanes.  Ties go to the larger block (fewer
// copies of the operator table).
constexpr int MAX_THREADS64 = 192;
// per: threads' tasks per element (its nodes); perf: face nodes.
inline int pick_epb64(int E, int per, int cn, int perf = 0, int cf = 0) {
  static const int sms = [] {
    int dev = 0, n = 0;
    if (cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || n < 1)
      n = 152;
    return n;
  }();
  int best = 1;
  long best_cost = 0;
  for (int epb = 1; epb == 1 || (epb * per + 31) / 32 * 32 <= MAX_THREADS64; ++epb) {
    const int wn = (epb * per + 31) / 32, wf = (epb * perf + 31) / 32;
    const long blocks = (E + epb - 1) / epb;
    const long cost = (blocks + sms - 1) / sms * (cn * wn + cf * wf);
    if (epb == 1 || cost <= best_cost) {
      best = epb;
      best_cost = cost;
    }
  }
  return best;
}

// Launches: programmatic dependents of the kernel before (dg_pdl.cuh), waiting first thing, so that
// a launch's latency overlaps that kernel's tail.  They do not let the next kernel start early:
// blocks that arrive while others still compute land unevenly, and the SM with the most blocks sets
// the time (64 x 64, p = 3: 191 us a step with an early trigger, 141 without).
//
// Bound by the FP64 pipe.  64 x 64, p = 3 in 2D: a step of three volume and three surface launches
// 172 -> 141 us (what the update reads requested where it is used: 147; ahead of the face work: no gain,
// and 3% slower where the grid has several waves, for the registers it holds).
template <int P, int DIM>
__global__ void __launch_bounds__(MAX_THREADS64)
k_volume(const Params prm, int epb, const double *__restrict__ w, double *__restrict__ rvol,
         double *__restrict__ tr) {
  using G = Geom<P, DIM, false, false>;
  constexpr int P1 = G::P1, NP = G::NP, NFK = G::NFK, NK = G::NK;
  constexpr int P11 = P1 * P1;
  extern __shared__ double s_mem[];
  grid_dependency_wait();
  double *s_op = s_mem;                    // Dx, Dy, Dhx, Dhy
  double *s_f = s_mem + 4 * P11;           // [G::NSTAGE][epb * NP]
  const int fs = epb * NP;                 // nodes of the block: stride between staged fields

  for (int t = threadIdx.x; t < 4 * P11; t += blockDim.x) s_op[t] = prm.ops[t];
  const double *Dx = s_op, *Dy = s_op + P11, *Dhx = s_op + 2 * P11, *Dhy = s_op + 3 * P11;

  const int le_raw = threadIdx.x / NP;
  const bool lane = le_raw < epb;
  const int le = lane ? le_raw : epb - 1;  // padding lanes mirror the last element, write nothing
  const int a = threadIdx.x % NP;
  const int e = blockIdx.x * epb + le;
  const int N = prm.N;
  const bool act = lane && e < prm.E && in_bounds(prm.status, (long long)e * NP + a, N);
  const int i = a % P1, j = DIM == 2 ? a / P1 : 0;
  const long n = (long)(act ? e : 0) * NP + a;
  const int sn = le * NP + a;              // the node in the staged fields
  const int sx = le * NP + P1 * j;         // its x-line (stride 1) and y-line (stride P1)
  const int sy = le * NP + i;

  double q[NV];
#pragma unroll
  for (int v = 0; v < NV; ++v) q[v] = act ? __ldca(w + (long)v * N + n) : (v == M1 || v == M2 ? 1.0 : 0.0);
  const double phi = q[PHI], psi = q[PSI];
  const double rho = q[M1] + q[M2];
  const double ir = rcp64_rn(rho);
  const double u = q[RU] * ir;
  const double v = DIM == 2 ? q[RV] * ir : 0.0;
  // sg_pressure, its divisions sharing the reciprocals
  const double rv0 = DIM == 2 ? q[RV] : 0.0;
  const double rhok = div64_rn(__dmul_rn(0.5, __dadd_rn(__dmul_rn(q[RU], q[RU]), __dmul_rn(rv0, rv0))), rho, ir);
  const double phi2 = __dsub_rn(1.0, phi);
  const double Cm = __dadd_rn(__dmul_rn(phi, prm.C1), __dmul_rn(phi2, prm.C2));
  const double den = __dadd_rn(__dmul_rn(phi, prm.g1), __dmul_rn(phi2, prm.g2));
  const double iden = rcp64_rn(den);
  const double Pr = div64_rn(__dsub_rn(__dsub_rn(q[RE], rhok), Cm), den, iden);
  const double B = fma(Pr, prm.Bp, prm.dC);
  const double k = 0.5 * fma(v, v, u * u);
  const double X = Pr + div64_rn(Pr + Cm, den, iden);  // rho c^2
  // Non-physical state: rho <= 0, a mixture 1/(gamma - 1) <= 0, or P + Pinf_mix <= 0, i.e.
  // rho c^2 <= 0 (Sec. 2 mixture rules).
  if (prm.check_finite && act && (nonpositive64(rho) || nonpositive64(den) || nonpositive64(X)))
    atomicOr(prm.status, STATUS_NONPHYSICAL);

  if (lane) {
    s_f[0 * fs + sn] = phi;
    s_f[1 * fs + sn] = psi;
  }
  __syncthreads();

  // Broken gradients: sum-factorised contractions along the two GLL lines.
  double gpx = 0.0, gpy = 0.0, gsx = 0.0, gsy = 0.0;
#pragma unroll
  for (int c = 0; c < P1; ++c) {
    const double dx = Dx[i * P1 + c];
    const int ax = sx + c;
    gpx = c ? fma(dx, s_f[0 * fs + ax], gpx) : dx * s_f[0 * fs + ax];
    gsx = c ? fma(dx, s_f[1 * fs + ax], gsx) : dx * s_f[1 * fs + ax];
    if (DIM == 2) {
      const double dy = Dy[j * P1 + c];
      const int ay = sy + P1 * c;
      gpy = c ? fma(dy, s_f[0 * fs + ay], gpy) : dy * s_f[0 * fs + ay];
      gsy = c ? fma(dy, s_f[1 * fs + ay], gsy) : dy * s_f[1 * fs + ay];
    }
  }

  // The transport term keeps the broken gradients; with grad_lift the gradients of phi and psi
  // become BR1-lifted: at a face node, M^-1 w_f (f+ - f-) / 2 along the outward normal, f+ the
  // neighbour's value at the coincident node (none at walls and pressure boundaries).
  const double bpx = gpx, bpy = gpy, bsx = gsx, bsy = gsy;
  if (prm.grad_lift && act && (i == 0 || i == P || (DIM == 2 && (j == 0 || j == P)))) {
    const OpsLayout Lo{P1, NP};
    const double im = __ldca(prm.ops + Lo.invM() + a);
    auto lift = [&](int f, int kk, double &gx_phi, double &gx_psi, double sgn) {
      const int e2 = neighbour(prm, e, f);
      if (e2 < 0) return;
      const int f2 = f ^ 1;
      const int a2 = f2 == 0 ? P1 * kk : f2 == 1 ? P + P1 * kk : f2 == 2 ? kk : kk + P1 * P;
      const long n2 = (long)e2 * NP + a2;
      if (!in_bounds(prm.status, n2, N)) return;
      const double wf = DIM == 2 ? __ldca(prm.ops + (f < 2 ? Lo.wfx() : Lo.wfy()) + kk) : 1.0;
      const double c = sgn * 0.5 * im * wf;
      gx_phi += c * (__ldca(w + (long)PHI * N + n2) - phi);
      gx_psi += c * (__ldca(w + (long)PSI * N + n2) - psi);
    };
    const int kx = DIM == 2 ? j : 0;
    if (i == 0) lift(0, kx, gpx, gsx, -1.0);
    if (i == P) lift(1, kx, gpx, gsx, 1.0);
    if (DIM == 2 && j == 0) lift(2, i, gpy, gsy, -1.0);
    if (DIM == 2 && j == P) lift(3, i, gpy, gsy, 1.0);
  }

  // Interface normal from the level set (zero where |grad psi| < 1e-12).
  const double g2 = fma(gsy, gsy, gsx * gsx);
  double nx = 0.0, ny = 0.0;
  if (has_gradient(g2)) {
    const double r = rsqrt(g2);
    nx = gsx * r;
    ny = gsy * r;
  }
  const double sphi = phi * phi2;
  const double a1x = prm.Gamma * fma(prm.eps, gpx, -(sphi * nx));
  const double a1y = DIM == 2 ? prm.Gamma * fma(prm.eps, gpy, -(sphi * ny)) : 0.0;

  // Conservative fluxes (moved to the right-hand side), per equation:
  // m_l u -+ rho0_l a_1, rho u u + P - drho0 a_1 u, (rho E + P) u - cE a_1.
  const double cE = fma(prm.drho0, k, B);
  const double dax = prm.drho0 * a1x, H = q[RE] + Pr;
  double F[G::NSTAGE];
  F[0] = -a1x;
  F[2] = fma(q[M1], u, -(prm.rho01 * a1x));
  F[4] = fma(q[M2], u, prm.rho02 * a1x);
  F[6] = fma(-dax, u, fma(q[RU], u, Pr));
  F[10] = fma(H, u, -(cE * a1x));
  if (DIM == 2) {
    const double day = prm.drho0 * a1y;
    F[1] = -a1y;
    F[3] = fma(q[M1], v, -(prm.rho01 * a1y));
    F[5] = fma(q[M2], v, prm.rho02 * a1y);
    F[7] = fma(q[RU], v, -(day * u));
    F[8] = fma(q[RV], u, -(dax * v));
    F[9] = fma(-day, v, fma(q[RV], v, Pr));
    F[11] = fma(H, v, -(cE * a1y));
  } else {
    F[8] = q[RV] * u;
  }
  __syncthreads();
  if (lane) {
#pragma unroll
    for (int s = 0; s < G::NSTAGE; ++s)
      if (DIM == 2 || !(s & 1)) s_f[s * fs + sn] = F[s];
  }
  __syncthreads();

  // Volume term: M^-1 sum_k w_k J grad(l_a)(x_k) . F_k = Dhx F^x + Dhy F^y.
  double R[NV];
#pragma unroll
  for (int eq = 0; eq < 6; ++eq) {
    double acc = 0.0;
#pragma unroll
    for (int c = 0; c < P1; ++c) {
      const double fx = s_f[2 * eq * fs + sx + c];
      acc = c ? fma(Dhx[i * P1 + c], fx, acc) : Dhx[i * P1 + c] * fx;
      if (DIM == 2) acc = fma(Dhy[j * P1 + c], s_f[(2 * eq + 1) * fs + sy + P1 * c], acc);
    }
    R[eq == 0 ? PHI : eq + 1] = acc;
  }
  // Non-conservative transport of phi and psi (Sec. 3: treated as a source), broken gradients.
  R[PHI] -= fma(v, bpy, u * bpx);
  R[PSI] = -fma(v, bsy, u * bsx);
  if (prm.gravity) {
    R[RU] += rho * prm.gx;
    R[RV] += rho * prm.gy;
    R[RE] += rho * (prm.gx * u + prm.gy * v);
  }
  if (act) {
#pragma unroll
    for (int vv = 0; vv < NV; ++vv) rvol[(long)vv * N + n] = R[vv];
  }

  // Face traces.
  const bool onW = i == 0, onE = i == P;
  const bool onS = DIM == 2 && j == 0, onN = DIM == 2 && j == P;
  if (act && (onW || onE || onS || onN)) {
    const double c = sqrt64_rn(X * ir);  // mixture sound speed
    const double tx[T_GPHI] = {phi, psi, q[M1], q[M2], q[RU], q[RV], q[RE], u, v, Pr, c, B};
    const long base = (long)e * NFK;
    const long stride = (long)prm.E * NFK;
    auto put = [&](int f, int kk, double gn, double nn) {
      const long o = base + f * NK + kk;
      if (!in_bounds(prm.status, o, stride)) return;
#pragma unroll
      for (int qf = 0; qf < T_GPHI; ++qf) tr[qf * stride + o] = tx[qf];
      tr[T_GPHI * stride + o] = gn;
      tr[T_N * stride + o] = nn;
    };
    const int kx = DIM == 2 ? j : 0;
    if (onW) put(0, kx, gpx, nx);
    if (onE) put(1, kx, gpx, nx);
    if (onS) put(2, i, gpy, ny);
    if (onN) put(3, i, gpy, ny);
  }
}

// Per axis and node of a face, the products of the face weight wf that a face node would otherwise
// form again: wf / 2, wf, wf rho01, wf (-rho02) and -wf / 2 Gamma eps.
enum FaceTable { FT_HALF = 0, FT_W, FT_W1, FT_W2, FT_SYM, NFT };

template <int P, int DIM>
__global__ void __launch_bounds__(MAX_THREADS64)
k_surface(const Params prm, int epb, int mode, double dt, const double *__restrict__ w0,
          const double *__restrict__ ws, const double *__restrict__ rvol, const double *__restrict__ tr,
          double *__restrict__ out) {
  using G = Geom<P, DIM, false, false>;
  constexpr int P1 = G::P1, NP = G::NP, NFK = G::NFK, NK = G::NK, NT = NT_INVISCID;
  constexpr int NS = NV + 6;            // planes: surface integrand, lifting coefficients
  constexpr int OPN = 2 * P1 * P1 + NP; // Dx, Dy, invM
  const OpsLayout L{P1, NP};
  extern __shared__ double s_mem[];
  grid_dependency_wait();
  double *s_op = s_mem;                 // Dx, Dy, invM
  double *s_ft = s_op + OPN;            // [2][NFT][P1]
  double *s_s = s_ft + 2 * NFT * P1;    // [NS][epb * NFK]
  const int fs = epb * NFK;

  for (int t = threadIdx.x; t < OPN; t += blockDim.x)
    s_op[t] = prm.ops[t < 2 * P1 * P1 ? t : L.invM() + t - 2 * P1 * P1];
  for (int t = threadIdx.x; t < 2 * P1; t += blockDim.x) {
    const double wf = prm.ops[(t < P1 ? L.wfx() : L.wfy()) + t % P1];
    double *r = s_ft + (t < P1 ? 0 : NFT * P1) + t % P1;
    r[FT_HALF * P1] = 0.5 * wf;
    r[FT_W * P1] = wf;
    r[FT_W1 * P1] = wf * prm.rho01;
    r[FT_W2 * P1] = wf * -prm.rho02;
    r[FT_SYM * P1] = -0.5 * wf * prm.Gamma * prm.eps;
  }
  __syncthreads();
  const double *Dx = s_op, *Dy = s_op + P1 * P1, *invM = s_op + 2 * P1 * P1;
  const long stride = (long)prm.E * NFK;
  const int le = threadIdx.x / NP, a = threadIdx.x % NP;
  const int e = blockIdx.x * epb + le;
  const int N = prm.N;
  const long n = (long)e * NP + a;
  const bool act = le < epb && e < prm.E && in_bounds(prm.status, n, N);
  if (prm.dt_dev) dt = __ldca(prm.dt_dev);

  // Phase 1: numerical fluxes at the block's face nodes.  S and the terms below carry a factor two
  // where the formula averages or halves (exact).
  for (int g = threadIdx.x; g < fs; g += blockDim.x) {
    const int fe = blockIdx.x * epb + g / NFK, t = g % NFK;
    if (fe >= prm.E) break;
    const int f = t / NK, kk = t % NK;
    const int e2 = neighbour(prm, fe, f);
    const bool wall = e2 < 0;
    const bool xf = f < 2;
    const int sm = (f & 1) ? 0 : (int)0x80000000;  // sign of m
    double Tm[NT], Tp[NT];
    const long om = (long)fe * NFK + t;
    const bool okm = in_bounds(prm.status, om, stride);
#pragma unroll
    for (int qf = 0; qf < NT; ++qf) Tm[qf] = okm ? __ldca(tr + qf * stride + om) : (qf == T_M1 ? 1.0 : 0.0);
    if (!wall) {
      const long op = (long)e2 * NFK + (f ^ 1) * NK + kk;
      const bool okp = in_bounds(prm.status, op, stride);
#pragma unroll
      for (int qf = 0; qf < NT; ++qf) Tp[qf] = okp ? __ldca(tr + qf * stride + op) : Tm[qf];
    } else {
#pragma unroll
      for (int qf = 0; qf < NT; ++qf) Tp[qf] = Tm[qf];
      const int bc = prm.bc[f];
      if (bc == BC_SLIP) {  // reverse the normal component only
        if (xf) { Tp[T_RU] = -Tm[T_RU]; Tp[T_U] = -Tm[T_U]; }
        else    { Tp[T_RV] = -Tm[T_RV]; Tp[T_V] = -Tm[T_V]; }
      } else if (bc == BC_PRESSURE) {
        // exterior state: own phase field and partial densities, at rest, at p_bc;
        // rho E from the stiffened-gas relation, then the closure of that state
        const double phi = Tm[T_PHI], phi2 = __dsub_rn(1.0, phi);
        const double den0 = __dadd_rn(__dmul_rn(phi, prm.g1), __dmul_rn(phi2, prm.g2));
        const double Cm0 = __dadd_rn(__dmul_rn(phi, prm.C1), __dmul_rn(phi2, prm.C2));
        const double rho = Tm[T_M1] + Tm[T_M2];
        Tp[T_RU] = Tp[T_RV] = Tp[T_U] = Tp[T_V] = 0.0;
        Tp[T_RE] = __dadd_rn(__dmul_rn(prm.p_bc[f], den0), Cm0);
        double Cm, den;
        const double Pg = sg_pressure(prm, phi, rho, 0.0, 0.0, Tp[T_RE], &Cm, &den);
        Tp[T_P] = Pg;
        Tp[T_C] = sqrt((Pg + (Pg + Cm) / den) / rho);
        Tp[T_B] = fma(Pg, prm.Bp, prm.dC);
      } else {              // no-slip: reverse the velocity
        Tp[T_RU] = -Tm[T_RU]; Tp[T_U] = -Tm[T_U];
        Tp[T_RV] = -Tm[T_RV]; Tp[T_V] = -Tm[T_V];
      }
    }
    const double unm = flip64(xf ? Tm[T_U] : Tm[T_V], sm);
    const double unp = flip64(xf ? Tp[T_U] : Tp[T_V], sm);
    const double lam = max_nonneg64(fabs(unm) + Tm[T_C], fabs(unp) + Tp[T_C]);
    const double *ft = s_ft + (xf ? 0 : NFT * P1) + kk;
    const double hw = ft[FT_HALF * P1];

    // Lax-Friedrichs flux {F}.m - lambda [[w]], [[w]] = (w+ - w-)/2, times -wf.
    double S[NV];
    {
      const double pmx = xf ? flip64(Tm[T_P], sm) : 0.0, pmy = xf ? 0.0 : flip64(Tm[T_P], sm);
      const double ppx = xf ? flip64(Tp[T_P], sm) : 0.0, ppy = xf ? 0.0 : flip64(Tp[T_P], sm);
      const double Fs[5] = {fma(Tp[T_M1], unp, Tm[T_M1] * unm), fma(Tp[T_M2], unp, Tm[T_M2] * unm),
                            fma(Tp[T_RU], unp, ppx) + fma(Tm[T_RU], unm, pmx),
                            fma(Tp[T_RV], unp, ppy) + fma(Tm[T_RV], unm, pmy),
                            fma(Tp[T_RE] + Tp[T_P], unp, (Tm[T_RE] + Tm[T_P]) * unm)};
#pragma unroll
      for (int c = 0; c < 5; ++c) {
        const int vv = M1 + c;
        S[vv] = -hw * __dsub_rn(Fs[c], __dmul_rn(lam, Tp[vv] - Tm[vv]));
      }
    }
    // Quasi-conservative transport: (lambda - m.u-) [[phi]], same for psi.
    const double jump = Tp[T_PHI] - Tm[T_PHI];
    const double hl = hw * (lam - unm);
    S[PHI] = hl * jump;
    S[PSI] = hl * (Tp[T_PSI] - Tm[T_PSI]);

    double lift[6] = {0, 0, 0, 0, 0, 0};
    if (!wall) {
      // SIP flux of a_1: Gamma [eps ({grad phi}.m + eta (phi+ - phi-)) - {phi(1-phi) n}.m]
      const double gn = flip64(Tp[T_GPHI] + Tm[T_GPHI], sm);
      const double sharp = flip64(fma(Tp[T_PHI] * (1.0 - Tp[T_PHI]), Tp[T_N], Tm[T_PHI] * (1.0 - Tm[T_PHI]) * Tm[T_N]), sm);
      const double ahat =
          0.5 * prm.Gamma * fma(prm.eps, fma(xf ? prm.eta2_x : prm.eta2_y, jump, gn), -sharp);
      // face coefficients of the a_1-derived terms
      const double km2 = fma(Tm[T_V], Tm[T_V], Tm[T_U] * Tm[T_U]), kp2 = fma(Tp[T_V], Tp[T_V], Tp[T_U] * Tp[T_U]);
      const double cu = prm.hdr * (Tp[T_U] + Tm[T_U]), cv = prm.hdr * (Tp[T_V] + Tm[T_V]);
      const double cE = fma(0.5, Tp[T_B] + Tm[T_B], __dmul_rn(0.5 * prm.hdr, kp2 + km2));
      const double sym = ft[FT_SYM * P1] * jump;
      const double wf = ft[FT_W * P1];
      S[PHI] = fma(wf, ahat, S[PHI]);
      S[M1] = fma(ft[FT_W1 * P1], ahat, S[M1]);
      S[M2] = fma(ft[FT_W2 * P1], ahat, S[M2]);
      S[RU] = fma(wf * cu, ahat, S[RU]);
      S[RV] = fma(wf * cv, ahat, S[RV]);
      S[RE] = fma(wf * cE, ahat, S[RE]);
      lift[0] = sym;
      lift[1] = prm.rho01 * sym;
      lift[2] = -prm.rho02 * sym;
      lift[3] = cu * sym;
      lift[4] = cv * sym;
      lift[5] = cE * sym;
    }
#pragma unroll
    for (int vv = 0; vv < NV; ++vv) s_s[vv * fs + g] = S[vv];
#pragma unroll
    for (int c = 0; c < 6; ++c) s_s[(NV + c) * fs + g] = lift[c];
  }
  __syncthreads();

  // Phase 2: gather onto the element's nodes, lift the symmetric term along
  // the normal lines, apply M^-1, add the volume part, write L or the stage.
  if (!act) return;
  // what the update reads is requested here, before the shared-memory gather, in one run
  double rv[NV], wn[NV], w0n[NV];
#pragma unroll
  for (int vv = 0; vv < NV; ++vv) rv[vv] = __ldca(rvol + (long)vv * N + n);
  if (mode != MODE_RHS) {
#pragma unroll
    for (int vv = 0; vv < NV; ++vv) wn[vv] = __ldca(ws + (long)vv * N + n);
    if (mode != MODE_S1) {
#pragma unroll
      for (int vv = 0; vv < NV; ++vv) w0n[vv] = __ldca(w0 + (long)vv * N + n);
    }
  }
  const int i = a % P1, j = DIM == 2 ? a / P1 : 0;
  const int kx = DIM == 2 ? j : 0;
  const int gb = le * NFK;
  double acc[NV];
  {
    // a line has two different end nodes, so a node lies on at most one face per axis
    const bool onx = i == 0 || i == P, ony = DIM == 2 && (j == 0 || j == P);
    const int gx = gb + (i == P ? NK : 0) + kx, gy = gb + (j == P ? 3 : 2) * NK + i;
#pragma unroll
    for (int vv = 0; vv < NV; ++vv) acc[vv] = onx ? s_s[vv * fs + gx] : 0.0;
    if (ony) {
#pragma unroll
      for (int vv = 0; vv < NV; ++vv) acc[vv] += s_s[vv * fs + gy];
    }
  }
  {
    const int slot[6] = {PHI, M1, M2, RU, RV, RE};
    const double lw = -Dx[0 * P1 + i], le_ = Dx[P * P1 + i];
#pragma unroll
    for (int c = 0; c < 6; ++c)
      if (DIM == 2 || c != 4)
        acc[slot[c]] += fma(s_s[(NV + c) * fs + gb + NK + kx], le_, s_s[(NV + c) * fs + gb + kx] * lw);
    if (DIM == 2) {
      const double ls = -Dy[0 * P1 + j], ln = Dy[P * P1 + j];
#pragma unroll
      for (int c = 0; c < 6; ++c)
        acc[slot[c]] += fma(s_s[(NV + c) * fs + gb + 3 * NK + i], ln, s_s[(NV + c) * fs + gb + 2 * NK + i] * ls);
    }
  }
  const double im = invM[a];
  bool bad = false;
#pragma unroll
  for (int vv = 0; vv < NV; ++vv) {
    const long o = (long)vv * N + n;
    double r = fma(acc[vv], im, rv[vv]);
    if (mode != MODE_RHS) {
      r = fma(dt, r, wn[vv]);
      if (mode == MODE_S2) r = fma(0.25, r, 0.75 * w0n[vv]);
      else if (mode == MODE_S3) r = fma(2.0 / 3.0, r, (1.0 / 3.0) * w0n[vv]);
    }
    bad |= !finite64(r);
    out[o] = r;
  }
  if (prm.check_finite && bad) atomicOr(prm.status, STATUS_NONFINITE);
}

template <int P, int DIM>
cudaError_t launch_volume(const Params &prm, const double *w, double *rvol, double *trace, cudaStream_t s) {
  using G = Geom<P, DIM, false, false>;
  const int epb = pick_epb64(prm.E, G::NP, 1), threads = (epb * G::NP + 31) / 32 * 32;
  const size_t smem = sizeof(double) * (4 * G::P1 * G::P1 + (size_t)G::NSTAGE * epb * G::NP);
  return launch_dependent(k_volume<P, DIM>, (prm.E + epb - 1) / epb, threads, smem, s, prm, epb, w, rvol, trace);
}

template <int P, int DIM>
cudaError_t launch_surface(const Params &prm, int mode, double dt, const double *w0, const double *ws,
                           const double *rvol, const double *trace, double *out, cudaStream_t s) {
  using G = Geom<P, DIM, false, false>;
  // a face node costs about as much as a node here
  const int epb = pick_epb64(prm.E, G::NP, 1, G::NFK, 1), threads = (epb * G::NP + 31) / 32 * 32;
  const size_t smem =
      sizeof(double) * (2 * G::P1 * G::P1 + G::NP + 2 * NFT * G::P1 + (size_t)(NV + 6) * epb * G::NFK);
  return launch_dependent(k_surface<P, DIM>, (prm.E + epb - 1) / epb, threads, smem, s, prm, epb, mode, dt, w0, ws,
                          rvol, trace, out);
}

template <int P, int DIM>
KernelSet make_set() {
  return KernelSet{&launch_volume<P, DIM>, &launch_surface<P, DIM>, NT_INVISCID};
}

}  // namespace dgpf
