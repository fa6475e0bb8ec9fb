// dg_kin.cuh -- kinematic mode (Sec. 4.1): the phase field and the level set
// advected by a prescribed analytical velocity, FP64 (GB300, sm_103a).
//
//   d(phi)/dt + u . grad(phi) = div a_1,   a_1 = Gamma (eps grad phi - phi (1 - phi) n),
//   d(psi)/dt + u . grad(psi) = 0,         n = grad psi / |grad psi|,
//
// with the discretisation of the phi and psi rows of the full scheme: the
// weak-form volume term of -a_1 (sum-factorised Dhat contractions), the
// non-conservative transport -u . grad f at the nodes, the transport flux
// (lambda - m.u-) [[f]] with lambda = max(|u-.m|, |u+.m|) -- the advection
// speed alone, as the kinematic system has no sound speed -- and the SIP flux
// of a_1 with its lifted symmetric term.  The nodal velocity is a uniform field
// as given, or, for the Rider-Kothe vortex, the discrete curl of its stream
// function interpolated at each element's nodes (discretely divergence-free,
// normal components continuous across faces: the phase field's mass is then
// conserved to round-off).  Time integration is the classical four-stage
// Runge-Kutta method: a volume launch on the state (k_kin_volume), then one
// launch per stage (k_kin_stage: face fluxes from the traces, M^-1, the stage
// update and the volume part of the next stage on the result, which the
// thread of each node holds).  Periodic meshes only.
#pragma once

#include <math_constants.h>

#include "dg_common.cuh"
#include "dg_kernels_fp64.cuh"

namespace dgpf {

enum { VEL_UNIFORM = 0, VEL_RIDER_KOTHE = 1 };
// What a kinematic stage kernel writes: the right-hand side, or one stage of
// classical RK4 (w0: step start, acc: k1 + 2 k2 + 2 k3 so far).
enum KinMode { KIN_RHS = 0, KIN_K1 = 1, KIN_K2 = 2, KIN_K3 = 3, KIN_K4 = 4 };

// Constants of one triangle type of the split-rectangle mesh (dg_tri.cuh): det = d(x,y)/d(r,s),
// its inverse, the inverse-map derivatives, and per edge f the outward unit normal m, half the
// edge length and its reciprocal, the penalty eta_tri / h_e and the reference components of
// grad l . m (gr = rx m0 + ry m1, gs = sx m0 + sy m1).
struct TriConst {
  double det, idet, rx, ry, sx, sy;
  double m0[3], m1[3], hl[3], ihl[3], eta[3], gr[3], gs[3];
};

struct KinParams {
  int nx, ny, E, N;
  double x0, y0, hx, hy;
  double Gamma, eps, eta_x, eta_y;
  double Ge, Gp_x, Gp_y;   // Gamma eps, 2 Gamma eps eta
  int vel;                 // VEL_UNIFORM or VEL_RIDER_KOTHE
  double u0, v0, T;        // uniform velocity; Rider-Kothe period
  double xc, yc;           // Rider-Kothe vortex centre
  double eta_tri;          // triangles: c_ip (p+1)(p+2); the edge penalty is eta_tri / h_e
  TriConst tc[2];          // triangles: the two element types
  const double *vel_tab;   // spatial velocity factor U at every node (rectangles) or quadrature point
                           // (triangles), see kin_velocity_factor
  const double *ops;       // operator table (OpsLayout)
  const double *xi;        // GLL nodes on [-1, 1]
  const double *kt;        // device: step sizes and time factors of the captured sequence (KinTime)
  int check_finite;
  unsigned *status;
};

// Prescribed velocity (Sec. 4.1), u(x, t) = c(t) U(x): the Rider-Kothe vortex with
// c = cos(pi t / T) and U = (sin^2(pi X) sin(2 pi Y), -sin(2 pi X) sin^2(pi Y)), or c = 1 and
// U = (u0, v0).  U does not change between stages: it is evaluated once per node (rectangles) or
// quadrature point (triangles) when the context is created, into KinParams::vel_tab, and a stage
// multiplies by c -- the FP64 sines would otherwise cost more than the scheme.
__device__ __forceinline__ void kin_velocity_factor(const KinParams &kp, double x, double y, double *U,
                                                    double *V) {
  if (kp.vel == VEL_RIDER_KOTHE) {
    const double X = x - kp.xc + 0.5, Y = y - kp.yc + 0.5;
    const double sx = sin(CUDART_PI * X), sy = sin(CUDART_PI * Y);
    *U = sx * sx * sin(2.0 * CUDART_PI * Y);
    *V = -sin(2.0 * CUDART_PI * X) * sy * sy;
  } else {
    *U = kp.u0;
    *V = kp.v0;
  }
}

// What the stage kernels of a captured sequence read from device memory, set before every launch of
// the sequence: dt/2, dt, dt/6 and the velocity's time factor c at every stage, stage st of step k
// at index KT_C + 4 k + st.  A cosine in every block would cost half of a stage kernel's FP64 work.
enum KinTime { KT_HALF = 0, KT_DT, KT_SIXTH, KT_C };
constexpr int KIN_MAX_STEPS = 8;  // steps of the longest captured sequence
constexpr int KT_SIZE = KT_C + 4 * KIN_MAX_STEPS;

__device__ __forceinline__ double kin_time_factor(const KinParams &kp, double t) {
  return kp.vel == VEL_RIDER_KOTHE ? cos(CUDART_PI * t / kp.T) : 1.0;
}

// Spatial factor of the Rider-Kothe stream function, u = d(Psi)/dy and v = -d(Psi)/dx:
// Psi = sin^2(pi X) sin^2(pi Y) / pi.
__device__ __forceinline__ double kin_stream_factor(const KinParams &kp, double x, double y) {
  const double sx = sin(CUDART_PI * (x - kp.xc + 0.5)), sy = sin(CUDART_PI * (y - kp.yc + 0.5));
  return sx * sx * sy * sy / CUDART_PI;
}

// U at every node of the rectangles, [N][2]: a uniform field as given; the vortex as the
// discrete curl of its stream function at the element's nodes, U = sum_c Dy[j][c] Psi(i, c),
// V = -sum_c Dx[i][c] Psi(c, j) (Dx, Dy: the (2/h) D rows of the operator table).
template <int P>
__global__ void k_kin_velocity_table(const KinParams kp, double *__restrict__ tab) {
  constexpr int P1 = P + 1, NP = P1 * P1;
  const long n = (long)blockIdx.x * blockDim.x + threadIdx.x;
  if (n >= kp.N) return;
  const int e = (int)(n / NP), a = (int)(n % NP), i = a % P1, j = a / P1;
  const int ex = e % kp.nx, ey = e / kp.nx;
  const double x = kp.x0 + kp.hx * (ex + 0.5 * (__ldg(kp.xi + i) + 1.0));
  const double y = kp.y0 + kp.hy * (ey + 0.5 * (__ldg(kp.xi + j) + 1.0));
  if (kp.vel != VEL_RIDER_KOTHE) {
    kin_velocity_factor(kp, x, y, &tab[2 * n], &tab[2 * n + 1]);
    return;
  }
  const OpsLayout L{P1, NP};
  double U = 0.0, V = 0.0;
  for (int c = 0; c < P1; ++c) {
    const double xc = kp.x0 + kp.hx * (ex + 0.5 * (__ldg(kp.xi + c) + 1.0));
    const double yc = kp.y0 + kp.hy * (ey + 0.5 * (__ldg(kp.xi + c) + 1.0));
    U = fma(__ldg(kp.ops + L.Dy() + j * P1 + c), kin_stream_factor(kp, x, yc), U);
    V = fma(-__ldg(kp.ops + L.Dx() + i * P1 + c), kin_stream_factor(kp, xc, y), V);
  }
  tab[2 * n] = U;
  tab[2 * n + 1] = V;
}

template <int P>
cudaError_t launch_kin_velocity_table(const KinParams &kp, double *tab, cudaStream_t s) {
  k_kin_velocity_table<P><<<(unsigned)((kp.N + 255) / 256), 256, 0, s>>>(kp, tab);
  return cudaGetLastError();
}

// Periodic neighbour across face f (0 W, 1 E, 2 S, 3 N).
__device__ __forceinline__ int kin_neighbour(const KinParams &kp, int e, int f) {
  const int ex = e % kp.nx, ey = e / kp.nx;
  switch (f) {
    case 0: return ex > 0 ? e - 1 : e + kp.nx - 1;
    case 1: return ex < kp.nx - 1 ? e + 1 : e - kp.nx + 1;
    case 2: return ey > 0 ? e - kp.nx : e + kp.nx * (kp.ny - 1);
    default: return ey < kp.ny - 1 ? e + kp.nx : e - kp.nx * (kp.ny - 1);
  }
}

// Node index of face node kk of face f (0 W, 1 E, 2 S, 3 N) in the x-fastest GLL order.
template <int P>
__device__ __forceinline__ int kin_face_node(int f, int kk) {
  constexpr int P1 = P + 1;
  return f == 0 ? kk * P1 : (f == 1 ? P + kk * P1 : (f == 2 ? kk : kk + P * P1));
}

// Face-trace fields, one plane per field: phi, psi and a_1 along the face's axis.
constexpr int KIN_NT = 3;

// Volume part of one stage at the thread's node (phi, psi), at velocity c U: broken gradients, n,
// a_1, the volume term of -a_1 (D^ contractions) and the non-conservative transport; writes the
// volume part and the face traces.  Every thread of the block calls it (it synchronises the block).
// s_op: Dx, Dy, Dhx, Dhy; s_f: two fields of fs values.
template <int P>
__device__ __forceinline__ void kin_volume_part(const KinParams &kp, const double *s_op, double *s_f, int fs, int le,
                                                int a, int e, bool lane, bool act, double phi, double psi, double2 U,
                                                double c, double *__restrict__ rvol, double *__restrict__ tr) {
  using G = Geom<P, 2, false, false>;
  constexpr int P1 = G::P1, NP = G::NP, NFK = G::NFK, NK = G::NK, P11 = P1 * P1;
  const double *Dx = s_op, *Dy = s_op + P11, *Dhx = s_op + 2 * P11, *Dhy = s_op + 3 * P11;
  const int i = a % P1, j = a / P1, sn = le * NP + a, sx = le * NP + P1 * j, sy = le * NP + i;
  const long n = (long)e * NP + a;
  __syncthreads();
  if (lane) {
    s_f[sn] = phi;
    s_f[fs + sn] = psi;
  }
  __syncthreads();
  double gpx = 0.0, gpy = 0.0, gsx = 0.0, gsy = 0.0;
#pragma unroll
  for (int k = 0; k < P1; ++k) {
    const double dx = Dx[i * P1 + k], dy = Dy[j * P1 + k];
    gpx = k ? fma(dx, s_f[sx + k], gpx) : dx * s_f[sx];
    gsx = k ? fma(dx, s_f[fs + sx + k], gsx) : dx * s_f[fs + sx];
    gpy = k ? fma(dy, s_f[sy + P1 * k], gpy) : dy * s_f[sy];
    gsy = k ? fma(dy, s_f[fs + sy + P1 * k], gsy) : dy * s_f[fs + sy];
  }
  // a_1 = Gamma (eps grad phi - phi (1 - phi) grad psi / |grad psi|), n = 0 unless |grad psi| >= 1e-12 (so a
  // NaN there does not reach phi)
  const double g2 = fma(gsy, gsy, gsx * gsx);
  double a1x, a1y;
  if (has_gradient(g2)) {
    const double Gn = kp.Gamma * fma(-phi, phi, phi) * rsqrt64(g2);
    a1x = fma(kp.Ge, gpx, -(Gn * gsx));
    a1y = fma(kp.Ge, gpy, -(Gn * gsy));
  } else {
    a1x = kp.Ge * gpx;
    a1y = kp.Ge * gpy;
  }
  __syncthreads();
  if (lane) {
    s_f[sn] = a1x;
    s_f[fs + sn] = a1y;
  }
  __syncthreads();
  double R = 0.0;
#pragma unroll
  for (int k = 0; k < P1; ++k) {
    const double ax = s_f[sx + k];
    R = k ? fma(Dhx[i * P1 + k], ax, R) : Dhx[i * P1] * ax;
    R = fma(Dhy[j * P1 + k], s_f[fs + sy + P1 * k], R);
  }
  if (!act) return;
  rvol[n] = -fma(c, fma(U.y, gpy, U.x * gpx), R);
  rvol[kp.N + n] = -(c * fma(U.y, gsy, U.x * gsx));
  const long stride = (long)kp.E * NFK;
  auto put = [&](int f, int kk, double an) {
    const long o = (long)e * NFK + f * NK + kk;
    if (!in_bounds(kp.status, o, stride)) return;
    tr[o] = phi;
    tr[stride + o] = psi;
    tr[2 * stride + o] = an;
  };
  if (i == 0) put(0, j, a1x);
  if (i == P) put(1, j, a1x);
  if (j == 0) put(2, i, a1y);
  if (j == P) put(3, i, a1y);
}

// The volume part of a sequence's first stage, on the state w (time factor kt[ic]).
template <int P>
__global__ void __launch_bounds__(MAX_THREADS64)
k_kin_volume(const KinParams kp, int epb, int ic, const double *__restrict__ w, double *__restrict__ rvol,
             double *__restrict__ tr) {
  using G = Geom<P, 2, false, false>;
  constexpr int P11 = G::P1 * G::P1, NP = G::NP;
  extern __shared__ double s_mem[];
  grid_dependency_wait();
  for (int t = threadIdx.x; t < 4 * P11; t += blockDim.x) s_mem[t] = kp.ops[t];
  const int le_raw = threadIdx.x / NP, a = threadIdx.x % NP;
  const bool lane = le_raw < epb;
  const int le = lane ? le_raw : epb - 1, e0 = blockIdx.x * epb + le;
  const bool act = lane && e0 < kp.E && in_bounds(kp.status, (long long)e0 * NP + a, kp.N);
  const int e = act ? e0 : 0;
  const long n = (long)e * NP + a;
  const double2 U = __ldg(reinterpret_cast<const double2 *>(kp.vel_tab) + n);
  kin_volume_part<P>(kp, s_mem, s_mem + 4 * P11, epb * NP, le, a, e, lane, act, act ? __ldca(w + n) : 0.0,
                     act ? __ldca(w + kp.N + n) : 0.0, U, __ldca(kp.kt + KT_C + ic), rvol, tr);
}

// One stage of the kinematic mode: at every face node the transport flux (lambda - m.u-) [[f]] and
// the SIP flux of a_1 with its lifted symmetric term, from the traces of both sides; M^-1 (in the
// tables cf and lw), the volume part and the right-hand side or an RK4 stage:
//   K1: acc = L,        r = w0 + dt/2 L
//   K2: acc += 2 L,     r = w0 + dt/2 L
//   K3: acc += 2 L,     r = w0 + dt L
//   K4: r = w0 + dt/6 (acc + L), written to w0 (each node by the thread that read it);
// then, unless last, the volume part of the next stage on r (time factor kt[KT_C + ic + 1]; stage
// index ic of the captured sequence), into rvol (the node's own value was read before) and the
// other trace buffer, which neighbouring blocks of this launch do not read.  r itself is written (out)
// by K4, and by every stage that is the last before a volume launch.
// Bound by the FP64 pipe: about 65 operations per node at p = 3, where a stage that evaluated the
// neighbours' gradients and normals at every face node itself took about 150 (64 x 64, p = 3: an RK4
// step 85 -> 44 us).
template <int P>
__global__ void __launch_bounds__(MAX_THREADS64)
k_kin_stage(const KinParams kp, int epb, int mode, int ic, bool last, double *w0, double *__restrict__ acc,
            double *rvol, const double *__restrict__ tr, double *__restrict__ tr_out, double *out) {
  using G = Geom<P, 2, false, false>;
  constexpr int P1 = G::P1, NP = G::NP, NFK = G::NFK, NK = G::NK, P11 = P1 * P1;
  const OpsLayout L{P1, NP};
  extern __shared__ double s_mem[];
  double *s_op = s_mem, *s_cf = s_op + 4 * P11, *s_lw = s_cf + 2;
  double *s_f = s_lw + 4 * P1;           // [2][epb * NP]
  double *s_s = s_f + 2 * epb * NP;      // [3][epb * NFK]: twice the flux of phi and psi, Gamma eps [[phi]]
  const int fs = epb * NFK, N = kp.N;
  grid_dependency_wait();
  for (int t = threadIdx.x; t < 4 * P11; t += blockDim.x) s_op[t] = kp.ops[t];
  for (int t = threadIdx.x; t < 2 + 4 * P1; t += blockDim.x) s_cf[t] = kp.ops[L.cf() + t];
  const double c = __ldca(kp.kt + KT_C + ic);
  const double2 *vt = reinterpret_cast<const double2 *>(kp.vel_tab);
  const long stride = (long)kp.E * NFK;

  const int le_raw = threadIdx.x / NP, a = threadIdx.x % NP;
  const bool lane = le_raw < epb;
  const int le = lane ? le_raw : epb - 1, e0 = blockIdx.x * epb + le;
  const bool act = lane && e0 < kp.E && in_bounds(kp.status, (long long)e0 * NP + a, N);
  // (idle lanes take their own block's first element: another block's nodes may be being written)
  const int e = act ? e0 : blockIdx.x * epb;
  const long n = (long)e * NP + a;
  double r[2], base[2] = {0.0, 0.0};
#pragma unroll
  for (int v = 0; v < 2; ++v) {
    r[v] = __ldca(rvol + (long)v * N + n);
    if (mode != KIN_RHS) base[v] = __ldca(w0 + (long)v * N + n);
  }

  for (int g = threadIdx.x; g < fs; g += blockDim.x) {
    const int fe = blockIdx.x * epb + g / NFK, t = g % NFK;
    if (fe >= kp.E) break;
    const int f = t / NK, kk = t % NK, e2 = kin_neighbour(kp, fe, f);
    const bool xf = f < 2;
    const int sm = (f & 1) ? 0 : (int)0x80000000;  // sign of m
    const long om = (long)fe * NFK + t, op = (long)e2 * NFK + (f ^ 1) * NK + kk;
    const long nm = (long)fe * NP + kin_face_node<P>(f, kk), np = (long)e2 * NP + kin_face_node<P>(f ^ 1, kk);
    double flux = 0.0, fpsi = 0.0, gej = 0.0;
    if (in_bounds(kp.status, om, stride) && in_bounds(kp.status, op, stride) && in_bounds(kp.status, nm, N) &&
        in_bounds(kp.status, np, N)) {
      const double jphi = __ldca(tr + op) - __ldca(tr + om);
      const double jpsi = __ldca(tr + stride + op) - __ldca(tr + stride + om);
      const double asum = __ldca(tr + 2 * stride + op) + __ldca(tr + 2 * stride + om);
      const double2 Um = __ldg(vt + nm), Up = __ldg(vt + np);
      const double um = flip64(xf ? Um.x : Um.y, sm), up = xf ? Up.x : Up.y;
      // lambda - m.u- with lambda = |c| max(|U- . m|, |U+ . m|)
      const double lu = fma(-c, um, fabs(c) * max_nonneg64(fabs(um), fabs(up)));
      gej = kp.Ge * jphi;
      flux = fma(lu, jphi, fma(xf ? kp.Gp_x : kp.Gp_y, jphi, flip64(asum, sm)));
      fpsi = lu * jpsi;
    }
    s_s[g] = flux;
    s_s[fs + g] = fpsi;
    s_s[2 * fs + g] = gej;
  }
  __syncthreads();
  const int i = a % P1, j = a / P1, gb = le * NFK;
  if (i == 0 || i == P) {
    const int g = gb + (i == 0 ? 0 : NK) + j;
    r[0] = fma(s_cf[0], s_s[g], r[0]);
    r[1] = fma(s_cf[0], s_s[fs + g], r[1]);
  }
  if (j == 0 || j == P) {
    const int g = gb + (j == 0 ? 2 : 3) * NK + i;
    r[0] = fma(s_cf[1], s_s[g], r[0]);
    r[1] = fma(s_cf[1], s_s[fs + g], r[1]);
  }
  {
    const double *lift = s_s + 2 * fs + gb;
    r[0] = fma(s_lw[i], lift[j], r[0]);
    r[0] = fma(s_lw[P1 + i], lift[NK + j], r[0]);
    r[0] = fma(s_lw[2 * P1 + j], lift[2 * NK + i], r[0]);
    r[0] = fma(s_lw[3 * P1 + j], lift[3 * NK + i], r[0]);
  }
  if (mode != KIN_RHS) {
    const double h = __ldca(kp.kt + (mode == KIN_K4 ? KT_SIXTH : (mode == KIN_K3 ? KT_DT : KT_HALF)));
#pragma unroll
    for (int v = 0; v < 2; ++v) {
      const long o = (long)v * N + n;
      double Lv = r[v];
      if (act) {
        if (mode == KIN_K1) {
          acc[o] = Lv;
        } else {
          const double q = acc[o];
          if (mode == KIN_K4) Lv += q;
          else acc[o] = fma(2.0, Lv, q);
        }
      }
      r[v] = fma(h, Lv, base[v]);
    }
  }
  if (act) {
    if (kp.check_finite && !(finite64(r[0]) && finite64(r[1]))) atomicOr(kp.status, STATUS_NONFINITE);
    if (mode == KIN_RHS || mode == KIN_K4 || last) {
      out[n] = r[0];
      out[N + n] = r[1];
    }
  }
  if (last) return;
  kin_volume_part<P>(kp, s_op, s_f, epb * NP, le, a, e, lane, act, act ? r[0] : 0.0, act ? r[1] : 0.0, __ldg(vt + n),
                     __ldca(kp.kt + KT_C + ic + 1), rvol, tr_out);
}

struct KinKernels {
  cudaError_t (*volume)(const KinParams &, int ic, const double *w, double *rvol, double *tr, cudaStream_t);
  cudaError_t (*stage)(const KinParams &, int mode, int ic, bool last, double *w0, double *acc, double *rvol,
                       const double *tr, double *tr_out, double *out, cudaStream_t);
  cudaError_t (*velocity_table)(const KinParams &, double *tab, cudaStream_t);
};

template <int P>
cudaError_t launch_kin_volume(const KinParams &kp, int ic, const double *w, double *rvol, double *tr, cudaStream_t s) {
  using G = Geom<P, 2, false, false>;
  const int epb = pick_epb64(kp.E, G::NP, 1), threads = (epb * G::NP + 31) / 32 * 32;
  const size_t smem = sizeof(double) * (4 * G::P1 * G::P1 + 2 * (size_t)epb * G::NP);
  return launch_dependent(k_kin_volume<P>, (kp.E + epb - 1) / epb, threads, smem, s, kp, epb, ic, w, rvol, tr);
}

template <int P>
cudaError_t launch_kin_stage(const KinParams &kp, int mode, int ic, bool last, double *w0, double *acc, double *rvol,
                             const double *tr, double *tr_out, double *out, cudaStream_t s) {
  using G = Geom<P, 2, false, false>;
  // (a node costs about five times a face node)
  const int epb = pick_epb64(kp.E, G::NP, 5, G::NFK, 1), threads = (epb * G::NP + 31) / 32 * 32;
  const size_t smem =
      sizeof(double) * (4 * G::P1 * G::P1 + 2 + 4 * G::P1 + (size_t)epb * (2 * G::NP + 3 * G::NFK));
  return launch_dependent(k_kin_stage<P>, (kp.E + epb - 1) / epb, threads, smem, s, kp, epb, mode, ic, last, w0, acc,
                          rvol, tr, tr_out, out);
}

bool kin_kernels(int p, KinKernels *out);

}  // namespace dgpf
