// dg_reinit.cuh -- level-set re-initialisation (end of Sec. 3), FP64.
//
// In pseudo-time tau, from psi0 = phi - 1/2:
//   d(psi)/d(tau) = S (1 - |grad psi|) + div(nu grad psi),   S = tanh(psi0 / (2 eps |grad psi0|)),
// the hyperbolic term a nodal source on the broken gradient, the diffusion
// with the SIP flux nu ({grad psi}.m + eta (psi+ - psi-)) and its lifted
// symmetric term (no flux through walls), three-stage SSP Runge-Kutta.  The
// sign of the hyperbolic term is the one under which |grad psi| relaxes to 1
// (printed with the opposite sign, it grows at the interface).  Only psi
// changes; phi and every other field of the state are left as they are.
#pragma once

#include "dg_common.cuh"
#include "dg_kernels_fp64.cuh"

namespace dgpf {

struct ReinitParams {
  int nx, ny, E, N;
  int bc[4];
  double eps, nu;
  double eta2_x, eta2_y;  // 2 eta
  const double *ops;  // operator table (OpsLayout)
  unsigned *status;   // the context's status word (the bounds-checked build latches STATUS_BOUNDS)
};

__device__ __forceinline__ int ri_neighbour(const ReinitParams &rp, int e, int f) {
  const int ex = e % rp.nx, ey = e / rp.nx;
  switch (f) {
    case 0: return ex > 0 ? e - 1 : (rp.bc[0] == BC_PERIODIC ? e + rp.nx - 1 : -1);
    case 1: return ex < rp.nx - 1 ? e + 1 : (rp.bc[1] == BC_PERIODIC ? e - rp.nx + 1 : -1);
    case 2: return ey > 0 ? e - rp.nx : (rp.bc[2] == BC_PERIODIC ? e + rp.nx * (rp.ny - 1) : -1);
    default: return ey < rp.ny - 1 ? e + rp.nx : (rp.bc[3] == BC_PERIODIC ? e - rp.nx * (rp.ny - 1) : -1);
  }
}

// Broken gradient of the shared-memory field f of element slot le at node (i, j).
template <int P1, int DIM, int EPB, int NP>
__device__ __forceinline__ void ri_grad(const double *Dx, const double *Dy, const double (*f)[NP], int le, int i,
                                        int j, double *gx, double *gy) {
  double sx = 0.0, sy = 0.0;
#pragma unroll
  for (int c = 0; c < P1; ++c) {
    sx = fma(Dx[i * P1 + c], f[le][c + P1 * j], sx);
    if (DIM == 2) sy = fma(Dy[j * P1 + c], f[le][i + P1 * c], sy);
  }
  *gx = sx;
  *gy = sy;
}

// Smeared sign S from psi0 = phi - 1/2 (S = sign(psi0) where |grad psi0| < 1e-12),
// and psi <- psi0.  w: the state, phi at w[0..N), psi at w[N..2N).
template <int P, int DIM>
__global__ void __launch_bounds__(Geom<P, DIM, false, false>::THREADS)
k_ri_sign(const ReinitParams rp, double *w, double *S) {
  using G = Geom<P, DIM, false, false>;
  constexpr int P1 = G::P1, NP = G::NP, EPB = G::EPB, P11 = P1 * P1;
  __shared__ double s_op[2 * P11];
  __shared__ double s_f[EPB][NP];
  for (int t = threadIdx.x; t < 2 * P11; t += blockDim.x) s_op[t] = rp.ops[t];
  const int le_raw = threadIdx.x / NP;
  const bool lane = le_raw < EPB;
  const int le = lane ? le_raw : EPB - 1;
  const int a = threadIdx.x % NP;
  const int e = blockIdx.x * EPB + le;
  const bool act = lane && e < rp.E && in_bounds(rp.status, (long long)e * NP + a, rp.N);
  const int i = a % P1, j = DIM == 2 ? a / P1 : 0;
  const long n = (long)(act ? e : 0) * NP + a;
  const double p0 = act ? w[n] - 0.5 : 0.0;
  if (lane) s_f[le][a] = p0;
  __syncthreads();
  double gx, gy;
  ri_grad<P1, DIM, EPB, NP>(s_op, s_op + P11, s_f, le, i, j, &gx, &gy);
  const double gm = sqrt(gx * gx + gy * gy);
  const double sg = (gm < 1e-12 || !(rp.eps > 0.0)) ? (p0 > 0.0 ? 1.0 : (p0 < 0.0 ? -1.0 : 0.0))
                                                    : tanh(p0 / (2.0 * rp.eps * gm));
  if (act) {
    S[n] = sg;
    w[rp.N + n] = p0;
  }
}

// Volume part of one stage at the thread's node: S (1 - |grad psi|) + M^-1 int grad l . (-nu grad
// psi) into rvol, and the traces (psi, d psi / d axis).  Every thread of the block calls it (it
// synchronises the block).  s_op: Dx, Dy, Dhx, Dhy; s_f: two fields of fs values.
template <int P, int DIM>
__device__ __forceinline__ void ri_volume_part(const ReinitParams &rp, const double *s_op, double *s_f, int fs, int le,
                                               int a, int e, bool lane, bool act, double ps,
                                               const double *__restrict__ S, double *__restrict__ rvol,
                                               double *__restrict__ tr) {
  using G = Geom<P, DIM, false, false>;
  constexpr int P1 = G::P1, NP = G::NP, NFK = G::NFK, NK = G::NK, P11 = P1 * P1;
  const double *Dx = s_op, *Dy = s_op + P11, *Dhx = s_op + 2 * P11, *Dhy = s_op + 3 * P11;
  const int i = a % P1, j = DIM == 2 ? a / P1 : 0, sn = le * NP + a, sx = le * NP + P1 * j, sy = le * NP + i;
  const long n = (long)e * NP + a;
  __syncthreads();
  if (lane) s_f[sn] = ps;
  __syncthreads();
  double gx = 0.0, gy = 0.0;
#pragma unroll
  for (int c = 0; c < P1; ++c) {
    gx = c ? fma(Dx[i * P1 + c], s_f[sx + c], gx) : Dx[i * P1] * s_f[sx];
    if (DIM == 2) gy = c ? fma(Dy[j * P1 + c], s_f[sy + P1 * c], gy) : Dy[j * P1] * s_f[sy];
  }
  __syncthreads();
  if (lane) {
    s_f[sn] = gx;
    if (DIM == 2) s_f[fs + sn] = gy;
  }
  __syncthreads();
  double R = 0.0;
#pragma unroll
  for (int c = 0; c < P1; ++c) {
    R = c ? fma(Dhx[i * P1 + c], s_f[sx + c], R) : Dhx[i * P1] * s_f[sx];
    if (DIM == 2) R = fma(Dhy[j * P1 + c], s_f[fs + sy + P1 * c], R);
  }
  if (!act) return;
  const double gm = sqrt64(DIM == 2 ? fma(gy, gy, gx * gx) : gx * gx);
  rvol[n] = fma(-rp.nu, R, __ldca(S + n) * (1.0 - gm));
  const long stride = (long)rp.E * NFK;
  auto put = [&](int f, int kk, double gn) {
    const long o = (long)e * NFK + f * NK + kk;
    if (!in_bounds(rp.status, o, stride)) return;
    tr[o] = ps;
    tr[stride + o] = gn;
  };
  const int kx = DIM == 2 ? j : 0;
  if (i == 0) put(0, kx, gx);
  if (i == P) put(1, kx, gx);
  if (DIM == 2 && j == 0) put(2, i, gy);
  if (DIM == 2 && j == P) put(3, i, gy);
}

// The volume part of the first stage.
template <int P, int DIM>
__global__ void __launch_bounds__(MAX_THREADS64)
k_ri_volume(const ReinitParams rp, int epb, const double *__restrict__ psi, const double *__restrict__ S,
            double *__restrict__ rvol, double *__restrict__ tr) {
  using G = Geom<P, DIM, false, false>;
  constexpr int P11 = G::P1 * G::P1, NP = G::NP;
  extern __shared__ double s_mem[];
  grid_dependency_wait();
  for (int t = threadIdx.x; t < 4 * P11; t += blockDim.x) s_mem[t] = rp.ops[t];
  const int le_raw = threadIdx.x / NP, a = threadIdx.x % NP;
  const bool lane = le_raw < epb;
  const int le = lane ? le_raw : epb - 1, e0 = blockIdx.x * epb + le;
  const bool act = lane && e0 < rp.E && in_bounds(rp.status, (long long)e0 * NP + a, rp.N);
  const int e = act ? e0 : 0;
  ri_volume_part<P, DIM>(rp, s_mem, s_mem + 4 * P11, epb * NP, le, a, e, lane, act,
                         act ? __ldca(psi + (long)e * NP + a) : 0.0, S, rvol, tr);
}

// One stage: SIP flux and lifted symmetric term from the traces of both sides, M^-1 (in the tables cf
// and lw), the volume part, one SSP-RK3 stage of psi (mode MODE_S1..S3), then, unless last, the
// volume part of the next stage on the result, which the thread of each node holds, into rvol (the
// node's own value was read before) and the other trace buffer, which neighbouring blocks of this
// launch do not read.  psi: the step start, overwritten by stage 3 (each node by the thread that
// read it); ws: the stage state, written and read back by the node's thread.  One launch per stage
// instead of two: at 64 x 64, p = 3 the two took 8 us each, half of it launch and load latency
// (50 iterations 2,420 -> 1,100 us).
template <int P, int DIM>
__global__ void __launch_bounds__(MAX_THREADS64)
k_ri_stage(const ReinitParams rp, int epb, int mode, double dtau, bool last, double *psi, double *__restrict__ ws,
           const double *__restrict__ S, double *rvol, const double *__restrict__ tr, double *__restrict__ tr_out) {
  using G = Geom<P, DIM, false, false>;
  constexpr int P1 = G::P1, NP = G::NP, NFK = G::NFK, NK = G::NK, P11 = P1 * P1;
  const OpsLayout L{P1, NP};
  extern __shared__ double s_mem[];
  double *s_op = s_mem, *s_cf = s_op + 4 * P11, *s_lw = s_cf + 2;
  double *s_f = s_lw + 4 * P1;          // [2][epb * NP]
  double *s_s = s_f + 2 * epb * NP;     // [2][epb * NFK]: twice the flux, nu [[psi]]
  const int fs = epb * NFK;
  grid_dependency_wait();
  for (int t = threadIdx.x; t < 4 * P11; t += blockDim.x) s_op[t] = rp.ops[t];
  for (int t = threadIdx.x; t < 2 + 4 * P1; t += blockDim.x) s_cf[t] = rp.ops[L.cf() + t];
  const long stride = (long)rp.E * NFK;
  const int le_raw = threadIdx.x / NP, a = threadIdx.x % NP;
  const bool lane = le_raw < epb;
  const int le = lane ? le_raw : epb - 1, e0 = blockIdx.x * epb + le;
  const bool act = lane && e0 < rp.E && in_bounds(rp.status, (long long)e0 * NP + a, rp.N);
  const int e = act ? e0 : 0;
  const long n = (long)e * NP + a;
  // (idle lanes read no node: another block may be writing it)
  double p0 = 0.0, pw = 0.0, r = 0.0;
  if (act) {
    p0 = __ldca(psi + n);
    r = __ldca(rvol + n);
    pw = mode == MODE_S1 ? p0 : __ldca(ws + n);
  }

  for (int g = threadIdx.x; g < fs; g += blockDim.x) {
    const int fe = blockIdx.x * epb + g / NFK, t = g % NFK;
    if (fe >= rp.E) break;
    const int f = t / NK, kk = t % NK, e2 = ri_neighbour(rp, fe, f);
    double flux = 0.0, lift = 0.0;
    const long om = (long)fe * NFK + t, op = (long)(e2 >= 0 ? e2 : 0) * NFK + (f ^ 1) * NK + kk;
    if (e2 >= 0 && in_bounds(rp.status, om, stride) && in_bounds(rp.status, op, stride)) {
      const double nj = rp.nu * (__ldca(tr + op) - __ldca(tr + om));
      const double gs = flip64(__ldca(tr + stride + op) + __ldca(tr + stride + om), (f & 1) ? 0 : (int)0x80000000);
      flux = fma(f < 2 ? rp.eta2_x : rp.eta2_y, nj, rp.nu * gs);
      lift = nj;
    }
    s_s[g] = flux;
    s_s[fs + g] = lift;
  }
  __syncthreads();
  const int i = a % P1, j = DIM == 2 ? a / P1 : 0, kx = DIM == 2 ? j : 0, gb = le * NFK;
  if (i == 0 || i == P) r = fma(s_cf[0], s_s[gb + (i == 0 ? 0 : NK) + kx], r);
  if (DIM == 2 && (j == 0 || j == P)) r = fma(s_cf[1], s_s[gb + (j == 0 ? 2 : 3) * NK + i], r);
  r = fma(s_lw[i], s_s[fs + gb + kx], r);
  r = fma(s_lw[P1 + i], s_s[fs + gb + NK + kx], r);
  if (DIM == 2) {
    r = fma(s_lw[2 * P1 + j], s_s[fs + gb + 2 * NK + i], r);
    r = fma(s_lw[3 * P1 + j], s_s[fs + gb + 3 * NK + i], r);
  }
  r = fma(dtau, r, pw);
  if (mode == MODE_S2) r = fma(0.75, p0, 0.25 * r);
  else if (mode == MODE_S3) r = fma(1.0 / 3.0, p0, (2.0 / 3.0) * r);
  if (act) {
    if (mode == MODE_S3) psi[n] = r;
    else ws[n] = r;
  }
  if (last) return;
  ri_volume_part<P, DIM>(rp, s_op, s_f, epb * NP, le, a, e, lane, act, act ? r : 0.0, S, rvol, tr_out);
}

template <int P, int DIM>
cudaError_t launch_ri_sign(const ReinitParams &rp, double *w, double *S, cudaStream_t s) {
  using G = Geom<P, DIM, false, false>;
  k_ri_sign<P, DIM><<<(rp.E + G::EPB - 1) / G::EPB, G::THREADS, 0, s>>>(rp, w, S);
  return cudaGetLastError();
}

template <int P, int DIM>
cudaError_t launch_ri_volume(const ReinitParams &rp, const double *psi, const double *S, double *rvol, double *tr,
                             cudaStream_t s) {
  using G = Geom<P, DIM, false, false>;
  const int epb = pick_epb64(rp.E, G::NP, 1), threads = (epb * G::NP + 31) / 32 * 32;
  const size_t smem = sizeof(double) * (4 * G::P1 * G::P1 + 2 * (size_t)epb * G::NP);
  return launch_dependent(k_ri_volume<P, DIM>, (rp.E + epb - 1) / epb, threads, smem, s, rp, epb, psi, S, rvol, tr);
}

template <int P, int DIM>
cudaError_t launch_ri_stage(const ReinitParams &rp, int mode, double dtau, bool last, double *psi, double *ws,
                            const double *S, double *rvol, const double *tr, double *tr_out, cudaStream_t s) {
  using G = Geom<P, DIM, false, false>;
  // (a node costs about seven times a face node)
  const int epb = pick_epb64(rp.E, G::NP, 7, G::NFK, 1), threads = (epb * G::NP + 31) / 32 * 32;
  const size_t smem =
      sizeof(double) * (4 * G::P1 * G::P1 + 2 + 4 * G::P1 + (size_t)epb * (2 * G::NP + 2 * G::NFK));
  return launch_dependent(k_ri_stage<P, DIM>, (rp.E + epb - 1) / epb, threads, smem, s, rp, epb, mode, dtau, last, psi,
                          ws, S, rvol, tr, tr_out);
}

struct ReinitKernels {
  cudaError_t (*sign)(const ReinitParams &, double *w, double *S, cudaStream_t);
  cudaError_t (*volume)(const ReinitParams &, const double *psi, const double *S, double *rvol, double *tr,
                        cudaStream_t);
  cudaError_t (*stage)(const ReinitParams &, int mode, double dtau, bool last, double *psi, double *ws,
                       const double *S, double *rvol, const double *tr, double *tr_out, cudaStream_t);
  int nfk;
};

bool reinit_kernels(int p, int dim, ReinitKernels *out);

}  // namespace dgpf
