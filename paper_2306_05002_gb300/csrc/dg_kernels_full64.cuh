// dg_kernels_full64.cuh -- FP64 kernels of the right-hand side with viscous stress or surface
// tension (2D), the same two launches and the same scheme as dg_kernels_fp64.cuh (GB300, sm_103a).
//
// On GB300 the FP64 pipe (two operations per clock and SM) bounds this path, so these kernels are
// written to the fewest FP64 instructions: operator tables are premultiplied (2/h, M^-1 and the
// face weights), a_1's and the energy's face coefficients are formed once per node and travel in
// the trace, the terms of the partial densities that repeat the phase field's are added as
// multiples of it, reciprocals and square roots are single third-order steps (dg_math64.cuh), and
// signs, comparisons and index work are integer.  The pressure keeps the operation order of the
// stiffened-gas formula where it cancels (~4 digits against sum phi_l gamma_l Pinf_l/(gamma_l-1)).
//
// Rising bubble on 20 x 40 elements, p = 4 (viscous, surface tension): an SSP-RK3 step 139 -> 68 us;
// 25 us of that from the elements per block (pick_epb64), 6 us from loading the update's inputs
// ahead of the face work and dependent launches.
//
// The inviscid kernels of dg_kernels_fp64.cuh keep the operation order that the discrete adjoint
// differentiates; contexts with viscous stress or surface tension have no adjoint, so their
// operations may be regrouped.
#pragma once

#include "dg_kernels_fp64.cuh"

namespace dgpf {

// Face-trace record of these kernels (one plane per field): the fields T_PHI..T_C, then
enum TraceFull {
  V_CE = T_C + 1,    // (rho01 - rho02) k + B: a_1's coefficient in the energy flux
  V_A1,              // a_1 along the axis normal to the face
  V_TX, V_TY, V_MU   // viscous: tau . e_axis and mixture mu
};
constexpr int NV_INVISCID = V_A1 + 1;
constexpr int NV_VISCOUS = V_MU + 1;

template <int P, bool VISC, bool ST>
__global__ void __launch_bounds__(MAX_THREADS64)
k_volume_full(const Params prm, int epb, const double *__restrict__ w, double *__restrict__ rvol,
         double *__restrict__ tr) {
  using G = Geom<P, 2, VISC, ST>;
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
  const int i = a % P1, j = a / P1;
  const long n = (long)(act ? e : 0) * NP + a;
  const int sn = le * NP + a;              // the node in the staged fields
  const int sx = le * NP + P1 * j;         // its x-line (stride 1) and y-line (stride P1)
  const int sy = le * NP + i;

  double q[NV];
#pragma unroll
  for (int v = 0; v < NV; ++v) q[v] = act ? __ldca(w + (long)v * N + n) : (v == M1 || v == M2 ? 1.0 : 0.0);
  const double phi = q[PHI], psi = q[PSI];
  const double rho = q[M1] + q[M2];
  const double ir = rcp64(rho);
  const double u = q[RU] * ir;
  const double v = q[RV] * ir;
  const double k = 0.5 * (fma(v, v, u * u));
  const double den = fma(phi, prm.dg, prm.g2);
  const double iden = rcp64(den);
  // the pressure, in the formula's order where it cancels (sg_pressure)
  const double Cm = mixture_constant(prm, phi);
  const double Pr = __dsub_rn(fma(-rho, k, q[RE]), Cm) * iden;
  const double X = fma(Pr + Cm, iden, Pr);  // rho c^2 = P + (P + Cm) / den
  const double cE = fma(prm.drho0, k, fma(Pr, prm.Bp, prm.dC));  // a_1's coefficient in the energy flux
  // Non-physical state: rho <= 0, a mixture 1/(gamma - 1) <= 0, or P + Pinf_mix <= 0, i.e.
  // rho c^2 <= 0 (Sec. 2 mixture rules).
  if (prm.check_finite && act && (nonpositive64(rho) || nonpositive64(den) || nonpositive64(X)))
    atomicOr(prm.status, STATUS_NONPHYSICAL);

  if (lane) {
    s_f[0 * fs + sn] = phi;
    s_f[1 * fs + sn] = psi;
    if (VISC) {
      s_f[2 * fs + sn] = u;
      s_f[3 * fs + sn] = v;
    }
  }
  __syncthreads();

  // Broken gradients: sum-factorised contractions along the two GLL lines.
  double gpx = 0.0, gpy = 0.0, gsx = 0.0, gsy = 0.0, gux = 0.0, guy = 0.0, gvx = 0.0, gvy = 0.0;
#pragma unroll
  for (int c = 0; c < P1; ++c) {
    const double dx = Dx[i * P1 + c];
    const int ax = sx + c;
    gpx = c ? fma(dx, s_f[0 * fs + ax], gpx) : dx * s_f[0 * fs + ax];
    gsx = c ? fma(dx, s_f[1 * fs + ax], gsx) : dx * s_f[1 * fs + ax];
    if (VISC) {
      gux = c ? fma(dx, s_f[2 * fs + ax], gux) : dx * s_f[2 * fs + ax];
      gvx = c ? fma(dx, s_f[3 * fs + ax], gvx) : dx * s_f[3 * fs + ax];
    }
    const double dy = Dy[j * P1 + c];
    const int ay = sy + P1 * c;
    gpy = c ? fma(dy, s_f[0 * fs + ay], gpy) : dy * s_f[0 * fs + ay];
    gsy = c ? fma(dy, s_f[1 * fs + ay], gsy) : dy * s_f[1 * fs + ay];
    if (VISC) {
      guy = c ? fma(dy, s_f[2 * fs + ay], guy) : dy * s_f[2 * fs + ay];
      gvy = c ? fma(dy, s_f[3 * fs + ay], gvy) : dy * s_f[3 * fs + ay];
    }
  }

  // The transport term keeps the broken gradients; with grad_lift the gradients of phi and psi
  // become BR1-lifted: at a face node, M^-1 w_f (f+ - f-) / 2 along the outward normal, f+ the
  // neighbour's value at the coincident node (none at walls and pressure boundaries).
  const double bpx = gpx, bpy = gpy, bsx = gsx, bsy = gsy;
  if (prm.grad_lift && act && (i == 0 || i == P || j == 0 || j == P)) {
    const OpsLayout Lo{P1, NP};
    const double im = __ldca(prm.ops + Lo.invM() + a);
    auto lift = [&](int f, int kk, double &gx_phi, double &gx_psi, double sgn) {
      const int e2 = neighbour(prm, e, f);
      if (e2 < 0) return;
      const int f2 = f ^ 1;
      const int a2 = f2 == 0 ? P1 * kk : f2 == 1 ? P + P1 * kk : f2 == 2 ? kk : kk + P1 * P;
      const long n2 = (long)e2 * NP + a2;
      if (!in_bounds(prm.status, n2, N)) return;
      const double wf = __ldca(prm.ops + (f < 2 ? Lo.wfx() : Lo.wfy()) + kk);
      const double c = sgn * 0.5 * im * wf;
      gx_phi += c * (__ldca(w + (long)PHI * N + n2) - phi);
      gx_psi += c * (__ldca(w + (long)PSI * N + n2) - psi);
    };
    const int kx = j;
    if (i == 0) lift(0, kx, gpx, gsx, -1.0);
    if (i == P) lift(1, kx, gpx, gsx, 1.0);
    if (j == 0) lift(2, i, gpy, gsy, -1.0);
    if (j == P) lift(3, i, gpy, gsy, 1.0);
  }

  // Interface normal from the level set (zero where |grad psi| < 1e-12).
  const double g2 = fma(gsy, gsy, gsx * gsx);
  double nx = 0.0, ny = 0.0;
  if (has_gradient(g2)) {
    const double r = rsqrt64(g2);
    nx = gsx * r;
    ny = gsy * r;
  }
  const double Gs = prm.Gamma * fma(-phi, phi, phi);  // Gamma phi (1 - phi)
  const double a1x = fma(prm.Ge, gpx, -(Gs * nx));
  const double a1y = fma(prm.Ge, gpy, -(Gs * ny));

  // Viscous stress tau = 2 mu (S - div(u)/3 I), mixture mu.
  double txx = 0.0, txy = 0.0, tyy = 0.0, mu = 0.0;
  if (VISC) {
    mu = prm.mu1 * phi + prm.mu2 * (1.0 - phi);
    const double div3 = (gux + gvy) * (1.0 / 3.0);
    const double mu2 = mu + mu;
    txx = mu2 * (gux - div3);
    tyy = mu2 * (gvy - div3);
    txy = mu * (guy + gvx);
  }

  // Curvature kappa = -div n from the nodal normal.
  double kappa = 0.0;
  if (ST) {
    if (lane) {
      s_f[4 * fs + sn] = nx;
      s_f[5 * fs + sn] = ny;
    }
    __syncthreads();
    double dv = 0.0;
#pragma unroll
    for (int c = 0; c < P1; ++c) {
      dv = fma(Dx[i * P1 + c], s_f[4 * fs + sx + c], dv);
      dv = fma(Dy[j * P1 + c], s_f[5 * fs + sy + P1 * c], dv);
    }
    kappa = -dv;
  }

  // Fluxes to contract.  The a_1 parts of the partial densities' fluxes (-rho01 a_1, +rho02 a_1)
  // are multiples of the phase field's flux -a_1 and are added after the contraction.
  double F[G::NSTAGE];
  F[0] = a1x;
  F[1] = a1y;
  F[2] = q[M1] * u;
  F[3] = q[M1] * v;
  F[4] = q[M2] * u;
  F[5] = q[M2] * v;
  const double gx = fma(-prm.drho0, a1x, q[RU]);  // mass flux less (rho01 - rho02) a_1
  F[6] = fma(gx, u, Pr);
  F[8] = gx * v;
  const double H = q[RE] + Pr;
  F[10] = fma(H, u, -(cE * a1x));
  const double gy = fma(-prm.drho0, a1y, q[RV]);
  F[7] = gy * u;
  F[9] = fma(gy, v, Pr);
  F[11] = fma(H, v, -(cE * a1y));
  if (VISC) {
    F[6] -= txx;
    F[7] -= txy;
    F[8] -= txy;
    F[9] -= tyy;
    F[10] = fma(-txx, u, fma(-txy, v, F[10]));
    F[11] = fma(-txy, u, fma(-tyy, v, F[11]));
  }
  __syncthreads();
  if (lane) {
#pragma unroll
    for (int s = 0; s < G::NSTAGE; ++s) s_f[s * fs + sn] = F[s];
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
      acc = fma(Dhy[j * P1 + c], s_f[(2 * eq + 1) * fs + sy + P1 * c], acc);
    }
    R[eq == 0 ? PHI : eq + 1] = acc;
  }
  const double ra = R[PHI];  // contraction of +a_1
  R[M1] = fma(-prm.rho01, ra, R[M1]);
  R[M2] = fma(prm.rho02, ra, R[M2]);
  // Non-conservative transport of phi and psi (Sec. 3: treated as a source), broken gradients.
  R[PHI] = fma(-u, bpx, fma(-v, bpy, -ra));
  R[PSI] = fma(-u, bsx, -(v * bsy));
  if (prm.gravity) {
    R[RU] += rho * prm.gx;
    R[RV] += rho * prm.gy;
    R[RE] += rho * (prm.gx * u + prm.gy * v);
  }
  if (ST) {
    // CSF surface tension sigma kappa n delta, delta = |grad phi|.
    const double s = prm.sigma * kappa * sqrt64(gpx * gpx + gpy * gpy);
    R[RU] = fma(s, nx, R[RU]);
    R[RV] = fma(s, ny, R[RV]);
    R[RE] = fma(s, u * nx + v * ny, R[RE]);
  }
  if (act) {
#pragma unroll
    for (int vv = 0; vv < NV; ++vv) rvol[(long)vv * N + n] = R[vv];
  }

  // Face traces.
  const bool onW = i == 0, onE = i == P;
  const bool onS = j == 0, onN = j == P;
  if (act && (onW || onE || onS || onN)) {
    const double c = sqrt64(X * ir);  // mixture sound speed
    const double tx[V_A1] = {phi, psi, q[M1], q[M2], q[RU], q[RV], q[RE], u, v, Pr, c, cE};
    const long base = (long)e * NFK;
    const long stride = (long)prm.E * NFK;
    auto put = [&](int f, int kk, double an, double t1, double t2) {
      const long o = base + f * NK + kk;
      if (!in_bounds(prm.status, o, stride)) return;
#pragma unroll
      for (int qf = 0; qf < V_A1; ++qf) tr[qf * stride + o] = tx[qf];
      tr[V_A1 * stride + o] = an;
      if (VISC) {
        tr[V_TX * stride + o] = t1;
        tr[V_TY * stride + o] = t2;
        tr[V_MU * stride + o] = mu;
      }
    };
    const int kx = j;
    if (onW) put(0, kx, a1x, txx, txy);
    if (onE) put(1, kx, a1x, txx, txy);
    if (onS) put(2, i, a1y, txy, tyy);
    if (onN) put(3, i, a1y, txy, tyy);
  }
}

// Shared planes of the surface kernel, one value per face node of the block: twice the surface
// integrand of the seven equations, then what the symmetric SIP term carries along the normal
// line: Gamma eps [[phi]] alone and times the coefficients of momentum and energy.
enum SurfPlane { SP_S = 0, SP_LIFT = NV, SP_LU, SP_LV, SP_LE, NSP };

template <int P, bool VISC, bool ST>
__global__ void __launch_bounds__(MAX_THREADS64)
k_surface_full(const Params prm, int epb, int mode, double dt, const double *__restrict__ w0,
          const double *__restrict__ ws, const double *__restrict__ rvol, const double *__restrict__ tr,
          double *__restrict__ out) {
  using G = Geom<P, 2, VISC, ST>;
  constexpr int P1 = G::P1, NP = G::NP, NFK = G::NFK, NK = G::NK, NT = VISC ? NV_VISCOUS : NV_INVISCID;
  const OpsLayout L{P1, NP};
  extern __shared__ double s_mem[];
  grid_dependency_wait();
  double *s_lw = s_mem;                 // cf [2], lw [4][P1]
  double *s_s = s_mem + 2 + 4 * P1;     // [NSP][epb * NFK]
  const int fs = epb * NFK;

  for (int t = threadIdx.x; t < 2 + 4 * P1; t += blockDim.x) s_lw[t] = prm.ops[L.cf() + t];
  const long stride = (long)prm.E * NFK;
  const int le = threadIdx.x / NP, a = threadIdx.x % NP;
  const int e = blockIdx.x * epb + le;
  const int N = prm.N;
  const long n = (long)e * NP + a;
  const bool act = le < epb && e < prm.E && in_bounds(prm.status, n, N);
  // the node's inputs of the update, loaded ahead of the face work that hides their latency
  double rv[NV], wn[NV], w0n[NV];
#pragma unroll
  for (int vv = 0; vv < NV; ++vv) rv[vv] = wn[vv] = w0n[vv] = 0.0;
  if (act) {
#pragma unroll
    for (int vv = 0; vv < NV; ++vv) rv[vv] = __ldca(rvol + (long)vv * N + n);
    if (mode != MODE_RHS) {
#pragma unroll
      for (int vv = 0; vv < NV; ++vv) wn[vv] = __ldca(ws + (long)vv * N + n);
    }
    if (mode == MODE_S2 || mode == MODE_S3) {
#pragma unroll
      for (int vv = 0; vv < NV; ++vv) w0n[vv] = __ldca(w0 + (long)vv * N + n);
    }
  }
  if (prm.dt_dev) dt = __ldca(prm.dt_dev);

  // Phase 1: numerical fluxes at the block's face nodes, in the own frame (outward normal m = sg
  // e_axis), twice the flux and without the face weight: the gather's coefficients carry both.
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
      } else {              // no-slip: reverse the velocity
        Tp[T_RU] = -Tm[T_RU]; Tp[T_U] = -Tm[T_U];
        Tp[T_RV] = -Tm[T_RV]; Tp[T_V] = -Tm[T_V];
      }
    }
    const double unm = flip64(xf ? Tm[T_U] : Tm[T_V], sm);
    const double unp = flip64(xf ? Tp[T_U] : Tp[T_V], sm);
    const double lam = max_nonneg64(fabs(unm) + Tm[T_C], fabs(unp) + Tp[T_C]);
    const double jphi = Tp[T_PHI] - Tm[T_PHI];
    // a_1 at the face, twice: the SIP flux Gamma eps ({grad phi} . m + eta [phi]) - {Gamma phi (1 - phi) n} . m
    // is the mean of the two traces' own a_1 plus the penalty.  None crosses a wall.
    const double Gej = prm.Ge * jphi;
    const double eta2 = xf ? prm.eta2_x : prm.eta2_y;
    const double A = wall ? 0.0 : fma(eta2, Gej, flip64(Tm[V_A1] + Tp[V_A1], sm));

    // Lax-Friedrichs flux {F}.m - lambda [[w]], [[w]] = (w+ - w-)/2: -2 of it per equation.
    double S[NV];
#pragma unroll
    for (int vv = M1; vv <= RV; ++vv)
      S[vv] = fma(lam, Tp[vv] - Tm[vv], -fma(Tp[vv], unp, Tm[vv] * unm));
    const double Ps = flip64(Tm[T_P] + Tp[T_P], sm);
    const double Hm = Tm[T_RE] + Tm[T_P], Hp = Tp[T_RE] + Tp[T_P];
    S[RE] = fma(lam, Tp[T_RE] - Tm[T_RE], -fma(Hp, unp, Hm * unm));
    if (xf) S[RU] -= Ps;
    else S[RV] -= Ps;
    // Quasi-conservative transport (lambda - m.u-) [[phi]], same for psi; the SIP flux of a_1 and of
    // every a_1-derived term (coefficients averaged over the two sides).
    const double lu = lam - unm;
    const double du = prm.hdr * (Tm[T_U] + Tp[T_U]);
    const double dv = prm.hdr * (Tm[T_V] + Tp[T_V]);
    const double dE = 0.5 * (Tm[V_CE] + Tp[V_CE]);
    S[PHI] = fma(lu, jphi, A);
    S[PSI] = lu * (Tp[T_PSI] - Tm[T_PSI]);
    S[M1] = fma(prm.rho01, A, S[M1]);
    S[M2] = fma(-prm.rho02, A, S[M2]);
    S[RU] = fma(du, A, S[RU]);
    S[RV] = fma(dv, A, S[RV]);
    S[RE] = fma(dE, A, S[RE]);
    if (VISC) {
      const double em = 0.5 * eta2 * (Tp[V_MU] + Tm[V_MU]);  // 2 eta {mu}
      const double tx = flip64(Tm[V_TX] + Tp[V_TX], sm), ty = flip64(Tm[V_TY] + Tp[V_TY], sm);
      S[RU] = fma(em, Tp[T_U] - Tm[T_U], S[RU] + tx);
      S[RV] = fma(em, Tp[T_V] - Tm[T_V], S[RV] + ty);
      const double km = fma(Tm[T_V], Tm[T_V], Tm[T_U] * Tm[T_U]);
      const double kp = fma(Tp[T_V], Tp[T_V], Tp[T_U] * Tp[T_U]);
      const double tu = fma(Tm[V_TX], Tm[T_U], Tm[V_TY] * Tm[T_V]) + fma(Tp[V_TX], Tp[T_U], Tp[V_TY] * Tp[T_V]);
      S[RE] = fma(0.5 * em, kp - km, S[RE] + flip64(tu, sm));
    }
#pragma unroll
    for (int vv = 0; vv < NV; ++vv) s_s[vv * fs + g] = S[vv];
    s_s[SP_LIFT * fs + g] = Gej;  // zero at a wall: the ghost keeps the own phase field
    s_s[SP_LU * fs + g] = du * Gej;
    s_s[SP_LV * fs + g] = dv * Gej;
    s_s[SP_LE * fs + g] = dE * Gej;
  }
  __syncthreads();

  // Phase 2: gather onto the element's nodes, lift the symmetric term along
  // the normal lines (M^-1 is in the coefficients), add the volume part, write L or the stage.
  if (!act) return;
  const int i = a % P1, j = a / P1;
  const int kx = j;
  double r[NV];
#pragma unroll
  for (int vv = 0; vv < NV; ++vv) r[vv] = rv[vv];
  // (a line has two different end nodes, so a node lies on at most one face per axis)
  if (i == 0 || i == P) {
    const int g = le * NFK + (i == 0 ? 0 : NK) + kx;
#pragma unroll
    for (int vv = 0; vv < NV; ++vv) r[vv] = fma(s_lw[0], s_s[vv * fs + g], r[vv]);
  }
  if (j == 0 || j == P) {
    const int g = le * NFK + (j == 0 ? 2 : 3) * NK + i;
#pragma unroll
    for (int vv = 0; vv < NV; ++vv) r[vv] = fma(s_lw[1], s_s[vv * fs + g], r[vv]);
  }
  {
    const double *lw = s_lw + 2;
    double lp = 0.0;
#pragma unroll
    for (int f = 0; f < 4; ++f) {
      const int g = le * NFK + f * NK + (f < 2 ? kx : i);
      const double c = lw[f * P1 + (f < 2 ? i : j)];
      lp = f ? fma(c, s_s[SP_LIFT * fs + g], lp) : c * s_s[SP_LIFT * fs + g];
      r[RU] = fma(c, s_s[SP_LU * fs + g], r[RU]);
      r[RV] = fma(c, s_s[SP_LV * fs + g], r[RV]);
      r[RE] = fma(c, s_s[SP_LE * fs + g], r[RE]);
    }
    r[PHI] += lp;
    r[M1] = fma(prm.rho01, lp, r[M1]);
    r[M2] = fma(-prm.rho02, lp, r[M2]);
  }
  bool bad = false;
#pragma unroll
  for (int vv = 0; vv < NV; ++vv) {
    const long o = (long)vv * N + n;
    if (mode != MODE_RHS) {
      r[vv] = fma(dt, r[vv], wn[vv]);
      if (mode == MODE_S2) r[vv] = fma(0.75, w0n[vv], 0.25 * r[vv]);
      else if (mode == MODE_S3) r[vv] = fma(1.0 / 3.0, w0n[vv], (2.0 / 3.0) * r[vv]);
    }
    bad |= !finite64(r[vv]);
    out[o] = r[vv];
  }
  if (prm.check_finite && bad) atomicOr(prm.status, STATUS_NONFINITE);
}

template <int P, bool VISC, bool ST>
cudaError_t launch_volume_full(const Params &prm, const double *w, double *rvol, double *trace, cudaStream_t s) {
  using G = Geom<P, 2, VISC, ST>;
  const int epb = pick_epb64(prm.E, G::NP, 1), threads = (epb * G::NP + 31) / 32 * 32;
  const size_t smem = sizeof(double) * (4 * G::P1 * G::P1 + (size_t)G::NSTAGE * epb * G::NP);
  return launch_dependent(k_volume_full<P, VISC, ST>, (prm.E + epb - 1) / epb, threads, smem, s, prm, epb, w, rvol,
                          trace);
}

template <int P, bool VISC, bool ST>
cudaError_t launch_surface_full(const Params &prm, int mode, double dt, const double *w0, const double *ws,
                           const double *rvol, const double *trace, double *out, cudaStream_t s) {
  using G = Geom<P, 2, VISC, ST>;
  // face nodes cost about as much as nodes here (46 and 50 operations)
  const int epb = pick_epb64(prm.E, G::NP, 1, G::NFK, 1), threads = (epb * G::NP + 31) / 32 * 32;
  const size_t smem = sizeof(double) * (2 + 4 * G::P1 + (size_t)NSP * epb * G::NFK);
  return launch_dependent(k_surface_full<P, VISC, ST>, (prm.E + epb - 1) / epb, threads, smem, s, prm, epb, mode, dt,
                          w0, ws, rvol, trace, out);
}


template <int P, bool VISC, bool ST>
KernelSet make_set_full() {
  return KernelSet{&launch_volume_full<P, VISC, ST>, &launch_surface_full<P, VISC, ST>,
                   VISC ? NV_VISCOUS : NV_INVISCID};
}

// All families of one order.
template <int P>
bool kernels_fp64_p(int dim, bool viscous, bool st, KernelSet *out) {
  if (dim == 1) {
    if (viscous || st) return false;
    *out = make_set<P, 1>();
    return true;
  }
  if (!viscous && !st) *out = make_set<P, 2>();
  else if (viscous && !st) *out = make_set_full<P, true, false>();
  else if (!viscous && st) *out = make_set_full<P, false, true>();
  else *out = make_set_full<P, true, true>();
  return true;
}

}  // namespace dgpf
