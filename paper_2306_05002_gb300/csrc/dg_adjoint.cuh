// dg_adjoint.cuh -- discrete adjoint (vector-Jacobian product) of the FP64
// right-hand side, for the inviscid equations without surface tension
// (gravity allowed): mu = (dL/dw)^T lambda, written by hand in reverse mode.
//
// Three launches per product:
//   k_volume      (forward, dg_kernels_fp64.cuh) -- the face traces of w;
//   k_adj_face    per face node of the mesh: the adjoints of the trace records
//                 of both elements sharing the face;
//   k_adj_volume  per element: recomputes the node quantities and runs the
//                 reverse of fluxes, a_1, normal, gradients and closure, adds
//                 the trace adjoints, and writes
//                 out = a x + b mu + c y + d z   (fused combination used by
//                 the reverse of the SSP-RK3 stages).
//
// Face adjoints.  The Lax-Friedrichs fluxes and the SIP flux of every
// a_1-derived term are conservative: seen from the neighbour (normal -m, the
// two traces swapped) their contribution is the negative of the own one,
// with the same lambda.  So one reverse evaluation seeded with (own seed -
// neighbour seed) gives the adjoints of both traces; only the
// non-conservative transport terms of phi and psi have a seed on each side.
// Where the two one-sided speeds tie in
// lambda = max(|u-.m| + c-, |u+.m| + c+) the derivative is given to both
// sides, each as its own side (a set of measure zero: the jump there is what
// lambda multiplies).
//
// Both kernels are bound by the FP64 pipe (two operations per clock and SM),
// so they are written to the fewest FP64 instructions.  A face is evaluated
// once, by the element that has it as its west or south face, which writes
// both records (twice, once from each side, before): at p = 3 about 185
// operations per face node, half a face node per node, where the two-sided
// form took 330 per node.  k_adj_volume: about 260 operations per node where
// the statement-by-statement reverse took 385, by reversing the grouped
// forward expressions (mass fluxes less a_1 times velocity, one mixture
// reciprocal, u and k in place of momenta over rho) and adding one face
// record per axis.
#pragma once

#include "dg_kernels_fp64.cuh"

namespace dgpf {

// Node index of face node k on face f.
template <int P, int DIM>
__device__ __forceinline__ int face_node(int f, int k) {
  constexpr int P1 = P + 1;
  if (DIM == 1) return f == 0 ? 0 : P;
  switch (f) {
    case 0: return P1 * k;
    case 1: return P + P1 * k;
    case 2: return k;
    default: return k + P1 * P;
  }
}

// Adjoint of the line terms of one element's face (f, k): per equation that carries the symmetric SIP
// term, the sum over the normal line of lambda times the weight with which the term reaches the node
// (OpsLayout lw), added to sL with sign sgn.
template <int P, int DIM>
__device__ __forceinline__ void line_seeds(const double *__restrict__ lam, int N, int e, int f, int k,
                                           const double *lw, double sgn, double sL[6]) {
  constexpr int P1 = P + 1, NP = DIM == 2 ? P1 * P1 : P1;
  const long base = (long)e * NP;
  const int slot[6] = {PHI, M1, M2, RU, RV, RE};
#pragma unroll
  for (int l = 0; l < P1; ++l) {
    const int b = f < 2 ? (DIM == 2 ? l + P1 * k : l) : k + P1 * l;
    const double wgt = flip64(lw[f * P1 + l], sgn < 0.0 ? (int)0x80000000 : 0);
#pragma unroll
    for (int c = 0; c < 6; ++c)
      if (DIM == 2 || c != 4) sL[c] = fma(__ldca(lam + (long)slot[c] * N + base + b), wgt, sL[c]);
  }
}

template <int P, int DIM>
__global__ void __launch_bounds__(MAX_THREADS64)
k_adj_face(const Params prm, int epb, const double *__restrict__ lam, const double *__restrict__ tr,
           double *__restrict__ trbar) {
  using G = Geom<P, DIM, false, false>;
  constexpr int P1 = G::P1, NP = G::NP, NFK = G::NFK, NK = G::NK;
  constexpr int NO = DIM * NK;  // face nodes of an element's west and south faces
  constexpr int NT = NT_INVISCID;
  const OpsLayout L{P1, NP};
  __shared__ double s_lw[2 + 4 * P1];
  grid_dependency_wait();
  for (int t = threadIdx.x; t < 2 + 4 * P1; t += blockDim.x) s_lw[t] = prm.ops[L.cf() + t];
  __syncthreads();
  const long stride = (long)prm.E * NFK;
  const int N = prm.N;
  // the east and north faces of a mesh that ends in walls there are their own elements' work
  const bool ends = prm.bc[1] != BC_PERIODIC || (DIM == 2 && prm.bc[3] != BC_PERIODIC);
  const int ntask = epb * NO * (ends ? 2 : 1);

  for (int g = threadIdx.x; g < ntask; g += blockDim.x) {
    const int far = g >= epb * NO, g1 = g - far * epb * NO;
    const int e = blockIdx.x * epb + g1 / NO, t = g1 % NO;
    const int f = 2 * (t / NK) + far, kk = t % NK;
    if (e >= prm.E) continue;
    const int e2 = neighbour(prm, e, f);
    const bool wall = e2 < 0;
    if (far && !wall) continue;
    // the elements' nodes (line seeds) and face records
    if (!in_bounds(prm.status, (long long)e * NP + NP - 1, N) ||
        !in_bounds(prm.status, (long long)e * NFK + NFK - 1, stride))
      continue;
    if (!wall && (!in_bounds(prm.status, (long long)e2 * NP + NP - 1, N) ||
                  !in_bounds(prm.status, (long long)e2 * NFK + NFK - 1, stride)))
      continue;
    const bool xf = f < 2;
    const int sm = (f & 1) ? 0 : (int)0x80000000;  // sign of m
    double Tm[NT], Tp[NT];
    const long om = (long)e * NFK + f * NK + kk;
    const long op = (long)(wall ? e : e2) * NFK + (wall ? f : (f ^ 1)) * NK + kk;
#pragma unroll
    for (int q = 0; q < NT; ++q) Tm[q] = __ldca(tr + q * stride + om);
#pragma unroll
    for (int q = 0; q < NT; ++q) Tp[q] = __ldca(tr + q * stride + op);
    const bool flip_u = wall && (prm.bc[f] != BC_SLIP || xf), flip_v = wall && (prm.bc[f] != BC_SLIP || !xf);
    if (flip_u) { Tp[T_RU] = -Tm[T_RU]; Tp[T_U] = -Tm[T_U]; }
    if (flip_v) { Tp[T_RV] = -Tm[T_RV]; Tp[T_V] = -Tm[T_V]; }

    // Seeds.  cf carries the face weight, M^-1 and the halves of the averages and jumps: h[v] is the
    // seed of the conservative part of equation v, (own - neighbour); the transport of phi and psi
    // has one seed per side (so, sn).
    const double cf = s_lw[xf ? 0 : 1];
    const long nm = (long)e * NP + face_node<P, DIM>(f, kk);
    const long np = wall ? nm : (long)e2 * NP + face_node<P, DIM>(f ^ 1, kk);
    double h[NV], so[2], sn[2];
#pragma unroll
    for (int v = 0; v < NV; ++v) {
      const double lo = __ldca(lam + (long)v * N + nm), ln = wall ? 0.0 : __ldca(lam + (long)v * N + np);
      if (v < 2) {
        so[v] = cf * lo;
        sn[v] = cf * ln;
        h[v] = so[v] - sn[v];
      } else {
        h[v] = cf * (lo - ln);
      }
    }
    double bm[NT], bp[NT];

    // forward quantities
    const double unm = flip64(xf ? Tm[T_U] : Tm[T_V], sm), unp = flip64(xf ? Tp[T_U] : Tp[T_V], sm);
    const double Lm = fabs(unm) + Tm[T_C], Lp = fabs(unp) + Tp[T_C];
    const bool own = Lm >= Lp, other = Lp >= Lm;
    const double lm = own ? Lm : Lp;
    double blam = 0.0, bunm = 0.0, bunp = 0.0;

    // (a) Lax-Friedrichs part of the conservative equations: -({F}.m - lambda [[w]])
    const double am = -(lm + unm), ap = lm - unp;
#pragma unroll
    for (int v = M1; v <= RE; ++v) {
      blam = fma(Tp[v] - Tm[v], h[v], blam);
      bm[v] = am * h[v];
      bp[v] = ap * h[v];
      bunm = fma(-h[v], v == RE ? Tm[T_RE] + Tm[T_P] : Tm[v], bunm);
      bunp = fma(-h[v], v == RE ? Tp[T_RE] + Tp[T_P] : Tp[v], bunp);
    }
    const double hn = flip64(xf ? h[RU] : h[RV], sm);
    bm[T_P] = fma(-h[RE], unm, -hn);
    bp[T_P] = fma(-h[RE], unp, -hn);
    // (b) transport of phi and psi seen from this element, (lambda - m.u-) [[q]], and from the
    // neighbour, (lambda + m.u+) (q- - q+)/2
    const double lo = lm - unm, ln = lm + unp;
    const double jump = Tp[T_PHI] - Tm[T_PHI];
#pragma unroll
    for (int v = 0; v < 2; ++v) {
      const double j = v == 0 ? jump : Tp[T_PSI] - Tm[T_PSI];
      blam = fma(j, h[v], blam);
      bunm = fma(-j, so[v], bunm);
      bunp = fma(-j, sn[v], bunp);
      bp[v] = fma(lo, so[v], -(ln * sn[v]));
      bm[v] = -bp[v];
    }
#pragma unroll
    for (int q = T_U; q < NT; ++q)
      if (q != T_P) bm[q] = bp[q] = 0.0;
    // (c) SIP flux of a_1 and of every a_1-derived term (seed own - neighbour), twice the flux
    if (!wall) {
      double gL[6] = {0, 0, 0, 0, 0, 0};
      line_seeds<P, DIM>(lam, N, e, f, kk, s_lw + 2, 1.0, gL);
      line_seeds<P, DIM>(lam, N, e2, f ^ 1, kk, s_lw + 2, -1.0, gL);
      const double sp = fma(-Tp[T_PHI], Tp[T_PHI], Tp[T_PHI]), sM = fma(-Tm[T_PHI], Tm[T_PHI], Tm[T_PHI]);
      const double sharp = prm.Gamma * fma(sp, Tp[T_N], sM * Tm[T_N]);
      const double ahat = fma(xf ? prm.Gp_x : prm.Gp_y, jump, flip64(fma(prm.Ge, Tp[T_GPHI] + Tm[T_GPHI], -sharp), sm));
      const double km2 = DIM == 2 ? fma(Tm[T_V], Tm[T_V], Tm[T_U] * Tm[T_U]) : Tm[T_U] * Tm[T_U];
      const double kp2 = DIM == 2 ? fma(Tp[T_V], Tp[T_V], Tp[T_U] * Tp[T_U]) : Tp[T_U] * Tp[T_U];
      const double cu = prm.hdr * (Tp[T_U] + Tm[T_U]), cv = prm.hdr * (Tp[T_V] + Tm[T_V]);
      const double cE = 0.5 * fma(prm.hdr, kp2 + km2, Tp[T_B] + Tm[T_B]);
      const double gej = prm.Ge * jump;
      double H = fma(prm.rho01, h[M1], h[PHI]);  // half the adjoint of a_1 . m at the face
      H = fma(-prm.rho02, h[M2], H);
      H = fma(cu, h[RU], H);
      double Gq = fma(prm.rho01, gL[1], gL[0]);
      Gq = fma(-prm.rho02, gL[2], Gq);
      Gq = fma(cu, gL[3], Gq);
      if (DIM == 2) {
        H = fma(cv, h[RV], H);
        Gq = fma(cv, gL[4], Gq);
      }
      H = fma(cE, h[RE], H);
      Gq = fma(cE, gL[5], Gq);
      const double bcu = prm.hdr * fma(ahat, h[RU], gej * gL[3]);
      const double bcE = fma(ahat, h[RE], gej * gL[5]);
      const double bjump = prm.Ge * fma(xf ? prm.eta2_x : prm.eta2_y, H, Gq);
      bp[T_GPHI] = bm[T_GPHI] = flip64(prm.Ge * H, sm);
      const double GH = flip64(prm.Gamma * H, sm);
      bp[T_N] = -(sp * GH);
      bm[T_N] = -(sM * GH);
      bp[T_PHI] += fma(fma(2.0, Tp[T_PHI], -1.0), Tp[T_N] * GH, bjump);
      bm[T_PHI] += fma(fma(2.0, Tm[T_PHI], -1.0), Tm[T_N] * GH, -bjump);
      const double bk = prm.hdr * bcE;
      bp[T_U] = fma(Tp[T_U], bk, bcu);
      bm[T_U] = fma(Tm[T_U], bk, bcu);
      if (DIM == 2) {
        const double bcv = prm.hdr * fma(ahat, h[RV], gej * gL[4]);
        bp[T_V] = fma(Tp[T_V], bk, bcv);
        bm[T_V] = fma(Tm[T_V], bk, bcv);
      }
      bp[T_B] = bm[T_B] = 0.5 * bcE;
    }
    // (d) lambda = max of the one-sided speeds, then the normal velocities
    if (own) {
      bunm += unm > 0.0 ? blam : (unm < 0.0 ? -blam : 0.0);
      bm[T_C] = blam;
    }
    if (wall ? !own : other) {
      bunp += unp > 0.0 ? blam : (unp < 0.0 ? -blam : 0.0);
      bp[T_C] = blam;
    }
    if (xf) {
      bm[T_U] += flip64(bunm, sm);
      bp[T_U] += flip64(bunp, sm);
    } else {
      bm[T_V] += flip64(bunm, sm);
      bp[T_V] += flip64(bunp, sm);
    }
    // (e) a wall's ghost is a function of the own trace
    if (wall) {
#pragma unroll
      for (int q = 0; q < NT; ++q) {
        const bool neg = ((q == T_RU || q == T_U) && flip_u) || ((q == T_RV || q == T_V) && flip_v);
        bm[q] += neg ? -bp[q] : bp[q];
      }
    } else {
#pragma unroll
      for (int q = 0; q < NT; ++q) trbar[q * stride + op] = bp[q];
    }
#pragma unroll
    for (int q = 0; q < NT; ++q) trbar[q * stride + om] = bm[q];
  }
}

template <int P, int DIM>
__global__ void __launch_bounds__(MAX_THREADS64)
k_adj_volume(const Params prm, int epb, const double *__restrict__ w, const double *__restrict__ lam,
             const double *__restrict__ trbar, double *__restrict__ out, double ca, const double *__restrict__ xa,
             double cb, double cc, const double *__restrict__ yc, double cd, const double *__restrict__ zd) {
  using G = Geom<P, DIM, false, false>;
  constexpr int P1 = G::P1, NP = G::NP, NFK = G::NFK, NK = G::NK;
  constexpr int P11 = P1 * P1;
  extern __shared__ double s_mem[];
  double *s_op = s_mem;                    // Dx, Dy, Dhx, Dhy
  double *s_f = s_mem + 4 * P11;           // [6][epb * NP]
  const int fs = epb * NP;
  grid_dependency_wait();

  for (int t = threadIdx.x; t < 4 * P11; t += blockDim.x) s_op[t] = prm.ops[t];
  const double *Dx = s_op, *Dy = s_op + P11, *Dhx = s_op + 2 * P11, *Dhy = s_op + 3 * P11;

  const int le_raw = threadIdx.x / NP;
  const bool lane = le_raw < epb;
  const int le = lane ? le_raw : epb - 1;
  const int a = threadIdx.x % NP;
  const int e = blockIdx.x * epb + le;
  const int N = prm.N;
  const bool act = lane && e < prm.E && in_bounds(prm.status, (long long)e * NP + a, N);
  const int i = a % P1, j = DIM == 2 ? a / P1 : 0;
  const long n = (long)(act ? e : 0) * NP + a;
  const int sn = le * NP + a, sx = le * NP + P1 * j, sy = le * NP + i;

  // ---- forward recomputation
  double q[NV], lm[NV];
#pragma unroll
  for (int v = 0; v < NV; ++v) {
    q[v] = act ? __ldca(w + (long)v * N + n) : (v == M1 || v == M2 ? 1.0 : 0.0);
    lm[v] = act ? __ldca(lam + (long)v * N + n) : 0.0;
  }
  const double phi = q[PHI];
  const double rho = q[M1] + q[M2];
  const double ir = rcp64(rho);
  const double u = q[RU] * ir;
  const double v = DIM == 2 ? q[RV] * ir : 0.0;
  const double k = 0.5 * (DIM == 2 ? fma(v, v, u * u) : u * u);
  const double iden = rcp64(fma(phi, prm.dg, prm.g2));
  const double Cm = mixture_constant(prm, phi);
  const double Pr = __dsub_rn(fma(-rho, k, q[RE]), Cm) * iden;
  const double cE = fma(prm.drho0, k, fma(Pr, prm.Bp, prm.dC));
  if (lane) {
    s_f[0 * fs + sn] = phi;
    s_f[1 * fs + sn] = q[PSI];
  }
  __syncthreads();
  double gpx = 0.0, gpy = 0.0, gsx = 0.0, gsy = 0.0;
#pragma unroll
  for (int c = 0; c < P1; ++c) {
    const double dx = Dx[i * P1 + c];
    gpx = c ? fma(dx, s_f[0 * fs + sx + c], gpx) : dx * s_f[0 * fs + sx];
    gsx = c ? fma(dx, s_f[1 * fs + sx + c], gsx) : dx * s_f[1 * fs + sx];
    if (DIM == 2) {
      const double dy = Dy[j * P1 + c];
      gpy = c ? fma(dy, s_f[0 * fs + sy + P1 * c], gpy) : dy * s_f[0 * fs + sy];
      gsy = c ? fma(dy, s_f[1 * fs + sy + P1 * c], gsy) : dy * s_f[1 * fs + sy];
    }
  }
  const double g2 = DIM == 2 ? fma(gsy, gsy, gsx * gsx) : gsx * gsx;
  double nx = 0.0, ny = 0.0, rn = 0.0;
  const bool has_n = has_gradient(g2);
  if (has_n) {
    rn = rsqrt64(g2);
    nx = gsx * rn;
    ny = gsy * rn;
  }
  const double Gs = prm.Gamma * fma(-phi, phi, phi);
  const double a1x = fma(prm.Ge, gpx, -(Gs * nx));
  const double a1y = DIM == 2 ? fma(prm.Ge, gpy, -(Gs * ny)) : 0.0;

  // ---- reverse of the volume contraction: (x, y) = Dhat^T lambda, per equation
  __syncthreads();
  if (lane) {
    s_f[0 * fs + sn] = lm[PHI];
#pragma unroll
    for (int c = 1; c < 6; ++c) s_f[c * fs + sn] = lm[c + 1];
  }
  __syncthreads();
  double bx[6], by[6];
#pragma unroll
  for (int eq = 0; eq < 6; ++eq) {
    by[eq] = 0.0;
#pragma unroll
    for (int c = 0; c < P1; ++c) {
      const double dx = Dhx[c * P1 + i], fx = s_f[eq * fs + sx + c];
      bx[eq] = c ? fma(dx, fx, bx[eq]) : dx * fx;
      if (DIM == 2) {
        const double dy = Dhy[c * P1 + j], fy = s_f[eq * fs + sy + P1 * c];
        by[eq] = c ? fma(dy, fy, by[eq]) : dy * fy;
      }
    }
  }

  // face-trace adjoints of the faces this node lies on: at most one face per axis
  double T[T_GPHI], bgpx = 0.0, bgpy = 0.0, bnx = 0.0, bny = 0.0;
  {
    const long stride = (long)prm.E * NFK, eo = (long)(act ? e : 0) * NFK;
    const bool onx = act && (i == 0 || i == P), ony = DIM == 2 && act && (j == 0 || j == P);
    const long ox = eo + (i == P ? NK : 0) + (DIM == 2 ? j : 0), oy = eo + (j == P ? 3 : 2) * NK + i;
    const bool okx = onx && in_bounds(prm.status, ox, stride), oky = ony && in_bounds(prm.status, oy, stride);
#pragma unroll
    for (int f = 0; f < T_GPHI; ++f) T[f] = okx ? __ldca(trbar + f * stride + ox) : 0.0;
    if (okx) {
      bgpx = __ldca(trbar + T_GPHI * stride + ox);
      bnx = __ldca(trbar + T_N * stride + ox);
    }
    if (oky) {
#pragma unroll
      for (int f = 0; f < T_GPHI; ++f) T[f] += __ldca(trbar + f * stride + oy);
      bgpy = __ldca(trbar + T_GPHI * stride + oy);
      bny = __ldca(trbar + T_N * stride + oy);
    }
  }
  double *bw = T;  // adjoints of the state (T_PHI..T_RE), u, v, P, c and B start from the traces'
  double bu = T[T_U], bv = T[T_V], bP = T[T_P], brho = 0.0;
  const double bc = T[T_C];

  // fluxes: m_l u -+ rho0_l a_1, g u + P with g = rho u - drho0 a_1, (rho E + P) u - cE a_1
  const double gx = fma(-prm.drho0, a1x, q[RU]), H = q[RE] + Pr;
  const double bgx = DIM == 2 ? fma(bx[4], v, bx[3] * u) : bx[3] * u;
  bw[RU] += bgx;
  bu = fma(bx[3], gx, bu);
  bu = fma(bx[1], q[M1], bu);
  bu = fma(bx[2], q[M2], bu);
  bu = fma(bx[5], H, bu);
  bw[M1] = fma(bx[1], u, bw[M1]);
  bw[M2] = fma(bx[2], u, bw[M2]);
  double bH = bx[5] * u;
  bP += bx[3];
  double bcE = bx[5] * a1x;  // minus the adjoint of cE from the flux
  double ba1x = fma(prm.rho01, bx[1], bx[0]);  // minus the adjoint of a_1
  ba1x = fma(-prm.rho02, bx[2], ba1x);
  ba1x = fma(prm.drho0, bgx, ba1x);
  ba1x = fma(cE, bx[5], ba1x);
  double ba1y = 0.0;
  if (DIM == 2) {
    const double gy = fma(-prm.drho0, a1y, q[RV]);
    const double bgy = fma(by[4], v, by[3] * u);
    bw[RV] += bgy;
    bu = fma(by[3], gy, bu);
    bv = fma(bx[4], gx, bv);
    bv = fma(by[4], gy, bv);
    bv = fma(by[1], q[M1], bv);
    bv = fma(by[2], q[M2], bv);
    bv = fma(by[5], H, bv);
    bw[M1] = fma(by[1], v, bw[M1]);
    bw[M2] = fma(by[2], v, bw[M2]);
    bH = fma(by[5], v, bH);
    bP += by[4];
    bcE = fma(by[5], a1y, bcE);
    ba1y = fma(prm.rho01, by[1], by[0]);
    ba1y = fma(-prm.rho02, by[2], ba1y);
    ba1y = fma(prm.drho0, bgy, ba1y);
    ba1y = fma(cE, by[5], ba1y);
  } else {  // the unused y-momentum is carried as rho v u
    bw[RV] = fma(bx[4], u, bw[RV]);
    bu = fma(bx[4], q[RV], bu);
  }
  bw[RE] += bH;
  bP += bH;
  const double bk = -prm.drho0 * bcE, bB = T[T_B] - bcE;
  // non-conservative transport of phi and psi, gravity
  bgpx = fma(-lm[PHI], u, fma(-prm.Ge, ba1x, bgpx));
  bu = fma(-lm[PHI], gpx, bu);
  bu = fma(-lm[PSI], gsx, bu);
  double bgsx = -(lm[PSI] * u), bgsy = 0.0;
  bnx = fma(Gs, ba1x, bnx);
  double bs = nx * ba1x;  // Gamma bs: the adjoint of phi (1 - phi)
  if (DIM == 2) {
    bgpy = fma(-lm[PHI], v, fma(-prm.Ge, ba1y, bgpy));
    bv = fma(-lm[PHI], gpy, bv);
    bv = fma(-lm[PSI], gsy, bv);
    bgsy = -(lm[PSI] * v);
    bny = fma(Gs, ba1y, bny);
    bs = fma(ny, ba1y, bs);
  }
  if (prm.gravity) {
    brho += lm[RU] * prm.gx + lm[RV] * prm.gy + lm[RE] * (prm.gx * u + prm.gy * v);
    bu += lm[RE] * rho * prm.gx;
    bv += lm[RE] * rho * prm.gy;
  }
  bw[PHI] = fma(fma(-2.0, phi, 1.0), prm.Gamma * bs, bw[PHI]);
  // n = grad psi / |grad psi|
  if (has_n) {
    const double nn = DIM == 2 ? fma(ny, bny, nx * bnx) : nx * bnx;
    bgsx = fma(rn, fma(-nx, nn, bnx), bgsx);
    if (DIM == 2) bgsy = fma(rn, fma(-ny, nn, bny), bgsy);
  }
  // reverse of the gradient contractions (transpose over the element)
  __syncthreads();
  if (lane) {
    s_f[0 * fs + sn] = bgpx;
    s_f[1 * fs + sn] = bgpy;
    s_f[2 * fs + sn] = bgsx;
    s_f[3 * fs + sn] = bgsy;
  }
  __syncthreads();
#pragma unroll
  for (int c = 0; c < P1; ++c) {
    const double dx = Dx[c * P1 + i];
    bw[PHI] = fma(dx, s_f[0 * fs + sx + c], bw[PHI]);
    bw[PSI] = fma(dx, s_f[2 * fs + sx + c], bw[PSI]);
    if (DIM == 2) {
      const double dy = Dy[c * P1 + j];
      bw[PHI] = fma(dy, s_f[1 * fs + sy + P1 * c], bw[PHI]);
      bw[PSI] = fma(dy, s_f[3 * fs + sy + P1 * c], bw[PSI]);
    }
  }
  // closure: c (face nodes), B, k, P, u, v, rho
  double bCm = 0.0, bden = 0.0;
  bP = fma(prm.Bp, bB, bP);
  if (bc != 0.0) {  // c^2 = X / rho, X = P + (P + Cm) / den
    const double PC = (Pr + Cm) * iden;
    const double X = Pr + PC;
    const double t = 0.5 * bc * rsqrt64(X * ir) * ir;  // bc / (2 c rho): the adjoint of X
    bP = fma(t, 1.0 + iden, bP);
    bCm = t * iden;
    bden = -(bCm * PC);
    brho = fma(-t * X, ir, brho);
  }
  bu = fma(u, bk, bu);
  bv = fma(v, bk, bv);
  const double bPd = bP * iden;  // P = (rho E - rho k - Cm) / den
  bCm -= bPd;
  bden = fma(-bPd, Pr, bden);
  bw[RE] += bPd;
  bw[PHI] = fma(prm.C1 - prm.C2, bCm, fma(prm.dg, bden, bw[PHI]));
  // rho k = (ru^2 + rv^2) / (2 rho); u = ru / rho
  bw[RU] = fma(-bPd, u, fma(bu, ir, bw[RU]));
  if (DIM == 2) bw[RV] = fma(-bPd, v, fma(bv, ir, bw[RV]));
  brho = fma(bPd, k, brho);
  brho = fma(-ir, DIM == 2 ? fma(bv, v, bu * u) : bu * u, brho);
  bw[M1] += brho;
  bw[M2] += brho;

  if (!act) return;
#pragma unroll
  for (int vv = 0; vv < NV; ++vv) {
    const long o = (long)vv * N + n;
    double r = cb * bw[vv];
    if (xa) r = fma(ca, __ldca(xa + o), r);
    if (yc) r = fma(cc, __ldca(yc + o), r);
    if (zd) r = fma(cd, __ldca(zd + o), r);
    out[o] = r;
  }
}

struct AdjKernels {
  cudaError_t (*face)(const Params &, const double *lam, const double *trace, double *trbar, cudaStream_t);
  cudaError_t (*volume)(const Params &, const double *w, const double *lam, const double *trbar, double *out,
                        double ca, const double *xa, double cb, double cc, const double *yc, double cd,
                        const double *zd, cudaStream_t);
};

template <int P, int DIM>
cudaError_t launch_adj_face(const Params &prm, const double *lam, const double *trace, double *trbar,
                            cudaStream_t s) {
  constexpr int NO = DIM * Geom<P, DIM, false, false>::NK;
  const int epb = pick_epb64(prm.E, NO, 1), threads = (epb * NO + 31) / 32 * 32;
  return launch_dependent(k_adj_face<P, DIM>, (prm.E + epb - 1) / epb, threads, 0, s, prm, epb, lam, trace, trbar);
}

template <int P, int DIM>
cudaError_t launch_adj_volume(const Params &prm, const double *w, const double *lam, const double *trbar,
                              double *out, double ca, const double *xa, double cb, double cc, const double *yc,
                              double cd, const double *zd, cudaStream_t s) {
  using G = Geom<P, DIM, false, false>;
  const int epb = pick_epb64(prm.E, G::NP, 1), threads = (epb * G::NP + 31) / 32 * 32;
  const size_t smem = sizeof(double) * (4 * G::P1 * G::P1 + (size_t)6 * epb * G::NP);
  return launch_dependent(k_adj_volume<P, DIM>, (prm.E + epb - 1) / epb, threads, smem, s, prm, epb, w, lam, trbar,
                          out, ca, xa, cb, cc, yc, cd, zd);
}

template <int P>
bool adj_kernels_p(int dim, AdjKernels *out) {
  if (dim == 1) *out = {&launch_adj_face<P, 1>, &launch_adj_volume<P, 1>};
  else *out = {&launch_adj_face<P, 2>, &launch_adj_volume<P, 2>};
  return true;
}

bool adj_kernels(int p, int dim, AdjKernels *out);

}  // namespace dgpf
