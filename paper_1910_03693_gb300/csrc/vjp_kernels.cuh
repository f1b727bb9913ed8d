// Adjoint (VJP) kernels of the FR residual: the exact transpose of the
// linearisation that fr_jvp evaluates, in reverse order of the forward passes
//   trace -> face -> volume     becomes     volume^T -> face^T -> trace^T.
// Every adjoint value is written by exactly one thread into a slot it owns
// (element-face blocks), and gathered by the consumer: no floating-point
// atomics, so the result is deterministic.
//
// Buffers: fbar has the layout of fout (comp 0..NV-1: adjoint of F~^com,
// NV..2NV-1: adjoint of dq = q^com - q).  trbar uses the traces' element-face
// blocks, of which the first 2 NV components: the adjoint of the q trace with
// the tangential derivatives' adjoints already carried back to it (the face
// kernel holds whole faces, so it applies the transposed differentiation along
// the face's own axes itself), then the adjoint of the reference normal
// derivative.  The trace pass reads 2 NV instead of NV (1 + ND) components and
// no tangential sums.
//
// The pointwise fluxes are transposed in reverse mode (one sweep back through
// the formulas of physics.cuh); a forward-mode sweep per input column costs NV
// (volume) and 2 NV (common flux) evaluations of the dual arithmetic.  Measured
// with the columns and now: 24^3 hexahedra p = 4 FP32, volume 271 -> 140 us, face
// 245 -> 121 us, trace 149 -> 45 us, and the forward face pass 76 us replaced by
// the jumps' 26 us (VJP 806 -> 403 us); 12^3 FP64, volume 876 -> 277 us, face 827 ->
// 183 us, trace 182 -> 29 us.  FP64: the FP64 pipe bounds all but the jumps and
// the trace; FP32: the shared-memory lines and the face data's bytes.
#pragma once

#include "fused_jvp.cuh"

namespace frgb {

template <typename T>
__device__ __forceinline__ T sign_of(T x) { return x < T(0) ? T(-1) : T(1); }   // as dabs: +1 at 0

// qb += (d f_inv / dq)^T fb, f_inv[j][v] the inviscid flux (flux_inviscid).
template <int ND, typename T>
__device__ __forceinline__ void inviscid_adjoint(const T* q, const T (*fb)[ND + 2], T gamma, T* qb) {
  constexpr int NV = ND + 2;
  const T rinv = T(1) / q[0];
  T vel[ND], ub[ND], k = T(0);
#pragma unroll
  for (int i = 0; i < ND; ++i) {
    vel[i] = q[1 + i] * rinv;
    k += q[1 + i] * vel[i];
  }
  const T h = q[NV - 1] + (gamma - T(1)) * (q[NV - 1] - T(0.5) * k);   // rho E + p
  T pb = T(0), Eb = T(0), uu = T(0);
#pragma unroll
  for (int j = 0; j < ND; ++j) {
    pb += fb[j][1 + j] + fb[j][NV - 1] * vel[j];
    Eb += fb[j][NV - 1] * vel[j];
    T x = fb[j][NV - 1] * h;
#pragma unroll
    for (int i = 0; i < ND; ++i) x += fb[j][1 + i] * q[1 + i];
    ub[j] = x;
  }
  const T g1p = (gamma - T(1)) * pb;
#pragma unroll
  for (int i = 0; i < ND; ++i) {
    T x = fb[i][0] - g1p * vel[i] + ub[i] * rinv;
#pragma unroll
    for (int j = 0; j < ND; ++j) x += fb[j][1 + i] * vel[j];
    qb[1 + i] += x;
    uu += vel[i] * (T(0.5) * g1p * vel[i] - ub[i] * rinv);
  }
  qb[0] += uu;
  qb[NV - 1] += Eb + g1p;
}

// Transpose of the viscous flux f_v(q, G) (flux_viscous) at (q, G):
// qb += (d f_v / dq)^T fb and Gb = (d f_v / dG)^T fb.
template <int ND, typename T>
__device__ __forceinline__ void viscous_adjoint(const T* q, const T (*G)[ND + 2], const T (*fb)[ND + 2], T gamma, T mu,
                                                T kappa, T* qb, T (*Gb)[ND + 2]) {
  constexpr int NV = ND + 2;
  const T rinv = T(1) / q[0];
  T vel[ND], ub[ND], du[ND][ND], dub[ND][ND];
#pragma unroll
  for (int i = 0; i < ND; ++i) vel[i] = q[1 + i] * rinv;
  const T Es = q[NV - 1] * rinv;
#pragma unroll
  for (int i = 0; i < ND; ++i)
#pragma unroll
    for (int j = 0; j < ND; ++j) du[i][j] = (G[j][1 + i] - vel[i] * G[j][0]) * rinv;
  T div = T(0), tb = T(0);
#pragma unroll
  for (int i = 0; i < ND; ++i) {
    div += du[i][i];
    tb += fb[i][1 + i] + vel[i] * fb[i][NV - 1];
  }
  const T divb = -T(2.0 / 3.0) * mu * tb, lam = T(2.0 / 3.0) * mu * div;
#pragma unroll
  for (int i = 0; i < ND; ++i) {
    // tau_ij and its adjoint fb[j][1 + i] + u_i fb[j][E]; the energy row's u_i
    T x = T(0);
#pragma unroll
    for (int j = 0; j < ND; ++j) {
      T tau = mu * (du[i][j] + du[j][i]);
      if (i == j) tau -= lam;
      x += tau * fb[j][NV - 1];
      T b = mu * ((fb[j][1 + i] + vel[i] * fb[j][NV - 1]) + (fb[i][1 + j] + vel[j] * fb[i][NV - 1]));
      if (i == j) b += divb;
      dub[i][j] = b;
    }
    ub[i] = x;
  }
  T rb = T(0), Esb = T(0);    // rb: adjoint of log rho through every 1 / rho
#pragma unroll
  for (int j = 0; j < ND; ++j) {
    const T dEb = (gamma - T(1)) * kappa * fb[j][NV - 1];
    const T dE = (G[j][NV - 1] - Es * G[j][0]) * rinv;
    T g0 = -Es * dEb;
    rb -= dEb * dE;
    Esb -= dEb * G[j][0];
#pragma unroll
    for (int i = 0; i < ND; ++i) {
      ub[i] -= dEb * du[i][j];
      const T b = dub[i][j] - dEb * vel[i];
      Gb[j][1 + i] = b * rinv;
      g0 -= vel[i] * b;
      rb -= b * du[i][j];
      ub[i] -= b * (G[j][0] * rinv);
    }
    Gb[j][0] = g0 * rinv;
    Gb[j][NV - 1] = dEb * rinv;
  }
  Esb *= rinv;
#pragma unroll
  for (int i = 0; i < ND; ++i) {
    qb[1 + i] += ub[i] * rinv;
    rb -= ub[i] * vel[i];
  }
  rb -= Esb * Es;
  qb[NV - 1] += Esb * rinv;
  qb[0] += rb * rinv;
}

// qb += transpose of the normal flux (normal_flux) applied to fb, plus that of
// the wave speed |u.n| + c scaled by lamb.
template <int ND, typename T>
__device__ __forceinline__ void normal_flux_adjoint(const T* q, const T* n, T gamma, const T* fb, T lamb, T* qb) {
  constexpr int NV = ND + 2;
  const T rinv = T(1) / q[0];
  T mn = T(0), mu2 = T(0), x = T(0), pb = T(0);
#pragma unroll
  for (int i = 0; i < ND; ++i) {
    mn += q[1 + i] * n[i];
    mu2 += q[1 + i] * q[1 + i];
    x += fb[1 + i] * q[1 + i];
    pb += fb[1 + i] * n[i];
  }
  const T un = mn * rinv;
  const T pres = (gamma - T(1)) * (q[NV - 1] - T(0.5) * mu2 * rinv);
  T unb = x + fb[NV - 1] * (q[NV - 1] + pres), rb = T(0);
  pb += fb[NV - 1] * un;
  if (lamb != T(0)) {
    const T c = dsqrt(gamma * pres * rinv);
    const T cb = T(0.5) * lamb / c;
    unb += lamb * sign_of(un);
    pb += cb * gamma * rinv;
    rb -= T(0.5) * lamb * c;
  }
  const T g1p = (gamma - T(1)) * pb, mnb = fb[0] + unb * rinv;
#pragma unroll
  for (int i = 0; i < ND; ++i) qb[1 + i] += fb[1 + i] * un + mnb * n[i] - g1p * q[1 + i] * rinv;
  qb[NV - 1] += fb[NV - 1] * un + g1p;
  qb[0] += (rb - unb * un + T(0.5) * g1p * mu2 * rinv) * rinv;
}

// |u.n| + c as normal_flux computes it (the side of the maximum must be the one
// the forward pass took).
template <int ND, typename T>
__device__ __forceinline__ T wave_speed(const T* q, const T* n, T gamma) {
  constexpr int NV = ND + 2;
  const T rinv = T(1) / q[0];
  T mn = T(0), mu2 = T(0);
#pragma unroll
  for (int i = 0; i < ND; ++i) {
    mn += q[1 + i] * n[i];
    mu2 += q[1 + i] * q[1 + i];
  }
  const T pres = (gamma - T(1)) * (q[NV - 1] - T(0.5) * mu2 * rinv);
  return dabs(mn * rinv) + dsqrt(gamma * pres * rinv);
}

// (qLb, qRb) += (d Fn / d(qL, qR))^T Fnb of Rusanov's flux (rusanov, area included).
template <int ND, typename T>
__device__ __forceinline__ void rusanov_adjoint(const T* qL, const T* qR, const T* n, T absA, T gamma, const T* Fnb,
                                                T* qLb, T* qRb) {
  constexpr int NV = ND + 2;
  const T lamL = wave_speed<ND>(qL, n, gamma), lamR = wave_speed<ND>(qR, n, gamma);
  const bool right = lamR > lamL;     // the "-" side at a tie, as rusanov
  const T hl = T(0.5) * (right ? lamR : lamL);
  T half[NV], lamb = T(0);
#pragma unroll
  for (int v = 0; v < NV; ++v) {
    const T g = Fnb[v] * absA;
    half[v] = T(0.5) * g;
    lamb -= half[v] * (qR[v] - qL[v]);
    qLb[v] += hl * g;
    qRb[v] -= hl * g;
  }
  normal_flux_adjoint<ND>(qL, n, gamma, half, right ? T(0) : lamb, qLb);
  normal_flux_adjoint<ND>(qR, n, gamma, half, right ? lamb : T(0), qRb);
}

// The same for Roe's flux (roe): back through the wave strengths, Roe's
// averages and the two normal fluxes.
template <int ND, typename T>
__device__ __forceinline__ void roe_adjoint(const T* qL, const T* qR, const T* n, T absA, T gamma, const T* Fnb,
                                            T* qLb, T* qRb) {
  constexpr int NV = ND + 2;
  const T riL = T(1) / qL[0], riR = T(1) / qR[0];
  T uL[ND], uR[ND], kL = T(0), kR = T(0);
#pragma unroll
  for (int i = 0; i < ND; ++i) {
    uL[i] = qL[1 + i] * riL;
    uR[i] = qR[1 + i] * riR;
    kL += qL[1 + i] * uL[i];
    kR += qR[1 + i] * uR[i];
  }
  const T pL = (gamma - T(1)) * (qL[NV - 1] - T(0.5) * kL);
  const T pR = (gamma - T(1)) * (qR[NV - 1] - T(0.5) * kR);
  const T HL = (qL[NV - 1] + pL) * riL, HR = (qR[NV - 1] + pR) * riR;
  const T sL = dsqrt(qL[0]), sR = dsqrt(qR[0]);
  const T wi = T(1) / (sL + sR);
  T u[ND], du[ND], q2 = T(0), un = T(0), dun = T(0), udu = T(0);
#pragma unroll
  for (int i = 0; i < ND; ++i) {
    u[i] = (sL * uL[i] + sR * uR[i]) * wi;
    du[i] = uR[i] - uL[i];
    q2 += u[i] * u[i];
    un += u[i] * n[i];
    dun += du[i] * n[i];
    udu += u[i] * du[i];
  }
  const T H = (sL * HL + sR * HR) * wi;
  const T c2 = (gamma - T(1)) * (H - T(0.5) * q2);
  const T c = dsqrt(c2);
  const T rho = sL * sR;
  const T dp = pR - pL, drho = qR[0] - qL[0];
  const T ic2 = T(1) / c2;
  const T a1 = T(0.5) * (dp - rho * c * dun) * ic2;
  const T a3 = T(0.5) * (dp + rho * c * dun) * ic2;
  const T a2 = drho - dp * ic2;
  const T w1 = dabs(un - c), l2 = dabs(un), w3 = dabs(un + c);
  const T l1 = w1 * a1, l3 = w3 * a3;
  // adjoints of the dissipation d (Fn = (mean of the fluxes - d / 2) |A|)
  T half[NV], db[NV], dbu = T(0), dbn = T(0), dbdu = T(0);
#pragma unroll
  for (int v = 0; v < NV; ++v) {
    half[v] = T(0.5) * Fnb[v] * absA;
    db[v] = -half[v];
  }
#pragma unroll
  for (int i = 0; i < ND; ++i) {
    dbu += db[1 + i] * u[i];
    dbn += db[1 + i] * n[i];
    dbdu += db[1 + i] * du[i];
  }
  const T dE = db[NV - 1];
  const T s0 = db[0] + dbu + dE * H, s1 = dbn + dE * un;      // along (1, u, H) and (0, n, u.n)
  const T shear = dbdu - dun * dbn + dE * (udu - un * dun);
  const T l1b = s0 - c * s1, l3b = s0 + c * s1;
  const T a2b0 = db[0] + dbu + T(0.5) * dE * q2;
  const T l2b = a2 * a2b0 + rho * shear;
  T rhob = l2 * shear;
  T cb = (l3 - l1) * s1;
  T Hb = dE * (l1 + l3);
  T unb = dE * (c * (l3 - l1) - l2 * rho * dun);
  T dunb = -l2 * rho * s1;
  const T udub = l2 * rho * dE;
  T q2b = T(0.5) * l2 * a2 * dE;
  const T e1b = sign_of(un - c) * a1 * l1b, e3b = sign_of(un + c) * a3 * l3b;
  unb += e1b + e3b + sign_of(un) * l2b;
  cb += e3b - e1b;
  const T a1b = w1 * l1b, a3b = w3 * l3b, a2b = l2 * a2b0;
  T dpb = T(0.5) * ic2 * (a1b + a3b) - a2b * ic2;
  const T tb = T(0.5) * ic2 * (a3b - a1b);                     // adjoint of rho c dun
  rhob += tb * c * dun;
  cb += tb * rho * dun;
  dunb += tb * rho * c;
  const T ic2b = (a1b * a1 + a3b * a3) * c2 - a2b * dp;
  const T c2b = T(0.5) * cb / c - ic2b * ic2 * ic2;
  Hb += (gamma - T(1)) * c2b;
  q2b -= T(0.5) * (gamma - T(1)) * c2b;
  T uLb[ND], uRb[ND], sLb = Hb * (HL - H), sRb = Hb * (HR - H);
#pragma unroll
  for (int i = 0; i < ND; ++i) {
    const T ub = (l1 + l3 + l2 * a2) * db[1 + i] + udub * du[i] + unb * n[i] + T(2) * q2b * u[i];
    const T dub = l2 * rho * db[1 + i] + udub * u[i] + dunb * n[i];
    uLb[i] = ub * sL * wi - dub;
    uRb[i] = ub * sR * wi + dub;
    sLb += ub * (uL[i] - u[i]);
    sRb += ub * (uR[i] - u[i]);
  }
  sLb = sLb * wi + rhob * sR;
  sRb = sRb * wi + rhob * sL;
  auto side = [&](const T* q, const T* us, const T* usb, T ri, T p, T s, T sb, T Hsb, T pb, T rb, T* qb) {
    T rib = Hsb * (q[NV - 1] + p);
    const T pbt = pb + Hsb * ri;
    const T kb = -T(0.5) * (gamma - T(1)) * pbt;
#pragma unroll
    for (int i = 0; i < ND; ++i) {
      const T ub = usb[i] + kb * q[1 + i];
      qb[1 + i] += kb * us[i] + ub * ri;
      rib += ub * q[1 + i];
    }
    qb[NV - 1] += Hsb * ri + (gamma - T(1)) * pbt;
    qb[0] += rb + T(0.5) * sb / s - rib * ri * ri;
  };
  side(qL, uL, uLb, riL, pL, sL, sLb, Hb * sL * wi, -dpb, -a2b, qLb);
  side(qR, uR, uRb, riR, pR, sR, sRb, Hb * sR * wi, dpb, a2b, qRb);
  normal_flux_adjoint<ND>(qL, n, gamma, half, T(0), qLb);
  normal_flux_adjoint<ND>(qR, n, gamma, half, T(0), qRb);
}

template <int ND, typename T>
__device__ __forceinline__ void flux_adjoint(int kind, const T* qL, const T* qR, const T* n, T absA, T gamma,
                                             const T* Fnb, T* qLb, T* qRb) {
  if (kind == 1) roe_adjoint<ND>(qL, qR, n, absA, gamma, Fnb, qLb, qRb);
  else rusanov_adjoint<ND>(qL, qR, n, absA, gamma, Fnb, qLb, qRb);
}

// ---------------------------------------------------------------------------
// Primal jumps dq = q^com - q on every face (Navier-Stokes): all that the
// volume adjoint needs of the forward face pass.  Same CTAs as face_kernel;
// mixed groups stage the slave's q traces and project q^com back.
// ---------------------------------------------------------------------------
template <typename T, int ND>
__global__ void __launch_bounds__(kFaceThreads) jump_kernel(const __grid_constant__ FaceMulti<T> m) {
  constexpr int NV = ND + 2;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  int gi = 0;
  while (gi + 1 < m.ng && (int)blockIdx.x >= m.g[gi + 1].block0) ++gi;
  const FaceGroupRef& g = m.g[gi];
  const int Pm = g.Pm, Ps = g.Ps;
  const int NFPm = ND == 2 ? Pm : Pm * Pm;
  const int NFPs = ND == 2 ? Ps : Ps * Ps;
  const int lf = threadIdx.x / NFPm, t = threadIdx.x - lf * NFPm;
  const int64_t f0 = (int64_t)((int)blockIdx.x - g.block0) * g.fb;
  const bool valid = lf < g.fb && f0 + lf < g.n;
  T qM[NV], qG[NV];
  if (g.kind != 0) {
    if (!valid) return;
    const BndRec r = g.brecs[f0 + lf];
    load_trace_pt<ND>(m.trq, (const T*)nullptr, r.mt, 0, NV, NFPm, t, qM);
    ghost_state<ND>(qM, g.kind, m.qinf, qG);
#pragma unroll
    for (int v = 0; v < NV; ++v) m.fout[r.mo + (int64_t)(NV + v) * NFPm + t] = T(0.5) * (qM[v] + qG[v]) - qM[v];
    return;
  }
  FaceRec r{};
  if (valid) {
    r = g.recs[f0 + lf];
    load_trace_pt<ND>(m.trq, (const T*)nullptr, m.ct ? r.mt / m.nvt * m.ct : r.mt, 0, NV, NFPm, t, qM);
  }
  if (Pm == Ps) {
    if (!valid) return;
    const int u = orient_map(r.orient, t, Pm, ND);
    load_trace_pt<ND>(m.trq, (const T*)nullptr, m.ct ? r.st / m.nvt * m.ct : r.st, 0, NV, NFPs, u, qG);
#pragma unroll
    for (int v = 0; v < NV; ++v) {
      const T qc = T(0.5) * (qM[v] + qG[v]);
      m.fout[r.mo + (int64_t)(NV + v) * NFPm + t] = qc - qM[v];
      m.fout[r.so + (int64_t)(NV + v) * NFPs + u] = qc - qG[v];
    }
    return;
  }
  const MortarTab<T>& mt = m.mortar[Pm * (kPM + 1) + Ps];
  T* const sm = reinterpret_cast<T*>(smem_raw);
  const int fstride = NV * NFPm;
  const int nfaces = (int)min((int64_t)g.fb, (int64_t)g.n - f0), per = NV * NFPs;
  for (int k = threadIdx.x; k < nfaces * per; k += kFaceThreads) {
    const int f = k / per, o = k - f * per;
    sm[f * fstride + o] = m.trq[g.recs[f0 + f].st + o];
  }
  __syncthreads();
  const int u = valid ? orient_map(r.orient, t, Pm, ND) : 0;
  if (valid) {
    staged_at_mortar<ND, NV, 0>(sm + lf * fstride, (const T*)nullptr, mt, Ps, NFPs, u % Pm, ND == 2 ? 0 : u / Pm, qG);
#pragma unroll
    for (int v = 0; v < NV; ++v) {
      qG[v] = T(0.5) * (qM[v] + qG[v]);
      m.fout[r.mo + (int64_t)(NV + v) * NFPm + t] = qG[v] - qM[v];
    }
  }
  __syncthreads();
  if (valid) {
#pragma unroll
    for (int v = 0; v < NV; ++v) sm[lf * fstride + v * NFPm + u] = qG[v];
  }
  __syncthreads();
  const int lp = threadIdx.x / NFPs, pt = threadIdx.x - lp * NFPs;
  if (lp >= g.fb || f0 + lp >= g.n) return;
  const FaceRec rp = g.recs[f0 + lp];
  T acc[NV];
#pragma unroll
  for (int v = 0; v < NV; ++v) acc[v] = T(0);
  for (int mb = 0; mb < (ND == 2 ? 1 : Pm); ++mb) {
    const T wb = ND == 2 ? T(1) : mt.Pi[pt / Ps][mb];
    for (int ma = 0; ma < Pm; ++ma) {
      const T w = mt.Pi[pt % Ps][ma] * wb;
#pragma unroll
      for (int v = 0; v < NV; ++v) acc[v] += w * sm[lp * fstride + v * NFPm + ma + Pm * mb];
    }
  }
#pragma unroll
  for (int v = 0; v < NV; ++v)
    m.fout[rp.so + (int64_t)(NV + v) * NFPs + pt] = acc[v] - m.trq[rp.st + (int64_t)v * NFPs + pt];
}

// ---------------------------------------------------------------------------
// Volume adjoint.  One thread per solution point, epb elements per block.
// ---------------------------------------------------------------------------
template <typename T>
struct VolAdjArgs {
  const T* q;
  const T* w;
  T* out;              // partial q-bar (volume terms)
  const T* fout;       // primal jumps dq
  T* fbar;             // adjoints of F~^com and dq
  const int32_t* slot_elem;
  const BasisTab<T>* basis;
  GeoView<T> geo;
  T gamma, mu, kappa;
  int64_t state_base, out_base;
  int count, slot_begin;
};

// Adjoints of the values lifted from the faces of direction d: sums along every
// line with g_L' and g_R', one thread per line.  src(d): [NV][NSP] in shared
// memory; written to component c0 + v of the line's two faces.
template <typename T, int ND, int P, typename F>
__device__ __forceinline__ void face_line_sums(F src, const BasisTab<T>& B, T* fb, int c0, int lt) {
  using Sh = Shape<ND, P>;
  constexpr int NV = Sh::NV, NSP = Sh::NSP, NFP = Sh::NFP, FS = 3 * NV * NFP;
  for (int l = lt; l < ND * NFP; l += NSP) {
    const int d = l / NFP, t = l - d * NFP;
    const int base = line_sp<ND, P>(d, t, 0), stride = d == 0 ? 1 : (d == 1 ? P : P * P);
    const T* x = src(d) + base;
#pragma unroll
    for (int v = 0; v < NV; ++v) {
      T g0 = T(0), g1 = T(0);
#pragma unroll
      for (int k = 0; k < P; ++k) {
        const T y = x[v * NSP + k * stride];
        g0 += B.dg[0][k] * y;
        g1 += B.dg[1][k] * y;
      }
      fb[(2 * d + 0) * FS + (c0 + v) * NFP + t] = g0;
      fb[(2 * d + 1) * FS + (c0 + v) * NFP + t] = g1;
    }
  }
}

// DIAG: every metric S is diagonal (see trace_body).
// FP32: bound by the L1 data pipe (84 % of it at 20^3, p = 4, a third of the
// warps, which wait on their loads).  Three CTAs an SM for diagonal metrics from
// p = 2 (box, p = 2 / 3 / 5, 8.6-10.5M DOF: 119 / 124 / 145 us, with two 129 / 135 /
// 158); two at p = 1 (190, with three 195) and for full metrics, which need the
// registers (O-grid, p = 1..4: 81 us in all, with three 86).
template <typename T, int ND, int P, bool VISC, bool DIAG>
__global__ void __launch_bounds__(256, sizeof(T) != 4 ? 1 : (DIAG && P > 2 ? 3 : 2)) vol_adj_kernel(VolAdjArgs<T> a, int epb) {
  using Sh = Shape<ND, P>;
  constexpr int NV = Sh::NV, NF = Sh::NF, NSP = Sh::NSP, NFP = Sh::NFP;
  constexpr int FS = 3 * NV * NFP;
  constexpr int PER = (VISC ? 2 * NV + ND * NV : NV) * NSP;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  T* sm = reinterpret_cast<T*>(smem_raw);
  const int le = threadIdx.x / NSP;
  const int sp = threadIdx.x % NSP;
  const int64_t i = (int64_t)blockIdx.x * epb + le;
  const bool valid = le < epb && i < a.count;
  T* sdb = sm + le * PER;                            // div-bar [NV][NSP]
  T* sq = sdb + NV * NSP;                            // [NV][NSP]
  T* sgb = sq + NV * NSP;                            // gref-bar [ND][NV][NSP]
  const BasisTab<T>& B = a.basis[P];
  int idx[3];
  idx[0] = sp % P;
  idx[1] = (sp / P) % P;
  idx[2] = ND == 3 ? sp / (P * P) : 0;
  const int64_t e = valid ? a.slot_elem[a.slot_begin + i] : 0;
  const T* fo = a.fout + (valid ? a.out_base + i * NF * FS : 0);
  T* fb = a.fbar + (valid ? a.out_base + i * NF * FS : 0);

  T q[NV];
  T Sm[ND][ND];
  T Jinv = T(1);
  if (valid) {
#pragma unroll
    for (int d = 0; d < ND; ++d)
#pragma unroll
      for (int j = 0; j < ND; ++j) Sm[d][j] = (DIAG && d != j) ? T(0) : geo_vol(a.geo, e, d * ND + j, sp);
    Jinv = geo_vol(a.geo, e, ND * ND + 1, sp);
#pragma unroll
    for (int v = 0; v < NV; ++v) {
      q[v] = a.q[a.state_base + (i * NV + v) * NSP + sp];
      if (VISC) sq[v * NSP + sp] = q[v];
      sdb[v * NSP + sp] = -a.w[a.state_base + (i * NV + v) * NSP + sp] * Jinv;
    }
  }
  __syncthreads();

  T qb[NV];
#pragma unroll
  for (int v = 0; v < NV; ++v) qb[v] = T(0);
  if (valid) {
    face_line_sums<T, ND, P>([&](int) { return sdb; }, B, fb, 0, sp);
    // adjoint of the physical fluxes: S^T (Dh^T div-bar)
    T fbar[ND][NV];
    {
      T Fb[ND][NV];
#pragma unroll
      for (int d = 0; d < ND; ++d) {
        const int stride = d == 0 ? 1 : (d == 1 ? P : P * P);
        const int base = sp - idx[d] * stride;
#pragma unroll
        for (int v = 0; v < NV; ++v) {
          T acc = T(0);
#pragma unroll
          for (int k = 0; k < P; ++k) acc += B.Dh[k][idx[d]] * sdb[v * NSP + base + k * stride];
          Fb[d][v] = acc;
        }
      }
#pragma unroll
      for (int j = 0; j < ND; ++j)
#pragma unroll
        for (int v = 0; v < NV; ++v) {
          if (DIAG) {
            fbar[j][v] = Sm[j][j] * Fb[j][v];
          } else {
            T acc = T(0);
#pragma unroll
            for (int d = 0; d < ND; ++d) acc += Sm[d][j] * Fb[d][v];
            fbar[j][v] = acc;
          }
        }
    }
    inviscid_adjoint<ND>(q, fbar, a.gamma, qb);
    if (VISC) {
      T G[ND][NV];
      {
        T gref[ND][NV];
#pragma unroll
        for (int d = 0; d < ND; ++d) {
          const int stride = d == 0 ? 1 : (d == 1 ? P : P * P);
          const int base = sp - idx[d] * stride;
          const int tf = face_pt<ND, P>(d, idx);
#pragma unroll
          for (int v = 0; v < NV; ++v) {
            T acc = T(0);
#pragma unroll
            for (int k = 0; k < P; ++k) acc += B.D[idx[d]][k] * sq[v * NSP + base + k * stride];
#pragma unroll
            for (int s = 0; s < 2; ++s) acc += B.dg[s][idx[d]] * fo[(2 * d + s) * FS + (NV + v) * NFP + tf];
            gref[d][v] = acc;
          }
        }
#pragma unroll
        for (int j = 0; j < ND; ++j)
#pragma unroll
          for (int v = 0; v < NV; ++v) {
            if (DIAG) {
              G[j][v] = (Sm[j][j] * Jinv) * gref[j][v];
            } else {
              T acc = T(0);
#pragma unroll
              for (int d = 0; d < ND; ++d) acc += Sm[d][j] * gref[d][v];
              G[j][v] = acc * Jinv;
            }
          }
      }
      T Gb[ND][NV];
#pragma unroll
      for (int j = 0; j < ND; ++j)
#pragma unroll
        for (int v = 0; v < NV; ++v) fbar[j][v] = -fbar[j][v];     // f = f_inv - f_v
      viscous_adjoint<ND>(q, G, fbar, a.gamma, a.mu, a.kappa, qb, Gb);
#pragma unroll
      for (int d = 0; d < ND; ++d)
#pragma unroll
        for (int v = 0; v < NV; ++v) {
          T acc = T(0);
          if (DIAG) {
            acc = Sm[d][d] * Gb[d][v];
          } else {
#pragma unroll
            for (int j = 0; j < ND; ++j) acc += Sm[d][j] * Gb[j][v];
          }
          sgb[(d * NV + v) * NSP + sp] = acc * Jinv;
        }
    }
  }
  if (VISC) __syncthreads();
  if (!valid) return;
  if (VISC) {
    face_line_sums<T, ND, P>([&](int d) { return sgb + d * NV * NSP; }, B, fb, NV, sp);
#pragma unroll
    for (int d = 0; d < ND; ++d) {
      const int stride = d == 0 ? 1 : (d == 1 ? P : P * P);
      const int base = sp - idx[d] * stride;
#pragma unroll
      for (int v = 0; v < NV; ++v) {
        const T* line = sgb + (d * NV + v) * NSP + base;
        T acc = T(0);
#pragma unroll
        for (int k = 0; k < P; ++k) acc += B.D[k][idx[d]] * line[k * stride];
        qb[v] += acc;
      }
    }
  }
#pragma unroll
  for (int v = 0; v < NV; ++v) a.out[a.state_base + (i * NV + v) * NSP + sp] = qb[v];
}

// ---------------------------------------------------------------------------
// Face adjoint: every face in one launch, the CTAs of face_kernel (whole faces,
// one thread per mortar point).
// ---------------------------------------------------------------------------
template <typename T>
struct FaceAdjMulti {
  FaceMulti<T> f;      // trq: the primal traces; fout unused
  const T* fbar;       // adjoints of the face outputs
  T* trbar;            // adjoints of the traces
};

// Shared memory of one face, in values.  B: the tangential derivatives'
// adjoints of the master's side (and, conforming, of the slave's).  A (mixed):
// the slave's staged traces, lifting coefficients and face-output adjoints,
// then the mortar values of the slave's adjoints.
template <int ND, bool VISC>
struct AdjFace {
  static constexpr int NV = ND + 2;
  static constexpr int NT = VISC ? NV * (1 + ND) : NV;       // trace components, and adjoints of them
  static constexpr int NB = VISC ? 2 * NV : NV;              // face-output adjoints
  static constexpr int TG = VISC ? (ND - 1) * NV : 0;        // tangential adjoints
  __host__ __device__ static int a_size(int NFPm, int NFPs) {
    if (NFPm == NFPs) return 0;
    const int in = (NT + (VISC ? ND : 0) + NB) * NFPs, out = NT * NFPm;
    return in > out ? in : out;
  }
  __host__ __device__ static int stride(int NFPm, int NFPs) {
    return a_size(NFPm, NFPs) + (NFPm == NFPs ? 2 : 1) * TG * NFPm;
  }
};

// Reference-derivative adjoints at point t of face f from the physical-gradient
// adjoints: the normal direction's to nb, the tangential ones to shared memory
// [tangential axis][NV][NFP].
template <int ND, bool DIAG, typename T>
__device__ __forceinline__ void ref_adjoint(const GeoView<T>& g, int64_t e, int f, int t, int NFP, const T (*Gb)[ND + 2],
                                            T* nb, T* tang) {
  constexpr int NV = ND + 2;
  const T Jinv = geo_face(g, e, f, ND * ND + 1, t);
  const int dn = f >> 1;
#pragma unroll
  for (int d = 0; d < ND; ++d) {
    T row[ND];
#pragma unroll
    for (int j = 0; j < ND; ++j) row[j] = (DIAG && d != j) ? T(0) : geo_face(g, e, f, d * ND + j, t) * Jinv;
    const int slot = d > dn ? d - 1 : d;
#pragma unroll
    for (int v = 0; v < NV; ++v) {
      T acc = T(0);
      if (DIAG) {
        acc = row[d] * Gb[d][v];
      } else {
#pragma unroll
        for (int j = 0; j < ND; ++j) acc += row[j] * Gb[j][v];
      }
      if (d == dn) nb[v] = acc;
      else tang[(slot * NV + v) * NFP + t] = acc;
    }
  }
}

// One side's trace adjoints at its point t: the value's, with the transposed
// tangential differentiation of the face's tangential adjoints, and the normal
// derivative's.
template <int ND, bool VISC, typename T>
__device__ __forceinline__ void store_adj_side(T* o, int P, int NFP, int t, const T* vb, const T* nb, const T* tang,
                                               const BasisTab<T>& B) {
  constexpr int NV = ND + 2;
  const int ia = t % P, ib = ND == 2 ? 0 : t / P;
  T x[NV];
#pragma unroll
  for (int v = 0; v < NV; ++v) x[v] = vb[v];
  if (VISC) {
    for (int c = 0; c < P; ++c) {
      const T wa = B.D[c][ia], wb = ND == 3 ? B.D[c][ib] : T(0);
#pragma unroll
      for (int v = 0; v < NV; ++v) {
        x[v] += wa * tang[v * NFP + c + P * ib];
        if (ND == 3) x[v] += wb * tang[(NV + v) * NFP + ia + P * c];
      }
    }
  }
#pragma unroll
  for (int v = 0; v < NV; ++v) {
    o[v * NFP + t] = x[v];
    if (VISC) o[(NV + v) * NFP + t] = nb[v];
  }
}

template <typename T, int ND, bool VISC, bool DIAG>
__global__ void __launch_bounds__(kFaceThreads, sizeof(T) == 4 ? 4 : 1)
    face_adj_kernel(const __grid_constant__ FaceAdjMulti<T> am) {
  constexpr int NV = ND + 2;
  using AF = AdjFace<ND, VISC>;
  const FaceMulti<T>& m = am.f;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  int gi = 0;
  while (gi + 1 < m.ng && (int)blockIdx.x >= m.g[gi + 1].block0) ++gi;
  const FaceGroupRef& g = m.g[gi];
  const int Pm = g.Pm, Ps = g.Ps;
  const int NFPm = ND == 2 ? Pm : Pm * Pm;
  const int NFPs = ND == 2 ? Ps : Ps * Ps;
  const int lf = threadIdx.x / NFPm, t = threadIdx.x - lf * NFPm;
  const int64_t f0 = (int64_t)((int)blockIdx.x - g.block0) * g.fb;
  const bool valid = lf < g.fb && f0 + lf < g.n;
  const bool bnd = g.kind != 0, mixed = Pm != Ps, conf = !bnd && !mixed;
  const MortarTab<T>& mt = m.mortar[Pm * (kPM + 1) + Ps];
  T* const sm = reinterpret_cast<T*>(smem_raw);
  const int fstride = AF::stride(NFPm, NFPs), asize = AF::a_size(NFPm, NFPs);
  FaceRec r{};
  if (valid) {
    if (bnd) {
      const BndRec b = g.brecs[f0 + lf];
      r.mt = b.mt;
      r.mo = b.mo;
      r.me = b.me;
      r.mf = b.mf;
    } else {
      r = g.recs[f0 + lf];
    }
  }
  if (mixed) {
    const int nfaces = (int)min((int64_t)g.fb, (int64_t)g.n - f0);
    const int pq = AF::NT * NFPs, pb = AF::NB * NFPs;
    for (int k = threadIdx.x; k < nfaces * pq; k += kFaceThreads) {
      const int f = k / pq, o = k - f * pq;
      sm[f * fstride + o] = m.trq[g.recs[f0 + f].st + o];
    }
    for (int k = threadIdx.x; k < nfaces * pb; k += kFaceThreads) {
      const int f = k / pb, o = k - f * pb;
      sm[f * fstride + pq + o] = am.fbar[g.recs[f0 + f].so + o];
    }
    if (VISC) {
      const GeoView<T>& gs = m.geo[Ps];
      for (int k = threadIdx.x; k < nfaces * NFPs; k += kFaceThreads) {
        const int f = k / NFPs, pt = k - f * NFPs;
        const int64_t e = g.recs[f0 + f].se;
        const int sf = g.recs[f0 + f].sf;
        const T gJ = m.basis[Ps].dgf[sf & 1] * geo_face(gs, e, sf, ND * ND + 1, pt);
        T* c = sm + f * fstride + pq + pb;
#pragma unroll
        for (int j = 0; j < ND; ++j) c[j * NFPs + pt] = gJ * geo_face(gs, e, sf, (sf >> 1) * ND + j, pt);
      }
    }
    __syncthreads();
  }
  T qMb[NV], qSb[NV], nM[NV], nS[NV], Gb[ND][NV];
  T* const tangM = sm + lf * fstride + asize;
  T* const tangS = tangM + AF::TG * NFPm;     // conforming faces
  int u = 0;
  const T* const sq = sm + lf * fstride;      // staged slave (mixed)
  if (valid) {
    const int dm = r.mf >> 1, sm_ = r.mf & 1, ss = r.sf & 1;
    const GeoView<T>& geo_m = m.geo[Pm];
    if (!bnd) u = orient_map(r.orient, t, Pm, ND);
    const int ua = u % Pm, ub = ND == 2 ? 0 : u / Pm;
    T qM[NV], qS[NV];
    load_trace_pt<ND>(m.trq, (const T*)nullptr, r.mt, 0, NV, NFPm, t, qM);
    if (bnd) ghost_state<ND>(qM, g.kind, m.qinf, qS);
    else if (mixed) staged_at_mortar<ND, NV, 0>(sq, (const T*)nullptr, mt, Ps, NFPs, ua, ub, qS);
    else load_trace_pt<ND>(m.trq, (const T*)nullptr, r.st, 0, NV, NFPs, u, qS);
    T A[ND], n[ND];
    const T sgm = sm_ ? T(1) : T(-1), sgs = ss ? T(1) : T(-1);
    const T absA = geo_face(geo_m, r.me, r.mf, ND * ND + 2 + dm, t);
    const T inv_absA = geo_face(geo_m, r.me, r.mf, ND * ND + 2 + ND + dm, t);
#pragma unroll
    for (int j = 0; j < ND; ++j) {
      A[j] = sgm * geo_face(geo_m, r.me, r.mf, dm * ND + j, t);
      n[j] = A[j] * inv_absA;
    }
    // seeds: adjoints of the common flux, of q^com and of the two sides' q
    T Fnb[NV], qcb[NV];
    const T* fbm = am.fbar + r.mo;
#pragma unroll
    for (int v = 0; v < NV; ++v) {
      Fnb[v] = sgm * fbm[v * NFPm + t];
      qcb[v] = VISC ? fbm[(NV + v) * NFPm + t] : T(0);
      qMb[v] = VISC ? -qcb[v] : T(0);
      qSb[v] = T(0);
    }
    if (conf) {
      const T* fbs = am.fbar + r.so;
#pragma unroll
      for (int v = 0; v < NV; ++v) {
        Fnb[v] -= sgs * fbs[v * NFPs + u];
        if (VISC) {
          const T x = fbs[(NV + v) * NFPs + u];
          qcb[v] += x;
          qSb[v] -= x;
        }
      }
    } else if (mixed) {
      // transpose of the L2 projection onto the slave side
      const T* fbs = sq + AF::NT * NFPs;
      for (int pb = 0; pb < (ND == 2 ? 1 : Ps); ++pb) {
        const T wb = ND == 2 ? T(1) : mt.Pi[pb][ub];
        for (int pa = 0; pa < Ps; ++pa) {
          const T w = mt.Pi[pa][ua] * wb;
          const int pt = pa + Ps * pb;
#pragma unroll
          for (int v = 0; v < NV; ++v) {
            Fnb[v] -= sgs * w * fbs[v * NFPs + pt];
            if (VISC) qcb[v] += w * fbs[(NV + v) * NFPs + pt];
          }
        }
      }
    }
    flux_adjoint<ND>(m.flux, qM, qS, n, absA, m.gamma, Fnb, qMb, qSb);
    if (VISC) {
      T qc[NV], cM[ND], cS[ND];
#pragma unroll
      for (int v = 0; v < NV; ++v) qc[v] = T(0.5) * (qM[v] + qS[v]);
      const T gJ = m.basis[Pm].dgf[sm_] * geo_face(geo_m, r.me, r.mf, ND * ND + 1, t);
#pragma unroll
      for (int j = 0; j < ND; ++j) {
        cM[j] = gJ * geo_face(geo_m, r.me, r.mf, dm * ND + j, t);
        cS[j] = T(0);
      }
      T G[ND][NV];
      load_trace_pt<ND>(m.trq, (const T*)nullptr, r.mt, NV, ND * NV, NFPm, t, &G[0][0]);
      if (bnd) {
#pragma unroll
        for (int j = 0; j < ND; ++j)
#pragma unroll
          for (int v = 0; v < NV; ++v) G[j][v] += cM[j] * (qc[v] - qM[v]);
      } else {
        T GS[ND][NV];
        if (mixed) {
          staged_at_mortar<ND, ND, 0>(sq + (AF::NT + AF::NB) * NFPs, (const T*)nullptr, mt, Ps, NFPs, ua, ub, cS);
          staged_at_mortar<ND, ND * NV, 0>(sq + NV * NFPs, (const T*)nullptr, mt, Ps, NFPs, ua, ub, &GS[0][0]);
        } else {
          const GeoView<T>& geo_s = m.geo[Ps];
          const T gJs = m.basis[Ps].dgf[ss] * geo_face(geo_s, r.se, r.sf, ND * ND + 1, u);
#pragma unroll
          for (int j = 0; j < ND; ++j) cS[j] = gJs * geo_face(geo_s, r.se, r.sf, (r.sf >> 1) * ND + j, u);
          load_trace_pt<ND>(m.trq, (const T*)nullptr, r.st, NV, ND * NV, NFPs, u, &GS[0][0]);
        }
#pragma unroll
        for (int j = 0; j < ND; ++j)
#pragma unroll
          for (int v = 0; v < NV; ++v)
            G[j][v] = T(0.5) * (G[j][v] + cM[j] * (qc[v] - qM[v]) + GS[j][v] + cS[j] * (qc[v] - qS[v]));
      }
      // Fn -= sum_j f_v(q^com, G)[j] A_j (no energy flux through an adiabatic wall)
      T fvb[ND][NV];
#pragma unroll
      for (int j = 0; j < ND; ++j)
#pragma unroll
        for (int v = 0; v < NV; ++v) fvb[j][v] = (bnd && g.kind == -1 && v == NV - 1) ? T(0) : -Fnb[v] * A[j];
      viscous_adjoint<ND>(qc, G, fvb, m.gamma, m.mu, m.kappa, qcb, Gb);
      const T h = bnd ? T(1) : T(0.5);        // a boundary's gradient is the interior one alone
#pragma unroll
      for (int v = 0; v < NV; ++v) {
        T sM = T(0), sS = T(0);
#pragma unroll
        for (int j = 0; j < ND; ++j) {
          Gb[j][v] *= h;
          sM += cM[j] * Gb[j][v];
          sS += cS[j] * Gb[j][v];
        }
        qcb[v] += sM + sS;
        qMb[v] += T(0.5) * qcb[v] - sM;
        qSb[v] += T(0.5) * qcb[v] - sS;
      }
      ref_adjoint<ND, DIAG>(geo_m, r.me, r.mf, t, NFPm, Gb, nM, tangM);
      if (conf) ref_adjoint<ND, DIAG>(m.geo[Ps], r.se, r.sf, u, NFPs, Gb, nS, tangS);
    }
    // ghost-state transpose: the wall reverses momentum; the far-field state is constant
    if (bnd && g.kind == -1) {
      qMb[0] += qSb[0];
#pragma unroll
      for (int i = 0; i < ND; ++i) qMb[1 + i] -= qSb[1 + i];
      qMb[NV - 1] += qSb[NV - 1];
    }
  }
  if (VISC || mixed) __syncthreads();     // tangential adjoints written; staged traces read
  if (valid) {
    store_adj_side<ND, VISC>(am.trbar + r.mt, Pm, NFPm, t, qMb, nM, tangM, m.basis[Pm]);
    if (conf) store_adj_side<ND, VISC>(am.trbar + r.st, Ps, NFPs, u, qSb, nS, tangS, m.basis[Ps]);
    if (mixed) {
      T* sc = sm + lf * fstride + u;
#pragma unroll
      for (int v = 0; v < NV; ++v) sc[v * NFPm] = qSb[v];
      if (VISC) {
#pragma unroll
        for (int j = 0; j < ND; ++j)
#pragma unroll
          for (int v = 0; v < NV; ++v) sc[(NV + j * NV + v) * NFPm] = Gb[j][v];
      }
    }
  }
  if (!mixed) return;
  // the slave's side: transpose of its interpolation to the mortar, plus the
  // direct -dq-bar term, one thread per (face, slave point)
  __syncthreads();
  const int lp = threadIdx.x / NFPs, pt = threadIdx.x - lp * NFPs;
  const bool vp = lp < g.fb && f0 + lp < g.n;
  FaceRec rp{};
  T* const tang = sm + lp * fstride + asize;   // the master's tangential adjoints, read before the barrier above
  if (vp) {
    rp = g.recs[f0 + lp];
    const int pa = pt % Ps, pb = ND == 2 ? 0 : pt / Ps;
    const T* sc = sm + lp * fstride;
#pragma unroll
    for (int v = 0; v < NV; ++v) qSb[v] = VISC ? -am.fbar[rp.so + (int64_t)(NV + v) * NFPs + pt] : T(0);
    if (VISC) {
#pragma unroll
      for (int j = 0; j < ND; ++j)
#pragma unroll
        for (int v = 0; v < NV; ++v) Gb[j][v] = T(0);
    }
    for (int mb = 0; mb < (ND == 2 ? 1 : Pm); ++mb) {
      const T wb = ND == 2 ? T(1) : mt.I[mb][pb];
      for (int ma = 0; ma < Pm; ++ma) {
        const T w = mt.I[ma][pa] * wb;
        const int k = ma + Pm * mb;
#pragma unroll
        for (int v = 0; v < NV; ++v) qSb[v] += w * sc[v * NFPm + k];
        if (VISC) {
#pragma unroll
          for (int j = 0; j < ND; ++j)
#pragma unroll
            for (int v = 0; v < NV; ++v) Gb[j][v] += w * sc[(NV + j * NV + v) * NFPm + k];
        }
      }
    }
    if (VISC) ref_adjoint<ND, DIAG>(m.geo[Ps], rp.se, rp.sf, pt, NFPs, Gb, nS, tang);
  }
  if (VISC) __syncthreads();
  if (vp) store_adj_side<ND, VISC>(am.trbar + rp.st, Ps, NFPs, pt, qSb, nS, tang, m.basis[Ps]);
}

// Compact face adjoint (viscous, diagonal metrics, conforming faces; the
// transpose of the compact face passes): both sides' compact traces and
// face-output adjoints in, the tangential part of the common gradient taken
// from q^com (common_gradient) and transposed once a face.  24^3, p = 4, FP32:
// traces 81 -> 27 us, jumps 26 -> 24, face adjoint 121 -> 87 (VJP 384 -> 296); 12^3, FP64,
// traces 81 -> 32, face adjoint 183 -> 162.
template <typename T, int ND, int P>
__global__ void __launch_bounds__(128, sizeof(T) == 4 ? 4 : 2)
    cface_adj_kernel(CFaceArgs<T> a, const T* __restrict__ fbar, T* __restrict__ trbar) {
  constexpr int NV = ND + 2, NFP = ND == 2 ? P : P * P, CT = 2 * NV;
  constexpr int FB = NFP >= 128 ? 1 : 128 / NFP, SC = NV * NFP, ST = (ND - 1) * NV * NFP;
  __shared__ __align__(16) T sqc[FB * SC];
  __shared__ __align__(16) T stang[FB * ST];
  const int lf = threadIdx.x / NFP, t = threadIdx.x % NFP;
  const int64_t fidx = (int64_t)blockIdx.x * FB + lf;
  const bool valid = lf < FB && fidx < a.n;
  T* const qcs = sqc + min(lf, FB - 1) * SC;
  T* const tang = stang + min(lf, FB - 1) * ST;
  const BasisTab<T>& B = a.basis[P];
  FaceRec r{};
  CFaceGeo<T, ND> g{};
  T qM[NV], qS[NV], qMb[NV], qSb[NV], qcb[NV], nM[NV], nS[NV];
  const T *xm = nullptr, *xs = nullptr;
  if (valid) {
    r = a.recs[fidx];
    cface_geo<T, ND, P, true>(a, r, t, g);
    xm = a.trq + r.mt / a.nvt * CT + t;
    xs = a.trq + r.st / a.nvt * CT + g.u;
#pragma unroll
    for (int v = 0; v < NV; ++v) {
      qM[v] = xm[v * NFP];
      qS[v] = xs[v * NFP];
    }
    cface_common<ND, P, true, true, 0>(qM, qS, t, qcs);
  }
  cface_sync<ND, P, true, true>();
  if (valid) {
    const int dm = r.mf >> 1, sm = r.mf & 1, ss = r.sf & 1;
    const T sgm = sm ? T(1) : T(-1), sgs = ss ? T(1) : T(-1);
    T n[ND], Ad = T(0), h[ND], hM = T(0), hS = T(0);
#pragma unroll
    for (int j = 0; j < ND; ++j) {
      const T A = sgm * g.rowM[j];
      n[j] = A * g.inv_absA;
      h[j] = g.SfM[j][j] * g.JiM;
      if (j == dm) {
        Ad = A;
        hM = h[j];
        hS = g.SfS[j][j] * g.JiS;
      }
    }
    const T* fm = fbar + r.mo + t;
    const T* fs = fbar + r.so + g.u;
    T Fnb[NV];
#pragma unroll
    for (int v = 0; v < NV; ++v) {
      const T x = fm[(NV + v) * NFP], y = fs[(NV + v) * NFP];
      Fnb[v] = sgm * fm[v * NFP] - sgs * fs[v * NFP];
      qcb[v] = x + y;
      qMb[v] = -x;
      qSb[v] = -y;
    }
    flux_adjoint<ND>(a.flux, qM, qS, n, g.absA, a.gamma, Fnb, qMb, qSb);
    T qc[NV], dnM[NV], dnS[NV], Gc[ND][NV], fvb[ND][NV], Gcb[ND][NV];
#pragma unroll
    for (int v = 0; v < NV; ++v) {
      qc[v] = T(0.5) * (qM[v] + qS[v]);
      dnM[v] = xm[(NV + v) * NFP];
      dnS[v] = xs[(NV + v) * NFP];
    }
    common_gradient<T, ND, P, 0>(B, g, dm, t, B.dgf[sm], B.dgf[ss], qM, qS, qc, dnM, dnS, qcs, Gc);
#pragma unroll
    for (int j = 0; j < ND; ++j)
#pragma unroll
      for (int v = 0; v < NV; ++v) fvb[j][v] = j == dm ? -Fnb[v] * Ad : T(0);
    viscous_adjoint<ND>(qc, Gc, fvb, a.gamma, a.mu, a.kappa, qcb, Gcb);
    const T cM = B.dgf[sm] * hM, cS = B.dgf[ss] * hS;
#pragma unroll
    for (int v = 0; v < NV; ++v) {
      T gn = T(0);
#pragma unroll
      for (int j = 0; j < ND; ++j) {
        if (j == dm) gn = T(0.5) * Gcb[j][v];
        else tang[((j > dm ? j - 1 : j) * NV + v) * NFP + t] = h[j] * Gcb[j][v];
      }
      nM[v] = hM * gn;
      nS[v] = hS * gn;
      qcb[v] += (cM + cS) * gn;
      qMb[v] -= cM * gn;
      qSb[v] -= cS * gn;
    }
  }
  cface_sync<ND, P, true, true>();
  if (!valid) return;
  const int ia = t % P, ib = ND == 3 ? t / P : 0;
  T* om = trbar + r.mt + t;
  T* os = trbar + r.st + g.u;
  T wa[P], wb[P];
#pragma unroll
  for (int c = 0; c < P; ++c) {
    wa[c] = B.D[c][ia];
    wb[c] = ND == 3 ? B.D[c][ib] : T(0);
  }
#pragma unroll
  for (int v = 0; v < NV; ++v) {
    T x = qcb[v];
#pragma unroll
    for (int c = 0; c < P; ++c) {
      x += wa[c] * tang[v * NFP + c + P * ib];
      if (ND == 3) x += wb[c] * tang[(NV + v) * NFP + ia + P * c];
    }
    om[v * NFP] = qMb[v] + T(0.5) * x;
    om[(NV + v) * NFP] = nM[v];
    os[v * NFP] = qSb[v] + T(0.5) * x;
    os[(NV + v) * NFP] = nS[v];
  }
}

// ---------------------------------------------------------------------------
// Trace adjoint: every solution point gathers the value and normal-derivative
// adjoints at the ends of its three lines and adds them to the volume part.
// ---------------------------------------------------------------------------
template <typename T>
struct TraceAdjArgs {
  const T* trbar;
  T* out;              // in: volume part; out: full q-bar
  const BasisTab<T>* basis;
  int64_t state_base, trace_base;
  int count, nvt;
};

template <typename T, int ND, int P, bool VISC>
__global__ void __launch_bounds__(256) trace_adj_kernel(TraceAdjArgs<T> a) {
  using Sh = Shape<ND, P>;
  constexpr int NV = Sh::NV, NF = Sh::NF, NSP = Sh::NSP, NFP = Sh::NFP;
  const int64_t gid = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (gid >= (int64_t)a.count * NSP) return;
  const int sp = (int)(gid % NSP);
  const int64_t i = gid / NSP;
  const BasisTab<T>& B = a.basis[P];
  int idx[3];
  idx[0] = sp % P;
  idx[1] = (sp / P) % P;
  idx[2] = ND == 3 ? sp / (P * P) : 0;
  const T* tb = a.trbar + a.trace_base + i * NF * (int64_t)a.nvt * NFP;
  T acc[NV];
#pragma unroll
  for (int v = 0; v < NV; ++v) acc[v] = a.out[a.state_base + (i * NV + v) * NSP + sp];
#pragma unroll
  for (int f = 0; f < NF; ++f) {
    const T* blk = tb + f * a.nvt * NFP + face_pt<ND, P>(f >> 1, idx);
    const T e = B.ext[f & 1][idx[f >> 1]], de = B.dext[f & 1][idx[f >> 1]];
#pragma unroll
    for (int v = 0; v < NV; ++v) {
      acc[v] += e * blk[v * NFP];
      if (VISC) acc[v] += de * blk[(NV + v) * NFP];
    }
  }
#pragma unroll
  for (int v = 0; v < NV; ++v) a.out[a.state_base + (i * NV + v) * NSP + sp] = acc[v];
}

}  // namespace frgb
