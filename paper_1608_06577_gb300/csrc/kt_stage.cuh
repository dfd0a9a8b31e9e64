// kt_stage.cuh -- the fused KT + Heun stage kernels of the FP64 path (one launch per Runge-Kutta stage;
// stage_kernel, and stage_team_kernel for small grids) and what they share with the mixed path.
//
// One thread owns one physical cell and performs, in order (Sec. 4.3 steps 1-4 / 5-8):
//   a) for x, y, eta: generalised-minmod slopes of the 15 conserved components and of u^tau,
//      u^d on the 5-point stencil; half-cell extrapolations; local speeds a = max(|v+|,|v-|);
//      central-upwind fluxes at both faces; -(H_{i+1/2} - H_{i-1/2})/dx       (Eqs. Hflux, ax)
//   b) the source vector J = S + G of App. B: central differences of v P - v pi^{tau nu} +
//      pi^{d nu}, the geometric terms, and the relaxation sources built from theta, D u,
//      sigma, omega (App. A) with the coefficients of Eqs. (betaPi)-(lambdapiPi)
//   c) the Heun update in FP64: q* = q + dtau C[q]   or   q^{n+1} = (q^n + q* + dtau C[q*])/2
//   d) the FP64 inversion T^{tau mu} -> (e, u^mu) of Eq. (eInferred) at tau^{n+1}
//   e) the regulator of Eq. (regPimunu)
//   f) stores, including the ghost copies owned by boundary cells (Eqs. ghostCells_1/2)
// R is the arithmetic type of a) and b): double (KT_FP64) or float (KT_MIXED).
#pragma once
#include "kt_device.cuh"
#include "kt_mlp.cuh"

namespace kt {

template <typename R>
struct StageIO {
  const double* q_in;    // 15 fields, FP64 (q^n or q^*), read at the own cell for the Heun update
  const double* q_base;  // stage 2: q^n, read at the own cell only (aliases q_out)
  double* q_out;
  const R* qr_in;        // 15 fields in the stencil precision (FP64 mode: q_in itself; mixed: an
  R* qr_out;             // FP32 copy written by the previous stage); qr_out null in FP64 mode
  const R* u_in;         // 4 fields, stencil input (u^n or u^*)
  const R* u_prev;       // 4 fields, own cell only: u^{n-1} (stage 1) or u^n (stage 2)
  R* u_out;              // may alias u_prev (own cell only)
  const R* e_in;
  const R* p_in;
  R* e_out;
  R* p_out;
  const TauSlot* tau;    // this step's tau
  TauSlot* tau_next;     // stage 2: where the next step's goes (another slot), else null
  unsigned* status;
  unsigned* max_speed_bits;
  unsigned long long* counters;  // [0] Newton iterations, [1] regulated cells, [2] fallbacks
  const uint32_t* mlp_packed;  // learned start: packed weights (see kt_mlp.cuh), or null
  float* reg_out;        // stage 2: the regulation factor applied to pi^{n+1} at each cell, or null
  const R* fv;           // FP32, KT_IFACE_INVERT: v^m, v^p of the faces i+1/2 of x, y, eta (face_velocity_kernel)
};

// ------------------------------------------------------------------ a) the stencil
// Per direction d the cell has two faces, L = i-1/2 and R = i+1/2, each with a left (m) and a
// right (p) state.  With F = v q the central-upwind flux of Eq. (Hflux) is linear in the face
// states, H = (v^p - a)/2 q^p + (v^m + a)/2 q^m, so the velocities and speeds of a face are
// folded once into four weights per direction (times 1/dx, the R-face weights negated),
//   -(H_R - H_L)/dx = wLp q_L^p + wLm q_L^m + wRp q_R^p + wRm q_R^m,
// and, with the face states q_L^m = q_{i-1} + s_{i-1}/2, q_L^p = q_i - s_i/2, q_R^m = q_i + s_i/2,
// q_R^p = q_{i+1} - s_{i+1}/2, every component costs its three slopes and five multiply-adds:
//   (wLp + wRm) q_i + wLm (q_{i-1} + s_{i-1}/2) + wRp (q_{i+1} - s_{i+1}/2) + (wRm - wLp)/2 s_i,
// of which the q_i term is one multiply-add for all three directions.  (Seven per direction before, with
// the slopes combined first; with the regulator's pairs once and FP64 tests on integers three FP64
// 128^3 steps went from 39.2 to 36.5 ms, the Gubser grid from 4.43 to 4.13 ms.)
template <typename R>
struct Faces {
  R c0, wLm, wRp, hdW;   // c0 = wLp + wRm, hdW = (wRm - wLp)/2
  R vpl_h, vmi_h;        // v^d at i+1 and i-1, times 1/(2 dx)
  int s;                 // element stride of direction d
};

// Root-find of one extrapolated face state (KT_IFACE_INVERT): f(e) = e - E + M^2/A = 0 with
// A = E + P0(e) + Pi, safeguarded Newton in the stencil precision inside [e_min, E] from `guess`;
// returns A at the root (v^d = M^d / A), or false if the state has none (E <= 0, M^2 >= E^2, no
// convergence in 100 steps).  FP64: the cell root-find (stop at |de| <= 2^-50 E, below).  FP32: stop at
// |de| <= 2^-21 E; the residual in product form g = (e - E) A + M^2 = f A, so that a step takes two fast
// divisions (they only steer), and the interval's record in two vector loads.  Six of these per cell and
// stage bound such a step (face_velocity_kernel); with IEEE divisions and eos_interval's dependent loads six
// steps of a 72 x 64 x 40 box took 2.24 ms, so 1.66 ms, when each cell inverted the four states of both its
// faces.
__device__ __forceinline__ FaceSeg face_seg(const Params& P, float e) {
  const int n1 = P.eos_n - 2;
  const float g = (__logf(e) - P.lne0) * P.inv_h;
  int i = min((g > 0.f) ? (int)g : 0, n1);  // NaN compares false -> 0
  auto load = [&](int k) {
    const float4* p = reinterpret_cast<const float4*>(P.seg_face + k);
    const float4 a = __ldg(p), b = __ldg(p + 1);
    return FaceSeg{a.x, a.y, a.z, a.w, b.x, b.y, 0.f, 0.f};
  };
  FaceSeg s = load(i);
  if ((i > 0 && e < s.e0) || e >= s.e1) {  // next to a node the logarithm may miss by one
#pragma unroll 1
    for (int it = 0; it < 64 && i > 0 && e < P.seg_face[i].e0; ++it) --i;
#pragma unroll 1
    for (int it = 0; it < 64 && i < n1 && e >= P.seg_face[i].e1; ++it) ++i;
    s = load(i);
  }
  return s;
}
__device__ __forceinline__ bool face_root_table(const Params& P, float E, float M2, float Pi, float guess, float& A) {
  float lo = (P.e_min > 0.0) ? (float)P.e_min : 1e-30f, hi = E;
  float e = (guess >= lo && guess <= hi) ? guess : hi;
  const float EPi = E + Pi, stop = E * 0x1p-21f;
#pragma unroll 1
  for (int it = 0; it < 100; ++it) {
    const FaceSeg s = face_seg(P, e);
    const float d = e - s.e0;
    A = EPi + fmaf(d, fmaf(d, fmaf(d, s.a3, s.a2), s.a1), s.P0);
    const float c2 = fmaf(d, fmaf(d, 3.f * s.a3, 2.f * s.a2), s.a1);
    const float g = fmaf(e - E, A, M2);
    if (g == 0.f) return true;
    if ((g < 0.f) != (A < 0.f)) lo = e; else hi = e;
    float en = e - __fdividef(g, A - __fdividef(M2 * c2, A));
    if (!(en >= lo && en <= hi)) en = 0.5f * (lo + hi);
    const float de = en - e;
    e = en;
    if (fabsf(de) <= stop) {
      // P0 at the root by its slope: what that leaves out is below the rounding of a new evaluation (the error
      // of q after a step at u up to 4: 1.0e-8 so, 4.3e-8 with one)
      A = fmaf(c2, de, A);
      return true;
    }
  }
  return false;
}
__device__ __forceinline__ bool face_root_table(const Params& P, double E, double M2, double Pi, double guess, double& A);
template <typename R>
__device__ __forceinline__ bool face_root(const Params& P, R E, R M2, R Pi, R guess, R& A) {
  if (!pos(E) || !below(M2, E * E) || !finite(E)) return false;
  if (!P.eos_table) {  // (bulk pressure is evolved with a table EOS only)
    const R M = sqrt(M2);  // conformal closed form, cancellation-free
    const R e = rdiv(R(3) * (E - M) * (E + M), sqrt(fma(R(4) * E, E, R(-3) * M2)) + E);
    A = E + e * R(1.0 / 3.0) + Pi;
    return true;
  }
  return face_root_table(P, E, M2, Pi, guess, A);
}

// KT_IFACE_INVERT (literal reading of Sec. 3.1): the four extrapolated states along D -- left face
// m (from cell i-1) and p (from cell i), right face m (from cell i) and p (from cell i+1) -- of the
// components the root-find reads (T^{tau mu}, pi^{tau mu}, Pi), each inverted from the e of the cell
// it was extrapolated from; v^d = M^d / (E + P0 + Pi) at the root, 0 for a state without one.  FP64; in
// FP32 face_velocity_kernel has inverted every face once.
template <typename R, int D, bool TH1>
__device__ __forceinline__ void face_velocities_inverted(const Params& P, const Lattice& L, const StageIO<R>& io,
                                                         Idx<R> c, int s, R th, R gnn, R& vLm, R& vLp, R& vRm,
                                                         R& vRp) {
  const long long fs = L.fstride;
  const R h = R(0.5);
  R E4[4] = {R(0), R(0), R(0), R(0)}, M4[3][4] = {}, Pi4[4] = {R(0), R(0), R(0), R(0)};
#pragma unroll
  for (int k = 0; k < 9; ++k) {
    const int n = (k < 8) ? k : 14;
    const R* p = io.qr_in + n * fs;
    const R a2 = ld<R>(p, c - 2 * s), a1 = ld<R>(p, c - s), a0 = ld<R>(p, c), b1 = ld<R>(p, c + s),
            b2 = ld<R>(p, c + 2 * s);
    const R d0 = a1 - a2, d1 = a0 - a1, d2 = b1 - a0, d3 = b2 - b1;
    R sm, s0, sp;
    three_slopes<R, TH1>(d0, d1, d2, d3, th, sm, s0, sp);
    const R x[4] = {fma(h, sm, a1), fma(-h, s0, a0), fma(h, s0, a0), fma(-h, sp, b1)};
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      if (n == 0) E4[j] += x[j];
      else if (n == 4) E4[j] -= x[j];
      else if (n < 4) M4[n - 1][j] += x[j];
      else if (n < 8) M4[n - 5][j] -= x[j];
      else Pi4[j] = x[j];
    }
  }
  const R g[4] = {ld<R>(io.e_in, c - s), ld<R>(io.e_in, c), ld<R>(io.e_in, c), ld<R>(io.e_in, c + s)};
  R v[4];
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    const R M2 = fma(M4[0][j], M4[0][j], fma(M4[1][j], M4[1][j], gnn * M4[2][j] * M4[2][j]));
    R A;
    v[j] = face_root<R>(P, E4[j], M2, Pi4[j], g[j], A) ? sdiv(M4[D][j], A) : R(0);
  }
  vLm = v[0]; vLp = v[1]; vRm = v[2]; vRp = v[3];
}

// The same in FP32 for one face, i+1/2 of cell c: v^m from the state of cell i, v^p from that of i+1.
template <int D, bool TH1>
__device__ __forceinline__ void face_velocities_right(const Params& P, const float* q, const float* e, long long fs,
                                                      unsigned c, int s, float th, float gnn, float& vm, float& vp) {
  float E[2] = {0.f, 0.f}, M[3][2] = {}, Pi[2];
#pragma unroll
  for (int k = 0; k < 9; ++k) {
    const int n = (k < 8) ? k : 14;
    const float* p = q + n * fs;
    const float a1 = ld<float>(p, c - s), a0 = ld<float>(p, c), b1 = ld<float>(p, c + s), b2 = ld<float>(p, c + 2 * s);
    const float d1 = a0 - a1, d2 = b1 - a0, d3 = b2 - b1;
    float sm, s0, sp;
    three_slopes<float, TH1>(d1, d1, d2, d3, th, sm, s0, sp);
    const float x[2] = {fmaf(0.5f, s0, a0), fmaf(-0.5f, sp, b1)};
#pragma unroll
    for (int j = 0; j < 2; ++j) {
      if (n == 0) E[j] += x[j];
      else if (n == 4) E[j] -= x[j];
      else if (n < 4) M[n - 1][j] += x[j];
      else if (n < 8) M[n - 5][j] -= x[j];
      else Pi[j] = x[j];
    }
  }
  float v[2];
#pragma unroll
  for (int j = 0; j < 2; ++j) {
    const float M2 = fmaf(M[0][j], M[0][j], fmaf(M[1][j], M[1][j], rmul(rmul(gnn, M[2][j]), M[2][j])));
    float A;
    v[j] = face_root<float>(P, E[j], M2, Pi[j], ld<float>(e, j ? c + s : c), A) ? rdiv(M[D][j], A) : 0.f;
  }
  vm = v[0];
  vp = v[1];
}

// How the stencil reads u^mu around cell c: from the field arrays, through the read-only cache.
// (Staging u^mu in shared memory by TMA, like q, measured slower: the stencil's scattered u loads
// hit L1, which the larger shared-memory carve-out shrinks.)
template <typename R>
struct UGlobal {
  const R* u;
  long long fs;
  Idx<R> c;
  int sy, sz;  // row pitch, plane
  __device__ __forceinline__ R operator()(int m, int off) const { return ld<R>(u + m * fs, c + off); }
};
template <typename R>
__device__ __forceinline__ UGlobal<R> u_global(const Lattice& L, const StageIO<R>& io, Idx<R> c) {
  return UGlobal<R>{io.u_in, L.fstride, c, L.pitch, (int)L.plane};
}

// Velocity part of direction D: limited face states of u^tau and u^d and their ratio v^d
// (Sec. 3.1), the local speeds a = max(|v^p|, |v^m|) (Eq. ax), the central differences
// d_d u^mu and v^d_{i+1} - v^d_{i-1}, and the pressure part of S_c (App. B):
// -d_d (v^d P delta^nu_tau - g^{d nu} P), P = P0 + Pi.
template <typename R, int D, bool TH1, bool IFACE, typename UA>
__device__ __forceinline__ void face_setup(const Params& P, const Lattice& L, const StageIO<R>& io, Idx<R> c,
                                           const UA& ua, const R (&uc)[4], R inv_gnn, R sfac, R (&dq)[NQ],
                                           R (&du)[4][4], R& dvd, float& amax, Faces<R>& F) {
  const long long fs = L.fstride;
  const int s = (D == 0) ? 1 : ((D == 1) ? L.pitch : (int)L.plane);  // in the field arrays
  const int us = (D == 0) ? 1 : ((D == 1) ? ua.sy : ua.sz);           // where u is read
  const R hinv = pr<R>(P).half_inv_d[D];
  const R th = pr<R>(P).theta;

  R um1[4], up1[4];
#pragma unroll
  for (int m = 0; m < 4; ++m) {
    um1[m] = ua(m, -us);
    up1[m] = ua(m, us);
  }
  R vLm, vLp, vRm, vRp;
  if constexpr (IFACE && sizeof(R) == 4) {
    const R* vm = io.fv + 2 * D * fs;
    const R* vp = vm + fs;
    vLm = ld<R>(vm, c - s); vLp = ld<R>(vp, c - s);
    vRm = ld<R>(vm, c); vRp = ld<R>(vp, c);
  } else if constexpr (IFACE) {
    face_velocities_inverted<R, D, TH1>(P, L, io, c, s, th, sfac * sfac, vLm, vLp, vRm, vRp);
  } else {
    const R u0t = uc[0], u0d = uc[D + 1];
    const R um2t = ua(0, -2 * us), um2d = ua(D + 1, -2 * us);
    const R up2t = ua(0, 2 * us), up2d = ua(D + 1, 2 * us);
    R t0 = um1[0] - um2t, t1 = u0t - um1[0], t2 = up1[0] - u0t, t3 = up2t - up1[0];
    R d0 = um1[D + 1] - um2d, d1 = u0d - um1[D + 1], d2 = up1[D + 1] - u0d, d3 = up2d - up1[D + 1];
    R st_m, st_0, st_p, sd_m, sd_0, sd_p;
    three_slopes<R, TH1>(t0, t1, t2, t3, th, st_m, st_0, st_p);
    three_slopes<R, TH1>(d0, d1, d2, d3, th, sd_m, sd_0, sd_p);
    const R h = R(0.5);
    vLm = vdiv(fma(h, sd_m, um1[D + 1]), fma(h, st_m, um1[0]));
    vLp = vdiv(fma(-h, sd_0, u0d), fma(-h, st_0, u0t));
    vRm = vdiv(fma(h, sd_0, u0d), fma(h, st_0, u0t));
    vRp = vdiv(fma(-h, sd_p, up1[D + 1]), fma(-h, st_p, up1[0]));
  }
  const R aL = nmax(fabs(vLp), fabs(vLm));
  const R aR = nmax(fabs(vRp), fabs(vRm));
  const R aF = nmax(aL, aR);  // both faces: the first cell's left face is nobody's right face
  amax = fmaxf(amax, to_f32((D == 2) ? aF * sfac : aF));
  const R wLp = rmul(vLp - aL, hinv), wRm = rmul(-(vRm + aR), hinv);
  F.c0 = wLp + wRm;
  F.hdW = R(0.5) * (wRm - wLp);
  F.wLm = (vLm + aL) * hinv;
  F.wRp = (aR - vRp) * hinv;

#pragma unroll
  for (int m = 0; m < 4; ++m) du[D + 1][m] = rmul(up1[m] - um1[m], hinv);
  const R vpl = vdiv(up1[D + 1], up1[0]), vmi = vdiv(um1[D + 1], um1[0]);
  dvd = vpl - vmi;
  F.vpl_h = rmul(vpl, hinv);
  F.vmi_h = rmul(vmi, hinv);
  F.s = s;

  const R* q = io.qr_in;
  const R Ppl = ld<R>(io.p_in, c + s) + ld<R>(q + 14 * fs, c + s);
  const R Pmi = ld<R>(io.p_in, c - s) + ld<R>(q + 14 * fs, c - s);
  dq[0] -= fma(Ppl, F.vpl_h, -(Pmi * F.vmi_h));
  dq[D + 1] -= rmul((D == 2) ? (Ppl - Pmi) * inv_gnn : (Ppl - Pmi), hinv);
}

// An axis of one cell: its neighbours are copies of the cell, so every difference along it vanishes; the
// local speed is that of the cell itself.
template <typename R, int D>
__device__ __forceinline__ void face_none(const R (&uc)[4], R sfac, R (&du)[4][4], float& amax, Faces<R>& F) {
  const R a = fabs(vdiv(uc[D + 1], uc[0]));
  amax = fmaxf(amax, to_f32((D == 2) ? a * sfac : a));
  F.c0 = F.wLm = F.wRp = F.hdW = F.vpl_h = F.vmi_h = R(0);
  F.s = 0;
#pragma unroll
  for (int m = 0; m < 4; ++m) du[D + 1][m] = R(0);
}

// row nu of T^{tau nu} that component n feeds through -d_d(-v^d pi^{tau nu}) (first == true:
// n = pi^{tau nu}) or -d_d(pi^{d nu}) (n = pi^{d nu}); -1 if none
template <int D>
__device__ __forceinline__ int cross_row(int n, bool first) {
  if (first) return (n >= 4 && n <= 7) ? n - 4 : -1;
#pragma unroll
  for (int nu = 0; nu < 4; ++nu)
    if (n == pix(D + 1, nu)) return nu;
  return -1;
}

// dq[r] += v for a warp-uniform runtime row r (the switch keeps dq in registers)
template <typename R>
__device__ __forceinline__ void add_row(R (&dq)[NQ], int r, R v) {
  switch (r) {
    case 0: dq[0] += v; break;
    case 1: dq[1] += v; break;
    case 2: dq[2] += v; break;
    case 3: dq[3] += v; break;
    case 4: dq[4] += v; break;
    case 5: dq[5] += v; break;
    case 6: dq[6] += v; break;
    case 7: dq[7] += v; break;
    case 8: dq[8] += v; break;
    case 9: dq[9] += v; break;
    case 10: dq[10] += v; break;
    case 11: dq[11] += v; break;
    case 12: dq[12] += v; break;
    case 13: dq[13] += v; break;
    case 14: dq[14] += v; break;
    default: break;
  }
}

// one component along one direction: generalised-minmod reconstruction from the five-point FP32
// stencil p[-2s..2s] in shared memory (a0 = p[0] given) and the flux difference -(H_R - H_L)/dx without
// its q_i term, added to acc; a1, b1 return the neighbours for the central differences of S_c
template <bool TH1>
__device__ __forceinline__ float component_flux(const float* p, int s, float a0, float th, const Faces<float>& F,
                                                float& a1, float& b1, float acc) {
  const float a2 = p[-2 * s], b2 = p[2 * s];
  a1 = p[-s];
  b1 = p[s];
  const float d0 = a1 - a2, d1 = a0 - a1, d2 = b1 - a0, d3 = b2 - b1;
  float sm, s0, sp;
  three_slopes<float, TH1>(d0, d1, d2, d3, th, sm, s0, sp);
  acc = fma(F.wLm, fma(0.5f, sm, a1), acc);
  acc = fma(F.wRp, fma(-0.5f, sp, b1), acc);
  return fma(F.hdW, s0, acc);
}

// ---- paired FP32 arithmetic (the f32x2 instructions of the sm_100 family): two independent
// single-precision operations, each rounded to nearest as its scalar form, in one instruction
__device__ __forceinline__ unsigned long long pk2(float lo, float hi) {
  unsigned long long r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
  return r;
}
__device__ __forceinline__ void up2(unsigned long long v, float& lo, float& hi) {
  asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(v));
}
__device__ __forceinline__ unsigned long long sub2(unsigned long long a, unsigned long long b) {
  unsigned long long r;
  asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ unsigned long long add2(unsigned long long a, unsigned long long b) {
  unsigned long long r;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ unsigned long long mul2(unsigned long long a, unsigned long long b) {
  unsigned long long r;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ unsigned long long fma2(unsigned long long a, unsigned long long b, unsigned long long c) {
  unsigned long long r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
  return r;
}

// The x and y face weights of a cell as (x, y) pairs for the paired flux of component_rhs_xy.
struct FacesXY {
  unsigned long long wLm, wRp, hdW;
};
__device__ __forceinline__ FacesXY faces_xy(const Faces<float>& Fx, const Faces<float>& Fy) {
  return FacesXY{pk2(Fx.wLm, Fy.wLm), pk2(Fx.wRp, Fy.wRp), pk2(Fx.hdW, Fy.hdW)};
}

// Component n (warp-uniform) of the 15 conserved components, at a cell whose FP32 stencil starts at p in
// shared memory with strides 1, sy, sz: -div H in x, y, eta and the remaining S_c terms
// -d_d(-v^d pi^{tau nu} + pi^{d nu}) by central differences, added to dq.  The x and y directions are
// computed as pairs: the differences, bounds and five multiply-adds of the two share instructions; the
// limiter's min/max and the eta direction stay scalar.  With theta != 1 (96 x 96 x 64, theta = 1.3) the
// right-hand side took 82 us per launch with scalar directions and a sign test per slope, 76 us so.
template <bool TH1>
__device__ __forceinline__ void component_rhs_xy(const Params& P, int n, const float* p, int sy, int sz,
                                                 const FacesXY& W, const Faces<float>& Fx, const Faces<float>& Fy,
                                                 const Faces<float>& Fz, float th, float (&dq)[NQ]) {
  const float a0 = p[0];
  const float a2x = p[-2], a1x = p[-1], b1x = p[1], b2x = p[2];
  const float a2y = p[-2 * sy], a1y = p[-sy], b1y = p[sy], b2y = p[2 * sy];
  const unsigned long long A0 = pk2(a0, a0), A1 = pk2(a1x, a1y), B1 = pk2(b1x, b1y);
  const unsigned long long D0 = sub2(A1, pk2(a2x, a2y)), D1 = sub2(A0, A1), D2 = sub2(B1, A0),
                           D3 = sub2(pk2(b2x, b2y), B1);
  float d0x, d0y, d1x, d1y, d2x, d2y, d3x, d3y, smx, smy, s0x, s0y, spx, spy;
  up2(D0, d0x, d0y);
  up2(D1, d1x, d1y);
  up2(D2, d2x, d2y);
  up2(D3, d3x, d3y);
  // three_slopes for both directions
  if constexpr (TH1) {
    const float h1x = fmaxf(d1x, 0.f), h1y = fmaxf(d1y, 0.f), h2x = fmaxf(d2x, 0.f), h2y = fmaxf(d2y, 0.f);
    float l1x, l1y, l2x, l2y;
    up2(sub2(D1, pk2(h1x, h1y)), l1x, l1y);
    up2(sub2(D2, pk2(h2x, h2y)), l2x, l2y);
    smx = fminf(fmaxf(d0x, l1x), h1x);
    smy = fminf(fmaxf(d0y, l1y), h1y);
    s0x = fminf(fmaxf(d1x, l2x), h2x);
    s0y = fminf(fmaxf(d1y, l2y), h2y);
    spx = fminf(fmaxf(d3x, l2x), h2x);
    spy = fminf(fmaxf(d3y, l2y), h2y);
  } else {
    const unsigned long long T = pk2(th, th), H = pk2(0.5f, 0.5f);
    float h0x, h0y, l0x, l0y, h1x, h1y, l1x, l1y, h2x, h2y, l2x, l2y, h3x, h3y, l3x, l3y, cx, cy;
    const auto bounds = [&](unsigned long long D, float& hx, float& hy, float& lx, float& ly) {
      const unsigned long long t = mul2(T, D);
      float tx, ty;
      up2(t, tx, ty);
      hx = fmaxf(tx, 0.f);
      hy = fmaxf(ty, 0.f);
      up2(sub2(t, pk2(hx, hy)), lx, ly);
    };
    bounds(D0, h0x, h0y, l0x, l0y);
    bounds(D1, h1x, h1y, l1x, l1y);
    bounds(D2, h2x, h2y, l2x, l2y);
    bounds(D3, h3x, h3y, l3x, l3y);
    up2(mul2(H, add2(D0, D1)), cx, cy);
    smx = clamp_slope(cx, h0x, l0x, h1x, l1x);
    smy = clamp_slope(cy, h0y, l0y, h1y, l1y);
    up2(mul2(H, add2(D1, D2)), cx, cy);
    s0x = clamp_slope(cx, h1x, l1x, h2x, l2x);
    s0y = clamp_slope(cy, h1y, l1y, h2y, l2y);
    up2(mul2(H, add2(D2, D3)), cx, cy);
    spx = clamp_slope(cx, h2x, l2x, h3x, l3x);
    spy = clamp_slope(cy, h2y, l2y, h3y, l3y);
  }
  unsigned long long acc = mul2(W.wLm, fma2(pk2(0.5f, 0.5f), pk2(smx, smy), A1));
  acc = fma2(W.wRp, fma2(pk2(-0.5f, -0.5f), pk2(spx, spy), B1), acc);
  acc = fma2(W.hdW, pk2(s0x, s0y), acc);
  float accx, accy, a1z, b1z;
  up2(acc, accx, accy);
  const float accz =
      component_flux<TH1>(p, sz, a0, th, Fz, a1z, b1z, fmaf(Fx.c0 + Fy.c0 + Fz.c0, a0, accx + accy));
  add_row(dq, n, accz);
  if (n >= 4 && n <= 13) {  // pi components
    const int r0 = cross_row<0>(n, true);
    if (r0 >= 0)
      add_row(dq, r0, (Fx.vpl_h * b1x - Fx.vmi_h * a1x) + (Fy.vpl_h * b1y - Fy.vmi_h * a1y) +
                          (Fz.vpl_h * b1z - Fz.vmi_h * a1z));
    const int rx = cross_row<0>(n, false), ry = cross_row<1>(n, false), rz = cross_row<2>(n, false);
    const float* hinv = pr<float>(P).half_inv_d;
    if (rx >= 0) add_row(dq, rx, -(b1x - a1x) * hinv[0]);
    if (ry >= 0) add_row(dq, ry, -(b1y - a1y) * hinv[1]);
    if (rz >= 0) add_row(dq, rz, -(b1z - a1z) * hinv[2]);
  }
}

// All 15 components from global memory (FP64), all 32 lanes of the warp together.  An FP64 instruction
// costs its warp 64 cycles however many lanes are active, so work that cannot contribute is skipped by
// the whole warp: a component whose stencil is zero in every cell of the warp (pi and Pi of an ideal
// fluid, Pi of a conformal one) adds zero, and so does an axis of one cell, whose neighbours are all
// copies of it.  The next component's stencil is loaded while the current one computes: a grid with few
// warps has nothing else to cover the load latency with.
template <typename R>
struct Stencil13 {
  R a0, v[3][4];  // the cell and, per axis, i-2, i-1, i+1, i+2
};
template <typename R>
__device__ __forceinline__ Stencil13<R> load_stencil(const R* p, const bool (&on)[3], const int (&s)[3]) {
  Stencil13<R> q;
  q.a0 = ld<R>(p, 0LL);
#pragma unroll
  for (int d = 0; d < 3; ++d) {
    q.v[d][0] = q.v[d][1] = q.v[d][2] = q.v[d][3] = R(0);
    if (on[d]) {
      const long long e = s[d];
      q.v[d][0] = ld<R>(p, -2 * e); q.v[d][1] = ld<R>(p, -e); q.v[d][2] = ld<R>(p, e); q.v[d][3] = ld<R>(p, 2 * e);
    }
  }
  return q;
}
template <typename R>
__device__ __forceinline__ bool stencil_nonzero(const Stencil13<R>& q) {  // in any cell of the warp
  long long bits = __double_as_longlong(q.a0);
#pragma unroll
  for (int d = 0; d < 3; ++d)
#pragma unroll
    for (int k = 0; k < 4; ++k) bits |= __double_as_longlong(q.v[d][k]);
  return __any_sync(0xffffffffu, (bits << 1) != 0);
}
// -div H of one component, and for pi^{tau nu} the sum of the v^d pi^{tau nu} differences (mix)
template <typename R, bool TH1>
__device__ __forceinline__ void stencil_flux(const Stencil13<R>& q, R c0, const bool (&on)[3], const Faces<R> (&F)[3],
                                             R th, bool with_mix, R& acc, R& mix) {
  acc = rmul(c0, q.a0);
  mix = R(-0.0);
#pragma unroll
  for (int d = 0; d < 3; ++d) {
    if (!on[d]) continue;
    const R a1 = q.v[d][1], b1 = q.v[d][2];
    const R d0 = a1 - q.v[d][0], d1 = q.a0 - a1, d2 = b1 - q.a0, d3 = q.v[d][3] - b1;
    R sm, s0, sp;
    three_slopes<R, TH1>(d0, d1, d2, d3, th, sm, s0, sp);
    acc = fma(F[d].wLm, fma(R(0.5), sm, a1), acc);
    acc = fma(F[d].wRp, fma(R(-0.5), sp, b1), acc);
    acc = fma(F[d].hdW, s0, acc);
    if (with_mix) mix = fma(F[d].vpl_h, b1, fma(-F[d].vmi_h, a1, mix));
  }
}
template <typename R>
__device__ __forceinline__ R sum_c0(const Faces<R> (&F)[3], const bool (&on)[3]) {
  return (on[0] ? F[0].c0 : R(0)) + (on[1] ? F[1].c0 : R(0)) + (on[2] ? F[2].c0 : R(0));
}

template <typename R, bool TH1 = false>
__device__ __forceinline__ void conserved_fluxes(const Params& P, const Lattice& L, const StageIO<R>& io, Idx<R> c,
                                                 const Faces<R> (&F)[3], R (&dq)[NQ]) {
  const long long fs = L.fstride;
  const R th = pr<R>(P).theta;
  const bool on[3] = {L.nx > 1, L.ny > 1, L.nz > 1};
  const int s[3] = {F[0].s, F[1].s, F[2].s};
  const R c0 = sum_c0<R>(F, on);
  const R* p = io.qr_in + c;
  Stencil13<R> q = load_stencil<R>(p, on, s);
#pragma unroll
  for (int n = 0; n < NQ; ++n) {
    Stencil13<R> next;
    if (n + 1 < NQ) next = load_stencil<R>(p + (n + 1) * fs, on, s);
    if (stencil_nonzero<R>(q)) {
      R acc, mix;
      stencil_flux<R, TH1>(q, c0, on, F, th, n >= 4 && n <= 7, acc, mix);
#pragma unroll
      for (int d = 0; d < 3; ++d) {
        const int r = (d == 0) ? cross_row<0>(n, false) : ((d == 1) ? cross_row<1>(n, false) : cross_row<2>(n, false));
        if (on[d] && n >= 4 && n <= 13 && r >= 0) dq[r] = fma(q.v[d][1] - q.v[d][2], pr<R>(P).half_inv_d[d], dq[r]);
      }
      dq[n] += acc;
      if (n >= 4 && n <= 7) dq[n - 4] += mix;
    }
    q = next;
  }
}

// ------------------------------------------------------------- d) the root-find (Sec. 2.4)
// Positive doubles are ordered like their bit patterns read as integers, so the brackets and
// tolerances below are compared with integer instructions and the slow FP64 pipe only does
// arithmetic.
__device__ __forceinline__ long long obits(double x) { return __double_as_longlong(x); }
__device__ __forceinline__ long long abits(double x) { return __double_as_longlong(x) & 0x7fffffffffffffffLL; }
__device__ __forceinline__ double clamp_pos(double x, double lo, double hi) {  // lo, hi > 0; NaN -> hi
  return (obits(x) < obits(lo)) ? lo : ((obits(x) <= obits(hi)) ? x : hi);
}

// The interval of e > 0 in the FP64 table and its record: the single-precision log guess of
// eos_interval, checked against both ends of the interval in the same load; only a guess that
// misses (next to a node) searches as eos_interval does (integer comparisons of the bit patterns)
// and loads again.  The same interval as eos_interval, with one dependent load instead of three.
// Seg is RootSeg (FP64 path) or RootSegM (mixed precision); both start with e0, e1.
__device__ __forceinline__ RootSeg load_root_seg(const RootSeg* p) {
  const double2* d = reinterpret_cast<const double2*>(p);
  const double2 v0 = __ldg(d), v1 = __ldg(d + 1), v2 = __ldg(d + 2);
  const float4 v3 = __ldg(reinterpret_cast<const float4*>(p) + 3);
  return RootSeg{v0.x, v0.y, v1.x, v1.y, v2.x, v2.y, v3.x, v3.y, v3.z, v3.w};
}
__device__ __forceinline__ RootSegM load_root_seg(const RootSegM* p) {
  const double2* d = reinterpret_cast<const double2*>(p);
  const double2 v0 = __ldg(d), v1 = __ldg(d + 1);
  const float4 v2 = __ldg(reinterpret_cast<const float4*>(p) + 2);
  const float b3 = __ldg(reinterpret_cast<const float*>(p) + 12);
  return RootSegM{v0.x, v0.y, v1.x, v1.y, v2.x, v2.y, v2.z, v2.w, b3, 0.f, 0.f, 0.f};
}
template <typename Seg>
__device__ __forceinline__ Seg root_seg(const Params& P, const Seg* seg, double e) {
  const int n1 = P.eos_n - 2;
  const float g = (__logf(d2f_trunc(e)) - P.lne0) * P.inv_h;
  int i = min((g > 0.f) ? (int)g : 0, n1);  // NaN compares false -> 0
  const long long b = obits(e);
  Seg s = load_root_seg(seg + i);
  if ((i > 0 && b < obits(s.e0)) || b >= obits(s.e1)) {
#pragma unroll 1
    for (int it = 0; it < 64 && i > 0 && b < obits(seg[i].e0); ++it) --i;
#pragma unroll 1
    for (int it = 0; it < 64 && i < n1 && b >= obits(seg[i].e1); ++it) ++i;
    s = load_root_seg(seg + i);
  }
  return s;
}

// the interval's record for the FP64 path (RootSeg) or the mixed-precision one (RootSegM)
template <bool MIXED>
__device__ __forceinline__ auto path_seg(const Params& P, double e) {
  if constexpr (MIXED) return root_seg(P, P.seg_m, e);
  else return root_seg(P, P.seg_r, e);
}

// P0(e) in d = e - e0 on the interval's record: the cubic in FP64 (RootSeg), or (RootSegM) its
// leading part in FP64 with the correction d (a2 + d a3) to a1 formed in single precision from
// df, the single-precision d.
__device__ __forceinline__ double seg_P(const RootSeg& s, double d, float) {
  return fma(d, fma(d, fma(d, s.a3, s.a2), s.a1), s.P0);
}
__device__ __forceinline__ double seg_P(const RootSegM& s, double d, float df) {
  return fma(d, s.a1 + f2d_bits(df * fmaf(df, s.a3, s.a2)), s.P0);
}

// The residual in product form g(e) = (e - E) A(e) + M^2 = f(e) A(e), A = E + P0(e) + Pi > 0:
// the root and the sign of f(e) = e - E + M^2 / A of Eq. (eInferred), without a reciprocal.
// Also A, P0(e) and, in single precision, A (truncated) and A f'(e) = A - M^2 c_s^2 / A: the
// Newton step on f, e - f/f' = e - g/(A f'), then needs the FP64 product of g with a
// single-precision factor (which only sets the step length; f is nearly linear in e where M is
// small, g is not).  MIXED: P0 from the mixed-precision records (RootSegM), whose rounding of the
// cubic's correction term (~1e-13 of P0, in steps as d crosses single-precision values) is far
// below the learned start's 1e-10 acceptance but above the plain root-find's 2^-50 stop, so only
// the learned start's Newton steps use it.
struct Resid {
  double g, A, p0;
  float gp, Af;
};
template <bool MIXED>
__device__ __forceinline__ Resid residual(const Params& P, double e, double E, double EPi, double M2, float M2f) {
  const auto s = path_seg<MIXED>(P, e);
  const double d = e - s.e0;
  const float df = d2f_trunc(d);
  Resid r;
  r.p0 = seg_P(s, d, df);
  r.A = EPi + r.p0;
  const double em = e - E;
  r.g = fma(em, r.A, M2);
  const float c2 = fmaf(df, fmaf(df, s.b3, s.b2), s.b1);
  r.Af = d2f_trunc(r.A);
  r.gp = r.Af - __fdividef(M2f * c2, r.Af);
  return r;
}

// one Newton step on f: e - g / (A f')
__device__ __forceinline__ double newton_step(double e, const Resid& r) {
  return fma(-r.g, f2d_bits(__frcp_rn(r.gp)), e);
}

// P0(e) on the FP64 table
__device__ __forceinline__ double eos_P_pos(const Params& P, double e) {
  const RootSeg s = root_seg(P, P.seg_r, e);
  return seg_P(s, e - s.e0, 0.f);
}

// Plain root-find: safeguarded Newton inside the bracket [e_min, E] (a step that leaves it
// bisects), from `start` if it lies inside, else from E; stop at |de| <= 2^-50 E (g is known to
// about one ulp of E A), at most 100 steps.  Table EOS only.  The stop's bit pattern is E's with
// the exponent lowered by 50 (exact for E >= 2^-972; smaller E stops only at de = 0).
__device__ __forceinline__ unsigned rootfind_plain(const Params& P, double E, double EPi, double M2, float M2f,
                                                   double start, double& e, double& P0, unsigned& iters) {
  double lo = P.root_lo, hi = E;
  e = (obits(start) >= obits(lo) && obits(start) <= obits(hi)) ? start : hi;
  const long long stop = max(obits(E) - (50LL << 52), 0LL);
  int it;
  for (it = 0; it < 100; ++it) {
    const Resid r = residual<false>(P, e, E, EPi, M2, M2f);
    if (abits(r.g) == 0) break;
    if (obits(r.g) < 0) lo = e; else hi = e;
    double en = newton_step(e, r);
    if (!(obits(en) >= obits(lo) && obits(en) <= obits(hi))) en = 0.5 * (lo + hi);
    const double de = en - e;
    e = en;
    if (abits(de) <= stop) { ++it; break; }
  }
  iters += (unsigned)it;
  if (obits(e) < obits(P.e_min)) e = P.e_min;
  P0 = eos_P_pos(P, e);
  return (it >= 100) ? ST_INVERSION : 0u;
}

// (KT_IFACE_INVERT, FP64) A = E + P0 + Pi at the root of a face state.  The product form of rootfind_plain
// takes A > 0 for granted, which E + Pi > 0 guarantees.  A face state with a bulk pressure below -E (P0 > 0
// keeps the A of the cells around it positive) may start where A < 0: there f = e - E + M^2/A itself decides.
__device__ __noinline__ bool face_root_signed(const Params& P, double E, double M2, double Pi, double guess, double& A) {
  double lo = P.root_lo, hi = E;
  double e = (guess >= lo && guess <= hi) ? guess : hi;
  const double stop = E * 0x1p-50;
#pragma unroll 1
  for (int it = 0; it < 100; ++it) {
    const RootSeg s = root_seg(P, P.seg_r, e);
    const double d = e - s.e0;
    const double c2 = fma(d, fma(d, 3.0 * s.a3, 2.0 * s.a2), s.a1);
    A = E + seg_P(s, d, 0.f) + Pi;
    const double f = e - E + M2 / A;
    if (f == 0.0) return true;
    if (f < 0.0) lo = e; else hi = e;
    double en = e - f / (1.0 - M2 * c2 / (A * A));
    if (!(en >= lo && en <= hi)) en = 0.5 * (lo + hi);
    const double de = fabs(en - e);
    e = en;
    if (de <= stop) {
      A = E + eos_P_pos(P, (e < P.e_min) ? P.e_min : e) + Pi;
      return true;
    }
  }
  return false;
}
__device__ __forceinline__ bool face_root_table(const Params& P, double E, double M2, double Pi, double guess,
                                                double& A) {
  if (!pos(E + Pi)) return face_root_signed(P, E, M2, Pi, guess, A);
  double e, P0;
  unsigned its = 0;
  if (rootfind_plain(P, E, E + Pi, M2, d2f_trunc(M2), guess, e, P0, its)) return false;
  A = E + P0 + Pi;
  return true;
}

// ------------------------------------------------------------ d) inversion, FP64 (Sec. 2.4)
// T^{tau mu} -> (e, P0, u^mu) at tau (Eqs. eInferred-uiInferred): the safeguarded Newton of
// rootfind_plain from the cell's previous e; with the conformal EOS and no bulk pressure, the
// closed form.
__device__ __forceinline__ unsigned invert_fp64(const Params& P, double tau, const double (&qn)[NQ], double guess,
                                                double& e, double& P0, double (&uo)[4], unsigned& iters) {
  const double E = qn[0] - qn[4];
  const double Mx = qn[1] - qn[5], My = qn[2] - qn[6], Mn = qn[3] - qn[7];
  const double Pi = qn[14];
  const double gnn = P.milne ? tau * tau : 1.0;
  const double M2 = fma(Mx, Mx, fma(My, My, gnn * Mn * Mn));
  unsigned st = 0;
  if (!(obits(E) > 0) || !finite(E) || !finite(M2) || !(obits(M2) < obits(E * E))) {
    st = ST_INVERSION;
    e = (P.e_min > 0.0) ? P.e_min : 1e-30;
    P0 = eos_P(P, e);
  } else if (!P.eos_table) {  // (bulk pressure is evolved with a table EOS only)
    const double M = sqrt(M2);  // conformal closed form e = sqrt(4E^2 - 3M^2) - E, cancellation-free
    e = vdiv(3.0 * (E - M) * (E + M), sqrt(fma(4.0 * E, E, -3.0 * M2)) + E);
    if (obits(e) < obits(P.e_min)) e = P.e_min;
    P0 = e * (1.0 / 3.0);
  } else {
    st = rootfind_plain(P, E, E + Pi, M2, d2f_trunc(M2), guess, e, P0, iters);
  }
  if (st) {
    uo[0] = 1.0; uo[1] = uo[2] = uo[3] = 0.0;
  } else {
    const double Pt = P0 + Pi;
    const double ut = sqrt(vdiv(E + Pt, e + Pt));
    const double w = vdiv(1.0, (e + Pt) * ut);
    uo[0] = ut; uo[1] = Mx * w; uo[2] = My * w; uo[3] = Mn * w;
  }
  if (!finite(e) || !finite(uo[0]) || !finite(uo[1]) || !finite(uo[2]) || !finite(uo[3])) st |= ST_NONFINITE;
  return st;
}

// ------------------------------------------------------------ e) regulator (Sec. 3.2)
template <typename R>
__device__ __forceinline__ R regulator_factor(const Params& P, R gnn, R sqrt_gnn, R e, R P0, const R (&u)[4],
                                              const R (&pi)[4][4], R Pi) {
  // X^{ab} = Pi Delta^{ab} + pi^{ab}; PP = X^{ab} X_{ab} by powers of g_{eta eta} = -gnn, each pair once
  R X[4][4];
#pragma unroll
  for (int a = 0; a < 4; ++a) {
    const R Pu = Pi * u[a];
#pragma unroll
    for (int b = a; b < 4; ++b) X[a][b] = fma(-Pu, u[b], pi[a][b]);
  }
  X[0][0] += Pi;
  X[1][1] -= Pi;
  X[2][2] -= Pi;
  X[3][3] = fma(-Pi, sdiv(R(1), gnn), X[3][3]);
  const R Xd = fma(X[0][0], X[0][0], fma(X[1][1], X[1][1], X[2][2] * X[2][2]));
  const R Xo = fma(X[1][2], X[1][2], -fma(X[0][1], X[0][1], X[0][2] * X[0][2]));
  const R Xn = fma(X[1][3], X[1][3], fma(X[2][3], X[2][3], -(X[0][3] * X[0][3])));
  const R Xe = gnn * X[3][3];
  const R PP = fma(Xe, Xe, fma(R(2) * gnn, Xn, fma(R(2), Xo, Xd)));
  if (!pos(PP)) return R(1);
  const R ee = fma(R(3) * P0, P0, e * e);
  // a norm beyond the range is an infinite rho, which suppresses pi altogether (its product with 1/sqrt(PP)
  // = 0 below would be a NaN, which the maxima drop); with e^2 beyond it too nothing is known, and pi stays
  if (!finite(PP)) return finite(ee) ? R(0) : R(1);
  // (In FP32 with two hardware reciprocal roots: f is off the FP64 mode's by the same 2.3e-7 to 1.1e-6 rms as
  // with rounded roots and quotients, PP's own rounding, which cost 1% of a step.)
  const R rn = rsqrt_pos(PP);  // 1/sqrt(PP)
  R rho = PP * rn * rsqrt_pos(ee) * pr<R>(P).inv_rho_max;
  const R den = rn * pr<R>(P).inv_xi0_rho_max;
  const R tr = fma(-gnn, pi[3][3], pi[0][0] - pi[1][1] - pi[2][2]);
  rho = nmax(rho, fabs(tr) * den);
  const R gu = gnn * u[3], rg = P.milne ? sqrt_gnn : R(1);
#pragma unroll
  for (int l = 0; l < 4; ++l) {
    R o = fma(-gu, pi[l][3], fma(-u[2], pi[l][2], fma(-u[1], pi[l][1], pi[l][0] * u[0])));
    if (l == 3) o *= rg;
    rho = nmax(rho, fabs(o) * den);
  }
  if (below(rho, R(1e-4))) return R(1) - rho * rho * R(1.0 / 3.0);
  return sdiv(tanh(rho), rho);
}

// ---------------------------------------------------------------- f) stores with ghosts
template <typename R>
__device__ __forceinline__ void store_cell(const StageIO<R>& io, long long fs, Idx<R> t, const double (&qn)[NQ],
                                           const R (&qr)[NQ], const R (&uo)[4], R e, R P0) {
#pragma unroll
  for (int n = 0; n < NQ; ++n) put(io.q_out + n * fs, t, qn[n]);
  if (io.qr_out) {
#pragma unroll
    for (int n = 0; n < NQ; ++n) put(io.qr_out + n * fs, t, qr[n]);
  }
#pragma unroll
  for (int m = 0; m < 4; ++m) put(io.u_out + m * fs, t, uo[m]);
  put(io.e_out, t, e);
  put(io.p_out, t, P0);
}

// padded ghost coordinate g in {0, 1, n+2, n+3} that copies the physical padded coordinate p
__device__ __forceinline__ int ghost_source(int g, int n, int periodic) {
  if (periodic) return 2 + (((g - 2) % n) + n) % n;
  return (g < 2) ? 2 : n + 1;
}

// calls f(t) for the element index t = t0 of the padded cell (i, j, k) and of every ghost cell that
// copies it (Eqs. ghostCells_1/2, or the periodic images).  The ghosts of a boundary cell go through one
// rolled loop: unrolled, its twelve copies of the stores were most of the kernels' code.
template <typename I, typename F>
__device__ __forceinline__ void for_cell_and_ghosts(const Params& P, const Lattice& L, I t0, int i, int j, int k, F&& f) {
  f(t0);
  if (i > 3 && i < L.nx && j > 3 && j < L.ny && k > 3 && k < L.nz) return;  // interior cells own no ghost
#pragma unroll 1
  for (int a = 0; a < 12; ++a) {
    const int ax = a >> 2, g = a & 3;
    const int n = (ax == 0) ? L.nx : ((ax == 1) ? L.ny : L.nz), p = (ax == 0) ? i : ((ax == 1) ? j : k);
    const int pos = (g < 2) ? g : n + g;
    if (ghost_source(pos, n, P.periodic) != p) continue;
    const long long step = (ax == 0) ? 1 : ((ax == 1) ? (long long)L.pitch : L.plane);
    f((I)(t0 + (I)((pos - p) * step)));
  }
}

template <typename R>
__device__ __forceinline__ void store_with_ghosts(const Params& P, const Lattice& L, const StageIO<R>& io, int i,
                                                  int j, int k, const double (&qn)[NQ], const R (&qr)[NQ],
                                                  const R (&uo)[4], R e, R P0) {
  const long long fs = L.fstride;
  for_cell_and_ghosts(P, L, cell_idx<R>(L, i, j, k), i, j, k,
                      [&](Idx<R> t) { store_cell<R>(io, fs, t, qn, qr, uo, e, P0); });
}

// ---------------------------------------------------------------- a) + b) for one cell
// dq = C[q] of Eq. (semiDiscreteKT) at the cell c: -div H in x, y, eta plus the source vector
// J = S + G (App. B), in the stencil precision R, evaluated at tau.  In three parts: the cell's
// face data (velocities, speeds, flux weights, d_d u^mu, d_i v^i, pressure part of S_c), the 15
// components' fluxes (conserved_fluxes or a shared-memory loop), then the sources.
template <typename R>
struct CellGeom {
  R tau, gnn, inv_gnn;
};
template <typename R>
__device__ __forceinline__ CellGeom<R> cell_geom(const Params& P, double tau_src) {
  CellGeom<R> g;
  g.tau = from_f64<R>(tau_src);
  g.gnn = P.milne ? g.tau * g.tau : R(1);
  g.inv_gnn = P.milne ? sdiv(R(1), g.gnn) : R(1);
  return g;
}

// d_i v^i from the differences v^d_{i+1} - v^d_{i-1}
template <typename R>
__device__ __forceinline__ R divergence(const Params& P, const R (&d)[3]) {
  const R* h = pr<R>(P).half_inv_d;
  return fma(d[2], h[2], fma(d[1], h[1], rmul(d[0], h[0])));
}

// the three directions' face setups; uc returns u^mu at the cell
template <typename R, bool TH1, bool IFACE, typename UA>
__device__ __forceinline__ void cell_faces(const Params& P, const Lattice& L, const StageIO<R>& io, Idx<R> c,
                                           const UA& ua, const CellGeom<R>& G, R (&dq)[NQ], R (&uc)[4],
                                           R (&du)[4][4], R& dv, float& amax, Faces<R>& Fx, Faces<R>& Fy,
                                           Faces<R>& Fz) {
#pragma unroll
  for (int n = 0; n < NQ; ++n) dq[n] = R(-0.0);  // exact additive identity
#pragma unroll
  for (int m = 0; m < 4; ++m) uc[m] = ua(m, 0);
  const R sfac = P.milne ? G.tau : R(1);  // sqrt(-g_{eta eta}): speeds along eta in units of c
  R d[3] = {R(0), R(0), R(0)};
  if constexpr (sizeof(R) == 8 && !IFACE) {
    if (L.nx > 1) face_setup<R, 0, TH1, IFACE>(P, L, io, c, ua, uc, G.inv_gnn, sfac, dq, du, d[0], amax, Fx);
    else face_none<R, 0>(uc, R(1), du, amax, Fx);
    if (L.ny > 1) face_setup<R, 1, TH1, IFACE>(P, L, io, c, ua, uc, G.inv_gnn, sfac, dq, du, d[1], amax, Fy);
    else face_none<R, 1>(uc, R(1), du, amax, Fy);
    if (L.nz > 1) face_setup<R, 2, TH1, IFACE>(P, L, io, c, ua, uc, G.inv_gnn, sfac, dq, du, d[2], amax, Fz);
    else face_none<R, 2>(uc, sfac, du, amax, Fz);
  } else {
    face_setup<R, 0, TH1, IFACE>(P, L, io, c, ua, uc, G.inv_gnn, sfac, dq, du, d[0], amax, Fx);
    face_setup<R, 1, TH1, IFACE>(P, L, io, c, ua, uc, G.inv_gnn, sfac, dq, du, d[1], amax, Fy);
    face_setup<R, 2, TH1, IFACE>(P, L, io, c, ua, uc, G.inv_gnn, sfac, dq, du, d[2], amax, Fz);
  }
  dv = divergence<R>(P, d);
}

template <typename R, bool DIAG = false>
__device__ __forceinline__ void cell_sources(const Params& P, const Lattice& L, const StageIO<R>& io, Idx<R> c,
                                             const CellGeom<R>& G, const R (&uc)[4], R (&du)[4][4], R dv,
                                             R (&dq)[NQ], R* dg = nullptr);

template <typename R, bool TH1 = false, bool IFACE = false>
__device__ __forceinline__ void cell_rhs(const Params& P, const Lattice& L, const StageIO<R>& io, Idx<R> c,
                                         double tau_src, R (&dq)[NQ], float& amax) {
  const CellGeom<R> G = cell_geom<R>(P, tau_src);
  R uc[4], du[4][4];
  R dv;
  Faces<R> F[3];
  cell_faces<R, TH1, IFACE>(P, L, io, c, u_global(L, io, c), G, dq, uc, du, dv, amax, F[0], F[1], F[2]);
  conserved_fluxes<R, TH1>(P, L, io, c, F, dq);
  cell_sources<R>(P, L, io, c, G, uc, du, dv, dq);
}

// The source vector J = S + G of App. B at the cell, added to dq.  DIAG: also the validity
// diagnostics of Sec. 7 into dg[0..5]: tau_pi theta, tau_Pi theta (unfloored relaxation times),
// sqrt(pi.pi)/P0, |Pi|/P0, sqrt(J^{mu nu} J_{mu nu})/(2 eta sqrt(sigma.sigma)) and |J|/(zeta
// |theta|) with J^{mu nu}, J the second-order terms of Eq. (14_moment_terms) (no diffusion); a
// quantity whose channel is off, or whose denominator vanishes, is 0.
//
// The transport coefficients depend on e alone and nothing here reads the fluxes, so a kernel with warps
// to spare computes both beside them: `out` says where the terms go and may bring the coefficients.
template <typename R>
struct Transport {
  R T, lnd, es, rate_pi, rate_Pi, d;  // d = 1/3 - c_s^2
};
// T(e) and ln(1/3 - c_s^2)(e) are given; the rates are bounded by the step
template <typename R>
__device__ __forceinline__ void shear_transport(const Params& P, Transport<R>& tr) {
  tr.es = eta_over_s<R>(P, tr.T);
  const R rate = (tr.es > R(0)) ? ((P.eta.kind == 0) ? tr.T * pr<R>(P).eta_inv_5c0 : sdiv(tr.T, R(5) * tr.es)) : R(INFINITY);
  tr.rate_pi = nmin(rate, pr<R>(P).rate_max);
}
template <typename R>
__device__ __forceinline__ void bulk_transport(const Params& P, Transport<R>& tr) {
  tr.d = sexp(tr.lnd);
  // 1/tau_Pi = 15 (1/3 - c_s^2)^2 T / (zeta/s): both factors span hundreds of e-folds away from the
  // transition, so their quotient is formed in the exponent (Eq. (zetas), bounded below, divides)
  R rate;
  if (P.zeta.kind == 2) {
    const R z = pr<R>(P).zeta_c0 * zeta_over_s_paper<R>(tr.T * pr<R>(P).zeta_inv_c1);
    rate = (z > R(0)) ? sdiv(R(15) * tr.d * tr.d * tr.T, z) : R(INFINITY);
  } else {
    rate = R(15) * tr.T * sexp(fma(R(2), tr.lnd, -ln_zeta_over_s<R>(P, tr.T)));
  }
  tr.rate_Pi = nmin(rate, pr<R>(P).rate_max);
}
// the terms added to dq at once, the coefficients formed where they are used
template <typename R>
struct SourceDirect {
  static constexpr bool kHasTransport = false;
  Transport<R> tr;
  R (&dq)[NQ];
  __device__ __forceinline__ void conserved(int n, R it, R qn) { dq[n] = fma(-it, qn, dq[n]); }
  __device__ __forceinline__ void energy(R x) { dq[0] -= x; }
  __device__ __forceinline__ void shear(int n, R iu0, R s) { dq[n] = fma(iu0, s, dq[n]); }
  __device__ __forceinline__ void bulk(R x) { dq[14] += x; }
};

template <typename R, bool DIAG, typename Out>
__device__ __forceinline__ void cell_sources_to(const Params& P, const Lattice& L, const StageIO<R>& io, Idx<R> c,
                                                const CellGeom<R>& G, const R (&uc)[4], R (&du)[4][4], R dv,
                                                Out& out, R* dg) {
  if constexpr (DIAG) {
#pragma unroll
    for (int k = 0; k < 6; ++k) dg[k] = R(0);
  }
  const long long fs = L.fstride;
  const R tau = G.tau, gnn = G.gnn, inv_gnn = G.inv_gnn;
  // ---- b) sources at the cell
#pragma unroll
  for (int m = 0; m < 4; ++m) {
    du[0][m] = rmul(uc[m] - ld<R>(io.u_prev + m * fs, c), pr<R>(P).inv_dtau);  // backward difference
  }
  const R* q = io.qr_in;
  R pi[4][4];
#pragma unroll
  for (int a = 0; a < 4; ++a)
#pragma unroll
    for (int b = a; b < 4; ++b) {
      pi[a][b] = ld<R>(q + pix(a, b) * fs, c);
      pi[b][a] = pi[a][b];
    }
  const R Pic = ld<R>(q + 14 * fs, c);
  const R ec = ld<R>(io.e_in, c), P0c = ld<R>(io.p_in, c);
  const R Pt = P0c + Pic;
  const R it = P.milne ? tau * inv_gnn : R(0);  // Gamma^eta_{tau eta} = 1/tau
  const R tg = P.milne ? tau : R(0);         // Gamma^tau_{eta eta}

  // geometric sources of the conservation laws, Eqs. (dT001)-(dT0i1)
  {
    R Tnn = (ec + Pt) * uc[3] * uc[3] + Pt * inv_gnn + pi[3][3];
    out.energy(fma(tg, Tnn, rmul(ld<R>(q, c), it)));
    out.conserved(1, it, ld<R>(q + fs, c));
    out.conserved(2, it, ld<R>(q + 2 * fs, c));
    out.conserved(3, it, rmul(R(3), ld<R>(q + 3 * fs, c)));
  }

  if (P.shear_on || P.bulk_on) {
    const R gup[4] = {R(1), R(-1), R(-1), -inv_gnn};
    // u^m_{;a} = d_a u^m + Gamma^m_{a b} u^b in place of du[a][m] (only Gamma^eta_{tau eta} = 1/tau and
    // Gamma^tau_{eta eta} = tau)
    du[3][0] = fma(tg, uc[3], du[3][0]);
    du[0][3] = fma(it, uc[3], du[0][3]);
    du[3][3] = fma(it, uc[0], du[3][3]);
    const R theta = du[0][0] + du[1][1] + du[2][2] + du[3][3];
    const R th3 = rmul(theta, R(1.0 / 3.0));
    R D[4], hD[4], th3u[4];  // D u^m, half of it, theta u^m / 3
#pragma unroll
    for (int m = 0; m < 4; ++m) {
      D[m] = fma(uc[0], du[0][m], fma(uc[1], du[1][m], fma(uc[2], du[2][m], uc[3] * du[3][m])));
      hD[m] = R(0.5) * D[m];
      th3u[m] = th3 * uc[m];
    }
    // The relaxation terms of pi^{ab} are contractions of pi with matrices built from u^m_{;a}:
    //   I_1 = pi^{al} D u_l u^b + (a <-> b),  I_3 = pi^a_l omega^{bl} + (a <-> b),
    //   I_4 = pi^a_l sigma^{bl} / 2 + (a <-> b) - Delta^{ab} pi:sigma / 3,
    //   G_pi^{ab} = K^a_l pi^{lb} + (a <-> b), K^0_3 = tau u^eta, K^3_0 = u^eta/tau, K^3_3 = u^tau/tau
    // so -(I_1 - I_3 + (tau_pipi/tau_pi) I_4) - G_pi is ONE product with Y^{bl} = -u^b D u^l +
    // omega^{bl} - (tau_pipi/(2 tau_pi)) sigma^{bl}, and with G^{bl} = g^{bb} u^l_{;b} the u D terms of
    // omega (= (G^{lb} - G^{bl} - u^l D^b + u^b D^l)/2) combine to
    //   Y^{bl} = (G^{lb} - G^{bl})/2 - (u^b D^l + u^l D^b)/2 - (tau_pipi/(2 tau_pi)) sigma^{bl}.
    // Terms proportional to pi^{ab} itself go on the diagonal of the matrix.  One 4x4 product in place
    // of three (I_1, I_3, I_4), without nabla^a u^m and omega as arrays.  (Products that several sums
    // read are formed by rmul, so that no kernel contracts them into a different multiply-add.)
    // FP64 is bound by its pipe (one warp instruction per 19 cycles and SM), so every product saved
    // counts: three 128^3 steps with set and get 44.4 -> 39.2 ms; FP32, bound by issue: six learned
    // 128^3 steps 7.31 -> 7.18 ms, FP32 pi storage at 96x96x64 2.64 -> 2.52 ms.
    R G[4][4];
#pragma unroll
    for (int l = 0; l < 4; ++l) {
      G[0][l] = du[0][l];
      G[1][l] = -du[1][l];
      G[2][l] = -du[2][l];
      G[3][l] = rmul(gup[3], du[3][l]);
    }
    const R hk = R(0.5) * pr<R>(P).tpp;
    R sig[4][4], Y[4][4];  // sigma^{ab} (a <= b), Y^{bl}
#pragma unroll
    for (int a = 0; a < 4; ++a) {
      const R uD = rmul(uc[a], D[a]);
      const R sd = fma(th3u[a], uc[a], G[a][a] - uD);
      sig[a][a] = (a == 0) ? sd - th3 : ((a == 3) ? fma(-gup[3], th3, sd) : sd + th3);
      Y[a][a] = fma(-hk, sig[a][a], -uD);
#pragma unroll
      for (int b = a + 1; b < 4; ++b) {
        const R hW = fma(uc[a], hD[b], uc[b] * hD[a]);
        sig[a][b] = fma(th3u[a], uc[b], fma(R(0.5), G[a][b] + G[b][a], -hW));
        const R s = fma(-hk, sig[a][b], -hW), A = G[b][a] - G[a][b];
        Y[a][b] = fma(R(0.5), A, s);
        Y[b][a] = fma(R(-0.5), A, s);
      }
    }
    // pi^{mu nu} sigma_{mu nu}, by powers of g_{eta eta} = -gnn
    const R psd = fma(pi[0][0], sig[0][0], fma(pi[1][1], sig[1][1], pi[2][2] * sig[2][2]));
    const R pso = fma(pi[1][2], sig[1][2], -fma(pi[0][1], sig[0][1], pi[0][2] * sig[0][2]));
    const R psn = fma(pi[1][3], sig[1][3], fma(pi[2][3], sig[2][3], -(pi[0][3] * sig[0][3])));
    const R ps = fma(gnn, fma(gnn, pi[3][3] * sig[3][3], R(2) * psn), fma(R(2), pso, psd));

    // transport coefficients (Sec. 2.2) from T(e), ln(1/3 - c_s^2)(e)
    Transport<R>& tr = out.tr;
    if constexpr (!Out::kHasTransport) eos_T_lnd<R>(P, ec, tr.T, tr.lnd);
    const R iu0 = sdiv(R(1), uc[0]);

    if (P.shear_on) {
      const R eta_tp = (ec + P0c) * R(0.2);
      if constexpr (!Out::kHasTransport) shear_transport<R>(P, tr);
      const R tp3 = pr<R>(P).tpp * ps * R(1.0 / 3.0);
      const R csig = fma(R(1.2), Pic, R(2) * eta_tp);
      if constexpr (DIAG) {  // sums over the full tensor: off-diagonal pairs count twice
        const R glo[4] = {R(1), R(-1), R(-1), -gnn};
        R xs = R(0);
#pragma unroll
        for (int a = 0; a < 4; ++a)
#pragma unroll
          for (int b = a; b < 4; ++b) {
            R c = R(0);  // pi^a_l (omega^{bl} - (tau_pipi/(2 tau_pi)) sigma^{bl}) + (a <-> b)
#pragma unroll
            for (int l = 0; l < 4; ++l)
              c += glo[l] * (pi[a][l] * fma(uc[b], D[l], Y[b][l]) + pi[b][l] * fma(uc[a], D[l], Y[a][l]));
            const R w = glo[a] * glo[b] * ((a == b) ? R(1) : R(2));
            const R Dab = ((a == b) ? gup[a] : R(-0.0)) - uc[a] * uc[b];
            const R X = R(4.0 / 3.0) * theta * pi[a][b] - c - tp3 * Dab - R(1.2) * Pic * sig[a][b];  // -J^{ab}/tau_pi
            dg[2] += pi[a][b] * pi[a][b] * w;
            dg[4] += X * X * w;
            xs += sig[a][b] * sig[a][b] * w;
          }
        dg[0] = sdiv(R(5) * tr.es, tr.T) * theta;
        dg[4] = (xs > R(0)) ? sdiv(sqrt(dg[4]), R(2) * eta_tp * sqrt(xs)) : R(0);
      }
      // M^b_l = g_{ll} Y^{bl} - K^b_l, and on its diagonal half of the coefficient of pi^{ab}:
      // -1/tau_pi - 4 theta/3 (delta_pipi) + u^tau d_i v^i (S_pi's pi d_i v^i, taken inside the 1/u^tau)
      const R hc = rmul(R(0.5), fma(uc[0], dv, fma(R(-4.0 / 3.0), theta, -tr.rate_pi)));
      R M[4][4];
#pragma unroll
      for (int b = 0; b < 4; ++b) {
        M[b][0] = Y[b][0];
        M[b][1] = -Y[b][1];
        M[b][2] = -Y[b][2];
        M[b][3] = rmul(-gnn, Y[b][3]);
      }
      M[0][3] = fma(-tg, uc[3], M[0][3]);
      M[3][0] = fma(-it, uc[3], M[3][0]);
      M[3][3] = fma(-it, uc[0], M[3][3] + hc);
      M[0][0] += hc;
      M[1][1] += hc;
      M[2][2] += hc;
#pragma unroll
      for (int a = 0; a < 4; ++a) {
        const R tpu = tp3 * uc[a];
        // diagonal: twice pi^{al} M^a_l
        R h = fma(pi[a][0], M[a][0], fma(pi[a][1], M[a][1], fma(pi[a][2], M[a][2], pi[a][3] * M[a][3])));
        const R dg0 = (a == 0) ? tp3 : ((a == 3) ? gup[3] * tp3 : -tp3);
        h = fma(R(2), h, fma(csig, sig[a][a], fma(-tpu, uc[a], dg0)));
        out.shear(pix(a, a), iu0, h);
#pragma unroll
        for (int b = a + 1; b < 4; ++b) {
          R s = fma(csig, sig[a][b], -(tpu * uc[b]));
#pragma unroll
          for (int l = 0; l < 4; ++l) s = fma(pi[a][l], M[b][l], fma(pi[b][l], M[a][l], s));
          out.shear(pix(a, b), iu0, s);
        }
      }
    }
    if (P.bulk_on) {
      if constexpr (!Out::kHasTransport) bulk_transport<R>(P, tr);
      const R d = tr.d;
      const R zt = R(15) * d * d * (ec + P0c);
      const R IPi = fma(R(2.0 / 3.0) * Pic, theta, -(R(1.6) * d * ps));
      out.bulk(fma(fma(-tr.rate_Pi, Pic, fma(-zt, theta, -IPi)), iu0, rmul(Pic, dv)));
      if constexpr (DIAG) {
        const R lrate = R(2.70805020110221) + R(2) * tr.lnd + slog(tr.T) - ln_zeta_over_s<R>(P, tr.T);  // ln 15 + ...
        dg[1] = sexp(-lrate) * theta;
        dg[5] = (theta != R(0)) ? sdiv(fabs(IPi), zt * fabs(theta)) : R(0);
      }
    }
    if constexpr (DIAG) {
      dg[2] = sdiv(sqrt(dg[2]), P0c);
      dg[3] = sdiv(fabs(Pic), P0c);
    }
  }
}

template <typename R, bool DIAG>
__device__ __forceinline__ void cell_sources(const Params& P, const Lattice& L, const StageIO<R>& io, Idx<R> c,
                                             const CellGeom<R>& G, const R (&uc)[4], R (&du)[4][4], R dv,
                                             R (&dq)[NQ], R* dg) {
  SourceDirect<R> out{Transport<R>{}, dq};
  cell_sources_to<R, DIAG>(P, L, io, c, G, uc, du, dv, out, dg);
}

// The inversion's inputs at one cell (Eqs. eInferred-uiInferred): E = T^tt - pi^tt,
// M^i = T^ti - pi^ti, Pi and M^2 = M_x^2 + M_y^2 + g_nn M_n^2 in FP64; E and M^2 also truncated to
// single precision for the network's features, the Newton step factor and the quick test of
// M^2 < E^2.
struct InvIn {
  double E, Mx, My, Mn, Pi, M2;
  float Ef, M2f;
};
__device__ __forceinline__ InvIn inv_in(double gnn, double E, double Mx, double My, double Mn, double Pi) {
  InvIn v;
  v.E = E; v.Mx = Mx; v.My = My; v.Mn = Mn; v.Pi = Pi;
  v.M2 = fma(gnn * Mn, Mn, fma(My, My, Mx * Mx));
  v.Ef = d2f_trunc(E);
  v.M2f = d2f_trunc(v.M2);
  return v;
}

// The network's start for the root-find of the inversion inputs v: the conformal root corrected
// by y = r^2 z (r^2 = M^2/E^2, feature 1), e = E (e_conf/E) exp(y/10), with z the network's
// output for this cell at the start of the step (mlp_start_kernel).  The correction vanishes at
// rest, where e_conf = E is the root, and the network's BF16 error scales with it; cells with
// r^2 <= kMlpGateR2 start from e_conf.
__device__ __forceinline__ double learned_start(const InvIn& v, float z) {
  float x[MLP_IN], ecE;
  mlp_features(fmaxf(v.Ef, 1e-30f), v.M2f, d2f_trunc(v.Pi), x, ecE);
  const float y = (x[1] > kMlpGateR2) ? x[1] * z : 0.f;
  return f2d_bits(v.Ef * ecE * __expf(0.1f * y));
}

// ---------------------------------------------------------------- one cell (FP64)
// Cell o of an event (x fastest, then y, then eta).  The 32 lanes of a warp hold consecutive cells and
// stay together; lanes past the last cell repeat it and store nothing.
struct CellAt {
  long long c;
  int i, j, k;
  bool valid;
};
__device__ __forceinline__ CellAt cell_at(const Lattice& L, unsigned o) {
  const unsigned ncells = (unsigned)L.nx * (unsigned)L.ny * (unsigned)L.nz;
  CellAt a;
  a.valid = o < ncells;
  o = min(o, ncells - 1u);
  const unsigned row = o / (unsigned)L.nx;
  a.i = (int)(o - row * (unsigned)L.nx);
  a.k = (int)(row / (unsigned)L.ny);
  a.j = (int)row - a.k * L.ny;
  a.c = L.idx(a.i + 2, a.j + 2, a.k + 2);
  return a;
}

// Everything after dq = C[q]: c) the Heun update, d) the inversion, e) the regulator, f) the stores
template <typename R, int STAGE>
__device__ __forceinline__ void stage_finish(const Params& P, const Lattice& L, const StageIO<R>& io, const CellAt& at,
                                             double tau_out, const R (&dq)[NQ], unsigned& st, unsigned& nit,
                                             unsigned& nreg) {
  static_assert(sizeof(R) == 8, "the fused stage is the FP64 path; mixed precision uses kt_split.cuh");
  const long long fs = L.fstride, c = at.c;
  double qn[NQ];  // the new conserved state
  // ---- c) Heun update in FP64 (Eqs. step1-finalStep)
#pragma unroll
  for (int n = 0; n < NQ; ++n) {
    const double qi = __ldg(io.q_in + n * fs + c);
    if (STAGE == 1)
      qn[n] = fma(dq[n], pr<R>(P).dtau, qi);  // q* = q^n + dtau C[q^n]
    else  // q^{n+1} = (q^n + q* + dtau C[q*]) / 2
      qn[n] = fma(0.5, io.q_base[n * fs + c] + qi, dq[n] * pr<R>(P).half_dtau);
  }

  {
    // ---- d) inversion at tau^{n+1}
    double e, P0;
    R uo[4];
    const double guess = to_f64<R>(ld<R>(io.e_in, c));
    unsigned its = 0;
    const unsigned sti = invert_fp64(P, tau_out, qn, guess, e, P0, uo, its);
    if (!at.valid) return;
    st |= sti;
    nit += its;

    // the new state in the stencil precision (the copy the next stage's stencil reads)
    R qr[NQ];
#pragma unroll
    for (int n = 0; n < NQ; ++n) qr[n] = from_f64<R>(qn[n]);
    const R eR = from_f64<R>(e), P0R = from_f64<R>(P0);

    // ---- e) regulator
    if (P.regulate) {
      const R go = P.milne ? from_f64<R>(tau_out * tau_out) : R(1);
      R pm[4][4];
#pragma unroll
      for (int a = 0; a < 4; ++a)
#pragma unroll
        for (int b = a; b < 4; ++b) {
          pm[a][b] = qr[pix(a, b)];
          pm[b][a] = pm[a][b];
        }
      const R f = regulator_factor<R>(P, go, from_f64<R>(tau_out), eR, P0R, uo, pm, qr[14]);
      if (below(f, R(0.999))) ++nreg;
      if (STAGE == 2 && io.reg_out) io.reg_out[c] = to_f32(f);
      if (differs(f, R(1))) {
        const double fd = to_f64<R>(f);
#pragma unroll
        for (int n = 4; n < 14; ++n) {
          qn[n] *= fd;
          qr[n] *= f;
        }
      }
    }
#pragma unroll
    for (int n = 0; n < NQ; ++n)
      if (!finite(qr[n])) st |= ST_NONFINITE;

    // ---- f) stores
    store_with_ghosts<R>(P, L, io, at.i + 2, at.j + 2, at.k + 2, qn, qr, uo, eR, P0R);
  }
}

// tau^{n+1} for the next step, written by one thread of the second stage into another slot than the one
// this step's kernels read (a launch of its own cost 2 us per step: 4% of a small grid's)
__device__ __forceinline__ void advance_tau(const Params& P, const TauSlot* tau, TauSlot* tau_next, bool first) {
  if (tau_next && first) *tau_next = tau_slot(tau->tau_out, P.dtau, P.milne);
}

// The contiguous run [t0, t1) of the tile table that this block processes.  Tiles are ordered
// eta-fastest, so a block of a persistent grid walks up a column of tiles and the eta-neighbour
// planes read by its stencil are mostly still in its SM's L1.
__device__ __forceinline__ void tile_range(int ntiles, int& t0, int& t1) {
  const int per = (ntiles + (int)gridDim.x - 1) / (int)gridDim.x;
  t0 = (int)blockIdx.x * per;
  t1 = min(ntiles, t0 + per);
}

// ---------------------------------------------------------------- per-launch statistics
// status bits OR-ed, the largest local speed (float bits, all non-negative), and the Newton /
// regulated / fallback counters: warp reductions, then one set of atomics per block.  Every
// thread of the block calls this once, after its last cell.  SPEED, COUNTS: which of them the kernel has.
template <bool SPEED, bool COUNTS>
__device__ __forceinline__ void block_stats(unsigned* status, unsigned* max_speed_bits,
                                            unsigned long long* counters, unsigned st, float amax, unsigned nit,
                                            unsigned nreg, unsigned nfb) {
  __shared__ unsigned s_stat[5];
  const unsigned full = 0xffffffffu;
  const int tid = threadIdx.x + blockDim.x * (threadIdx.y + blockDim.y * threadIdx.z);
  if (tid < 5) s_stat[tid] = 0u;
  __syncthreads();
  const unsigned w_st = __reduce_or_sync(full, st);
  unsigned w_max = 0, w_it = 0, w_reg = 0, w_fb = 0;
  if (SPEED) w_max = __reduce_max_sync(full, __float_as_uint(amax));
  if (COUNTS) {
    w_it = __reduce_add_sync(full, nit);
    w_reg = __reduce_add_sync(full, nreg);
    w_fb = __reduce_add_sync(full, nfb);
  }
  if ((tid & 31) == 0) {
    if (w_st) atomicOr(&s_stat[0], w_st);
    if (SPEED) atomicMax(&s_stat[1], w_max);
    if (COUNTS) {
      atomicAdd(&s_stat[2], w_it);
      if (w_reg) atomicAdd(&s_stat[3], w_reg);
      if (w_fb) atomicAdd(&s_stat[4], w_fb);
    }
  }
  __syncthreads();
  if (tid < 5) {
    const unsigned v = s_stat[tid];
    if (tid == 0 && v) atomicOr(status, v);
    if (SPEED && tid == 1) atomicMax(max_speed_bits, v);
    if (COUNTS && tid >= 2 && v) atomicAdd(counters + tid - 2, (unsigned long long)v);
  }
}

// ---------------------------------------------------------------- the stage kernel (FP64)
// One warp per block and per 32 consecutive cells of an event.  The kernel is bound by the FP64 pipe:
// measured, one warp instruction per 19 cycles and SM from four warps on (64 cycles for a lone warp),
// the same with one active lane as with 32.  Hence cells in linear order (a 32-wide tile of a 37-cell
// row would leave 27 of 64 lanes idle at full cost), and blocks of one warp, so that a grid with few
// cells spreads over all SMs and no SM's last wave holds eight warps.  Against 256-thread tiles on a
// grid of resident blocks: shock tube of 200 cells, 80 steps, 9.03 -> 3.83 ms (with the one-cell axes
// and vanishing components skipped), Gubser grid 32 x 32 x 8, 20 steps, 4.13 -> 3.58 ms, three 128^3
// steps 36.5 -> 35.9 ms.
__device__ __forceinline__ void warp_stats(const StageIO<double>& io, unsigned st, float amax, unsigned nit,
                                           unsigned nreg) {
  const unsigned full = 0xffffffffu;
  const unsigned w_st = __reduce_or_sync(full, st), w_max = __reduce_max_sync(full, __float_as_uint(amax));
  const unsigned w_it = __reduce_add_sync(full, nit), w_reg = __reduce_add_sync(full, nreg);
  if ((threadIdx.x & 31) == 0) {
    if (w_st) atomicOr(io.status, w_st);
    atomicMax(io.max_speed_bits, w_max);
    if (w_it) atomicAdd(io.counters + 0, (unsigned long long)w_it);
    if (w_reg) atomicAdd(io.counters + 1, (unsigned long long)w_reg);
  }
}

// strips: (event, first cell) of every block; with a single event (n_events = 1) the block index says it
template <typename R, int STAGE, bool TH1, bool IFACE>
__global__ void __launch_bounds__(32, 8)
    stage_kernel(const Params P, const StageIO<R> io, const Lattice L0, const Lattice* __restrict__ lats,
                 const Tile* __restrict__ strips, int n_events) {
  unsigned st = 0, nit = 0, nreg = 0;
  float amax = 0.f;
  Lattice L = L0;
  unsigned first = 32u * blockIdx.x;
  if (n_events > 1) {
    const Tile s = strips[blockIdx.x];
    L = lats[s.event];
    first = (unsigned)s.i0;
  }
  const CellAt at = cell_at(L, first + threadIdx.x);
  const double tau_n = io.tau->tau, tau_out = io.tau->tau_out;
  R dq[NQ];
  cell_rhs<R, TH1, IFACE>(P, L, io, at.c, (STAGE == 1) ? tau_n : tau_out, dq, amax);
  stage_finish<R, STAGE>(P, L, io, at, tau_out, dq, st, nit, nreg);
  __syncwarp();
  if (STAGE == 2) advance_tau(P, io.tau, io.tau_next, blockIdx.x == 0 && threadIdx.x == 0);
  warp_stats(io, st, amax, nit, nreg);
}

// ---------------------------------------------------------------- the same for grids with few cells (FP64)
// With fewer strips than the chip has FP64 issue slots (four warps per SM) the kernel above is a serial
// chain of ~1,500 FP64 instructions at 64 cycles each while most units idle.  Here four warps share a
// strip.  Warps 0-2 take one axis each for the face setup and then every third component of the fluxes;
// warp 3 meanwhile computes the transport coefficients and then the sources (as long a chain as five
// components); warp 0 adds up and runs the update.  Values pass through shared memory and are added in
// the order of the one-warp kernel, so both give the same bits.  Gubser grid 32 x 32 x 8 (256 strips), 20
// steps: 2.24 ms with the sources in warp 0 after the fluxes, 2.05 ms beside them (3.39 ms with one warp per
// strip); shock tube of 7 strips, 80 steps, 3.50 ms with one warp, 2.94 ms here.
enum : int { TM_FACE = 0, TM_DU = 18, TM_DV = 30, TM_PR = 33, TM_ACC = 39, TM_MIX = 54, TM_DIFF = 58, TM_SRC = 70,
             TM_IU0 = 85, TM_VALUES = 86 };

// the source terms left in shared memory for warp 0 (rows 1-3: the components they multiply)
template <typename R>
struct SourceShared {
  static constexpr bool kHasTransport = true;
  Transport<R> tr;
  R (*sm)[32];
  int lane;
  __device__ __forceinline__ void conserved(int n, R, R qn) { sm[TM_SRC + n][lane] = qn; }
  __device__ __forceinline__ void energy(R x) { sm[TM_SRC][lane] = x; }
  __device__ __forceinline__ void shear(int n, R iu0, R s) {
    sm[TM_SRC + n][lane] = s;
    sm[TM_IU0][lane] = iu0;
  }
  __device__ __forceinline__ void bulk(R x) { sm[TM_SRC + 14][lane] = x; }
};

template <typename R, int D, bool TH1>
__device__ __forceinline__ void team_faces(const Params& P, const Lattice& L, const StageIO<R>& io, Idx<R> c,
                                           const CellGeom<R>& G, R (*sm)[32], float& amax) {
  const int lane = threadIdx.x & 31;
  const UGlobal<R> ua = u_global(L, io, c);
  const R sfac = P.milne ? G.tau : R(1);
  R uc[4], du[4][4], dq[NQ], dvd = R(0);
  Faces<R> F;
#pragma unroll
  for (int m = 0; m < 4; ++m) uc[m] = ua(m, 0);
  dq[0] = dq[D + 1] = R(-0.0);
  const int n = (D == 0) ? L.nx : ((D == 1) ? L.ny : L.nz);
  if (n > 1) face_setup<R, D, TH1, false>(P, L, io, c, ua, uc, G.inv_gnn, sfac, dq, du, dvd, amax, F);
  else face_none<R, D>(uc, (D == 2) ? sfac : R(1), du, amax, F);
  const R f[6] = {F.c0, F.wLm, F.wRp, F.hdW, F.vpl_h, F.vmi_h};
#pragma unroll
  for (int m = 0; m < 6; ++m) sm[TM_FACE + 6 * D + m][lane] = f[m];
#pragma unroll
  for (int m = 0; m < 4; ++m) sm[TM_DU + 4 * D + m][lane] = du[D + 1][m];
  sm[TM_DV + D][lane] = dvd;
  sm[TM_PR + 2 * D][lane] = dq[0];
  sm[TM_PR + 2 * D + 1][lane] = dq[D + 1];
}

template <typename R, int STAGE, bool TH1>
__global__ void __launch_bounds__(128, 2)
    stage_team_kernel(const Params P, const StageIO<R> io, const Lattice L0, const Lattice* __restrict__ lats,
                      const Tile* __restrict__ strips, int n_events) {
  __shared__ R sm[TM_VALUES][32];
  unsigned st = 0, nit = 0, nreg = 0;
  float amax = 0.f;
  Lattice L = L0;
  unsigned first = 32u * blockIdx.x;
  if (n_events > 1) {
    const Tile s = strips[blockIdx.x];
    L = lats[s.event];
    first = (unsigned)s.i0;
  }
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const CellAt at = cell_at(L, first + lane);
  const double tau_n = io.tau->tau, tau_out = io.tau->tau_out;
  const CellGeom<R> G = cell_geom<R>(P, (STAGE == 1) ? tau_n : tau_out);
  const long long fs = L.fstride, c = at.c;
  const bool on[3] = {L.nx > 1, L.ny > 1, L.nz > 1};
  const int s[3] = {1, L.pitch, (int)L.plane};
  const R* p = io.qr_in + c;
  Stencil13<R> q;
  SourceShared<R> src{Transport<R>{}, sm, lane};
  if (warp < 3) q = load_stencil<R>(p + warp * fs, on, s);  // in flight during the face setup
  if (warp == 0) team_faces<R, 0, TH1>(P, L, io, c, G, sm, amax);
  else if (warp == 1) team_faces<R, 1, TH1>(P, L, io, c, G, sm, amax);
  else if (warp == 2) team_faces<R, 2, TH1>(P, L, io, c, G, sm, amax);
  else if (P.shear_on || P.bulk_on) {
    eos_T_lnd<R>(P, ld<R>(io.e_in, c), src.tr.T, src.tr.lnd);
    if (P.shear_on) shear_transport<R>(P, src.tr);
    if (P.bulk_on) bulk_transport<R>(P, src.tr);
  }
  __syncthreads();
  if (warp == 3) {
    const R d[3] = {sm[TM_DV][lane], sm[TM_DV + 1][lane], sm[TM_DV + 2][lane]};
    R uc[4], du[4][4];
#pragma unroll
    for (int m = 0; m < 4; ++m) {
      uc[m] = ld<R>(io.u_in + m * fs, c);
#pragma unroll
      for (int a = 0; a < 3; ++a) du[a + 1][m] = sm[TM_DU + 4 * a + m][lane];
    }
    cell_sources_to<R, false>(P, L, io, c, G, uc, du, divergence<R>(P, d), src, nullptr);
  } else {
    Faces<R> F[3];
#pragma unroll
    for (int d = 0; d < 3; ++d)
      F[d] = Faces<R>{sm[TM_FACE + 6 * d][lane], sm[TM_FACE + 6 * d + 1][lane], sm[TM_FACE + 6 * d + 2][lane],
                      sm[TM_FACE + 6 * d + 3][lane], sm[TM_FACE + 6 * d + 4][lane], sm[TM_FACE + 6 * d + 5][lane], s[d]};
    const R c0 = sum_c0<R>(F, on), th = pr<R>(P).theta;
#pragma unroll 1
    for (int n = warp; n < NQ; n += 3) {
      const Stencil13<R> next = load_stencil<R>(p + min(n + 3, NQ - 1) * fs, on, s);
      R acc = R(-0.0), mix = R(-0.0);  // (adding -0 changes nothing)
      const bool any = stencil_nonzero<R>(q);
      if (any) stencil_flux<R, TH1>(q, c0, on, F, th, n >= 4 && n <= 7, acc, mix);
      sm[TM_ACC + n][lane] = acc;
      if (n >= 4 && n <= 7) sm[TM_MIX + n - 4][lane] = mix;
      if (n >= 4 && n <= 13) {
        const int r[3] = {cross_row<0>(n, false), cross_row<1>(n, false), cross_row<2>(n, false)};
#pragma unroll
        for (int d = 0; d < 3; ++d)
          if (r[d] >= 0) sm[TM_DIFF + 4 * d + r[d]][lane] = (any && on[d]) ? q.v[d][1] - q.v[d][2] : R(-0.0);
      }
      q = next;
    }
  }
  __syncthreads();
  if (warp > 0) {
    warp_stats(io, 0u, amax, 0u, 0u);
    return;
  }
  R dq[NQ];
#pragma unroll
  for (int n = 0; n < NQ; ++n) dq[n] = R(-0.0);
#pragma unroll
  for (int d = 0; d < 3; ++d) {
    dq[0] += sm[TM_PR + 2 * d][lane];
    dq[d + 1] += sm[TM_PR + 2 * d + 1][lane];
  }
#pragma unroll
  for (int n = 0; n < NQ; ++n) {
#pragma unroll
    for (int d = 0; d < 3; ++d) {
      const int r = (d == 0) ? cross_row<0>(n, false) : ((d == 1) ? cross_row<1>(n, false) : cross_row<2>(n, false));
      if (n >= 4 && n <= 13 && r >= 0) dq[r] = fma(sm[TM_DIFF + 4 * d + r][lane], pr<R>(P).half_inv_d[d], dq[r]);
    }
    dq[n] += sm[TM_ACC + n][lane];
    if (n >= 4 && n <= 7) dq[n - 4] += sm[TM_MIX + n - 4][lane];
  }
  SourceDirect<R> out{Transport<R>{}, dq};
  const R it = P.milne ? G.tau * G.inv_gnn : R(0);
  out.energy(sm[TM_SRC][lane]);
#pragma unroll
  for (int n = 1; n < 4; ++n) out.conserved(n, it, sm[TM_SRC + n][lane]);
  if (P.shear_on) {
#pragma unroll
    for (int n = 4; n < 14; ++n) out.shear(n, sm[TM_IU0][lane], sm[TM_SRC + n][lane]);
  }
  if (P.bulk_on) out.bulk(sm[TM_SRC + 14][lane]);
  stage_finish<R, STAGE>(P, L, io, at, tau_out, dq, st, nit, nreg);
  __syncwarp();
  if (STAGE == 2) advance_tau(P, io.tau, io.tau_next, blockIdx.x == 0 && threadIdx.x == 0);
  warp_stats(io, st, amax, nit, nreg);
}

}  // namespace kt
