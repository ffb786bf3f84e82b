// Massive-particle variant, m = 5 T0 (Sec. 2.3, Fig. m5-stencil): the fused
// stream + collide kernel, its helpers and the C ABI of
// include/rlbm_massive.h.
//
// One thread per site.  Per step (Eq. discrete-rbe): pull the 45 post-
// collision populations (periodic wrap or on-site bounce-back), moments
// N^a, T^ab as deviations from the rest values, Landau frame with the
// massive equation of state, equilibrium, Anderson-Witting relaxation,
// uniform force, store.  Every stored value is the relative deviation
// g_i = (f_i - f0_i) / f0_i from the rest populations f0_i = w_i / (m + 1)
// (f^eq at n = T = 1, u = 0).
//
// Equilibrium.  g^eq_i = (m + 1) m(p_i)^T G^-1 M(n, U, T) - 1 (projection
// of the Maxwell-Juttner distribution onto the polynomials of degree <= 3,
// Eq. feq-expansion-discrete; m the 16 monomials, G their Gram matrix
// under the weight function, M their Maxwell-Juttner moments).  The
// entries of (m + 1) m^T G^-1 reach 3e4 (1 and p0 are nearly collinear on
// the nodes), so the kernel never applies them to rounded O(delta) moments:
// with delta = (n - 1, T - 1, ux, uy),
//   g^eq_i = dn + L_i . (dT, ux, uy) + W_i . (quadratic monomials of delta)
//          + B_i . R3(delta),
// L and W exact per-node tables, and R3 the moments minus their linear and
// quadratic parts, written out below without cancellation (each term is a
// product of small factors).  The Maxwell-Juttner moments are
//   M[1] = n / (m + T),   M[p^a] = n U^a,   M[p^a p^b] = h U^a U^b - P eta^ab,
//   M[p^a p^b p^c] = alpha U^a U^b U^c - T h (U^a eta^bc + U^b eta^ac + U^c eta^ab),
// with P = n T, h = eps + P = n (m^2 + 3 m T + 3 T^2) / (m + T) and
// alpha = n (m^3 + 6 m^2 T + 15 m T^2 + 15 T^3) / (m + T) (rest-frame
// integrals of exp(-p0 / T) on the mass shell).
#include "rlbm_massive.h"

#include <cuda_runtime.h>

#include <cmath>
#include <cstdarg>
#include <cstdio>
#include <cstring>
#include <mutex>
#include <new>
#include <string>

#include "massive_tables.h"
#include "site.cuh"

namespace rlbm {
namespace massive {
namespace {

// physical constants at T0 = 1, m = 5
constexpr double kM = kMass;
constexpr double kM1 = kMass + 1;
constexpr double kE0 = (kM * kM + 2 * kM + 2) / kM1;            // eps at rest   37/6
constexpr double kH0 = (kM * kM + 3 * kM + 3) / kM1;            // eps + P       43/6
constexpr double kK1 = (2 * kM * kM + 6 * kM + 3) / (kM1 * kM1); // dh/dT          83/36
constexpr double kA0 = (kM * kM * kM + 6 * kM * kM + 15 * kM + 15) / kM1;   // alpha 365/6
constexpr double kC2 = kM * kM / (kM1 * kM1 * kM1);             // 25/216
constexpr double kSD0 = 2 * kM + 4 - kE0;                        // sqrt of the EOS discriminant at rest

// Tables of the step.  A class holds the vectors of one energy: axis (a, 0),
// diagonal (a, a), or eight (a, b) with a > b > 0.  By the square's symmetry a
// class needs one row for the radial part of g^eq, one for its (px^2 - py^2)
// part, one for its px py part and, per component magnitude, one for the part
// odd in that component; the pairs of the class follow by additions:
//   g^eq(a, b) even = A + C1 + C2, (-a, b): A + C1 - C2, (b, a): A - C1 + C2, ..
//   odd(a, b) = X_a + Y_b, (-a, b): -X_a + Y_b, (b, a): X_b + Y_a, ..
// 117 paired + 75 scalar operations per site in FP32 where 22 separate rows
// of 28 took 275 paired ones.
template <typename R> struct V2 { using T = double2; };
template <> struct V2<float> { using T = float2; };

// component functions: axis and diagonal classes one, classes of eight two
constexpr int kOddFns = 11;
__host__ __device__ constexpr int class_kind(int c) {      // 0 axis, 1 diagonal, 2 eight
  return c == 3 || c == 6 ? 2 : c == 1 || c == 4 || c == 7 ? 1 : 0;
}
__host__ __device__ constexpr int class_pair(int c) {      // first pair of class c
  return c == 0 ? 0 : c == 1 ? 2 : c == 2 ? 4 : c == 3 ? 6 : c == 4 ? 10 : c == 5 ? 12 : c == 6 ? 14
       : c == 7 ? 18 : 20;
}
__host__ __device__ constexpr int class_fn(int c) {        // first component function of class c
  return c <= 3 ? c : c <= 6 ? c + 1 : c + 2;
}

template <typename R>
struct MConsts {
  using V = typename V2<R>::T;
  // moments: f0 times 1, p0, (p^x v^x + p^y v^y) / 2, its difference, p^x v^y
  R mN0[kClasses], mE[kClasses], mPs[kClasses], mPd[kClasses], mPxy[kClasses];
  V mN[kOddFns], mM[kOddFns];   // f0 v and f0 p of the component, both lanes alike
  R A[kClasses][8];      // dT, dn dT, dT^2, ux^2 + uy^2, E0, E1, E2 + E4, E5 + E7 (9: rest)
  R C1[kClasses][3];     // ux^2 - uy^2, E2 - E4, E5 - E7
  R C2[kClasses][3];     // ux uy, E3, E6
  V O[kOddFns][7];       // (x, y) lanes alike: u, dn u, dT u, O0/O1, O2/O3, O4/O7, O6/O5
  V va[kOddFns], pa[kOddFns];   // v and p of the component, both lanes alike
  R p0[kClasses], rr[kClasses], dd[kClasses], pp[kClasses];   // (px^2 +- py^2) / 2, |px py|
  // (m + 1) G^-1 by symmetry.  Even rows, negated (the source takes them with
  // that sign): p0; px^2 + py^2 and its difference; px py; the same times p0.
  // Columns: 1, p0, px^2 + py^2, p0 (px^2 + py^2), or those of one parity.
  // Odd rows and columns px, p0 px, px^3, px py^2, in lanes with py, p0 py, ..
  R n1[4], nS[4], n0S[4], nD[2], n0D[2], nX[2], n0X[2];
  V gO[4][4];
  double f0[kQm], if0[kQm], ifl[kQm];      // 1 / f0 = if0 + ifl
};

__constant__ MConsts<float> c_f;
__constant__ MConsts<double> c_d;

template <typename R> __device__ __forceinline__ const MConsts<R>& mc();
template <> __device__ __forceinline__ const MConsts<float>& mc<float>() { return c_f; }
template <> __device__ __forceinline__ const MConsts<double>& mc<double>() { return c_d; }

constexpr int kMThreads = 64;

struct MGeom {
  int nx, ny, ldx;
  int px, py;            // periodic axes
  long long plane;       // elements per population plane
};

template <typename R>
struct MMacro {
  R ux, uy, gamma, gm1, r1;  // gm1 = gamma - 1, r1 = 1 / (1 + sqrt(1 - u^2))
  R dn, dT;                  // n - 1, T - 1
};

template <typename R>
struct MMom {
  R dN0, dNx, dNy;           // N^a - (1, 0, 0)
  R dE, Mx, My;              // T^00 - eps0, T^0x, T^0y
  R dPxx, dPxy, dPyy;        // T^ij - delta_ij
};

// Byte offsets, prepared on the host: from a site to the source of each pull
// (interior sites) and to each population plane.
struct MOffsets {
  long long pull[kQm], plane[kQm];
};

template <typename S>
__device__ __forceinline__ const S* at_bytes(const S* p, long long b) {
  return reinterpret_cast<const S*>(reinterpret_cast<const char*>(p) + b);
}
template <typename S>
__device__ __forceinline__ S* at_bytes(S* p, long long b) {
  return reinterpret_cast<S*>(reinterpret_cast<char*>(p) + b);
}

// A load that stays behind the wait for the predecessor's results (an ordinary
// read-only one may be moved above it), coherent because the predecessor may
// still write the buffer when this kernel starts.
__device__ __forceinline__ float ld_pull(const float* p, uint64_t policy) {
  float v;
  asm volatile("ld.global.L2::cache_hint.f32 %0, [%1], %2;\n" : "=f"(v) : "l"(p), "l"(policy) : "memory");
  return v;
}
__device__ __forceinline__ double ld_pull(const double* p, uint64_t) {
  double v;
  asm volatile("ld.global.f64 %0, [%1];\n" : "=d"(v) : "l"(p) : "memory");
  return v;
}

// Which group of an NS-way split holds class c (the rest vector: class 9).
// The groups hold about the same number of pairs.
__host__ __device__ constexpr int class_group(int ns, int c) {
  return ns == 1 || c <= 3 || c == 9 ? 0 : 1;
}
__host__ __device__ constexpr bool mine(int ns, int g, int p) {
  return class_group(ns, pair_class(p)) == g;
}

// ---------------------------------------------------------------------------
// Pull streaming: f_i(x) = f*_i(x - n_i); a source outside a walled axis
// bounces back (the opposite population of the destination site).
// ---------------------------------------------------------------------------
template <int NS, int G, typename S>
__device__ __forceinline__ void mpull(const S* __restrict__ src, const MGeom& g,
                                      const MOffsets& of, int x, int y, bool interior,
                                      uint64_t policy, S (&f)[kQm]) {
  const S* const here = src + ((long long)y * g.ldx + x);
  if (interior) {
#pragma unroll
    for (int i = 0; i < 2 * kPairs; ++i)
      if (mine(NS, G, i / 2)) f[i] = ld_pull(at_bytes(here, of.pull[i]), policy);
  } else {
#pragma unroll
    for (int i = 0; i < 2 * kPairs; ++i) {
      if (!mine(NS, G, i / 2)) continue;
      const int ex = i & 1 ? -pair_x(i / 2) : pair_x(i / 2);
      const int ey = i & 1 ? -pair_y(i / 2) : pair_y(i / 2);
      int sx = x - ex, sy = y - ey;
      bool in = true;
      if (ex != 0) {
        if (g.px) { sx += sx < 0 ? g.nx : 0; sx -= sx >= g.nx ? g.nx : 0; }
        else in = sx >= 0 && sx < g.nx;
      }
      if (ey != 0) {
        if (g.py) { sy += sy < 0 ? g.ny : 0; sy -= sy >= g.ny ? g.ny : 0; }
        else in = in && sy >= 0 && sy < g.ny;
      }
      const S* ptr = in ? src + (long long)i * g.plane + (long long)sy * g.ldx + sx
                        : at_bytes(here, of.plane[i ^ 1]);
      f[i] = ld_pull(ptr, policy);
    }
  }
  if (class_group(NS, 9) == G) f[kRestPop] = ld_pull(at_bytes(here, of.plane[kRestPop]), policy);
}

__device__ __forceinline__ bool site_interior(const MGeom& g, int x, int y) {
  return x >= kReach && x < g.nx - kReach && y >= kReach && y < g.ny - kReach;
}

// (x, y) lanes of FP32 (Blackwell's paired FMA) and of FP64 (two operations).
__device__ __forceinline__ float2 S2(float a) { return make_float2(a, a); }
__device__ __forceinline__ double2 S2(double a) { return make_double2(a, a); }
__device__ __forceinline__ float2 fma2(float2 a, float2 b, float2 c) { return __ffma2_rn(a, b, c); }
__device__ __forceinline__ float2 mul2(float2 a, float2 b) { return __fmul2_rn(a, b); }
__device__ __forceinline__ float2 add2(float2 a, float2 b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ double2 fma2(double2 a, double2 b, double2 c) {
  return make_double2(fma(a.x, b.x, c.x), fma(a.y, b.y, c.y));
}
__device__ __forceinline__ double2 mul2(double2 a, double2 b) { return make_double2(a.x * b.x, a.y * b.y); }
__device__ __forceinline__ double2 add2(double2 a, double2 b) { return make_double2(a.x + b.x, a.y + b.y); }
__device__ __forceinline__ float2 pair_of(float a, float b) { return make_float2(a, b); }
__device__ __forceinline__ double2 pair_of(double a, double b) { return make_double2(a, b); }
// sign pairs (constant memory, so that they cost no instruction to form in FP32)
__constant__ float2 c_pm = {1.f, -1.f};
__constant__ float2 c_mp = {-1.f, 1.f};
template <typename R> __device__ __forceinline__ typename V2<R>::T pm();
template <> __device__ __forceinline__ float2 pm<float>() { return c_pm; }
template <> __device__ __forceinline__ double2 pm<double>() { return make_double2(1.0, -1.0); }
template <typename R> __device__ __forceinline__ typename V2<R>::T mp();
template <> __device__ __forceinline__ float2 mp<float>() { return c_mp; }
template <> __device__ __forceinline__ double2 mp<double>() { return make_double2(-1.0, 1.0); }

// Moments class by class: the sums of a class that its symmetry leaves, once
// per monomial (170 operations per site, 148 instructions in FP32, where pair
// by pair took 212).
template <typename R>
struct MomSums {
  using V = typename V2<R>::T;
  R n0, e, ps, pd, xy;       // N^0, T^00, (T^xx + T^yy) / 2, (T^xx - T^yy) / 2, T^xy
  V n, m;                    // N^a, T^0a
};

template <int C, typename R>
__device__ __forceinline__ void class_moments(const R (&g)[kQm], MomSums<R>& s) {
  const MConsts<R>& c = mc<R>();
  constexpr int q = 2 * class_pair(C), kind = class_kind(C), f = class_fn(C);
  const R s0 = g[q] + g[q + 1], s1 = g[q + 2] + g[q + 3];
  const R o0 = g[q] - g[q + 1], o1 = g[q + 2] - g[q + 3];
  R S = s0 + s1;
  const R D = s0 - s1;
  if constexpr (kind == 0) {                   // (a, 0), (0, a)
    s.pd = fma(c.mPd[C], D, s.pd);
    const auto o = pair_of(o0, o1);
    s.n = fma2(c.mN[f], o, s.n);
    s.m = fma2(c.mM[f], o, s.m);
  } else if constexpr (kind == 1) {            // (a, a), (-a, a)
    s.xy = fma(c.mPxy[C], D, s.xy);
    const auto o = pair_of(o0 - o1, o0 + o1);
    s.n = fma2(c.mN[f], o, s.n);
    s.m = fma2(c.mM[f], o, s.m);
  } else {                                     // (a, b), (-a, b), (b, a), (-b, a)
    const R s2 = g[q + 4] + g[q + 5], s3 = g[q + 6] + g[q + 7];
    const R o2 = g[q + 4] - g[q + 5], o3 = g[q + 6] - g[q + 7];
    const R S1 = s2 + s3;
    s.pd = fma(c.mPd[C], S - S1, s.pd);
    s.xy = fma(c.mPxy[C], D + (s2 - s3), s.xy);
    S += S1;
    const auto oa = pair_of(o0 - o1, o2 + o3), ob = pair_of(o2 - o3, o0 + o1);
    s.n = fma2(c.mN[f + 1], ob, fma2(c.mN[f], oa, s.n));
    s.m = fma2(c.mM[f + 1], ob, fma2(c.mM[f], oa, s.m));
  }
  s.n0 = fma(c.mN0[C], S, s.n0);
  s.e = fma(c.mE[C], S, s.e);
  s.ps = fma(c.mPs[C], S, s.ps);
}

template <int NS, int G, typename R>
__device__ __forceinline__ MMom<R> mmoments(const R (&g)[kQm]) {
  const MConsts<R>& c = mc<R>();
  MomSums<R> s;
  s.n0 = s.e = s.ps = s.pd = s.xy = R(0);
  s.n = s.m = S2(R(0));
  if (class_group(NS, 0) == G) class_moments<0>(g, s);
  if (class_group(NS, 1) == G) class_moments<1>(g, s);
  if (class_group(NS, 2) == G) class_moments<2>(g, s);
  if (class_group(NS, 3) == G) class_moments<3>(g, s);
  if (class_group(NS, 4) == G) class_moments<4>(g, s);
  if (class_group(NS, 5) == G) class_moments<5>(g, s);
  if (class_group(NS, 6) == G) class_moments<6>(g, s);
  if (class_group(NS, 7) == G) class_moments<7>(g, s);
  if (class_group(NS, 8) == G) class_moments<8>(g, s);
  if (class_group(NS, 9) == G) {
    s.n0 = fma(c.mN0[9], g[kRestPop], s.n0);
    s.e = fma(c.mE[9], g[kRestPop], s.e);
  }
  MMom<R> m;
  m.dN0 = s.n0; m.dNx = s.n.x; m.dNy = s.n.y;
  m.dE = s.e; m.Mx = s.m.x; m.My = s.m.y;
  m.dPxx = s.ps + s.pd; m.dPxy = s.xy; m.dPyy = s.ps - s.pd;
  return m;
}

// Landau frame eps U^a = T^ab U_b: u = (Pi + eps I)^-1 M, Newton on
// eps - E + M.u(eps) (derivative 1 - u.u) from eps = E; n = U_a N^a; T from
// eps / n = (m^2 + 2 m T + 2 T^2) / (m + T).  The unknown is d = eps - E; FP64
// starts from the FP32 solution and needs one FP64 step as a rule (the
// reasoning stands at landau_d32 in site.cuh).
__device__ __forceinline__ bool mlandau_d32(float dE, float Mx, float My, float dPxx, float dPxy,
                                            float dPyy, float& d, float& ux, float& uy) {
  const float a0 = float(kH0) + dPxx, c0 = float(kH0) + dPyy, p2 = dPxy * dPxy;
  d = 0.f;
#pragma unroll 1
  for (int it = 0; it < 16; ++it) {
    const float deps = dE + d;
    const float a = a0 + deps, c = c0 + deps;
    const float inv = qrcp(fmaf(a, c, -p2));
    ux = fmaf(c, Mx, -(dPxy * My)) * inv;
    uy = fmaf(a, My, -(dPxy * Mx)) * inv;
    const float g = fmaf(Mx, ux, fmaf(My, uy, d));
    const float step = g * qrcp(fmaf(-ux, ux, fmaf(-uy, uy, 1.f)));
    d -= step;
    if (fabsf(step) <= 2e-7f * (float(kE0) + fabsf(deps))) {
      const float si = step * inv;
      const float vx = fmaf(c, ux, -(dPxy * uy)), vy = fmaf(a, uy, -(dPxy * ux));
      ux = fmaf(si, vx, ux);
      uy = fmaf(si, vy, uy);
      return true;
    }
  }
  return false;
}
__device__ __forceinline__ bool mlandau_frame(const MMom<float>& m, float& deps, float& ux, float& uy) {
  float d;
  const bool conv = mlandau_d32(m.dE, m.Mx, m.My, m.dPxx, m.dPxy, m.dPyy, d, ux, uy);
  deps = m.dE + d;
  return conv;
}
__device__ __forceinline__ bool mlandau_frame(const MMom<double>& m, double& deps, double& ux, double& uy) {
  float d32, ux32, uy32;
  const bool conv32 = mlandau_d32(trunc_f32(m.dE), trunc_f32(m.Mx), trunc_f32(m.My),
                                  trunc_f32(m.dPxx), trunc_f32(m.dPxy), trunc_f32(m.dPyy), d32,
                                  ux32, uy32);
  double d = conv32 ? widen_f64(d32) : 0.0;
  const double a0 = kH0 + m.dPxx + m.dE, c0 = kH0 + m.dPyy + m.dE, p2 = m.dPxy * m.dPxy;
  bool conv = false;
#pragma unroll 1
  for (int it = 0; it < 16; ++it) {
    const double a = a0 + d, c = c0 + d;
    const double inv = qrcp(fma(a, c, -p2));
    ux = fma(c, m.Mx, -(m.dPxy * m.My)) * inv;
    uy = fma(a, m.My, -(m.dPxy * m.Mx)) * inv;
    const double g = fma(m.Mx, ux, fma(m.My, uy, d));
    const double w = fma(-ux, ux, fma(-uy, uy, 1.0));
    const double step = g * qrcp(w);
    d -= step;
    if (fabsf(trunc_f32(step)) <= 1e-8f * (float(kE0) + fabsf(trunc_f32(m.dE) + trunc_f32(d)))) {
      const double si = step * inv;
      const double vx = fma(c, ux, -(m.dPxy * uy)), vy = fma(a, uy, -(m.dPxy * ux));
      ux = fma(si, vx, ux);
      uy = fma(si, vy, uy);
      conv = true;
      break;
    }
  }
  deps = m.dE + d;
  return conv;
}

// Fields of a site; returns its error bits.
template <typename R>
__device__ __forceinline__ unsigned mlandau(const MMom<R>& M, MMacro<R>& o) {
  R deps, ux, uy;
  const bool conv = mlandau_frame(M, deps, ux, uy);
  const R u2 = fma(ux, ux, uy * uy), w = R(1) - u2;
  const R gamma = qrsqrt(w);
  const R r1 = gamma * qrcp(R(1) + gamma);             // 1 / (1 + s), s = 1 / gamma
  const R gm1 = u2 * gamma * r1;                       // (gamma^2 - 1) / (gamma + 1)
  const R dNpar = fma(-uy, M.dNy, fma(-ux, M.dNx, M.dN0));   // U_a N^a / gamma - 1
  const R dn = fma(gm1, R(1) + dNpar, dNpar);
  // T - 1 = (de + sqrt(D) - sqrt(D0)) / 4,  D = e^2 + 4 m e - 4 m^2,  e = eps / n
  const R n = R(1) + dn;
  const R de = fma(R(-kE0), dn, deps) * qrcp(n);
  const R e = R(kE0) + de;
  const R D = fma(e, e + R(4 * kM), R(-4 * kM * kM));
  const R sD = D * qrsqrt(D);
  const R dT = R(0.25) * de * fma(e + R(kE0 + 4 * kM), qrcp(sD + R(kSD0)), R(1));
  o.ux = ux; o.uy = uy; o.gamma = gamma; o.gm1 = gm1; o.r1 = r1; o.dn = dn; o.dT = dT;
  unsigned bits = conv ? 0u : kErrNoConvergence;
  if (!(finite_bits(ux) && finite_bits(uy) && finite_bits(dn) && finite_bits(dT)))
    bits |= kErrNonFinite;
  else if (!(positive(w) && positive(n) && positive(R(1) + dT)))
    bits |= kErrUnphysical;
  return bits;
}

template <typename R>
__device__ __forceinline__ MMacro<R> macro_of(R n, R ux, R uy, R T) {
  MMacro<R> M;
  const R u2 = fma(ux, ux, uy * uy);
  M.ux = ux; M.uy = uy;
  M.gamma = qrsqrt(R(1) - u2);
  M.r1 = M.gamma * qrcp(R(1) + M.gamma);
  M.gm1 = u2 * M.gamma * M.r1;
  M.dn = n - R(1);
  M.dT = T - R(1);
  return M;
}

// Per-site part of the equilibrium: delta, its quadratic monomials and the
// third-order remainder R3 of the 16 moments (library order), combined by
// symmetry as the class tables want them.
template <typename R>
struct EqSite {
  using V = typename V2<R>::T;
  R dn, a[8];            // dT, dn dT, dT^2, ux^2 + uy^2, E0, E1, E2 + E4, E5 + E7
  R c1[3], c2[3];        // ux^2 - uy^2, E2 - E4, E5 - E7;  ux uy, E3, E6
  V o[7];                // (x, y): u, dn u, dT u, (O0, O1), (O2, O3), (O4, O7), (O6, O5)
  // for the source: alpha gamma^3, h gamma^2, T h at linear order, T h gamma -
  // h0, n gamma, M[1] - 1 / (m + 1)
  R ag3, hg2, Xl, Thgm, ng, d0;
};

template <typename R>
__device__ __forceinline__ EqSite<R> eq_site(const MMacro<R>& M) {
  const R m = R(kM), m1 = R(kM1), one = R(1);
  const R H0 = R(kH0), K1 = R(kK1), A0 = R(kA0);
  const R dn = M.dn, dT = M.dT, ux = M.ux, uy = M.uy;
  const R g = M.gamma, gm1 = M.gm1;
  const R u2 = ux * ux + uy * uy;
  const R T = one + dT;
  const R imT = qrcp(m + T);
  const R im1 = R(1.0 / kM1);
  const R gm1mh = u2 * (u2 * M.r1 + R(2) * gm1) * (R(0.5) * M.r1);                // gm1 - u^2/2
  const R phi = (m * m + R(3) * m * T + R(3) * T * T) * imT;                        // h / n
  const R kT = (R(3) * m1 * T + R(2) * m * m + R(3) * m) * imT * im1;               // (phi(T) - phi(1)) / dT
  const R aT = (m * m * m + R(6) * m * m * T + R(15) * m * T * T + R(15) * T * T * T) * imT;   // alpha / n
  const R kaT = R(5) * (R(3) * m1 * T * T + R(3) * m1 * m1 * T + m * (m * m + R(3) * m + R(3))) * imT * im1;
  const R dh = dn * phi + dT * kT;                                  // h - h0
  const R dT2 = dT * dT;
  const R dhq = dn * dT * kT + dT2 * (m * m) * imT * (im1 * im1);     // dh - h0 dn - k1 dT
  const R da = dn * aT + dT * kaT;                                  // alpha - alpha0
  const R g2 = g * g;
  const R g2m1 = g2 * u2;                                           // gamma^2 - 1
  const R g3m1 = gm1 * (g2 + g + one);                              // gamma^3 - 1
  const R hg2m = dh * g2 + H0 * g2m1;                               // h gamma^2 - h0
  const R hg2mq = dhq * g2 + (H0 * dn + K1 * dT) * g2m1 + H0 * g2m1;
  const R ag3m = da * g2 * g + A0 * g3m1;                           // alpha gamma^3 - alpha0
  const R ag3 = A0 + ag3m;                                          // alpha gamma^3
  const R Xlin = H0 * dn + (K1 + H0) * dT;
  const R XmXl = dhq + dT * dh;                                     // (T h - h0) - Xlin
  const R XmXl2 = dn * dT * (K1 + H0) + dT2 * (K1 + R(kC2));        // its quadratic part
  const R XmXl3 = dn * dT2 * (m * m) * imT * (im1 * im1) - dT2 * dT * (m * m) * imT * (im1 * im1 * im1)
                + dT * dhq;
  const R Rthg = XmXl * g + (Xlin + H0) * gm1;                      // T h gamma - h0 - Xlin
  const R Rthg3 = XmXl3 * g + XmXl2 * gm1 + Xlin * gm1 + H0 * gm1mh;
  const R uxx = ux * ux, uxy = ux * uy, uyy = uy * uy;
  EqSite<R> e;
  e.dn = dn;
  const R ud = uxx - uyy;
  e.a[0] = dT; e.a[1] = dn * dT; e.a[2] = dT2; e.a[3] = u2;
  e.d0 = (dn * m1 - dT) * imT * im1;
  e.a[4] = e.d0 * dT2 * (im1 * im1);
  e.a[5] = gm1mh + gm1 * dn;
  e.a[6] = hg2m * u2;                                // E2 + E4
  e.a[7] = ag3m * u2 + R(2) * Rthg3;                 // E5 + E7
  e.c1[0] = ud; e.c1[1] = hg2m * ud; e.c1[2] = ag3m * ud;
  e.c2[0] = uxy; e.c2[1] = hg2m * uxy; e.c2[2] = ag3m * uxy;
  const R ngm = gm1 * (one + dn);
  const typename V2<R>::T u = pair_of(ux, uy);
  e.o[0] = u;
  e.o[1] = mul2(S2(dn), u);
  e.o[2] = mul2(S2(dT), u);
  e.o[3] = mul2(S2(ngm), u);                         // O0, O1
  e.o[4] = mul2(S2(hg2mq), u);                       // O2, O3
  const R R3t = R(3) * Rthg;
  e.o[5] = mul2(pair_of(ag3 * uxx + R3t, ag3 * uyy + R3t), u);       // px^3, py^3
  e.o[6] = mul2(pair_of(ag3 * uyy + Rthg, ag3 * uxx + Rthg), u);     // px py^2, px^2 py
  e.ag3 = ag3; e.hg2 = H0 + hg2m; e.Xl = Xlin + H0; e.Thgm = Rthg + Xlin; e.ng = ngm + dn;
  return e;
}

// Even and odd parts of g^eq of the couple h (two pairs: lanes pair 2 q, 2 q +
// 1) of class C: axis (a, 0), (0, a); else (a, b), (-a, b) and, h = 1 in a
// class of eight, (b, a), (-b, a).
template <typename R>
struct ClassEq {
  using V = typename V2<R>::T;
  R A, C1, C2;
  V F1, F2;        // component functions of the larger and the smaller component
};

template <int C, typename R>
__device__ __forceinline__ ClassEq<R> class_eq(const EqSite<R>& e) {
  const MConsts<R>& c = mc<R>();
  ClassEq<R> k;
  k.A = fma(c.A[C][0], e.a[0], e.dn);
#pragma unroll
  for (int i = 1; i < 8; ++i) k.A = fma(c.A[C][i], e.a[i], k.A);
  k.C1 = k.C2 = R(0);
  if (class_kind(C) != 1)
    k.C1 = fma(c.C1[C][2], e.c1[2], fma(c.C1[C][1], e.c1[1], c.C1[C][0] * e.c1[0]));
  if (class_kind(C) != 0)
    k.C2 = fma(c.C2[C][2], e.c2[2], fma(c.C2[C][1], e.c2[1], c.C2[C][0] * e.c2[0]));
  constexpr int f = class_fn(C);
  k.F1 = mul2(c.O[f][0], e.o[0]);
#pragma unroll
  for (int i = 1; i < 7; ++i) k.F1 = fma2(c.O[f][i], e.o[i], k.F1);
  k.F2 = k.F1;
  if (class_kind(C) == 2) {
    k.F2 = mul2(c.O[f + 1][0], e.o[0]);
#pragma unroll
    for (int i = 1; i < 7; ++i) k.F2 = fma2(c.O[f + 1][i], e.o[i], k.F2);
  }
  return k;
}

template <int C, int H, typename R>
__device__ __forceinline__ void couple_eq(const ClassEq<R>& k, typename V2<R>::T& ev,
                                          typename V2<R>::T& od) {
  if (class_kind(C) == 0) {
    ev = fma2(S2(k.C1), pm<R>(), S2(k.A));
    od = k.F1;
  } else {
    const R e = class_kind(C) == 1 ? k.A : H ? k.A - k.C1 : k.A + k.C1;
    ev = fma2(S2(k.C2), pm<R>(), S2(e));
    const R X = H ? k.F2.x : k.F1.x, Y = H ? k.F1.y : k.F2.y;
    od = fma2(S2(X), pm<R>(), S2(Y));
  }
}

template <typename R>
__device__ __forceinline__ R eq_rest(const EqSite<R>& e) {
  const MConsts<R>& c = mc<R>();
  R ev = fma(c.A[9][0], e.a[0], e.dn);
#pragma unroll
  for (int i = 1; i < 8; ++i) ev = fma(c.A[9][i], e.a[i], ev);
  return ev;
}

// Forcing: with D(p) = g^eq as a polynomial (coefficients d = (m+1) G^-1 dM,
// dM the full moment deviations), the relative source is
//   F^ext_i / f0_i = (F.v_i)(1 + g^eq_i) - (F.v_i) dD/dp0(p_i) - F.grad_xy D(p_i).
template <typename R>
struct ForceSite {
  using V = typename V2<R>::T;
  R b1, bS, bD, bX;      // 1 - dD/dp0, even part: b1 + bS rr + bD (px^2 - py^2) / 2 + bX px py
  V a;                   // dD/dp0, odd part: a.x px + a.y py
  R h1, hp0, hS, hD, hX; // F.grad_xy D, even part, alike (h1 + hp0 p0 + ..)
  V nh, nh0;             // -F.grad_xy D, odd part: (nh + nh0 p0) . p
};

// The rows of (m + 1) G^-1 in the combinations that x <-> y leaves uncoupled:
// 20 even products and 16 on (x, y) lanes (66 without).
template <typename R>
__device__ __forceinline__ ForceSite<R> force_site(const EqSite<R>& e, R Fx, R Fy) {
  using V = typename V2<R>::T;
  const MConsts<R>& c = mc<R>();
  const R dn = e.dn, dT = e.a[0], u2 = e.a[3], ud = e.c1[0], uxy = e.c2[0];
  const R P1 = dn + dT + e.a[1];                      // P - 1
  // deviations of the moments: 1, p0, px^2 + py^2, p0 (px^2 + py^2) ..
  const R M[4] = {e.d0, e.ng, fma(e.hg2, u2, P1 + P1), fma(e.ag3, u2, e.Thgm + e.Thgm)};
  const R MD[2] = {e.hg2 * ud, e.ag3 * ud}, MX[2] = {e.hg2 * uxy, e.ag3 * uxy};
  const V u = e.o[0];
  // .. and px, p0 px, px^3, px py^2 with their y partners
  const V MO[4] = {mul2(S2(R(1) + e.ng), u), mul2(S2(e.hg2), u), fma2(S2(R(3) * e.Xl), u, e.o[5]),
                   fma2(S2(e.Xl), u, e.o[6])};
  auto row4 = [&](const R (&t)[4]) { return fma(t[3], M[3], fma(t[2], M[2], fma(t[1], M[1], t[0] * M[0]))); };
  const R n1 = row4(c.n1), nS = row4(c.nS), n0S = row4(c.n0S);
  const R nD = fma(c.nD[1], MD[1], c.nD[0] * MD[0]), n0D = fma(c.n0D[1], MD[1], c.n0D[0] * MD[0]);
  const R nX = fma(c.nX[1], MX[1], c.nX[0] * MX[0]), n0X = fma(c.n0X[1], MX[1], c.n0X[0] * MX[0]);
  V d[4];
#pragma unroll
  for (int k = 0; k < 4; ++k)
    d[k] = fma2(c.gO[k][3], MO[3], fma2(c.gO[k][2], MO[2], fma2(c.gO[k][1], MO[1], mul2(c.gO[k][0], MO[0]))));
  ForceSite<R> f;
  f.b1 = R(1) + n1; f.bS = n0S; f.bD = n0D; f.bX = n0X;
  f.a = d[1];
  f.h1 = fma(Fx, d[0].x, Fy * d[0].y);
  f.hp0 = fma(Fx, d[1].x, Fy * d[1].y);
  // d[2] = (px^3, py^3), d[3] = (px py^2, px^2 py)
  const R cx = R(3) * Fx * d[2].x, cy = R(3) * Fy * d[2].y, qx = Fx * d[3].x, qy = Fy * d[3].y;
  const R xx = cx + qy, yy = cy + qx;
  f.hS = xx + yy; f.hD = xx - yy;
  f.hX = R(2) * fma(Fx, d[3].y, Fy * d[3].x);
  f.nh = pair_of(fma(Fx, nS + nD, Fy * nX), fma(Fy, nS - nD, Fx * nX));
  f.nh0 = pair_of(fma(Fx, n0S + n0D, Fy * n0X), fma(Fy, n0S - n0D, Fx * n0X));
  return f;
}

// ---------------------------------------------------------------------------
// Collision of one site and store: class by class, two pairs at a time on (x,
// y) lanes, then each pair on lanes (population 2 p, its opposite 2 p + 1).
// The force's source of a population of pair p with sign s = +-1 is
//   s (F.v (1 - Ae) - Ho + F.v g^eq_s) - (F.v Ao + He)
// with Ae, Ao / He, Ho the even / odd parts of dD/dp0 / F.grad_xy D; B = 1 - Ae
// and N = -Ho are what force_site prepares.
// ---------------------------------------------------------------------------
template <typename R>
struct MRelax {
  R gt, Fx, Fy;
  typename V2<R>::T gu, F;       // gamma u / tau, F
};

template <int C, typename R, bool FORCE>
__device__ __forceinline__ void class_relax(const R (&g)[kQm], const EqSite<R>& e,
                                            const ForceSite<R>& fs, const MRelax<R>& r,
                                            R* __restrict__ out, const MOffsets& of) {
  using V = typename V2<R>::T;
  const MConsts<R>& c = mc<R>();
  const ClassEq<R> k = class_eq<C>(e);
  constexpr int kind = class_kind(C), f = class_fn(C);
  R eB = R(0), eH = R(0), dB = R(0), dH = R(0), xB = R(0), xH = R(0);
  V Nc = S2(R(0));
  if (FORCE) {
    eB = fma(fs.bS, c.rr[C], fs.b1);
    eH = fma(fs.hS, c.rr[C], fma(fs.hp0, c.p0[C], fs.h1));
    if (kind != 1) { dB = fs.bD * c.dd[C]; dH = fs.hD * c.dd[C]; }
    if (kind != 0) { xB = fs.bX * c.pp[C]; xH = fs.hX * c.pp[C]; }
    Nc = fma2(fs.nh0, S2(c.p0[C]), fs.nh);
  }
#pragma unroll
  for (int h = 0; h < (kind == 2 ? 2 : 1); ++h) {
    V ev, od, wv, B = S2(R(0)), He = B, Ao = B, N = B, Fv = B;
    if (h == 0) couple_eq<C, 0>(k, ev, od);
    else couple_eq<C, 1>(k, ev, od);
    if (kind == 0) {
      wv = mul2(r.gu, c.va[f]);
      if (FORCE) {
        Fv = mul2(r.F, c.va[f]);
        B = fma2(S2(dB), pm<R>(), S2(eB));
        He = fma2(S2(dH), pm<R>(), S2(eH));
        Ao = mul2(fs.a, c.pa[f]);
        N = mul2(Nc, c.pa[f]);
      }
    } else {
      // x component of the couple's pairs: function fx, y component: fy
      const int fx = kind == 1 ? f : f + h, fy = kind == 1 ? f : f + 1 - h;
      wv = fma2(S2(r.gu.x * c.va[fx].x), pm<R>(), S2(r.gu.y * c.va[fy].x));
      if (FORCE) {
        Fv = fma2(S2(r.F.x * c.va[fx].x), pm<R>(), S2(r.F.y * c.va[fy].x));
        const R a = h ? eB - dB : eB + dB, b = h ? eH - dH : eH + dH;
        B = fma2(S2(xB), pm<R>(), S2(a));
        He = fma2(S2(xH), pm<R>(), S2(b));
        Ao = fma2(S2(fs.a.x * c.pa[fx].x), pm<R>(), S2(fs.a.y * c.pa[fy].x));
        N = fma2(S2(Nc.x * c.pa[fx].x), pm<R>(), S2(Nc.y * c.pa[fy].x));
      }
    }
    V al = S2(R(0)), be = al;
    if (FORCE) {
      al = fma2(Fv, B, N);
      be = fma2(Fv, Ao, He);
    }
#pragma unroll
    for (int l = 0; l < 2; ++l) {
      const int p = class_pair(C) + 2 * h + l;
      const R evp = l ? ev.y : ev.x, odp = l ? od.y : od.x, w = l ? wv.y : wv.x;
      const V om = fma2(S2(w), mp<R>(), S2(r.gt));            // gamma (1 -+ v.u) / tau
      const V geq = fma2(S2(odp), pm<R>(), S2(evp));          // ev +- od
      const V G = pair_of(g[2 * p], g[2 * p + 1]);
      V o = fma2(om, fma2(G, S2(R(-1)), geq), G);
      if (FORCE) {
        const R Fp = l ? Fv.y : Fv.x, a = l ? al.y : al.x, b = l ? be.y : be.x;
        o = fma2(fma2(S2(Fp), geq, S2(a)), pm<R>(), add2(o, S2(-b)));
      }
      *at_bytes(out, of.plane[2 * p]) = o.x;
      *at_bytes(out, of.plane[2 * p + 1]) = o.y;
    }
  }
}

// Parking of the gathered populations (FP32): between the moments and the
// relaxation they wait in shared memory, [4 populations][thread], 16 bytes an
// entry, and come back class by class.  128 -> 80 registers, 16 -> 24 warps per
// SM: 2048 x 2048 sites with a force 280 -> 262 us per step, 1024 x 512 41.2 ->
// 40.4 (20 warps 264 and 40.7, 28 warps spill: 292 and 42.8; 200 x 150, less
// than a wave, 9.1 us both ways).  The accesses are volatile so that the
// compiler cannot keep the register copies alive instead.
template <typename R> struct MPark { static constexpr bool kOn = sizeof(R) == 4; };
constexpr int kParkStride = kMThreads * 16;

__device__ __forceinline__ void park_all(uint32_t a, const float (&g)[kQm]) {
#pragma unroll
  for (int v = 0; v < kQm / 4; ++v)
    asm volatile("st.shared.v4.f32 [%0], {%1, %2, %3, %4};\n"
                 :: "r"(a + v * kParkStride), "f"(g[4 * v]), "f"(g[4 * v + 1]), "f"(g[4 * v + 2]), "f"(g[4 * v + 3])
                 : "memory");
  asm volatile("st.shared.f32 [%0], %1;\n" :: "r"(a + kQm / 4 * kParkStride), "f"(g[kRestPop]) : "memory");
}
template <int C>
__device__ __forceinline__ void unpark(uint32_t a, float (&g)[kQm]) {
  constexpr int v0 = class_pair(C) / 2, n = class_kind(C) == 2 ? 2 : 1;
#pragma unroll
  for (int v = v0; v < v0 + n; ++v)
    asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];\n"
                 : "=f"(g[4 * v]), "=f"(g[4 * v + 1]), "=f"(g[4 * v + 2]), "=f"(g[4 * v + 3])
                 : "r"(a + v * kParkStride) : "memory");
}

template <int C, int NS, int G, typename R, bool FORCE>
__device__ __forceinline__ void class_step(R (&g)[kQm], const EqSite<R>& e, const ForceSite<R>& fs,
                                           const MRelax<R>& r, R* __restrict__ out, const MOffsets& of,
                                           uint32_t park) {
  if constexpr (class_group(NS, C) == G) {
    if constexpr (MPark<R>::kOn) unpark<C>(park, g);
    class_relax<C, R, FORCE>(g, e, fs, r, out, of);
  }
}

template <int NS, int G, typename R, bool FORCE>
__device__ __forceinline__ void mcollide_store(R (&g)[kQm], const MMacro<R>& M, R inv_tau,
                                               R Fx, R Fy, R* __restrict__ out, const MOffsets& of,
                                               uint32_t park) {
  const EqSite<R> e = eq_site(M);
  MRelax<R> r;
  r.gt = M.gamma * inv_tau;
  r.gu = mul2(S2(r.gt), pair_of(M.ux, M.uy));
  r.F = pair_of(Fx, Fy);
  ForceSite<R> fs{};
  if (FORCE) fs = force_site(e, Fx, Fy);
  class_step<0, NS, G, R, FORCE>(g, e, fs, r, out, of, park);
  class_step<1, NS, G, R, FORCE>(g, e, fs, r, out, of, park);
  class_step<2, NS, G, R, FORCE>(g, e, fs, r, out, of, park);
  class_step<3, NS, G, R, FORCE>(g, e, fs, r, out, of, park);
  class_step<4, NS, G, R, FORCE>(g, e, fs, r, out, of, park);
  class_step<5, NS, G, R, FORCE>(g, e, fs, r, out, of, park);
  class_step<6, NS, G, R, FORCE>(g, e, fs, r, out, of, park);
  class_step<7, NS, G, R, FORCE>(g, e, fs, r, out, of, park);
  class_step<8, NS, G, R, FORCE>(g, e, fs, r, out, of, park);
  if (class_group(NS, 9) == G) {
    if constexpr (MPark<R>::kOn)
      asm volatile("ld.shared.f32 %0, [%1];\n" : "=f"(g[kRestPop]) : "r"(park + kQm / 4 * kParkStride) : "memory");
    R orr = fma(r.gt, eq_rest(e) - g[kRestPop], g[kRestPop]);
    if (FORCE) orr -= fma(fs.hp0, R(kM), fs.h1);
    *at_bytes(out, of.plane[kRestPop]) = orr;
  }
}

// ---------------------------------------------------------------------------
// Kernels.  Steps are chained launches (programmatic dependent launch): the
// next step's blocks are placed early and wait for this one's results before
// their first access.  FP32 1024 x 512 with a force: 57.6 -> 45.0 us per step
// by the class tables and the prepared offsets, -> 41 us by moments per class
// and the source's symmetric rows, -> 40.4 with 24 instead of 16 warps per SM
// (28 us is the HBM time; instruction issue bounds it).
// ---------------------------------------------------------------------------
__device__ __forceinline__ void chain_release() {
  asm volatile("griddepcontrol.launch_dependents;\n" ::: "memory");
}
__device__ __forceinline__ void chain_wait() {
  asm volatile("griddepcontrol.wait;\n" ::: "memory");
}
__device__ __forceinline__ uint64_t mpolicy(bool evict_first) {
  uint64_t a, b;
  asm("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(a));
  asm("createpolicy.fractional.L2::evict_normal.b64 %0, 1.0;" : "=l"(b));
  return evict_first ? a : b;
}

struct MLaunch {
  int reverse, evict_first;
  int early;             // let the next step's blocks be placed while this one runs
};

// Warps take 32 consecutive sites of a row, two per block.
template <typename R, bool FORCE>
__device__ __forceinline__ void mstep_body(const R* __restrict__ src, R* __restrict__ dst,
                                           const MGeom& geo, const MOffsets& of, const MLaunch& ml,
                                           R inv_tau, R Fx, R Fy, unsigned* __restrict__ err) {
  if (ml.early) chain_release();
  const unsigned per_row = (unsigned)(geo.nx + 31) / 32;
  const unsigned block = ml.reverse ? gridDim.x - 1 - blockIdx.x : blockIdx.x;
  const unsigned t = block * (kMThreads / 32) + threadIdx.x / 32;
  const int y = (int)(t / per_row), x0 = (int)(t - (unsigned)y * per_row) * 32;
  const int x = x0 + (int)(threadIdx.x % 32);
  const uint64_t policy = mpolicy(ml.evict_first);
  chain_wait();
  if (x >= geo.nx || y >= geo.ny) return;
  R g[kQm];
  mpull<1, 0>(src, geo, of, x, y, site_interior(geo, x0, y) && site_interior(geo, x0 + 31, y), policy, g);
  MMacro<R> M;
  const MMom<R> mom = mmoments<1, 0>(g);
  uint32_t park = 0;
  if constexpr (MPark<R>::kOn) {
    __shared__ __align__(16) unsigned char area[(kQm / 4 + 1) * kParkStride];
    park = (uint32_t)__cvta_generic_to_shared(area) + threadIdx.x * 16u;
    park_all(park, g);
  }
  const unsigned bits = mlandau(mom, M);
  mcollide_store<1, 0, R, FORCE>(g, M, inv_tau, Fx, Fy, dst + (long long)y * geo.ldx + x, of, park);
  if (bits) atomicOr(err, bits);
}

// FP32: at most 80 registers (24 warps per SM; MPark).
template <typename R, bool FORCE>
__global__ void __launch_bounds__(kMThreads, sizeof(R) == 4 ? 12 : 1)
k_mstep(const R* __restrict__ src, R* __restrict__ dst, const __grid_constant__ MGeom geo,
        const __grid_constant__ MOffsets of, MLaunch ml, R inv_tau, R Fx, R Fy,
        unsigned* __restrict__ err) {
  mstep_body<R, FORCE>(src, dst, geo, of, ml, inv_tau, Fx, Fy, err);
}

// FP64, few sites: two warps share 32 sites (consecutive in row-major order,
// across row ends), each with the populations of some classes.  A warp
// instruction of the FP64 pipe takes 66 cycles of its SM sub-partition, so
// below one warp per sub-partition a step lasts as long as one warp's chain.
// 97 x 70 sites with a force: 78 -> 38 us per step.  Two and not four: four
// repeat the Landau solve and the coefficients once more each, which pays for
// one solver alone (64 x 64 28 us, two warps 34) but not where several share
// the GPU (eight of 64 x 64, each on its own stream, per step of all: four 194
// us, two 112, one thread per site 136).
template <int NS, int G, bool FORCE>
__device__ __forceinline__ void msplit_group(const double* __restrict__ src, double* __restrict__ dst,
                                             const MGeom& geo, const MOffsets& of, double inv_tau,
                                             double Fx, double Fy, unsigned* __restrict__ err,
                                             MMom<double>* part, int x, int y, bool in, bool interior) {
  const int lane = threadIdx.x % 32;
  double g[kQm];
  if (in) {
    mpull<NS, G>(src, geo, of, x, y, interior, 0, g);
    part[G * 32 + lane] = mmoments<NS, G>(g);
  }
  // a barrier that the warps meet at from NS places in the code
  asm volatile("bar.sync 1, %0;\n" :: "n"(32 * NS) : "memory");
  if (!in) return;
  MMom<double> m = part[lane];
#pragma unroll
  for (int k = 1; k < NS; ++k) {
    const MMom<double>& q = part[k * 32 + lane];
    m.dN0 += q.dN0; m.dNx += q.dNx; m.dNy += q.dNy;
    m.dE += q.dE; m.Mx += q.Mx; m.My += q.My;
    m.dPxx += q.dPxx; m.dPxy += q.dPxy; m.dPyy += q.dPyy;
  }
  MMacro<double> M;
  const unsigned bits = mlandau(m, M);
  mcollide_store<NS, G, double, FORCE>(g, M, inv_tau, Fx, Fy, dst + (long long)y * geo.ldx + x, of, 0);
  if (G == 0 && bits) atomicOr(err, bits);
}

template <int NS, bool FORCE>
__global__ void __launch_bounds__(32 * NS)
k_mstep_split(const double* __restrict__ src, double* __restrict__ dst,
              const __grid_constant__ MGeom geo, const __grid_constant__ MOffsets of,
              double inv_tau, double Fx, double Fy, unsigned* __restrict__ err) {
  __shared__ MMom<double> part[NS * 32];
  const long long n = (long long)blockIdx.x * 32 + threadIdx.x % 32;
  const bool in = n < (long long)geo.nx * geo.ny;
  const int y = in ? (int)(n / geo.nx) : 0, x = in ? (int)(n - (long long)y * geo.nx) : 0;
  const bool interior = __all_sync(0xffffffffu, !in || site_interior(geo, x, y));
  chain_wait();
  const int w = threadIdx.x / 32;
  if (w == 0) msplit_group<NS, 0, FORCE>(src, dst, geo, of, inv_tau, Fx, Fy, err, part, x, y, in, interior);
  else msplit_group<NS, 1, FORCE>(src, dst, geo, of, inv_tau, Fx, Fy, err, part, x, y, in, interior);
}

template <typename R>
__global__ void __launch_bounds__(128) k_mmoments(const R* __restrict__ src,
                                                  const __grid_constant__ MGeom geo,
                                                  const __grid_constant__ MOffsets of,
                                                  double* __restrict__ n, double* __restrict__ ux,
                                                  double* __restrict__ uy, double* __restrict__ T,
                                                  unsigned* __restrict__ err) {
  const int x = blockIdx.x * 32 + threadIdx.x, y = blockIdx.y * 4 + threadIdx.y;
  if (x >= geo.nx || y >= geo.ny) return;
  const int x0 = blockIdx.x * 32;
  R g[kQm];
  mpull<1, 0>(src, geo, of, x, y, site_interior(geo, x0, y) && site_interior(geo, x0 + 31, y),
              mpolicy(false), g);
  MMacro<R> M;
  const unsigned bits = mlandau(mmoments<1, 0>(g), M);
  const long long o = (long long)y * geo.nx + x;
  if (n) n[o] = 1.0 + as_f64(M.dn);
  if (ux) ux[o] = as_f64(M.ux);
  if (uy) uy[o] = as_f64(M.uy);
  if (T) T[o] = 1.0 + as_f64(M.dT);
  if (bits) atomicOr(err, bits);
}

template <int C, typename R>
__device__ __forceinline__ void class_init(const EqSite<R>& e, R* __restrict__ out, const MOffsets& of) {
  const ClassEq<R> k = class_eq<C>(e);
#pragma unroll
  for (int h = 0; h < (class_kind(C) == 2 ? 2 : 1); ++h) {
    typename V2<R>::T ev, od;
    if (h == 0) couple_eq<C, 0>(k, ev, od);
    else couple_eq<C, 1>(k, ev, od);
    const int p = class_pair(C) + 2 * h;
    *at_bytes(out, of.plane[2 * p]) = ev.x + od.x;
    *at_bytes(out, of.plane[2 * p + 1]) = ev.x - od.x;
    *at_bytes(out, of.plane[2 * p + 2]) = ev.y + od.y;
    *at_bytes(out, of.plane[2 * p + 3]) = ev.y - od.y;
  }
}

template <typename R>
__global__ void __launch_bounds__(128) k_minit(R* __restrict__ dst, const __grid_constant__ MGeom geo,
                                               const __grid_constant__ MOffsets of,
                                               const double* __restrict__ n,
                                               const double* __restrict__ ux, const double* __restrict__ uy,
                                               const double* __restrict__ T, unsigned* __restrict__ err) {
  const int x = blockIdx.x * 32 + threadIdx.x, y = blockIdx.y * 4 + threadIdx.y;
  if (x >= geo.nx || y >= geo.ny) return;
  const long long o = (long long)y * geo.nx + x;
  const double u2 = ux[o] * ux[o] + uy[o] * uy[o];
  if (!(u2 < 1.0 && n[o] > 0.0 && T[o] > 0.0)) { atomicOr(err, kErrUnphysical); return; }
  const MMacro<R> M = macro_of<R>(R(n[o]), R(ux[o]), R(uy[o]), R(T[o]));
  const EqSite<R> e = eq_site(M);
  R* out = dst + (long long)y * geo.ldx + x;
  class_init<0>(e, out, of);
  class_init<1>(e, out, of);
  class_init<2>(e, out, of);
  class_init<3>(e, out, of);
  class_init<4>(e, out, of);
  class_init<5>(e, out, of);
  class_init<6>(e, out, of);
  class_init<7>(e, out, of);
  class_init<8>(e, out, of);
  *at_bytes(out, of.plane[kRestPop]) = eq_rest(e);
}

// state I/O: delta_i = f0_i g_i in FP64, dense [45][ny][nx]
template <typename R>
__global__ void k_mget(const R* __restrict__ src, MGeom geo, double* __restrict__ delta) {
  const long long nsite = (long long)geo.nx * geo.ny;
  for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < nsite * kQm;
       t += (long long)gridDim.x * blockDim.x) {
    const int i = (int)(t / nsite);
    const long long r = t - i * nsite;
    const int y = (int)(r / geo.nx), x = (int)(r - (long long)y * geo.nx);
    delta[t] = (double)src[(long long)i * geo.plane + (long long)y * geo.ldx + x] * mc<R>().f0[i];
  }
}

template <typename R>
__global__ void k_mset(R* __restrict__ dst, MGeom geo, const double* __restrict__ delta) {
  const long long nsite = (long long)geo.nx * geo.ny;
  for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < nsite * kQm;
       t += (long long)gridDim.x * blockDim.x) {
    const int i = (int)(t / nsite);
    const long long r = t - i * nsite;
    const int y = (int)(r / geo.nx), x = (int)(r - (long long)y * geo.nx);
    // delta / f0 with 1 / f0 in two parts
    dst[(long long)i * geo.plane + (long long)y * geo.ldx + x] =
        (R)over(delta[t], mc<R>().if0[i], mc<R>().ifl[i]);
  }
}

// sum over sites of |u - u_prev|^2 and |u|^2 into acc[0], acc[1] (FP64):
// warp shuffles, one pair of atomics per warp
__global__ void k_mresidual(const double* __restrict__ uxp, const double* __restrict__ uyp,
                            const double* __restrict__ ux, const double* __restrict__ uy,
                            long long nsite, double* __restrict__ acc) {
  double a = 0.0, b = 0.0;
  for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < nsite;
       t += (long long)gridDim.x * blockDim.x) {
    const double dx = ux[t] - uxp[t], dy = uy[t] - uyp[t];
    a = fma(dx, dx, fma(dy, dy, a));
    b = fma(ux[t], ux[t], fma(uy[t], uy[t], b));
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    a += __shfl_xor_sync(0xffffffffu, a, o);
    b += __shfl_xor_sync(0xffffffffu, b, o);
  }
  if ((threadIdx.x & 31) == 0) {
    atomicAdd(acc, a);
    atomicAdd(acc + 1, b);
  }
}

// ---------------------------------------------------------------------------
// Host side
// ---------------------------------------------------------------------------
thread_local std::string g_error;

template <typename R>
void fill_consts(const Tables& t, MConsts<R>& c) {
  using V = typename V2<R>::T;
  auto fn = [&](int f, int p) {       // part of pair p's row odd in px
    const double o[7] = {t.LX[p], t.WO[p][0], t.WO[p][2], t.BO[p][0], t.BO[p][2], t.BO[p][4], t.BO[p][6]};
    for (int k = 0; k < 7; ++k) c.O[f][k] = V{(R)o[k], (R)o[k]};
    c.va[f] = V{(R)t.vx[p], (R)t.vx[p]};
    c.pa[f] = V{(R)t.mvO[p][0], (R)t.mvO[p][0]};
    c.mN[f] = V{(R)t.mNx[p], (R)t.mNx[p]};
    c.mM[f] = V{(R)t.mMx[p], (R)t.mMx[p]};
  };
  for (int k = 0; k < kClasses - 1; ++k) {
    const int p = class_pair(k);
    const double a[8] = {t.LT[p], t.WE[p][0], t.WE[p][1], 0.5 * (t.WE[p][2] + t.WE[p][4]), t.BE[p][0],
                         t.BE[p][1], 0.5 * (t.BE[p][2] + t.BE[p][4]), 0.5 * (t.BE[p][5] + t.BE[p][7])};
    for (int q = 0; q < 8; ++q) c.A[k][q] = (R)a[q];
    c.C1[k][0] = (R)(0.5 * (t.WE[p][2] - t.WE[p][4]));
    c.C1[k][1] = (R)(0.5 * (t.BE[p][2] - t.BE[p][4]));
    c.C1[k][2] = (R)(0.5 * (t.BE[p][5] - t.BE[p][7]));
    c.C2[k][0] = (R)t.WE[p][3]; c.C2[k][1] = (R)t.BE[p][3]; c.C2[k][2] = (R)t.BE[p][6];
    c.mN0[k] = (R)t.mN0[p]; c.mE[k] = (R)t.mE[p]; c.mPxy[k] = (R)t.mPxy[p];
    c.mPs[k] = (R)(0.5 * (t.mPxx[p] + t.mPyy[p]));
    c.mPd[k] = (R)(0.5 * (t.mPxx[p] - t.mPyy[p]));
    c.p0[k] = (R)t.mvE[p][1];
    c.rr[k] = (R)(0.5 * (t.mvE[p][2] + t.mvE[p][4]));
    c.dd[k] = (R)(0.5 * (t.mvE[p][2] - t.mvE[p][4]));
    c.pp[k] = (R)t.mvE[p][3];
    fn(class_fn(k), p);
    if (class_kind(k) == 2) fn(class_fn(k) + 1, p + 2);
  }
  const double a[8] = {t.restLT, t.restWE[0], t.restWE[1], 0.5 * (t.restWE[2] + t.restWE[4]), t.restBE[0],
                       t.restBE[1], 0.5 * (t.restBE[2] + t.restBE[4]), 0.5 * (t.restBE[5] + t.restBE[7])};
  for (int q = 0; q < 8; ++q) c.A[kClasses - 1][q] = (R)a[q];
  for (int q = 0; q < 3; ++q) c.C1[kClasses - 1][q] = c.C2[kClasses - 1][q] = R(0);
  c.p0[kClasses - 1] = (R)kM;
  c.rr[kClasses - 1] = c.dd[kClasses - 1] = c.pp[kClasses - 1] = R(0);
  c.mN0[kClasses - 1] = (R)t.restN0; c.mE[kClasses - 1] = (R)t.restE;
  c.mPs[kClasses - 1] = c.mPd[kClasses - 1] = c.mPxy[kClasses - 1] = R(0);
  const auto& gi = t.gi;
  const int col[4] = {0, 1, 2, 5};     // monomials 1, p0, px^2, p0 px^2 (py^2: 4, 7)
  for (int k = 0; k < 4; ++k) {
    c.n1[k] = (R)-gi[1][col[k]];
    c.nS[k] = (R)-(gi[2][col[k]] + gi[4][col[k]]);
    c.n0S[k] = (R)-(gi[5][col[k]] + gi[7][col[k]]);
  }
  for (int k = 0; k < 2; ++k) {
    const int b = k ? 5 : 2, x = k ? 6 : 3;
    c.nD[k] = (R)-(gi[2][b] - gi[4][b]);
    c.n0D[k] = (R)-(gi[5][b] - gi[7][b]);
    c.nX[k] = (R)-gi[3][x];
    c.n0X[k] = (R)-gi[6][x];
  }
  const int odd[4] = {8, 10, 12, 14};  // px, p0 px, px^3, px py^2
  for (int k = 0; k < 4; ++k)
    for (int b = 0; b < 4; ++b) c.gO[k][b] = V{(R)gi[odd[k]][odd[b]], (R)gi[odd[k]][odd[b]]};
  for (int i = 0; i < kQm; ++i) {
    c.f0[i] = t.f0[i];
    c.if0[i] = 1.0 / t.f0[i];
    c.ifl[i] = std::fma(-t.f0[i], c.if0[i], 1.0) / t.f0[i];
  }
}

std::mutex g_upload_mu;
bool g_uploaded[64];

}  // namespace
}  // namespace massive
}  // namespace rlbm

using namespace rlbm::massive;

struct rlbm_massive_ctx {
  rlbm_massive_config cfg;
  MGeom geo;
  MOffsets of;
  int sms;
  size_t l2, elem;
  void* buf[2];
  int cur;
  unsigned* err;
  double* scratch;
  size_t scratch_bytes;
  long long steps, launches;
  std::string msg;
};

namespace {

int fail(rlbm_massive_ctx* c, int code, const char* fmt, ...) {
  char b[512];
  va_list ap;
  va_start(ap, fmt);
  std::vsnprintf(b, sizeof b, fmt, ap);
  va_end(ap);
  if (c) c->msg = b; else g_error = b;
  return code;
}

int cuda_fail(rlbm_massive_ctx* c, cudaError_t e, const char* what) {
  return fail(c, RLBM_ECUDA, "%s: %s", what, cudaGetErrorString(e));
}

int upload_tables(int dev) {
  const Tables& t = tables();
  if (!t.ok) return fail(nullptr, RLBM_EINVAL, "massive quadrature: %s", t.msg);
  std::lock_guard<std::mutex> lock(g_upload_mu);
  if (dev < 0 || dev >= 64) return fail(nullptr, RLBM_ECUDA, "device index %d", dev);
  if (g_uploaded[dev]) return RLBM_OK;
  static MConsts<float> hf;
  static MConsts<double> hd;
  fill_consts(t, hf);
  fill_consts(t, hd);
  cudaError_t e = cudaMemcpyToSymbol(c_f, &hf, sizeof hf);
  if (e == cudaSuccess) e = cudaMemcpyToSymbol(c_d, &hd, sizeof hd);
  if (e != cudaSuccess) return fail(nullptr, RLBM_ECUDA, "constant upload: %s", cudaGetErrorString(e));
  g_uploaded[dev] = true;
  return RLBM_OK;
}

cudaStream_t stream_of(const rlbm_massive_ctx* c) { return (cudaStream_t)c->cfg.stream; }

dim3 grid_of(const MGeom& g) { return dim3((g.nx + 31) / 32, (g.ny + 3) / 4); }

int need_scratch(rlbm_massive_ctx* c, size_t bytes) {
  if (c->scratch_bytes >= bytes) return RLBM_OK;
  if (c->scratch) { cudaStreamSynchronize(stream_of(c)); cudaFree(c->scratch); c->scratch = nullptr; }
  c->scratch_bytes = 0;
  cudaError_t e = cudaMalloc((void**)&c->scratch, bytes);
  if (e != cudaSuccess) return fail(c, RLBM_ENOMEM, "scratch cudaMalloc(%zu): %s", bytes, cudaGetErrorString(e));
  c->scratch_bytes = bytes;
  return RLBM_OK;
}

int grid_1d(long long work) {
  long long b = (work + 255) / 256;
  return (int)(b < 4096 ? (b < 1 ? 1 : b) : 4096);
}

}  // namespace

namespace {

template <typename... P, typename... A>
void launch_chained(cudaStream_t st, void (*k)(P...), unsigned grid, int block, size_t smem, A... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(grid);
  cfg.blockDim = dim3(block);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute at;
  at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at.val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = &at;
  cfg.numAttrs = 1;
  cudaLaunchKernelEx(&cfg, k, P(args)...);
}

int launch_steps(rlbm_massive_ctx* c, int nsteps) {
  const bool force = c->cfg.Fx != 0.0 || c->cfg.Fy != 0.0;
  const cudaStream_t st = stream_of(c);
  const size_t bytes = (size_t)c->geo.plane * kQm * c->elem;
  const long long warps = (long long)((c->geo.nx + 31) / 32) * c->geo.ny;
  const unsigned grid = (unsigned)((warps + kMThreads / 32 - 1) / (kMThreads / 32));
  // FP64: two warps per 32 sites up to two such tiles per SM (one warp per SM
  // sub-partition)
  const long long tiles = ((long long)c->geo.nx * c->geo.ny + 31) / 32;
  const bool split = tiles <= 2 * c->sms;
  for (int s = 0; s < nsteps; ++s) {
    const void* src = c->buf[c->cur];
    void* dst = c->buf[c->cur ^ 1];
    // order and L2 policy of the pulls (FP32): the rules of the massless step
    // (launch_single in prec_impl.cuh)
    MLaunch ml;
    ml.evict_first = bytes <= 2 * c->l2;
    // as in the massless step, FP64 of up to two blocks per SM keeps the next
    // step's blocks from gathering on the SMs it leaves idle
    ml.early = c->elem != 8 || grid > 2u * (unsigned)c->sms;
    ml.reverse = c->cur && bytes <= 4 * c->l2;
    if (c->elem == 8) {
      const double it = 1.0 / c->cfg.tau, fx = c->cfg.Fx, fy = c->cfg.Fy;
      const double* a = (const double*)src;
      double* b = (double*)dst;
      if (split)
        launch_chained(st, force ? k_mstep_split<2, true> : k_mstep_split<2, false>, (unsigned)tiles, 64, 0,
                       a, b, c->geo, c->of, it, fx, fy, c->err);
      else
        launch_chained(st, force ? k_mstep<double, true> : k_mstep<double, false>, grid, kMThreads, 0, a, b,
                       c->geo, c->of, ml, it, fx, fy, c->err);
    } else {
      const float it = (float)(1.0 / c->cfg.tau), fx = (float)c->cfg.Fx, fy = (float)c->cfg.Fy;
      launch_chained(st, force ? k_mstep<float, true> : k_mstep<float, false>, grid, kMThreads, 0,
                     (const float*)src, (float*)dst, c->geo, c->of, ml, it, fx, fy, c->err);
    }
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return cuda_fail(c, e, "step kernel");
    c->cur ^= 1;
    ++c->steps;
    ++c->launches;
  }
  return RLBM_OK;
}

int velocity_planes(rlbm_massive_ctx* c, double* ux, double* uy) {
  if (c->elem == 8)
    k_mmoments<double><<<grid_of(c->geo), dim3(32, 4), 0, stream_of(c)>>>((const double*)c->buf[c->cur], c->geo, c->of, nullptr, ux, uy, nullptr, c->err);
  else
    k_mmoments<float><<<grid_of(c->geo), dim3(32, 4), 0, stream_of(c)>>>((const float*)c->buf[c->cur], c->geo, c->of, nullptr, ux, uy, nullptr, c->err);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return cuda_fail(c, e, "moments kernel");
  ++c->launches;
  return RLBM_OK;
}

}  // namespace

extern "C" {

int rlbm_massive_quadrature(double* v0, double window[2], double w[10], double p0[10]) {
  const Tables& t = tables();
  if (!t.ok) return fail(nullptr, RLBM_EINVAL, "massive quadrature: %s", t.msg);
  if (v0) *v0 = t.v0;
  if (window) { window[0] = t.window_lo; window[1] = t.window_hi; }
  for (int k = 0; k < kClasses; ++k) {
    if (w) w[k] = t.w_class[k];
    if (p0) p0[k] = t.p0_class[k];
  }
  return RLBM_OK;
}

int rlbm_massive_stencil(int vx[45], int vy[45]) {
  if (!vx || !vy) return fail(nullptr, RLBM_EINVAL, "NULL output");
  for (int p = 0; p < kPairs; ++p) {
    vx[2 * p] = pair_x(p); vy[2 * p] = pair_y(p);
    vx[2 * p + 1] = -pair_x(p); vy[2 * p + 1] = -pair_y(p);
  }
  vx[kRestPop] = vy[kRestPop] = 0;
  return RLBM_OK;
}

int rlbm_massive_create(const rlbm_massive_config* cfg, rlbm_massive_ctx** out) {
  if (!out) return fail(nullptr, RLBM_EINVAL, "out is NULL");
  *out = nullptr;
  if (!cfg) return fail(nullptr, RLBM_EINVAL, "config is NULL");
  if (cfg->nx < kReach + 1 || cfg->ny < kReach + 1 || cfg->nx > (1 << 17) || cfg->ny > (1 << 17))
    return fail(nullptr, RLBM_EINVAL, "nx, ny must be in [5, 131072]");
  if (!(cfg->tau > 0.5 && cfg->tau < 1e6)) return fail(nullptr, RLBM_EINVAL, "tau must be in (0.5, 1e6)");
  if (!(std::fabs(cfg->Fx) < 1e-2 && std::fabs(cfg->Fy) < 1e-2))
    return fail(nullptr, RLBM_EINVAL, "|F| must be < 1e-2");
  if (cfg->prec != RLBM_F64 && cfg->prec != RLBM_F32)
    return fail(nullptr, RLBM_EINVAL, "precision must be RLBM_F64 or RLBM_F32");
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return fail(nullptr, RLBM_ECUDA, "cudaGetDevice: %s", cudaGetErrorString(e));
  int r = upload_tables(dev);
  if (r) return r;
  rlbm_massive_ctx* c = new (std::nothrow) rlbm_massive_ctx();
  if (!c) return fail(nullptr, RLBM_ENOMEM, "host allocation failed");
  c->cfg = *cfg;
  c->elem = cfg->prec == RLBM_F64 ? 8 : 4;
  c->geo.nx = cfg->nx; c->geo.ny = cfg->ny;
  c->geo.ldx = (cfg->nx + 31) / 32 * 32;
  c->geo.px = cfg->periodic_x ? 1 : 0; c->geo.py = cfg->periodic_y ? 1 : 0;
  c->geo.plane = (long long)c->geo.ldx * cfg->ny;
  for (int i = 0; i < kQm; ++i) {
    const int s = i & 1 ? -1 : 1;
    const long long back = i == kRestPop ? 0 : s * ((long long)pair_y(i / 2) * c->geo.ldx + pair_x(i / 2));
    c->of.plane[i] = (long long)i * c->geo.plane * (long long)c->elem;
    c->of.pull[i] = c->of.plane[i] - back * (long long)c->elem;
  }
  int l2 = 0;
  if (cudaDeviceGetAttribute(&c->sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess ||
      cudaDeviceGetAttribute(&l2, cudaDevAttrL2CacheSize, dev) != cudaSuccess) {
    delete c;
    return fail(nullptr, RLBM_ECUDA, "device attributes");
  }
  c->l2 = (size_t)l2;
  const size_t bytes = (size_t)c->geo.plane * kQm * c->elem;
  for (int b = 0; b < 2; ++b) {
    e = cudaMalloc(&c->buf[b], bytes);
    if (e != cudaSuccess) {
      rlbm_massive_destroy(c);
      return fail(nullptr, RLBM_ENOMEM, "cudaMalloc(%zu): %s", bytes, cudaGetErrorString(e));
    }
  }
  e = cudaMalloc((void**)&c->err, sizeof(unsigned));
  if (e == cudaSuccess) e = cudaMemset(c->err, 0, sizeof(unsigned));
  if (e == cudaSuccess) e = cudaMemset(c->buf[0], 0, bytes);
  if (e != cudaSuccess) {
    rlbm_massive_destroy(c);
    return fail(nullptr, RLBM_ECUDA, "setup: %s", cudaGetErrorString(e));
  }
  *out = c;
  return RLBM_OK;
}

int rlbm_massive_init(rlbm_massive_ctx* c, const double* n, const double* ux, const double* uy,
                      const double* T, int device_ptrs) {
  if (!c) return fail(nullptr, RLBM_EINVAL, "ctx is NULL");
  const long long ns = (long long)c->geo.nx * c->geo.ny;
  const size_t bytes = (size_t)c->geo.plane * kQm * c->elem;
  cudaError_t e;
  if (!n && !ux && !uy && !T) {
    e = cudaMemsetAsync(c->buf[0], 0, bytes, stream_of(c));
    if (e != cudaSuccess) return cuda_fail(c, e, "memset");
  } else {
    if (!n || !ux || !uy || !T) return fail(c, RLBM_EINVAL, "give all four fields or none");
    const double* f[4] = {n, ux, uy, T};
    if (!device_ptrs) {
      int r = need_scratch(c, 4 * ns * sizeof(double));
      if (r) return r;
      for (int k = 0; k < 4; ++k) {
        e = cudaMemcpyAsync(c->scratch + k * ns, f[k], ns * sizeof(double), cudaMemcpyHostToDevice, stream_of(c));
        if (e != cudaSuccess) return cuda_fail(c, e, "field upload");
        f[k] = c->scratch + k * ns;
      }
    }
    if (c->elem == 8)
      k_minit<double><<<grid_of(c->geo), dim3(32, 4), 0, stream_of(c)>>>((double*)c->buf[0], c->geo, c->of, f[0], f[1], f[2], f[3], c->err);
    else
      k_minit<float><<<grid_of(c->geo), dim3(32, 4), 0, stream_of(c)>>>((float*)c->buf[0], c->geo, c->of, f[0], f[1], f[2], f[3], c->err);
    e = cudaGetLastError();
    if (e != cudaSuccess) return cuda_fail(c, e, "init kernel");
    ++c->launches;
    e = cudaStreamSynchronize(stream_of(c));
    if (e != cudaSuccess) return cuda_fail(c, e, "init");
    unsigned bits = 0;
    e = cudaMemcpy(&bits, c->err, sizeof bits, cudaMemcpyDeviceToHost);
    if (e != cudaSuccess) return cuda_fail(c, e, "error word");
    if (bits) {
      cudaMemset(c->err, 0, sizeof(unsigned));
      return fail(c, RLBM_EINVAL, "init fields: need |u| < 1, n > 0, T > 0");
    }
  }
  c->cur = 0;
  c->steps = 0;
  return RLBM_OK;
}



int rlbm_massive_step(rlbm_massive_ctx* c, int nsteps, double* residual) {
  if (!c) return fail(nullptr, RLBM_EINVAL, "ctx is NULL");
  if (nsteps < 0) return fail(c, RLBM_EINVAL, "nsteps < 0");
  if (!residual) return launch_steps(c, nsteps);
  if (nsteps < 1) return fail(c, RLBM_EINVAL, "a residual needs nsteps >= 1");
  const long long ns = (long long)c->geo.nx * c->geo.ny;
  int r = need_scratch(c, 4 * ns * sizeof(double) + 2 * sizeof(double));
  if (r) return r;
  double* up = c->scratch;             // u(t - 1): x, y planes; u(t): x, y planes; sums
  double* acc = c->scratch + 4 * ns;
  if ((r = launch_steps(c, nsteps - 1))) return r;
  if ((r = velocity_planes(c, up, up + ns))) return r;
  if ((r = launch_steps(c, 1))) return r;
  if ((r = velocity_planes(c, up + 2 * ns, up + 3 * ns))) return r;
  cudaError_t e = cudaMemsetAsync(acc, 0, 2 * sizeof(double), stream_of(c));
  if (e != cudaSuccess) return cuda_fail(c, e, "memset");
  k_mresidual<<<grid_1d(ns), 256, 0, stream_of(c)>>>(up, up + ns, up + 2 * ns, up + 3 * ns, ns, acc);
  e = cudaGetLastError();
  if (e != cudaSuccess) return cuda_fail(c, e, "residual kernel");
  ++c->launches;
  double h[2];
  e = cudaMemcpyAsync(h, acc, sizeof h, cudaMemcpyDeviceToHost, stream_of(c));
  if (e == cudaSuccess) e = cudaStreamSynchronize(stream_of(c));
  if (e != cudaSuccess) return cuda_fail(c, e, "residual readback");
  *residual = h[1] > 0.0 ? std::sqrt(h[0] / h[1]) : (h[0] > 0.0 ? INFINITY : 0.0);
  return rlbm_massive_check(c);
}



int rlbm_massive_moments(rlbm_massive_ctx* c, double* n, double* ux, double* uy, double* T,
                         int device_ptrs) {
  if (!c) return fail(nullptr, RLBM_EINVAL, "ctx is NULL");
  const long long ns = (long long)c->geo.nx * c->geo.ny;
  double* d[4] = {n, ux, uy, T};
  if (!device_ptrs) {
    int r = need_scratch(c, 4 * ns * sizeof(double));
    if (r) return r;
    for (int k = 0; k < 4; ++k) d[k] = c->scratch + k * ns;
  }
  if (c->elem == 8)
    k_mmoments<double><<<grid_of(c->geo), dim3(32, 4), 0, stream_of(c)>>>((const double*)c->buf[c->cur], c->geo, c->of, d[0], d[1], d[2], d[3], c->err);
  else
    k_mmoments<float><<<grid_of(c->geo), dim3(32, 4), 0, stream_of(c)>>>((const float*)c->buf[c->cur], c->geo, c->of, d[0], d[1], d[2], d[3], c->err);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return cuda_fail(c, e, "moments kernel");
  ++c->launches;
  if (!device_ptrs) {
    double* h[4] = {n, ux, uy, T};
    for (int k = 0; k < 4; ++k) {
      if (!h[k]) continue;
      e = cudaMemcpyAsync(h[k], d[k], ns * sizeof(double), cudaMemcpyDeviceToHost, stream_of(c));
      if (e != cudaSuccess) return cuda_fail(c, e, "moments download");
    }
    e = cudaStreamSynchronize(stream_of(c));
    if (e != cudaSuccess) return cuda_fail(c, e, "moments");
  }
  return RLBM_OK;
}

int rlbm_massive_get_state(rlbm_massive_ctx* c, double* delta, int device_ptrs) {
  if (!c || !delta) return fail(c, RLBM_EINVAL, "NULL argument");
  const long long work = (long long)c->geo.nx * c->geo.ny * kQm;
  double* d = delta;
  if (!device_ptrs) {
    int r = need_scratch(c, work * sizeof(double));
    if (r) return r;
    d = c->scratch;
  }
  if (c->elem == 8) k_mget<double><<<grid_1d(work), 256, 0, stream_of(c)>>>((const double*)c->buf[c->cur], c->geo, d);
  else k_mget<float><<<grid_1d(work), 256, 0, stream_of(c)>>>((const float*)c->buf[c->cur], c->geo, d);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return cuda_fail(c, e, "state kernel");
  ++c->launches;
  if (!device_ptrs) {
    e = cudaMemcpyAsync(delta, d, work * sizeof(double), cudaMemcpyDeviceToHost, stream_of(c));
    if (e == cudaSuccess) e = cudaStreamSynchronize(stream_of(c));
    if (e != cudaSuccess) return cuda_fail(c, e, "state download");
  }
  return RLBM_OK;
}

int rlbm_massive_set_state(rlbm_massive_ctx* c, const double* delta, int device_ptrs) {
  if (!c || !delta) return fail(c, RLBM_EINVAL, "NULL argument");
  const long long work = (long long)c->geo.nx * c->geo.ny * kQm;
  const double* d = delta;
  if (!device_ptrs) {
    int r = need_scratch(c, work * sizeof(double));
    if (r) return r;
    cudaError_t e = cudaMemcpyAsync(c->scratch, delta, work * sizeof(double), cudaMemcpyHostToDevice, stream_of(c));
    if (e != cudaSuccess) return cuda_fail(c, e, "state upload");
    d = c->scratch;
  }
  if (c->elem == 8) k_mset<double><<<grid_1d(work), 256, 0, stream_of(c)>>>((double*)c->buf[0], c->geo, d);
  else k_mset<float><<<grid_1d(work), 256, 0, stream_of(c)>>>((float*)c->buf[0], c->geo, d);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return cuda_fail(c, e, "state kernel");
  ++c->launches;
  c->cur = 0;
  c->steps = 0;
  if (!device_ptrs) {
    e = cudaStreamSynchronize(stream_of(c));
    if (e != cudaSuccess) return cuda_fail(c, e, "state upload");
  }
  return RLBM_OK;
}

int rlbm_massive_check(rlbm_massive_ctx* c) {
  if (!c) return fail(nullptr, RLBM_EINVAL, "ctx is NULL");
  cudaError_t e = cudaStreamSynchronize(stream_of(c));
  if (e != cudaSuccess) return cuda_fail(c, e, "sync");
  unsigned bits = 0;
  e = cudaMemcpy(&bits, c->err, sizeof bits, cudaMemcpyDeviceToHost);
  if (e != cudaSuccess) return cuda_fail(c, e, "error word");
  if (!bits) return RLBM_OK;
  cudaMemset(c->err, 0, sizeof(unsigned));
  return fail(c, RLBM_ENAN, "device error bits 0x%x (1 non-finite, 2 |u| >= 1 or n, T <= 0, "
              "4 Landau solve not converged)", bits);
}

long long rlbm_massive_steps_done(const rlbm_massive_ctx* c) { return c ? c->steps : -1; }
long long rlbm_massive_launch_count(const rlbm_massive_ctx* c) { return c ? c->launches : -1; }

void rlbm_massive_destroy(rlbm_massive_ctx* c) {
  if (!c) return;
  cudaStreamSynchronize(stream_of(c));
  for (int b = 0; b < 2; ++b) if (c->buf[b]) cudaFree(c->buf[b]);
  if (c->err) cudaFree(c->err);
  if (c->scratch) cudaFree(c->scratch);
  delete c;
}

const char* rlbm_massive_last_error(const rlbm_massive_ctx* c) {
  return c ? c->msg.c_str() : g_error.c_str();
}

}  // extern "C"
