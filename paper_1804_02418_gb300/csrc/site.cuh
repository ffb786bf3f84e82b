// Per-site arithmetic of the relativistic lattice Boltzmann step
// (Eq. discrete-rbe, the per-site algorithm at the end of Sec. 2, App. A-B).
//
// Everything here works on relative deviations from the rest equilibrium
// (n = T = 1, u = 0, where f^eq_i = w_i):  g_i = (f_i - w_i) / w_i, the value
// every storage type keeps (16-bit storage scaled by s); delta_i = w_i g_i.
// Rest values of the moments (N = (1,0,0), T = diag(2,1,1)) are added
// analytically, and the
// equilibrium coefficients are written in terms of the small quantities
// n - 1, T - 1, gamma - 1 and T gamma - 1, so FP32 arithmetic keeps full
// relative precision on the O(u) flux-carrying parts.
//
// The equilibrium.  Q(p) = sum_k a^(k) J^(k)(p) (App. A polynomials, App. B
// projections) is, on the massless shell p = p0 (1, v) and with
//     W = T gamma - 1,  (X, Y) = T gamma u,  z(v) = W + X vx + Y vy,
// a cubic in the shell energy whose coefficients are polynomials in z alone:
//     Q - 1 = q0 + p0 (kappa z + lambda) + p0^2 z (mu z + D) + p0^3 z^3 / 6,
//     D = W^2 - X^2 - Y^2,               q0 = W^2 + r^2/2 - W (1 + W^2 + 3 r^2/2),
//     kappa = 1 - 3 W + 6 W^2 + 3 r^2/2, lambda = D (1 - 3 W),
//     mu = 1/2 - 5 W / 2,                r^2 = X^2 + Y^2
// (App. A-B multiplied out with vx^2 + vy^2 = 1 and the mass shell
// (1 + W)^2 = T^2 + r^2).  W, X, Y and everything built from them vanish at
// rest, so the small quantities keep their relative precision.  One scalar z
// per direction replaces the 15 polynomial coefficients of q_m(v): the
// per-site set-up is about 25 operations and a direction's cubic about 8.
// Measured against the expansion in monomials of v (15 coefficients, about
// 110 operations to form, 46 paired instructions per direction pair with a
// force instead of 24; Landau solve in FP64 throughout), whole passes of
// init + steps + fields: FP64 1024 x 512 with force 10.82 -> 7.49 ms (10
// steps; bound by the FP64 pipe), FP64 64 x 64 3.11 -> 2.48 ms (100 steps),
// FP16 storage 4096 x 2048 7.81 -> 6.94 ms (20 steps; bound by the FMA pipe),
// FP32 1024 x 512 1.91 -> 1.81 ms (50 steps).
#pragma once
#include <cuda_runtime.h>
#include <cuda_fp16.h>
#include <cuda_bf16.h>
#include <stdint.h>

#include <type_traits>

namespace rlbm {

constexpr int kQ = 48;
constexpr int kDirs = 12;
constexpr int kShells = 4;
constexpr int kRadius = 5;
constexpr int kMaxContacts = 4;

// Stencil G = {(+-3,+-4)_FS, (+-5,0)_FS} (Sec. 2.3); opposite of d is d ^ 1.
__host__ __device__ constexpr int hop_x(int d) {
  return d == 0 ? 3 : d == 1 ? -3 : d == 2 ? -3 : d == 3 ? 3 : d == 4 ? 4 : d == 5 ? -4
       : d == 6 ? -4 : d == 7 ? 4 : d == 8 ? 5 : d == 9 ? -5 : 0;
}
__host__ __device__ constexpr int hop_y(int d) {
  return d == 0 ? 4 : d == 1 ? -4 : d == 2 ? 4 : d == 3 ? -4 : d == 4 ? 3 : d == 5 ? -3
       : d == 6 ? 3 : d == 7 ? -3 : d == 8 ? 0 : d == 9 ? 0 : d == 10 ? 5 : -5;
}
__host__ __device__ constexpr int dir_kind(int d) { return d < 8 ? 0 : 1; }

// Quadrature constants (refined Sec. 2.3 values), uploaded once per module.
template <typename R>
struct QuadConsts {
  R p0[kShells];            // shell energies p0_j
  R wp0[2][kShells];        // w p0_j / s   (moments of the stored s g; s = 1 above 16 bits)
  R wp0sq[2][kShells];      // w p0_j^2 / s
  R dec_s, enc_s;           // 16-bit storage scale: 1 / s, s (the 16-bit kernels compute on s g)
  double wd[2][kShells];    // w in FP64: state I/O converts g <-> delta = w g in FP64
  double iwd[2][kShells], iwl[2][kShells];   // 1 / w = iwd + iwl
  // Conservation projection (reduced precision): correction
  // w_2j (l0 + l1 p0_j + p0_j (lx vx + ly vy)) on the (5,0)-type directions,
  // (l0, l1) = P (rN, rE), (lx, ly) = px (rX, rY).
  R P00, P01, P10, P11, px;
  // Operand pairs of the paired FP32 arithmetic (FP32 kernels only).  Pair
  // lanes are (direction d, its opposite d + 1) in the collision and (shell
  // j, shell j + 1) in the relaxation; a constant pair read from here costs
  // nothing as an operand, a literal pair of two different values would.
  float2 vxo[kDirs / 2], vyo[kDirs / 2];   // (vx, -vx), (vy, -vy) of direction pair q = d / 2
  float2 vxy[kDirs / 2];      // (vx, vy) of direction 2q
  float2 vsq[kDirs / 2];      // (vx^2, vx vy) of direction 2q
  float2 wab[2][kShells];     // (w p0_j / s, w p0_j^2 / s) by direction kind
  float2 p01, p23;            // (p0_0, p0_1), (p0_2, p0_3)
};

// Geometry and physics of one sample as seen by the kernels.
struct DevSample {
  int nx, ny, ldx;                    // ldx: row pitch in elements
  int periodic_x, periodic_y;
  int ncontacts;
  long long plane;                    // elements per population plane
  long long site0;                    // first site of this sample in the flat u / mask arrays
  long long off[2];                   // element offsets of the two buffers (batched launches)
  double inv_tau;
  double Fx, Fy;
  // the same in FP32, for the FP32 arithmetic (a conversion per thread would
  // run on the FP64 pipe)
  float inv_tau_f, Fx_f, Fy_f, inv_cg_f;
  int cedge[kMaxContacts], clo[kMaxContacts], chi[kMaxContacts];
  // electric force of the local capacitance approximation (Sec. 3): coupling
  // e^2 / C_g (0: none) and two planes of n - 1 in the arithmetic type, same
  // site indexing as a population plane; dn[cur] holds the previous step's
  // density, dn[cur ^ 1] receives this step's
  double inv_cg;
  void* dn[2];
  int cur;
};

// Error bits of the device error word.
constexpr unsigned kErrNonFinite = 1u;
constexpr unsigned kErrUnphysical = 2u;
constexpr unsigned kErrNoConvergence = 4u;
constexpr unsigned kErrTimeout = 8u;      // a bounded wait inside a kernel gave up

__device__ __forceinline__ bool finite_bits(float a) {
  return (__float_as_uint(a) & 0x7f800000u) != 0x7f800000u;
}
__device__ __forceinline__ bool finite_bits(double a) {
  return ((unsigned)__double2hiint(a) & 0x7ff00000u) != 0x7ff00000u;
}

// v / w for a weight w: the product with 1 / w held as hi + lo, rounded once
// (error below half an ulp and 2^-50 of one, as the division's, in 2 instead
// of about 10 FP64 operations).  An infinite v stays what it is: lo may have
// the other sign or be 0.
__device__ __forceinline__ double over(double v, double hi, double lo) {
  return finite_bits(v) ? fma(v, hi, v * lo) : v;
}
template <class C>
__device__ __forceinline__ double over_weight(double v, int kind, int j, const C& c) {
  return over(v, c.iwd[kind][j], c.iwl[kind][j]);
}

// ---------------------------------------------------------------------------
// Storage codecs.  The four shells of one (direction, site) are stored side by
// side, so one aligned vector access moves them (16 B for FP32, 32 B for FP64,
// 8 B for 16-bit storage).  The loads are written as assembly with a memory
// clobber: the compiler may move an ordinary read-only load above the wait
// for the predecessor's results (chain_wait).  They are coherent loads, not
// ld.global.nc: a chained step is resident while its predecessor still writes
// the buffer it will read, and .nc is defined only for memory that nothing
// writes during the whole kernel.
// ---------------------------------------------------------------------------
template <typename S> struct Codec;
template <> struct Codec<double> {
  using R = double;
  __device__ static void load4(const double* p, uint64_t, double* o) {
    asm volatile("ld.global.v2.f64 {%0, %1}, [%2];\n" : "=d"(o[0]), "=d"(o[1]) : "l"(p) : "memory");
    asm volatile("ld.global.v2.f64 {%0, %1}, [%2];\n" : "=d"(o[2]), "=d"(o[3]) : "l"(p + 2) : "memory");
  }
  // from shared memory (32-bit shared-window address)
  __device__ static void load4s(uint32_t a, double* o) {
    asm volatile("ld.shared.v2.f64 {%0, %1}, [%2];\n" : "=d"(o[0]), "=d"(o[1]) : "r"(a));
    asm volatile("ld.shared.v2.f64 {%0, %1}, [%2];\n" : "=d"(o[2]), "=d"(o[3]) : "r"(a + 16));
  }
  __device__ static void store4(double* p, const double* v) {
    reinterpret_cast<double2*>(p)[0] = make_double2(v[0], v[1]);
    reinterpret_cast<double2*>(p)[1] = make_double2(v[2], v[3]);
  }
  // stored relative deviation g <-> deviation delta = f - w (state I/O, in
  // FP64; the round trip can move a value by one ulp)
  template <class C> __device__ static double decode(double v, int kind, int j, const C& c) {
    return v * c.wd[kind][j];
  }
  template <class C> __device__ static double encode(double v, int kind, int j, const C& c) {
    return over_weight(v, kind, j, c);
  }
};
template <> struct Codec<float> {
  using R = float;
  // policy: an L2 eviction policy (pull_policy); the other types' loads take none
  __device__ static void load4(const float* p, uint64_t policy, float* o) {
    asm volatile("ld.global.L2::cache_hint.v4.f32 {%0, %1, %2, %3}, [%4], %5;\n"
                 : "=f"(o[0]), "=f"(o[1]), "=f"(o[2]), "=f"(o[3]) : "l"(p), "l"(policy) : "memory");
  }
  __device__ static void load4s(uint32_t a, float* o) {
    asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];\n"
                 : "=f"(o[0]), "=f"(o[1]), "=f"(o[2]), "=f"(o[3]) : "r"(a));
  }
  __device__ static void store4(float* p, const float* v) {
    *reinterpret_cast<float4*>(p) = make_float4(v[0], v[1], v[2], v[3]);
  }
  // in FP64: delta = g w to 1e-16, and delta / w rounds back to g exactly
  template <class C> __device__ static double decode(float v, int kind, int j, const C& c) {
    return double(v) * c.wd[kind][j];
  }
  template <class C> __device__ static float encode(double v, int kind, int j, const C& c) {
    return float(over_weight(v, kind, j, c));
  }
};
template <typename H> struct Codec16 {
  using R = float;
  __device__ static float tof(H h);
  __device__ static H fromf(float f);
  // two stored values <-> two floats (one conversion instruction per pair)
  __device__ static float2 unpack2(uint32_t u);
  __device__ static uint32_t pack2(float a, float b);
  __device__ static void load4(const H* p, uint64_t, float* o) {
    uint2 u;
    asm volatile("ld.global.v2.b32 {%0, %1}, [%2];\n" : "=r"(u.x), "=r"(u.y) : "l"(p) : "memory");
    const float2 a = unpack2(u.x), b = unpack2(u.y);   // s g: the kernels work scaled
    o[0] = a.x; o[1] = a.y; o[2] = b.x; o[3] = b.y;
  }
  __device__ static void load4s(uint32_t a, float* o) {
    uint2 u;
    asm volatile("ld.shared.v2.u32 {%0, %1}, [%2];\n" : "=r"(u.x), "=r"(u.y) : "r"(a));
    const float2 x = unpack2(u.x), y = unpack2(u.y);
    o[0] = x.x; o[1] = x.y; o[2] = y.x; o[3] = y.y;
  }
  __device__ static void store4(H* p, const float* v) {
    *reinterpret_cast<uint2*>(p) = make_uint2(pack2(v[0], v[1]), pack2(v[2], v[3]));
  }
  // stored s g <-> deviation delta = f - w (state I/O, in FP64: exact round trip)
  template <class C> __device__ static double decode(H v, int kind, int j, const C& c) {
    return double(tof(v)) * double(c.dec_s) * c.wd[kind][j];
  }
  template <class C> __device__ static H encode(double v, int kind, int j, const C& c) {
    return fromf(float(over_weight(v, kind, j, c) * double(c.enc_s)));
  }
};
template <> __device__ inline float2 Codec16<__half>::unpack2(uint32_t u) {
  __half2 h;
  memcpy(&h, &u, sizeof u);
  return __half22float2(h);
}
template <> __device__ inline uint32_t Codec16<__half>::pack2(float a, float b) {
  const __half2 h = __floats2half2_rn(a, b);
  uint32_t u;
  memcpy(&u, &h, sizeof u);
  return u;
}
template <> __device__ inline float2 Codec16<__nv_bfloat16>::unpack2(uint32_t u) {
  __nv_bfloat162 h;
  memcpy(&h, &u, sizeof u);
  return __bfloat1622float2(h);
}
template <> __device__ inline uint32_t Codec16<__nv_bfloat16>::pack2(float a, float b) {
  const __nv_bfloat162 h = __floats2bfloat162_rn(a, b);
  uint32_t u;
  memcpy(&u, &h, sizeof u);
  return u;
}
template <> __device__ inline float Codec16<__half>::tof(__half h) { return __half2float(h); }
template <> __device__ inline __half Codec16<__half>::fromf(float f) { return __float2half_rn(f); }
template <> __device__ inline float Codec16<__nv_bfloat16>::tof(__nv_bfloat16 h) { return __bfloat162float(h); }
template <> __device__ inline __nv_bfloat16 Codec16<__nv_bfloat16>::fromf(float f) { return __float2bfloat16_rn(f); }
template <> struct Codec<__half> : Codec16<__half> {};
template <> struct Codec<__nv_bfloat16> : Codec16<__nv_bfloat16> {};

// ---------------------------------------------------------------------------
// Macroscopic state of one site (deviation form).
// ---------------------------------------------------------------------------
template <typename R>
struct Macro {
  R ux, uy;
  R gamma, gm1;   // gamma and gamma - 1
  R dn, dT;       // n - 1, T - 1
  R deps;         // eps - 2
  R invT;         // 1 / T
};

// Reciprocal and reciprocal square root of a positive number.  FP32: the
// hardware approximations (1 - 2 ulp, far below the FP32 storage rounding the
// arithmetic feeds).  FP64: the hardware's approximation (relative error
// below 2^-18) refined by one step of third order from the residual
// e = 1 - a r (Householder's method; e^3 < 2^-54), 3 and 5 FP64 operations:
// the FP64 pipe retires 1/70 of the FP32 rate and bounds the FP64 step.
__device__ __forceinline__ float qrcp(float a) {
  float r;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(a));
  return r;
}
__device__ __forceinline__ double qrcp(double a) {
  double r;
  asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(r) : "d"(a));
  double e = fma(-a, r, 1.0);
  e = fma(e, e, e);
  return fma(r, e, r);
}
__device__ __forceinline__ float qrsqrt(float a) { return rsqrtf(a); }
__device__ __forceinline__ double qrsqrt(double a) {
  double y;
  asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(a));
  const double e = fma(-(a * y), y, 1.0);
  return fma(y * e, fma(e, 0.375, 0.5), y);
}

// double <-> float by moving bits (integer operations, off the FP64 pipe, on
// which conversions run too): toward zero, values below the normal FP32 range
// become 0, values above it (and NaN) infinity.
__device__ __forceinline__ float trunc_f32(double d) {
  const unsigned hi = (unsigned)__double2hiint(d), lo = (unsigned)__double2loint(d);
  const unsigned mag = hi & 0x7fffffffu;
  unsigned m = ((mag - (896u << 20)) << 3) | (lo >> 29);
  if (mag < (897u << 20)) m = 0u;
  if (mag >= (1151u << 20)) m = 0x7f800000u;
  return __uint_as_float((hi & 0x80000000u) | m);
}
// exact for normal numbers and zero; infinity and NaN become NaN
__device__ __forceinline__ double widen_f64(float f) {
  const unsigned b = __float_as_uint(f), mag = b & 0x7fffffffu;
  unsigned hi = (mag >> 3) + (896u << 20), lo = b << 29;
  if (mag < 0x00800000u) hi = lo = 0u;
  if (mag >= 0x7f800000u) hi = 0x7ff80000u;
  return __hiloint2double((int)((b & 0x80000000u) | hi), (int)lo);
}

// double(a), off the FP64 pipe for normal numbers and zero
__device__ __forceinline__ double as_f64(double a) { return a; }
__device__ __forceinline__ double as_f64(float a) {
  const unsigned e = __float_as_uint(a) & 0x7f800000u;
  return (e - 0x00800000u) < 0x7f000000u || a == 0.f ? widen_f64(a) : double(a);
}

// a > 0 (false for NaN) without a compare on the FP64 pipe; for numbers that
// are no subnormal ones (sums with 1 or 2)
__device__ __forceinline__ bool positive(float a) { return a > 0.f; }
__device__ __forceinline__ bool positive(double a) {
  const int hi = __double2hiint(a);
  return hi > 0 && hi <= 0x7ff00000;
}

// Moment deviations from 48 streamed deviations.
template <typename R>
struct Moments {
  R dN0, dNx, dNy;              // N^a - (1, 0, 0)
  R dE, Mx, My, dPxx, dPxy, dPyy; // T^ab - diag(2, 1, 1)
};

// In FP64 the sums are formed per group of four directions (velocities v, -v
// and their mirror images; group 2: the axes), so that three warps can share a
// site's populations and get the same bits.  With A_d = sum_j w p0_j g_dj,
// B_d = sum_j w p0_j^2 g_dj and |v| = (a, b) in a group: N = sum A, X = sum A
// sign(vx), Y = sum A sign(vy); E, MX, MY alike from B; S = sum B sign(vx vy)
// (group 2: the part of E on the x axis).
template <typename R>
struct GroupSums {
  R N, X, Y, E, MX, MY, S;
};

template <int G, typename R, class C>
__device__ __forceinline__ GroupSums<R> group_sums(const R* f, const C& qc) {
  constexpr int k = G == 2 ? 1 : 0;
  R A[4], B[4];
#pragma unroll
  for (int d = 0; d < 4; ++d) {
    A[d] = f[4 * d] * qc.wp0[k][0];
    B[d] = f[4 * d] * qc.wp0sq[k][0];
#pragma unroll
    for (int j = 1; j < kShells; ++j) {
      A[d] = fma(f[4 * d + j], qc.wp0[k][j], A[d]);
      B[d] = fma(f[4 * d + j], qc.wp0sq[k][j], B[d]);
    }
  }
  GroupSums<R> s;
  if (G == 2) {                    // (1,0) (-1,0) (0,1) (0,-1)
    s.N = (A[0] + A[1]) + (A[2] + A[3]);
    s.X = A[0] - A[1];
    s.Y = A[2] - A[3];
    s.S = B[0] + B[1];
    s.E = s.S + (B[2] + B[3]);
    s.MX = B[0] - B[1];
    s.MY = B[2] - B[3];
  } else {                         // (a,b) (-a,-b) (-a,b) (a,-b)
    const R pA = A[0] + A[1], qA = A[2] + A[3], mA = A[0] - A[1], nA = A[3] - A[2];
    const R pB = B[0] + B[1], qB = B[2] + B[3], mB = B[0] - B[1], nB = B[3] - B[2];
    s.N = pA + qA;
    s.X = mA + nA;
    s.Y = mA - nA;
    s.E = pB + qB;
    s.MX = mB + nB;
    s.MY = mB - nB;
    s.S = pB - qB;
  }
  return s;
}

template <typename R>
__device__ __forceinline__ Moments<R> add_groups(const GroupSums<R>& g, const GroupSums<R>& h,
                                                 const GroupSums<R>& a) {
  Moments<R> m;
  m.dN0 = (g.N + h.N) + a.N;
  m.dNx = fma(g.X, R(0.6), fma(h.X, R(0.8), a.X));
  m.dNy = fma(g.Y, R(0.8), fma(h.Y, R(0.6), a.Y));
  m.dE = (g.E + h.E) + a.E;
  m.Mx = fma(g.MX, R(0.6), fma(h.MX, R(0.8), a.MX));
  m.My = fma(g.MY, R(0.8), fma(h.MY, R(0.6), a.MY));
  m.dPxx = fma(g.E, R(0.36), fma(h.E, R(0.64), a.S));
  m.dPxy = (g.S + h.S) * R(0.48);
  m.dPyy = m.dE - m.dPxx;   // massless shells: T^00 = T^xx + T^yy exactly
  return m;
}

template <typename R, class C>
__device__ __forceinline__ Moments<R> moments_scalar(const R (&f)[kQ], const C& qc) {
  return add_groups(group_sums<0>(f, qc), group_sums<1>(f + 16, qc), group_sums<2>(f + 32, qc));
}

// ---------------------------------------------------------------------------
// Paired FP32 arithmetic.  Blackwell retires two FP32 fused multiply-adds per
// instruction on a register pair (the same per-lane rounding as two scalar
// ones); the FP32 step is bound by its instruction issue, so its collision is
// written on pairs.  A pair whose lanes hold the same value ("splat") costs
// nothing extra as an operand.
// ---------------------------------------------------------------------------
__device__ __forceinline__ float2 S2(float a) { return make_float2(a, a); }
__device__ __forceinline__ float2 fma2(float2 a, float2 b, float2 c) { return __ffma2_rn(a, b, c); }
__device__ __forceinline__ float2 mul2(float2 a, float2 b) { return __fmul2_rn(a, b); }
__device__ __forceinline__ float2 add2(float2 a, float2 b) { return __fadd2_rn(a, b); }

// The moments of moments() on pairs: lanes (A_d, B_d) of one direction,
// A_d = sum_j w p0_j g_dj, B_d = sum_j w p0_j^2 g_dj.
template <class C>
__device__ __forceinline__ Moments<float> moments_paired(const float (&f)[kQ], const C& qc) {
  float2 NE = S2(0.f), NxMx = S2(0.f), NyMy = S2(0.f), PP = S2(0.f);
#pragma unroll
  for (int d = 0; d < kDirs; d += 2) {
    const int k = dir_kind(d);
    float2 ABp = mul2(S2(f[4 * d]), qc.wab[k][0]);
    float2 ABn = mul2(S2(f[4 * d + 4]), qc.wab[k][0]);
#pragma unroll
    for (int j = 1; j < kShells; ++j) {
      ABp = fma2(S2(f[4 * d + j]), qc.wab[k][j], ABp);
      ABn = fma2(S2(f[4 * d + 4 + j]), qc.wab[k][j], ABn);
    }
    const float2 e = add2(ABp, ABn);                 // (A_e, B_e): even parts
    const float2 o = fma2(ABn, S2(-1.f), ABp);       // (A_o, B_o): odd parts
    const float vx = float(hop_x(d)) / 5.f, vy = float(hop_y(d)) / 5.f;
    if (d == 0) {
      NE = e;
      NxMx = mul2(o, S2(vx));
      NyMy = mul2(o, S2(vy));
      PP = mul2(S2(e.y), qc.vsq[d / 2]);
    } else {
      NE = add2(NE, e);
      if (hop_x(d) != 0) NxMx = fma2(o, S2(vx), NxMx);
      if (hop_y(d) != 0) NyMy = fma2(o, S2(vy), NyMy);
      if (hop_x(d) != 0) PP = fma2(S2(e.y), qc.vsq[d / 2], PP);
    }
  }
  Moments<float> m;
  m.dN0 = NE.x; m.dE = NE.y;
  m.dNx = NxMx.x; m.Mx = NxMx.y;
  m.dNy = NyMy.x; m.My = NyMy.y;
  m.dPxx = PP.x; m.dPxy = PP.y;
  m.dPyy = m.dE - m.dPxx;   // massless shells: T^00 = T^xx + T^yy exactly
  return m;
}

// Moment deviations of 48 streamed relative deviations: paired in FP32,
// scalar in FP64.
template <typename R, class C>
__device__ __forceinline__ Moments<R> moments(const R (&f)[kQ], const C& qc) {
  if constexpr (std::is_same<R, float>::value) return moments_paired(f, qc);
  else return moments_scalar(f, qc);
}

// Landau frame eps U^a = T^ab U_b:  u = (Pi + eps I)^-1 M, eps = E - M.u,
// Newton on g(eps) = eps - E + M.u(eps), g' = 1 - u.u, from eps0 = E.
// Then n = U_a N^a and the massless EOS eps = 2 n T.
//
// The unknown of the FP32 iteration is d = eps - E = -M.u, which keeps its
// relative precision.  FP64 starts from the FP32 solution (its error is about
// 1e-7 u^2) and takes Newton steps until one is below 1e-8 (2 + |deps|): the
// next would be its square times u^2 / (3 (1 - u^2)), below the FP64 rounding
// (which 1 / (1 - u^2) magnifies alike), so one FP64 step is the rule.  The
// slope is FP64 too: one of FP32 leaves 1.5e-7 of the step, T off by 7.3e-16 at
// |u| = 0.1 - 0.3 (3 operations of about 700 per site: 1024 x 512, 10 steps,
// 7.36 -> 7.39 ms).
// After the last step u follows by its derivative, du = (Pi + eps I)^-1 u step.
__device__ __forceinline__ bool landau_d32(float dE, float Mx, float My, float dPxx, float dPxy,
                                           float dPyy, float& d, float& ux, float& uy) {
  const float a0 = 3.f + dPxx, c0 = 3.f + dPyy, p2 = dPxy * dPxy;
  d = 0.f;
#pragma unroll 1
  for (int it = 0; it < 12; ++it) {
    const float deps = dE + d;
    const float a = a0 + deps, c = c0 + deps;
    const float inv = qrcp(fmaf(a, c, -p2));
    ux = fmaf(c, Mx, -(dPxy * My)) * inv;
    uy = fmaf(a, My, -(dPxy * Mx)) * inv;
    const float g = fmaf(Mx, ux, fmaf(My, uy, d));
    const float step = g * qrcp(fmaf(-ux, ux, fmaf(-uy, uy, 1.f)));
    d -= step;
    if (fabsf(step) <= 2e-7f * (2.f + fabsf(deps))) {
      const float si = step * inv;
      const float vx = fmaf(c, ux, -(dPxy * uy)), vy = fmaf(a, uy, -(dPxy * ux));
      ux = fmaf(si, vx, ux);
      uy = fmaf(si, vy, uy);
      return true;
    }
  }
  return false;
}

__device__ __forceinline__ bool landau_frame(const Moments<float>& m, float& deps, float& ux,
                                             float& uy) {
  float d;
  const bool conv = landau_d32(m.dE, m.Mx, m.My, m.dPxx, m.dPxy, m.dPyy, d, ux, uy);
  deps = m.dE + d;
  return conv;
}

__device__ __forceinline__ bool landau_frame(const Moments<double>& m, double& deps, double& ux,
                                             double& uy) {
  float d32, ux32, uy32;
  const bool conv32 = landau_d32(trunc_f32(m.dE), trunc_f32(m.Mx), trunc_f32(m.My),
                                 trunc_f32(m.dPxx), trunc_f32(m.dPxy), trunc_f32(m.dPyy), d32,
                                 ux32, uy32);
  // an FP32 iteration that did not converge (|u| near 1) may have left the
  // root's side: then from eps = E
  double d = conv32 ? widen_f64(d32) : 0.0;
  const double a0 = 3.0 + m.dPxx + m.dE, c0 = 3.0 + m.dPyy + m.dE, p2 = m.dPxy * m.dPxy;
  bool conv = false;
#pragma unroll 1
  for (int it = 0; it < 12; ++it) {
    const double a = a0 + d, c = c0 + d;
    const double inv = qrcp(fma(a, c, -p2));
    ux = fma(c, m.Mx, -(m.dPxy * m.My)) * inv;
    uy = fma(a, m.My, -(m.dPxy * m.Mx)) * inv;
    const double g = fma(m.Mx, ux, fma(m.My, uy, d));
    const double w = fma(-ux, ux, fma(-uy, uy, 1.0));
    const double step = g * qrcp(w);
    d -= step;
    if (fabsf(trunc_f32(step)) <= 1e-8f * (2.f + fabsf(trunc_f32(m.dE) + trunc_f32(d)))) {
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

// Error bits of a site's fields; kErrUnphysical only where they are finite.
template <typename R>
__device__ __forceinline__ unsigned landau(const Moments<R>& m, Macro<R>& o) {
  R deps, ux, uy;
  const bool conv = landau_frame(m, deps, ux, uy);
  const R u2 = fma(ux, ux, uy * uy);
  const R w = R(1) - u2;
  const R gamma = qrsqrt(w);
  const R gm1 = u2 * gamma * (gamma * qrcp(R(1) + gamma));   // (gamma^2 - 1) / (gamma + 1)
  const R dNpar = fma(-uy, m.dNy, fma(-ux, m.dNx, m.dN0));   // U_a N^a / gamma - 1
  const R dn = fma(gm1, R(1) + dNpar, dNpar);                // n - 1
  const R n = R(1) + dn, eps = R(2) + deps;
  const R r = qrcp(n * eps);                                 // 1 / (n eps): both quotients below
  const R dT = fma(R(-2), dn, deps) * (R(0.5) * (eps * r));  // T - 1 = (eps - 2 n) / (2 n)
  o.ux = ux; o.uy = uy; o.gamma = gamma; o.gm1 = gm1; o.dn = dn; o.dT = dT; o.deps = deps;
  // 1 / T = 2 n / eps; in FP32, where three roundings more show, from T
  if constexpr (sizeof(R) == 4) o.invT = qrcp(R(1) + dT);
  else o.invT = (n + n) * (n * r);
  unsigned bits = conv ? 0u : kErrNoConvergence;
  if (!(finite_bits(ux) && finite_bits(uy) && finite_bits(dn) && finite_bits(dT)))
    bits |= kErrNonFinite;
  else if (!(positive(w) && positive(n) && positive(eps)))
    bits |= kErrUnphysical;
  return bits;
}

// Site coefficients of (f^eq - w) / w = e0 + p0 e1 + p0^2 e2 + p0^3 e3,
//   e1 = kap z + lam, e2 = z (mu z + D), e3 = nu z^3   (header comment),
// all times n / T; nT = n / T and nmT = (n - T) / T carry the storage scale.
template <typename R>
struct EqCoeffs {
  R W, X, Y;
  R e0, kap, lam, mu, D, nu;
};

template <typename R>
__device__ __forceinline__ EqCoeffs<R> eq_coeffs(const Macro<R>& M, R nT, R nmT) {
  EqCoeffs<R> c;
  const R W = fma(M.dT, M.gamma, M.gm1);                 // T gamma - 1
  const R X = fma(W, M.ux, M.ux), Y = fma(W, M.uy, M.uy);  // T gamma u, rounded once
  const R r2 = fma(X, X, Y * Y), W2 = W * W;
  const R h = fma(R(1.5), r2, R(1));                     // 1 + 3 r^2 / 2
  const R q0 = fma(-W, W2 + h, fma(R(0.5), r2, W2));
  const R t = fma(R(-3), W, R(1));                       // 1 - 3 W
  c.W = W; c.X = X; c.Y = Y;
  c.e0 = fma(nT, q0, nmT);
  c.D = nT * (W2 - r2);
  c.lam = c.D * t;
  c.kap = nT * fma(R(-3), W, fma(R(6), W2, h));
  c.mu = nT * fma(R(-2.5), W, R(0.5));
  c.nu = nT * R(1.0 / 6.0);
  return c;
}

// Per-direction cubic R_0 + R_1 p0 + R_2 p0^2 + R_3 p0^3 such that the new
// deviation of shell j is  (1 - omega_d) g_dj + sum_m R_m p0_j^m:
//   omega_d (f^eq - w) / w  +  F^ext / w,
// with omega_d = gamma (1 - v_d.u) / tau (= p^m U_m / (p^0 tau) on the massless shell).
// Forcing (force F per particle, dt = 1):
//   F^ext / w = (n/T) [ (F.v) Q - F.grad Q ]  at p = p0 (1, v),
// grad along the shell (grad p0 = v).  Q depends on the momentum through p0
// and y = p0 z = W p0 + X px + Y py, so with phi = F.v, f = F.(X, Y) and
// psi = F.grad y = W phi + f
//   F.grad Q = phi (lambda + D y) + psi (kappa + D p0 + 2 mu y + y^2 / 2);
// psi is linear in phi, and everything that multiplies phi or stands alone is
// gathered per site:
//   R_0 = o e0 + a0 phi + b0
//   R_1 = o e1 + z (a1 phi + b1) + a2 phi + b2
//   R_2 = o e2 + z^2 (a3 phi + b3)
//   R_3 = o e3,                        o = omega + phi = gt + (F - gt u).v.
// FP32 rounds omega, of order 1, by more than phi's digits and needs omega and
// 1 - omega to add up to 1: there R_0 and R_1 take omega alone, with phi e0 and
// phi e1 in a0, a1 and a2; R_2 and R_3 are of second order in z.  After 2,000
// steps of a closed box at F = 2e-6 (256 x 128) the error of n - 1 is 5.5e-8,
// 1.2e-7 with phi in omega.
template <typename R>
struct ForceCoeffs {
  R a0, b0, a1, b1, a2, b2, a3, b3;
};

template <typename R>
__device__ __forceinline__ ForceCoeffs<R> force_coeffs(const EqCoeffs<R>& c, R Fx, R Fy, R scl) {
  ForceCoeffs<R> k;
  const R f = fma(Fx, c.X, Fy * c.Y);
  const R m2 = R(-2) * c.mu, n3 = R(-3) * c.nu;
  k.a0 = fma(-c.W, c.kap, scl - c.lam);
  k.b0 = -(f * c.kap);
  k.a1 = fma(m2, c.W, -c.D);
  k.b1 = m2 * f;
  k.a2 = -(c.D * c.W);
  if constexpr (sizeof(R) == 4) {
    k.a0 += c.e0;
    k.a1 += c.kap;
    k.a2 += c.lam;
  }
  k.b2 = -(c.D * f);
  k.a3 = n3 * c.W;
  k.b3 = n3 * f;
  return k;
}

// What a direction's cubic needs beside c: gt = gamma / tau, gt u and F; FP64
// also 1 - gt.
template <typename R>
struct RelaxSite {
  R gt, omgt, gux, guy, Fx, Fy;
};

// The cubic of one direction from its z, o = omega + phi and phi = F.v.
template <typename R, bool FORCE>
__device__ __forceinline__ void direction_cubic(const EqCoeffs<R>& c, const ForceCoeffs<R>& k,
                                                R z, R o, R phi, R (&Rm)[4]) {
  const R e1 = fma(c.kap, z, c.lam);
  const R e2 = z * fma(c.mu, z, c.D);
  const R z2 = z * z;
  const R e3 = (c.nu * z) * z2;
  if (FORCE) {
    Rm[0] = fma(o, c.e0, fma(phi, k.a0, k.b0));
    Rm[1] = fma(o, e1, fma(z, fma(phi, k.a1, k.b1), fma(phi, k.a2, k.b2)));
    Rm[2] = fma(o, e2, z2 * fma(phi, k.a3, k.b3));
  } else {
    Rm[0] = o * c.e0;
    Rm[1] = o * e1;
    Rm[2] = o * e2;
  }
  Rm[3] = o * e3;
}

// Cubics and 1 - omega of directions d (even) and d + 1 (opposite velocity).
template <typename R, bool FORCE>
__device__ __forceinline__ void pair_cubics(const int d, const EqCoeffs<R>& c,
                                            const ForceCoeffs<R>& k, const RelaxSite<R>& s,
                                            R (&Rp)[4], R (&Rn)[4], R& omcp, R& omcn) {
  const R vx = R(hop_x(d)) / R(5), vy = R(hop_y(d)) / R(5);
  R zo, go, phi;
  if (hop_y(d) == 0) {            // v = (1, 0)
    zo = c.X; go = s.gux; phi = s.Fx;
  } else if (hop_x(d) == 0) {     // v = (0, 1)
    zo = c.Y; go = s.guy; phi = s.Fy;
  } else {
    zo = fma(c.X, vx, c.Y * vy);
    go = fma(s.gux, vx, s.guy * vy);
    phi = FORCE ? fma(s.Fx, vx, s.Fy * vy) : R(0);
  }
  const R oo = FORCE ? phi - go : -go;
  omcp = s.omgt + go;
  omcn = s.omgt - go;
  direction_cubic<R, FORCE>(c, k, c.W + zo, s.gt + oo, phi, Rp);
  direction_cubic<R, FORCE>(c, k, c.W - zo, s.gt - oo, -phi, Rn);
}

}  // namespace rlbm
