// Kernels of the fused relativistic LBM step, templated on the storage type.
//
// Stored values are relative deviations g = (f - w) / w from the rest weights
// (times s in 16-bit storage, where the kernels also compute on s g).
//
// Layout in HBM (per sample): two ping-pong buffers, each 12 direction planes
// of `plane` sites (row-major, row pitch ldx a multiple of 32, plane a
// multiple of 64 sites).  A site of direction plane d holds the four shells of
// direction d side by side:
//     element (d, site, j) = buffer[(d * plane + site) * 4 + j].
// The four shells share their pull offset n_d, so one aligned vector access
// moves them (the shift by n_d keeps the 16 / 32 / 8-byte alignment because
// it moves by whole sites).
//
// One thread updates one site.  Pull scheme: the thread gathers the 12 vectors
// arriving at its site (each warp reads 32 consecutive sites of a shifted row:
// coalesced), applies the boundary rules, collides in registers and writes 12
// vectors of its own site into the other buffer.
#pragma once
#include <type_traits>

#include "site.cuh"

namespace rlbm {

constexpr int kBX = 128;   // threads per block along x; one block row per y

// FORCE template argument of the step kernels: no force, a uniform force per
// particle, or a uniform force plus the electric force of the local
// capacitance approximation (its own instantiation, so that the others do not
// carry its registers).
constexpr int kForceNone = 0, kForceUniform = 1, kForceLca = 2;

template <typename R>
struct StepAux {
  R* uprev;              // [sites] x 2 velocity plane for the residual (or null)
  double* acc;           // [2] residual accumulators (sum |du|^2, sum |u|^2)
  unsigned* err;         // device error word
};

__device__ __forceinline__ long long vec_index(const DevSample& s, int d, long long site) {
  return ((long long)d * s.plane + site) * 4;
}

// Index of the contact whose ghost strip holds the (outside) source (sx, sy).
__device__ __forceinline__ int contact_of(const DevSample& s, int sx, int sy) {
#pragma unroll
  for (int k = 0; k < kMaxContacts; ++k) {
    if (k >= s.ncontacts) break;
    const int e = s.cedge[k];
    const int t = (e < 2) ? sx : sy;
    const bool side = e == 0 ? (sy < 0) : e == 1 ? (sy >= s.ny) : e == 2 ? (sx < 0) : (sx >= s.nx);
    if (side && t >= s.clo[k] && t < s.chi[k]) return k;
  }
  return -1;
}

// A thread's site vector in direction plane 0 of the two buffers, and the
// byte offsets from there to the 12 vectors it pulls (interior sites) and to
// the 12 direction planes it stores.  The single-sample kernel takes the
// offsets from its parameters (constant memory: two additions per access);
// formed from the descriptor by each thread they cost about 100 integer
// instructions per site, most of them on the pipe that bounds the 16-bit step.
template <typename S>
struct Tile {
  const S* in;
  S* out;
  uint64_t policy;     // L2 policy of the pulled vectors
};

template <typename S>
__host__ __device__ constexpr long long pull_offset(int d, long long plane, long long ldx) {
  return ((long long)d * plane - ((long long)hop_y(d) * ldx + hop_x(d))) * (long long)(4 * sizeof(S));
}
template <typename S>
__host__ __device__ constexpr long long plane_offset(int d, long long plane) {
  return (long long)d * plane * (long long)(4 * sizeof(S));
}

struct StepOffsets {        // prepared on the host
  long long pull_[kDirs], plane_[kDirs];
  __device__ __forceinline__ long long pull(int d) const { return pull_[d]; }
  __device__ __forceinline__ long long plane(int d) const { return plane_[d]; }
};
template <typename S>
struct SampleOffsets {      // from the descriptor
  long long p;
  int ldx;
  __device__ __forceinline__ long long pull(int d) const { return pull_offset<S>(d, p, ldx); }
  __device__ __forceinline__ long long plane(int d) const { return plane_offset<S>(d, p); }
};

template <typename T>
__device__ __forceinline__ T* byte_ptr(T* base, long long bytes) {
  using B = typename std::conditional<std::is_const<T>::value, const char, char>::type;
  return reinterpret_cast<T*>(reinterpret_cast<B*>(base) + bytes);
}

// L2 policy of the pulls, FP32 storage (the other types' loads take none).
// Each stored value is read once per step and its line is next written a step
// later, so when a buffer is not much larger than the L2 the lines just read
// should leave first and the ones just written (the next step's input) stay;
// see launch_single for the rule.
__device__ __forceinline__ uint64_t pull_policy(bool evict_first) {
  uint64_t a, b;
  asm("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(a));
  asm("createpolicy.fractional.L2::evict_normal.b64 %0, 1.0;" : "=l"(b));
  return evict_first ? a : b;
}

// Gathers the 48 streamed deviations arriving at (x, y).
// Directions D0 .. D0 + ND - 1 into f[0 .. 4 ND).
template <typename S, bool INTERIOR, int D0, int ND, class C, class O>
__device__ __forceinline__ void pull(const S* __restrict__ fin, const Tile<S>& tl, const O& of,
                                     const DevSample& s, int x, int y,
                                     const typename Codec<S>::R* __restrict__ ghost, const C& qc,
                                     typename Codec<S>::R* f0) {
  typename Codec<S>::R* const f = f0 - 4 * D0;
#pragma unroll
  for (int d = D0; d < D0 + ND; ++d) {
    const int dx = hop_x(d), dy = hop_y(d);
    if (INTERIOR) {
      Codec<S>::load4(byte_ptr(tl.in, of.pull(d)), tl.policy, &f[4 * d]);
    } else {
      int sx = x - dx, sy = y - dy;
      if (s.periodic_x) sx = sx < 0 ? sx + s.nx : (sx >= s.nx ? sx - s.nx : sx);
      if (s.periodic_y) sy = sy < 0 ? sy + s.ny : (sy >= s.ny ? sy - s.ny : sy);
      const bool inside = (unsigned)sx < (unsigned)s.nx && (unsigned)sy < (unsigned)s.ny;
      if (inside) {
        Codec<S>::load4(fin + vec_index(s, d, (long long)sy * s.ldx + sx), tl.policy, &f[4 * d]);
      } else {
        const int owner = contact_of(s, sx, sy);
        if (owner >= 0) {
#pragma unroll
          for (int j = 0; j < kShells; ++j) f[4 * d + j] = ghost[owner * kQ + 4 * d + j];
        } else {
          // bounce-back: post-collision population of the opposite direction, same shell
          Codec<S>::load4(byte_ptr(tl.in, of.plane(d ^ 1)), tl.policy, &f[4 * d]);
        }
      }
    }
  }
}

// ---------------------------------------------------------------------------
// Shared-memory staging of the pull.  For one tile (a row segment of BX sites
// starting at x0 in row y) the 12 arriving populations come from 12 row
// segments, one per direction plane: plane d, row y - dy_d, columns
// x0 - dx_d .. x0 - dx_d + BX - 1.  Each segment is contiguous in HBM (whole
// site vectors), so the persistent batched kernel moves it with one bulk
// asynchronous copy (cp.async.bulk, completion counted in bytes on an
// mbarrier) into a shared-memory slot row while the block still computes the
// previous tile.  Columns outside the sample are clipped (their sites take the
// boundary rules, as in pull()); a segment that wraps around a periodic x edge
// is not staged and read directly.  Copies move whole 16-byte granules:
// 16-bit storage (8-byte vectors) rounds a segment out to even sites, and the
// slot index of column c is c - (a & ~(G - 1)), a = x0 - dx_d, G sites per
// granule.
// ---------------------------------------------------------------------------
// Parking of the gathered populations (16-bit storage).  After the moments
// are formed, the 48 values of a site leave the registers for a shared-memory
// area laid out [direction][thread] (16 bytes per entry: conflict-free) and
// come back one direction pair at a time for the relaxation.  This frees
// about 40 registers per thread, so more warps are resident to hide the
// latency of the long per-site arithmetic.  The accesses are volatile so that
// the compiler cannot keep the register copies alive instead.  FP16 storage,
// 4096 x 2048: 274 us per step, 289 without.  FP32 storage runs as well from
// registers at its five blocks per SM, without the 36 shared accesses per
// thread (1024 x 512: 27.1 -> 26.5 us per step, 200 x 150: 6.0 -> 5.9).
template <typename S> struct Park { static constexpr bool kOn = sizeof(S) == 2; };

// Bytes of the parking area of a block of `threads` threads.
template <typename S>
__host__ __device__ constexpr size_t park_bytes(int threads) {
  return Park<S>::kOn ? (size_t)kDirs * threads * 16 : 0;
}

__device__ __forceinline__ void park_store(uint32_t a, const float* v) {
  asm volatile("st.shared.v4.f32 [%0], {%1, %2, %3, %4};\n"
               :: "r"(a), "f"(v[0]), "f"(v[1]), "f"(v[2]), "f"(v[3]) : "memory");
}
__device__ __forceinline__ void park_load(uint32_t a, float* v) {
  asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];\n"
               : "=f"(v[0]), "=f"(v[1]), "=f"(v[2]), "=f"(v[3]) : "r"(a) : "memory");
}

// Control block after the two buffers: full[2] (mbarriers, 8 B each),
// released[2] (+ pad), tiles[2] (int4), masks[2], abort flag (+ pad).
constexpr size_t kStageCtlBytes = 16 + 16 + 32 + 8 + 8;

template <typename S>
struct Stage {
  static constexpr int kVecBytes = 4 * (int)sizeof(S);
  static constexpr int kG = kVecBytes >= 16 ? 1 : 16 / kVecBytes;   // sites per granule
  template <int BX> __host__ __device__ static constexpr int slots() { return BX + 2 * (kG - 1); }
  // elements of one buffer (12 slot rows)
  template <int BX> __host__ __device__ static constexpr int buf_elems() { return kDirs * slots<BX>() * 4; }
  // dynamic shared memory of the kernel: two buffers, then the control block
  template <int BX> __host__ __device__ static constexpr size_t smem_bytes() {
    return 2 * (size_t)buf_elems<BX>() * sizeof(S) + kStageCtlBytes +
           park_bytes<S>(BX);
  }
};

constexpr long long kStageSpinCycles = 2000000000LL;   // about 1 s at 2 GHz

__device__ __forceinline__ uint32_t smem_addr(const void* p) {
  return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}


__device__ __forceinline__ void stage_bar_init(uint32_t bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;\n" :: "r"(bar), "r"(count) : "memory");
}


// Bounded wait for the completion of the phase with the given parity: gives
// up (false) once more than `limit` clock cycles have passed.  The first probe
// does not block (test_wait), so a limit shorter than a copy's latency gives up
// at once; later probes may suspend the thread for a while (try_wait).
__device__ __forceinline__ bool stage_wait(uint32_t bar, uint32_t parity,
                                           long long limit = kStageSpinCycles) {
  const long long t0 = clock64();
  uint32_t ok;
  asm volatile(
      "{\n .reg .pred p;\n mbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2;\n"
      " selp.u32 %0, 1, 0, p;\n}\n"
      : "=r"(ok) : "r"(bar), "r"(parity) : "memory");
  while (!ok) {
    if (clock64() - t0 > limit) return false;
    asm volatile(
        "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n"
        " selp.u32 %0, 1, 0, p;\n}\n"
        : "=r"(ok) : "r"(bar), "r"(parity) : "memory");
  }
  return true;
}

// Issued by the 32 lanes of one warp (lane d < 12 copies direction d): the
// segments of tile (x0, y) of sample s into `buf`; *mask gets bit d for every
// staged direction and *tile the tile (sample, x0, y).  One arrive with the
// expected byte count (release semantics: mask and tile become visible to the
// waiting threads) completes the phase together with the copies.
template <typename S, int BX>
__device__ __forceinline__ void stage_issue(const S* __restrict__ fin, const DevSample& s, int x0,
                                            int y, S* buf, uint32_t bar, unsigned* mask,
                                            int4* tile, int sample) {
  constexpr int G = Stage<S>::kG, VB = Stage<S>::kVecBytes, SL = Stage<S>::template slots<BX>();
  const int lane = threadIdx.x & 31;
  const int nv = min(BX, s.nx - x0);
  bool ok = false;
  uint32_t bytes = 0, dst = 0;
  const S* src = nullptr;
  if (lane < kDirs) {
    const int d = lane, dx = hop_x(d), dy = hop_y(d);
    int sy = y - dy;
    if (s.periodic_y) sy = sy < 0 ? sy + s.ny : (sy >= s.ny ? sy - s.ny : sy);
    if ((unsigned)sy < (unsigned)s.ny) {
      const int a = x0 - dx;
      int lo = a, hi = a + nv;
      const bool wraps = s.periodic_x && (lo < 0 || hi > s.nx);
      if (!s.periodic_x) { lo = max(lo, 0); hi = min(hi, s.nx); }
      if (!wraps && lo < hi) {
        const int lor = lo & ~(G - 1), hir = (hi + G - 1) & ~(G - 1);
        ok = true;
        bytes = (uint32_t)(hir - lor) * VB;
        src = fin + vec_index(s, d, (long long)sy * s.ldx + lor);
        dst = smem_addr(buf + ((long long)d * SL + (lor - (a & ~(G - 1)))) * 4);
      }
    }
  }
  const unsigned m = __ballot_sync(0xffffffffu, ok);
  uint32_t total = bytes;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) total += __shfl_xor_sync(0xffffffffu, total, o);
  if (lane == 0) {
    *mask = m;
    *tile = make_int4(sample, x0, y, 0);
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;\n"
                 :: "r"(bar), "r"(total) : "memory");
  }
  __syncwarp();
  if (ok)
    asm volatile(
        "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];\n"
        :: "r"(dst), "l"(src), "r"(bytes), "r"(bar) : "memory");
}

// The staged slot rows of a tile.
template <typename S, int BX>
struct StagedSrc {
  uint32_t buf;     // shared-window address of the tile's slot rows
  unsigned mask;    // bit d: direction d staged
  int x0;           // first column of the tile
};

// pull() with staged segments: a source inside the sample whose direction is
// staged is read from shared memory; everything else as in pull().
template <typename S, bool INTERIOR, int BX, class C>
__device__ __forceinline__ void pull_staged(const S* __restrict__ fin, const DevSample& s, int x,
                                            int y, const typename Codec<S>::R* __restrict__ ghost,
                                            const C& qc, const StagedSrc<S, BX>& st,
                                            typename Codec<S>::R (&f)[kQ]) {
  constexpr int G = Stage<S>::kG, SL = Stage<S>::template slots<BX>();
  constexpr int VB = Stage<S>::kVecBytes;
  const long long site = (long long)y * s.ldx + x;
  const uint64_t pol = pull_policy(false);
  const int i = x - st.x0;
  if (INTERIOR && __builtin_expect(st.mask == (1u << kDirs) - 1u, 1)) {
#pragma unroll
    for (int d = 0; d < kDirs; ++d)
      Codec<S>::load4s(st.buf + (uint32_t)((d * SL + i + ((st.x0 - hop_x(d)) & (G - 1))) * VB),
                        &f[4 * d]);
    return;
  }
#pragma unroll
  for (int d = 0; d < kDirs; ++d) {
    const int dx = hop_x(d), dy = hop_y(d);
    const bool staged = (st.mask >> d) & 1u;
    const uint32_t sp = st.buf + (uint32_t)((d * SL + i + ((st.x0 - dx) & (G - 1))) * VB);
    if (INTERIOR) {
      if (staged) Codec<S>::load4s(sp, &f[4 * d]);
      else Codec<S>::load4(fin + vec_index(s, d, site - ((long long)dy * s.ldx + dx)), pol,
                           &f[4 * d]);
    } else {
      int sx = x - dx, sy = y - dy;
      if (s.periodic_x) sx = sx < 0 ? sx + s.nx : (sx >= s.nx ? sx - s.nx : sx);
      if (s.periodic_y) sy = sy < 0 ? sy + s.ny : (sy >= s.ny ? sy - s.ny : sy);
      const bool inside = (unsigned)sx < (unsigned)s.nx && (unsigned)sy < (unsigned)s.ny;
      if (inside) {
        if (staged) Codec<S>::load4s(sp, &f[4 * d]);
        else Codec<S>::load4(fin + vec_index(s, d, (long long)sy * s.ldx + sx), pol, &f[4 * d]);
      } else {
        const int owner = contact_of(s, sx, sy);
        if (owner >= 0) {
#pragma unroll
          for (int j = 0; j < kShells; ++j) f[4 * d + j] = ghost[owner * kQ + 4 * d + j];
        } else {
          Codec<S>::load4(fin + vec_index(s, d ^ 1, site), pol, &f[4 * d]);
        }
      }
    }
  }
}

template <typename R>
__device__ __forceinline__ void block_reduce_add2(double a, double b, double* acc) {
  __shared__ double sa[32], sb[32];
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    a += __shfl_xor_sync(0xffffffffu, a, o);
    b += __shfl_xor_sync(0xffffffffu, b, o);
  }
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  if (lane == 0) { sa[warp] = a; sb[warp] = b; }
  __syncthreads();
  if (warp == 0) {
    const int nw = blockDim.x >> 5;
    a = lane < nw ? sa[lane] : 0.0;
    b = lane < nw ? sb[lane] : 0.0;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      a += __shfl_xor_sync(0xffffffffu, a, o);
      b += __shfl_xor_sync(0xffffffffu, b, o);
    }
    if (lane == 0) {
      atomicAdd(acc, a);
      atomicAdd(acc + 1, b);
    }
  }
}

// Warp sums of (a, b) added to acc[0], acc[1] by lane 0 (no block barrier).
__device__ __forceinline__ void warp_reduce_add2(double a, double b, double* acc) {
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

// New relative deviations of the four shells of a direction from its cubic:
// out_j = (1 - omega) g_j + R0 + R1 p0_j + R2 p0_j^2 + R3 p0_j^3
// (delta = w g: the weight w_j drops out of the update).  omc = 1 - omega.
template <typename R, class C>
__device__ __forceinline__ void relax_shells(const R (&Rm)[4], R omc, const C& qc, R* f) {
#pragma unroll
  for (int j = 0; j < kShells; ++j) {
    const R p = qc.p0[j];
    const R val = fma(fma(fma(Rm[3], p, Rm[2]), p, Rm[1]), p, Rm[0]);
    f[j] = fma(omc, f[j], val);
  }
}

// Gradient of the previous step's n - 1 at (x, y) over one hop (5 sites, the
// length unit of c = 1): (a(x + 5) - a(x - 5)) / 2 where both exist, the
// forward or backward difference over 5 sites next to a walled edge, wrapped
// on periodic axes (Sec. 3, local capacitance approximation; a difference over
// neighbouring sites would drive density structure finer than a hop).
// The previous step may still write the plane when this kernel starts:
// coherent loads behind the wait, as the pulls (Codec::load4).
__device__ __forceinline__ float ld_plane(const float* p) {
  float v;
  asm volatile("ld.global.f32 %0, [%1];\n" : "=f"(v) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ double ld_plane(const double* p) {
  double v;
  asm volatile("ld.global.f64 %0, [%1];\n" : "=d"(v) : "l"(p) : "memory");
  return v;
}
template <typename R>
__device__ __forceinline__ void lca_gradient(const DevSample& s, const R* p, int x, int y, R& gx,
                                             R& gy) {
  constexpr int h = kRadius;
  int xm = x - h, xp = x + h, ym = y - h, yp = y + h;
  R hx = R(0.5), hy = R(0.5);
  if (s.periodic_x) { xm = xm < 0 ? xm + s.nx : xm; xp = xp >= s.nx ? xp - s.nx : xp; }
  else if (xm < 0) { xm = x; hx = R(1); }
  else if (xp >= s.nx) { xp = x; hx = R(1); }
  if (s.periodic_y) { ym = ym < 0 ? ym + s.ny : ym; yp = yp >= s.ny ? yp - s.ny : yp; }
  else if (ym < 0) { ym = y; hy = R(1); }
  else if (yp >= s.ny) { yp = y; hy = R(1); }
  const long long row = (long long)y * s.ldx;
  gx = (ld_plane(p + row + xp) - ld_plane(p + row + xm)) * hx;
  gy = (ld_plane(p + (long long)yp * s.ldx + x) - ld_plane(p + (long long)ym * s.ldx + x)) * hy;
}

// Whether the 32 sites of a warp (consecutive x of row y) pull only from
// inside the rectangle.
__device__ __forceinline__ bool warp_interior(const DevSample& s, int x, int y) {
  const int wx0 = x & ~31;
  return wx0 >= kRadius && wx0 + 32 + kRadius <= s.nx && y >= kRadius && y + kRadius < s.ny;
}

// Gathers the 48 deviations streamed into site (x < nx, y) from HBM.
template <typename S, int D0 = 0, int ND = kDirs, class C, class O>
__device__ __forceinline__ void gather(const S* __restrict__ fin, const Tile<S>& tl, const O& of,
                                       const DevSample& s, int x, int y,
                                       const typename Codec<S>::R* __restrict__ ghost, const C& qc,
                                       typename Codec<S>::R* f) {
  if (warp_interior(s, x, y)) pull<S, true, D0, ND>(fin, tl, of, s, x, y, ghost, qc, f);
  else pull<S, false, D0, ND>(fin, tl, of, s, x, y, ghost, qc, f);
}

// pair_cubics() on register pairs, lanes (d, d + 1): the two lanes differ only
// in the sign of v, which the constant pairs (vx, -vx), (vy, -vy) carry, so
// each instruction serves both directions.  Returns R0..R3 and 1 - omega.
template <bool FORCE, class C>
__device__ __forceinline__ void pair_cubics_paired(const int d, const EqCoeffs<float>& c,
                                                   const ForceCoeffs<float>& k,
                                                   const RelaxSite<float>& s, const C& qc,
                                                   float2 (&R)[4], float2& omc) {
  const int q = d / 2;
  const bool hx = hop_x(d) != 0, hy = hop_y(d) != 0;
  const float2 vx = qc.vxo[q], vy = qc.vyo[q];
  float2 z = S2(c.W);
  // o = omega rounded, omc = 1 - o without a rounding of its own near 1: their
  // sum is 1, so a population at its equilibrium stays (formed the other way
  // round it grows by up to 2^-25 a step)
  float2 o = S2(s.gt);
  if (hx) {
    z = fma2(S2(c.X), vx, z);
    o = fma2(S2(-s.gux), vx, o);
  }
  if (hy) {
    z = fma2(S2(c.Y), vy, z);
    o = fma2(S2(-s.guy), vy, o);
  }
  omc = fma2(o, S2(-1.f), S2(1.f));
  const float2 e1 = fma2(S2(c.kap), z, S2(c.lam));
  const float2 e2 = mul2(z, fma2(S2(c.mu), z, S2(c.D)));
  const float2 z2 = mul2(z, z);
  const float2 e3 = mul2(mul2(S2(c.nu), z), z2);
  if (FORCE) {
    float2 phi;
    if (hx && hy) phi = fma2(S2(s.Fx), vx, mul2(S2(s.Fy), vy));
    else if (hx) phi = mul2(S2(s.Fx), vx);
    else phi = mul2(S2(s.Fy), vy);
    R[0] = fma2(o, S2(c.e0), fma2(phi, S2(k.a0), S2(k.b0)));
    R[1] = fma2(o, e1, fma2(z, fma2(phi, S2(k.a1), S2(k.b1)), fma2(phi, S2(k.a2), S2(k.b2))));
    o = add2(o, phi);
    R[2] = fma2(o, e2, mul2(z2, fma2(phi, S2(k.a3), S2(k.b3))));
  } else {
    R[0] = mul2(o, S2(c.e0));
    R[1] = mul2(o, e1);
    R[2] = mul2(o, e2);
  }
  R[3] = mul2(o, e3);
}

// New relative deviations of the four shells of one direction on shell pairs:
// out_j = (1 - omega) g_j + R0 + R1 p0_j + R2 p0_j^2 + R3 p0_j^3.  With BAL the
// direction's moment change (sum_j w p0_j (out_j - g_j), sum_j w p0_j^2
// (out_j - g_j)) is returned in bal (the conservation projection's input).
template <bool BAL, class C>
__device__ __forceinline__ void relax_shells_paired(float R0, float R1, float R2, float R3,
                                                    float omc, int kind, const C& qc, float* f,
                                                    float2& bal) {
  const float2 v01 = fma2(fma2(fma2(S2(R3), qc.p01, S2(R2)), qc.p01, S2(R1)), qc.p01, S2(R0));
  const float2 v23 = fma2(fma2(fma2(S2(R3), qc.p23, S2(R2)), qc.p23, S2(R1)), qc.p23, S2(R0));
  const float2 i01 = make_float2(f[0], f[1]), i23 = make_float2(f[2], f[3]);
  const float2 o01 = fma2(S2(omc), i01, v01);
  const float2 o23 = fma2(S2(omc), i23, v23);
  if (BAL) {
    const float2 d01 = fma2(i01, S2(-1.f), o01), d23 = fma2(i23, S2(-1.f), o23);
    bal = mul2(S2(d01.x), qc.wab[kind][0]);
    bal = fma2(S2(d01.y), qc.wab[kind][1], bal);
    bal = fma2(S2(d23.x), qc.wab[kind][2], bal);
    bal = fma2(S2(d23.y), qc.wab[kind][3], bal);
  }
  f[0] = o01.x; f[1] = o01.y; f[2] = o23.x; f[3] = o23.y;
}

// collide_store() with FP32 arithmetic (FP32 and 16-bit storage) on register
// pairs: the same quantities in the same order of operations per population,
// with each instruction serving two directions or two shells.
template <typename S, int FORCE, int RES, int BT, class C, class O>
__device__ __forceinline__ void collide_store_paired(float (&f)[kQ], const Tile<S>& tl,
                                                     const O& of, const DevSample& s, int x, int y,
                                                     const StepAux<float>& aux, const C& qc,
                                                     double& r_du2, double& r_u2, uint32_t park,
                                                     const float* dn_prev, float* dn_next) {
  constexpr bool kProject = sizeof(S) == sizeof(float);
  const bool lca = FORCE == kForceLca && s.dn[0] != nullptr;
  float egx = 0.f, egy = 0.f;
  if (lca) lca_gradient(s, dn_prev, x, y, egx, egy);
  const Moments<float> m = moments(f, qc);
  constexpr uint32_t park_stride = BT * 16u;
  if constexpr (Park<S>::kOn) {
#pragma unroll
    for (int d = 0; d < kDirs; ++d) park_store(park + d * park_stride, &f[4 * d]);
  }
  Macro<float> M;
  const unsigned bad = landau(m, M);
  if (bad) atomicOr(aux.err, bad);

  const float scl = sizeof(S) == 2 ? qc.enc_s : 1.f;
  // n / T = 1 + (n - T) / T: the rounding of 1 / T reaches the small term only.
  // With o and X, Y each rounded once and the force kept out of o, the error of
  // u against 64 bits (50 to 100 steps, amplitude 1e-4) is 1.04e-7 at 1024 x 512
  // and 1.29e-7 with the electric force at 600 x 300; 1.16e-7 and 1.50e-7
  // otherwise, at the same speed.
  const float iTs = M.invT * scl, dnT = M.dn - M.dT;
  const EqCoeffs<float> c = eq_coeffs(M, fmaf(dnT, iTs, scl), dnT * iTs);
  const float Fx = lca ? fmaf(-s.inv_cg_f, egx, s.Fx_f) : s.Fx_f;
  const float Fy = lca ? fmaf(-s.inv_cg_f, egy, s.Fy_f) : s.Fy_f;
  RelaxSite<float> rs;
  rs.gt = M.gamma * s.inv_tau_f;
  rs.gux = rs.gt * M.ux; rs.guy = rs.gt * M.uy;
  rs.Fx = Fx; rs.Fy = Fy;
  ForceCoeffs<float> k{};
  if (FORCE != 0) k = force_coeffs(c, Fx, Fy, scl);
  if (lca) dn_next[(long long)y * s.ldx + x] = M.dn;
  // conservation projection: sums of the moment changes (N^0, T^00) and
  // (T^0x, T^0y), started with minus the forcing's target
  float2 accNE = S2(0.f), accXY = S2(0.f);
  if (kProject && FORCE != 0) {
    // forcing changes T^0a by (F.N_E, F N_E^0), N_E = n gamma (1, u)
    const float nG = fmaf(M.dn, M.gamma, M.gamma);
    accNE = make_float2(0.f, -(nG * fmaf(Fx, M.ux, Fy * M.uy)));
    accXY = make_float2(-(nG * Fx), -(nG * Fy));
  }
  // (5,0)-type pairs first: with FP32 storage they take the correction and
  // are kept for the end; the (3,4)-type pairs are stored as soon as done.
#pragma unroll
  for (int pi = 0; pi < kDirs / 2; ++pi) {
    const int d = (2 * pi + 8) % kDirs;
    const int kind = dir_kind(d);
    float2 R[4], omc;
    pair_cubics_paired<FORCE != 0>(d, c, k, rs, qc, R, omc);
    if constexpr (Park<S>::kOn) {
      park_load(park + d * park_stride, &f[4 * d]);
      park_load(park + (d + 1) * park_stride, &f[4 * d + 4]);
    }
    float2 bp, bn;
    relax_shells_paired<kProject>(R[0].x, R[1].x, R[2].x, R[3].x, omc.x, kind, qc, &f[4 * d], bp);
    relax_shells_paired<kProject>(R[0].y, R[1].y, R[2].y, R[3].y, omc.y, kind, qc, &f[4 * d + 4],
                                  bn);
    if (kProject) {
      accNE = add2(accNE, add2(bp, bn));
      accXY = fma2(S2(bp.y - bn.y), qc.vxy[d / 2], accXY);
    }
    if (!kProject || kind == 0) {
      Codec<S>::store4(byte_ptr(tl.out, of.plane(d)), &f[4 * d]);
      Codec<S>::store4(byte_ptr(tl.out, of.plane(d + 1)), &f[4 * d + 4]);
    }
  }
  if (kProject) {
    const float rN = accNE.x, rE = accNE.y;
    const float l0 = fmaf(qc.P00, rN, qc.P01 * rE);
    const float l1 = fmaf(qc.P10, rN, qc.P11 * rE);
    const float lx = qc.px * accXY.x, ly = qc.px * accXY.y;
#pragma unroll
    for (int d = 8; d < kDirs; ++d) {
      const float cd = l1 + (hop_x(d) > 0 ? lx : hop_x(d) < 0 ? -lx : hop_y(d) > 0 ? ly : -ly);
      // delta += w (l0 + p0 cd)
      const float2 t01 = fma2(S2(cd), qc.p01, S2(l0));
      const float2 t23 = fma2(S2(cd), qc.p23, S2(l0));
      const float2 o01 = add2(make_float2(f[4 * d], f[4 * d + 1]), t01);
      const float2 o23 = add2(make_float2(f[4 * d + 2], f[4 * d + 3]), t23);
      f[4 * d] = o01.x; f[4 * d + 1] = o01.y; f[4 * d + 2] = o23.x; f[4 * d + 3] = o23.y;
      Codec<S>::store4(byte_ptr(tl.out, of.plane(d)), &f[4 * d]);
    }
  }
  if (RES == 1) {
    const long long k = s.site0 + (long long)y * s.nx + x;
    aux.uprev[2 * k] = M.ux;
    aux.uprev[2 * k + 1] = M.uy;
  } else if (RES == 2) {
    const long long k = s.site0 + (long long)y * s.nx + x;
    const double dx = double(M.ux) - double(aux.uprev[2 * k]);
    const double dy = double(M.uy) - double(aux.uprev[2 * k + 1]);
    r_du2 = fma(dx, dx, fma(dy, dy, r_du2));
    r_u2 = fma(double(M.ux), double(M.ux), fma(double(M.uy), double(M.uy), r_u2));
  }
}

// Relaxation, force and store of directions D0 .. D0 + ND - 1 (f: their
// populations) for the site's fields M.
template <typename S, int FORCE, int D0, int ND, class C, class O>
__device__ __forceinline__ void relax_store_f64(double* f, const Tile<S>& tl, const O& of,
                                                const DevSample& s, const Macro<double>& M,
                                                bool lca, double egx, double egy, const C& qc) {
  using R = double;
  const EqCoeffs<R> c = eq_coeffs(M, fma(M.dn, M.invT, M.invT), (M.dn - M.dT) * M.invT);
  RelaxSite<R> rs;
  rs.gt = M.gamma * s.inv_tau;
  rs.omgt = R(1) - rs.gt;
  rs.gux = rs.gt * M.ux; rs.guy = rs.gt * M.uy;
  rs.Fx = lca ? fma(-s.inv_cg, egx, s.Fx) : s.Fx;
  rs.Fy = lca ? fma(-s.inv_cg, egy, s.Fy) : s.Fy;
  ForceCoeffs<R> k{};
  if (FORCE != 0) k = force_coeffs(c, rs.Fx, rs.Fy, R(1));
#pragma unroll
  for (int d = D0; d < D0 + ND; d += 2) {
    R Rp[4], Rn[4], omcp, omcn;
    pair_cubics<R, FORCE != 0>(d, c, k, rs, Rp, Rn, omcp, omcn);
    R* const g = f + 4 * (d - D0);
    relax_shells(Rp, omcp, qc, g);
    relax_shells(Rn, omcn, qc, g + 4);
    Codec<S>::store4(byte_ptr(tl.out, of.plane(d)), g);
    Codec<S>::store4(byte_ptr(tl.out, of.plane(d + 1)), g + 4);
  }
}

// The residual's part of a site: RES 1 keeps u, RES 2 adds |u - u_prev|^2 and |u|^2.
template <int RES>
__device__ __forceinline__ void residual_terms(const DevSample& s, int x, int y,
                                               const Macro<double>& M, const StepAux<double>& aux,
                                               double& r_du2, double& r_u2) {
  if (RES == 0) return;
  const long long j = s.site0 + (long long)y * s.nx + x;
  if (RES == 1) {
    aux.uprev[2 * j] = M.ux;
    aux.uprev[2 * j + 1] = M.uy;
  } else {
    const double dx = M.ux - aux.uprev[2 * j], dy = M.uy - aux.uprev[2 * j + 1];
    r_du2 = fma(dx, dx, fma(dy, dy, r_du2));
    r_u2 = fma(M.ux, M.ux, fma(M.uy, M.uy, r_u2));
  }
}

// Collision of the gathered deviations f of site (x < nx, y) and store of the
// 48 new deviations into fout.  RES: 0 nothing extra; 1 store u for the
// residual; 2 add |u - u_prev|^2 and |u|^2 to r_du2, r_u2 (the caller
// reduces them).  dn_prev / dn_next: the electric force's density planes of
// the previous and of this step (used when s.inv_cg != 0).
template <typename S, int FORCE, int RES, int BT, class C, class O>
__device__ __forceinline__ void collide_store(typename Codec<S>::R (&f)[kQ], const Tile<S>& tl,
                                              const O& of, const DevSample& s, int x, int y,
                                              const StepAux<typename Codec<S>::R>& aux,
                                              const C& qc, double& r_du2, double& r_u2,
                                              uint32_t park,
                                              const typename Codec<S>::R* dn_prev,
                                              typename Codec<S>::R* dn_next) {
  using R = typename Codec<S>::R;
  if constexpr (std::is_same<R, float>::value) {
    collide_store_paired<S, FORCE, RES, BT>(f, tl, of, s, x, y, aux, qc, r_du2, r_u2, park, dn_prev,
                                        dn_next);
  } else {
    // FP64 storage: the populations stay in registers (the FP64 pipe, not
    // latency, bounds this path), no conservation projection
    const bool lca = FORCE == kForceLca && s.dn[0] != nullptr;
    R egx = R(0), egy = R(0);
    if (lca) lca_gradient(s, dn_prev, x, y, egx, egy);
    Macro<R> M;
    const unsigned bad = landau(moments(f, qc), M);
    if (bad) atomicOr(aux.err, bad);
    if (lca) dn_next[(long long)y * s.ldx + x] = M.dn;
    relax_store_f64<S, FORCE, 0, kDirs>(f, tl, of, s, M, lca, egx, egy, qc);
    residual_terms<RES>(s, x, y, M, aux, r_du2, r_u2);
  }
}

// Fused stream + collide of site (x, y) (nothing if x >= nx).
template <typename S, int FORCE, int RES, int BT, class C, class O>
__device__ __forceinline__ void site_step(const S* __restrict__ fin, const Tile<S>& tl,
                                          const O& of, const DevSample& s, int x, int y,
                                          const typename Codec<S>::R* __restrict__ ghost,
                                          const StepAux<typename Codec<S>::R>& aux, const C& qc,
                                          double& r_du2, double& r_u2, uint32_t park, int cur) {
  using R = typename Codec<S>::R;
  if (x < s.nx) {
    R f[kQ];
    gather<S>(fin, tl, of, s, x, y, ghost, qc, f);
    // select, not s.dn[cur]: a runtime index would move the descriptor to local memory
    void* const prev = cur ? s.dn[1] : s.dn[0];
    void* const next = cur ? s.dn[0] : s.dn[1];
    collide_store<S, FORCE, RES, BT>(f, tl, of, s, x, y, aux, qc, r_du2, r_u2, park,
                                     static_cast<const R*>(prev), static_cast<R*>(next));
  }
}

// Row segments of 32 sites ("warp tiles") of one sample, numbered row by row.
struct WarpTiles {
  unsigned per_row, magic, count;   // magic = floor(2^32 / per_row)
  int evict_first;                  // L2 policy of the pulls (pull_policy; FP32 storage)
  int reverse;                      // walk the tiles from the last to the first
  int early;                        // let the next step's blocks be placed while this one runs
  __device__ __forceinline__ void row_of(unsigned t, unsigned& y, unsigned& r) const {
    // the product's high word is the quotient t / per_row or one below it
    y = __umulhi(t, magic);
    r = t - y * per_row;
    if (r >= per_row) { r -= per_row; ++y; }
  }
};

// Chained launches: a step kernel lets its successor start as soon as all of
// its own blocks run, and waits for its predecessor's results only before
// its first access to them.  A small FP64 step does not (WarpTiles::early): the
// next step's blocks would gather on the SMs that it leaves idle, several
// to an SM, and share the FP64 units there.
__device__ __forceinline__ void chain_release() {
  asm volatile("griddepcontrol.launch_dependents;\n" ::: "memory");
}
__device__ __forceinline__ void chain_wait() {
  asm volatile("griddepcontrol.wait;\n" ::: "memory");
}

// One sample: each warp of a block of BT threads updates one warp tile.
template <typename S, int FORCE, int RES, int BT, class C>
__device__ __forceinline__ void step_body(const S* __restrict__ fin, S* __restrict__ fout,
                                          const DevSample& s, const WarpTiles& wt,
                                          const StepOffsets& of,
                                          const typename Codec<S>::R* __restrict__ ghost,
                                          const StepAux<typename Codec<S>::R>& aux, const C& qc,
                                          unsigned char* park) {
  if (wt.early) chain_release();
  double r_du2 = 0.0, r_u2 = 0.0;
  const unsigned block = wt.reverse ? gridDim.x - 1 - blockIdx.x : blockIdx.x;
  unsigned y, r;
  const unsigned t = block * (BT / 32) + threadIdx.x / 32;
  wt.row_of(t, y, r);
  const int x = (int)(r * 32 + threadIdx.x % 32);
  const long long site = (long long)y * s.ldx + x;
  Tile<S> tl;
  tl.in = fin + 4 * site;
  tl.out = fout + 4 * site;
  tl.policy = pull_policy(wt.evict_first);
  chain_wait();
  site_step<S, FORCE, RES, BT>(fin, tl, of, s, t < wt.count ? x : s.nx, (int)y, ghost, aux, qc,
                               r_du2, r_u2, smem_addr(park) + threadIdx.x * 16u, s.cur);
  if (RES == 2) block_reduce_add2<typename Codec<S>::R>(r_du2, r_u2, aux.acc);
}

// FP64, one sample, few sites: three warps share the 32 sites of a warp tile,
// each with the populations of one group of four directions.  A warp
// instruction of the FP64 pipe takes 66 cycles of its SM sub-partition however
// many of its lanes are active, so a sample of fewer warp tiles than
// sub-partitions (608) is bound by the chain of one warp: about 690 FP64
// instructions.  Split, a warp runs about 320 (its third of the moments and
// the relaxation; the Landau solve and the coefficients are repeated).
// 64 x 64 sites: 22.9 -> 12.1 us per step; eight such samples at once, each on
// its own stream, 58 us per step of all (one thread per site, 1,026
// operations: 66).
template <typename S, int FORCE, int RES, int G, class C>
__device__ __forceinline__ void split_group(const S* __restrict__ fin, const Tile<S>& tl,
                                            const StepOffsets& of, const DevSample& s, int x,
                                            int y, const double* __restrict__ ghost,
                                            const StepAux<double>& aux, const C& qc,
                                            GroupSums<double>* part) {
  const int lane = threadIdx.x % 32;
  const bool in = x < s.nx;
  const bool lca = FORCE == kForceLca && s.dn[0] != nullptr;
  double f[16], egx = 0.0, egy = 0.0;
  if (in) {
    gather<S, 4 * G, 4>(fin, tl, of, s, x, y, ghost, qc, f);
    if (lca) lca_gradient(s, static_cast<const double*>(s.cur ? s.dn[1] : s.dn[0]), x, y, egx, egy);
    part[G * 32 + lane] = group_sums<G>(f, qc);
  }
  // a barrier that the three warps meet at from three places in the code
  asm volatile("bar.sync 1, 96;\n" ::: "memory");
  double r_du2 = 0.0, r_u2 = 0.0;
  if (in) {
    Macro<double> M;
    const unsigned bad = landau(add_groups(part[lane], part[32 + lane], part[64 + lane]), M);
    if (G == 0) {
      if (bad) atomicOr(aux.err, bad);
      if (lca) static_cast<double*>(s.cur ? s.dn[0] : s.dn[1])[(long long)y * s.ldx + x] = M.dn;
      residual_terms<RES>(s, x, y, M, aux, r_du2, r_u2);
    }
    relax_store_f64<S, FORCE, 4 * G, 4>(f, tl, of, s, M, lca, egx, egy, qc);
  }
  if (RES == 2 && G == 0) warp_reduce_add2(r_du2, r_u2, aux.acc);
}

template <typename S, int FORCE, int RES, class C>
__device__ __forceinline__ void split_body(const S* __restrict__ fin, S* __restrict__ fout,
                                           const DevSample& s, const WarpTiles& wt,
                                           const StepOffsets& of, const double* __restrict__ ghost,
                                           const StepAux<double>& aux, const C& qc,
                                           GroupSums<double>* part) {
  unsigned y, r;
  wt.row_of(wt.reverse ? gridDim.x - 1 - blockIdx.x : blockIdx.x, y, r);
  const int x = (int)(r * 32 + threadIdx.x % 32), g = threadIdx.x / 32;
  const long long site = (long long)y * s.ldx + x;
  Tile<S> tl;
  tl.in = fin + 4 * site;
  tl.out = fout + 4 * site;
  tl.policy = pull_policy(false);
  chain_wait();
  if (g == 0) split_group<S, FORCE, RES, 0>(fin, tl, of, s, x, (int)y, ghost, aux, qc, part);
  else if (g == 1) split_group<S, FORCE, RES, 1>(fin, tl, of, s, x, (int)y, ghost, aux, qc, part);
  else split_group<S, FORCE, RES, 2>(fin, tl, of, s, x, (int)y, ghost, aux, qc, part);
}

// Many samples of uneven size in one launch.  The work list is every row
// segment of BX sites of every sample ("tile"), numbered sample by sample;
// tile_start[k] is the first tile of sample k (tile_start[nsamples] = total).
// Blocks walk the list with a grid stride (persistent when the grid is a
// multiple of the SM count).  Sample k's buffers are base + samples[k].off[cur]
// (input) and base + samples[k].off[1 - cur] (output).
struct BatchArgs {
  const DevSample* samples;
  const long long* tile_start;
  int nsamples;
  int cur;
  long long ntiles;
  long long wait_limit;   // clock cycles a wait for a staged tile may take before it gives up
};

template <typename S, int FORCE, int RES, int BX, class C>
__device__ __forceinline__ void batch_body(S* __restrict__ base, const BatchArgs& b,
                                           const typename Codec<S>::R* __restrict__ ghost,
                                           const StepAux<typename Codec<S>::R>& aux, const C& qc,
                                           unsigned char* park) {
  const uint32_t my_park = smem_addr(park) + threadIdx.x * 16u;
  const uint64_t policy = pull_policy(false);
  chain_release();
  chain_wait();
#pragma unroll 1
  for (long long t = blockIdx.x; t < b.ntiles; t += gridDim.x) {
    int lo = 0, hi = b.nsamples;                 // tile_start[lo] <= t < tile_start[hi]
    while (hi - lo > 1) {
      const int mid = (lo + hi) >> 1;
      if (__ldg(b.tile_start + mid) <= t) lo = mid; else hi = mid;
    }
    const DevSample s = b.samples[lo];
    const long long lt = t - __ldg(b.tile_start + lo);
    const int tpr = (s.nx + BX - 1) / BX;
    const int y = (int)(lt / tpr);
    const int x = (int)(lt - (long long)y * tpr) * BX + threadIdx.x;
    const S* fin = base + (b.cur ? s.off[1] : s.off[0]);
    Tile<S> tl;
    const long long site = (long long)y * s.ldx + x;
    tl.in = fin + 4 * site;
    tl.out = base + (b.cur ? s.off[0] : s.off[1]) + 4 * site;
    tl.policy = policy;
    const SampleOffsets<S> of{s.plane, s.ldx};
    double r_du2 = 0.0, r_u2 = 0.0;
    site_step<S, FORCE, RES, BX>(fin, tl, of, s, x, y,
                             ghost + (long long)lo * kMaxContacts * kQ, aux, qc, r_du2, r_u2,
                             my_park, b.cur);
    // per-sample residual accumulators: acc[2 k], acc[2 k + 1]
    if (RES == 2) {
      block_reduce_add2<typename Codec<S>::R>(r_du2, r_u2, aux.acc + 2 * lo);
      __syncthreads();   // the reduction's shared scratch is reused by the next tile
    }
  }
}

// The batched step with staged pulls (persistent: gridDim.x blocks walk the
// tile list with a grid stride; the block's k-th tile is blockIdx.x + k G,
// G = gridDim.x).  Two slot-row buffers alternate: buffer b holds tiles
// k = b, b + 2, ... (use j = k / 2), and mbarrier full[b] completes phase j
// when tile 2 j + b has landed (one arrive with the byte count by the issuing
// warp, plus the copies' bytes).  Warp 0 fills both buffers up front; after
// that the last warp to finish gathering tile k (a shared counter per buffer)
// issues tile k + 2 into the buffer it just freed, so two tiles are always in
// flight or landed and no warp waits for another one.  Every wait is bounded
// (b.wait_limit cycles, about 1 s by default): a warp that gives up sets
// kErrTimeout and a shared abort flag, waits once more for the copies of both
// buffers (bounded by the full ~1 s whatever b.wait_limit is, so that no bulk
// copy into the block's shared memory is left in flight), and leaves the loop;
// the other warps leave at their next tile.
template <typename S, int FORCE, int RES, int BX, class C>
__device__ __forceinline__ void staged_batch_body(S* __restrict__ base, const BatchArgs& b,
                                                  const typename Codec<S>::R* __restrict__ ghost,
                                                  const StepAux<typename Codec<S>::R>& aux,
                                                  const C& qc, unsigned char* smem) {
  using R = typename Codec<S>::R;
  constexpr int BUF = Stage<S>::template buf_elems<BX>();
  constexpr int kWarps = BX / 32;
  S* stage = reinterpret_cast<S*>(smem);
  unsigned char* ctl = smem + 2 * (size_t)BUF * sizeof(S);
  uint64_t* full = reinterpret_cast<uint64_t*>(ctl);          // [2]
  unsigned* released = reinterpret_cast<unsigned*>(ctl + 16);  // [2] warps done gathering
  int4* tiles = reinterpret_cast<int4*>(ctl + 32);             // [2]: sample, x0, y
  unsigned* masks = reinterpret_cast<unsigned*>(ctl + 64);     // [2]
  volatile int* abort_flag = reinterpret_cast<volatile int*>(ctl + 72);
  const int tid = threadIdx.x, lane = tid & 31;
  const uint32_t my_park = smem_addr(ctl + kStageCtlBytes) + tid * 16u;
  const uint32_t full0 = smem_addr(&full[0]), full1 = smem_addr(&full[1]);
  const uint32_t buf0 = smem_addr(stage), buf1 = smem_addr(stage + BUF);
  auto full_bar = [&](int k) { return k ? full1 : full0; };
  const long long G = gridDim.x;
  long long t = blockIdx.x;
  if (t >= b.ntiles) return;
  if (tid == 0) {
    stage_bar_init(full0, 1);
    stage_bar_init(full1, 1);
    asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
    released[0] = released[1] = 0;
    *abort_flag = 0;
  }
  __syncthreads();

  // fills buffer `buf` with tile tt (all lanes of the calling warp)
  auto issue = [&](long long tt, int buf) {
    int lo = 0, hi = b.nsamples;                 // tile_start[lo] <= tt < tile_start[hi]
    while (hi - lo > 1) {
      const int mid = (lo + hi) >> 1;
      if (__ldg(b.tile_start + mid) <= tt) lo = mid; else hi = mid;
    }
    const DevSample& s = b.samples[lo];
    const long long lt = tt - __ldg(b.tile_start + lo);
    const int tpr = (s.nx + BX - 1) / BX;
    const int y = (int)(lt / tpr);
    const int x0 = (int)(lt - (long long)y * tpr) * BX;
    const S* fin = base + (b.cur ? s.off[1] : s.off[0]);
    asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");
    stage_issue<S, BX>(fin, s, x0, y, stage + (size_t)buf * BUF, full_bar(buf), &masks[buf],
                       &tiles[buf], lo);
  };

  if (tid < 32) {
    issue(t, 0);
    if (t + G < b.ntiles) issue(t + G, 1);
  }
#pragma unroll 1
  for (int it = 0;; ++it) {
    const int cb = it & 1;
    bool ok = !*abort_flag && stage_wait(full_bar(cb), (it >> 1) & 1, b.wait_limit);
    ok = __all_sync(0xffffffffu, ok);
    if (!ok) {
      if (lane == 0 && !*abort_flag) {
        *abort_flag = 1;
        atomicOr(aux.err, kErrTimeout);
      }
      // copies that may still be in flight into either buffer
      stage_wait(full_bar(cb), (it >> 1) & 1);
      if (t + G < b.ntiles) stage_wait(full_bar(cb ^ 1), ((it + 1) >> 1) & 1);
      break;
    }
    const int4 tl = tiles[cb];
    const StagedSrc<S, BX> src{cb ? buf1 : buf0, masks[cb], tl.y};
    const DevSample s = b.samples[tl.x];
    const int x = tl.y + tid;
    R f[kQ];
    if (x < s.nx) {
      const S* fin = base + (b.cur ? s.off[1] : s.off[0]);
      const R* gh = ghost + (long long)tl.x * kMaxContacts * kQ;
      if (warp_interior(s, x, tl.z)) pull_staged<S, true>(fin, s, x, tl.z, gh, qc, src, f);
      else pull_staged<S, false>(fin, s, x, tl.z, gh, qc, src, f);
    }
    __syncwarp();
    // the last warp done with this buffer refills it with tile k + 2
    if (t + 2 * G < b.ntiles) {
      unsigned last = 0;
      if (lane == 0) {
        // a compiler barrier too: this tile's shared reads stay before it
        unsigned prev;
        asm volatile("atom.shared.add.u32 %0, [%1], 1;\n"
                     : "=r"(prev) : "r"(smem_addr(&released[cb])) : "memory");
        last = prev == kWarps - 1;
      }
      last = __shfl_sync(0xffffffffu, last, 0);
      if (last) {
        if (lane == 0) released[cb] = 0;
        issue(t + 2 * G, cb);
      }
    }
    double r_du2 = 0.0, r_u2 = 0.0;
    Tile<S> dst;
    dst.in = nullptr;
    dst.out = base + (b.cur ? s.off[0] : s.off[1]) + 4 * ((long long)tl.z * s.ldx + x);
    const SampleOffsets<S> of{s.plane, s.ldx};
    if (x < s.nx)
      collide_store<S, FORCE, RES, BX>(f, dst, of, s, x, tl.z, aux, qc,
                                   r_du2, r_u2, my_park,
                                   static_cast<const R*>(b.cur ? s.dn[1] : s.dn[0]),
                                   static_cast<R*>(b.cur ? s.dn[0] : s.dn[1]));
    if (RES == 2) warp_reduce_add2(r_du2, r_u2, aux.acc + 2 * tl.x);
    t += G;
    if (t >= b.ntiles) break;
  }
}

// Macroscopic fields of the streamed populations (no collision).
template <typename S, class C>
__device__ __forceinline__ void moments_body(const S* __restrict__ fin, const DevSample& s,
                                             const typename Codec<S>::R* __restrict__ ghost,
                                             double* n, double* ux, double* uy, double* T,
                                             unsigned* err, const C& qc,
                                             typename Codec<S>::R* dn_out) {
  using R = typename Codec<S>::R;
  const int bx0 = blockIdx.x * kBX;
  const int x = bx0 + threadIdx.x;
  const int y = blockIdx.y;
  if (x >= s.nx) return;
  R f[kQ];
  Tile<S> tl;
  tl.in = fin + 4 * ((long long)y * s.ldx + x);
  tl.out = nullptr;
  tl.policy = pull_policy(false);
  gather<S>(fin, tl, SampleOffsets<S>{s.plane, s.ldx}, s, x, y, ghost, qc, f);
  const Moments<R> m = moments(f, qc);
  Macro<R> M;
  const unsigned bad = landau(m, M) & ~kErrUnphysical;
  if (bad) atomicOr(err, bad);
  const long long k = (long long)y * s.nx + x;
  if (n) n[k] = 1.0 + as_f64(M.dn);
  if (ux) ux[k] = as_f64(M.ux);
  if (uy) uy[k] = as_f64(M.uy);
  if (T) T[k] = 1.0 + as_f64(M.dT);
  if (dn_out) dn_out[(long long)y * s.ldx + x] = M.dn;
}

// Macroscopic state of site k of dense FP64 fields (n, u, T), formed in FP64
// and rounded once: FP32 would lose 1 - u^2 for |u| near 1 (gamma off by 3 % at
// 1 - u^2 = 1e-6, infinite at 1e-8).  17 FP64 operations and 6 conversions on
// the FP64 pipe, which bounds k_init in FP32 arithmetic: FP16 storage
// 4096 x 2048 361 us (268 MB in and 805 MB out; gamma in FP32 159 us, with
// IEEE divisions and square root 608 us).
template <typename R>
__device__ __forceinline__ Macro<R> field_macro(const double* n, const double* ux,
                                                const double* uy, const double* T, long long k,
                                                bool& ok) {
  Macro<R> M;
  const double vx = ux[k], vy = uy[k], nk = n[k], Tk = T[k];
  M.ux = R(vx);
  M.uy = R(vy);
  M.dn = R(nk - 1.0);
  M.dT = R(Tk - 1.0);
  M.deps = R(0);
  const double u2 = fma(vx, vx, vy * vy), w = 1.0 - u2;
  const double g = qrsqrt(w);
  M.gamma = R(g);
  M.gm1 = R(u2 * g * (g * qrcp(1.0 + g)));       // (gamma^2 - 1) / (gamma + 1)
  if constexpr (sizeof(R) == 8) M.invT = qrcp(R(1) + M.dT);
  else M.invT = R(1) / (R(1) + M.dT);
  ok = positive(w) && positive(nk) && positive(Tk) && finite_bits(nk) && finite_bits(Tk);
  // positive() takes no subnormal numbers
  if (!ok) ok = w > 0.0 && nk > 0.0 && Tk > 0.0 && finite_bits(nk) && finite_bits(Tk);
  return M;
}

// Equilibrium coefficients of the macroscopic state M as stored (16-bit
// storage holds s g).
template <typename S, class C>
__device__ __forceinline__ EqCoeffs<typename Codec<S>::R> stored_eq(
    const Macro<typename Codec<S>::R>& M, const C& qc) {
  using R = typename Codec<S>::R;
  const R iTs = sizeof(S) == 2 ? R(M.invT * qc.enc_s) : M.invT;
  return eq_coeffs(M, fma(M.dn, iTs, iTs), (M.dn - M.dT) * iTs);
}

// Relative deviations (f^eq - w) / w of the two directions d (even), d + 1
// from stored_eq(): vp, vn.
template <typename S, class C>
__device__ __forceinline__ void eq_pair(const EqCoeffs<typename Codec<S>::R>& c, int d,
                                        const C& qc, typename Codec<S>::R* vp,
                                        typename Codec<S>::R* vn) {
  using R = typename Codec<S>::R;
  const R vx = R(hop_x(d)) / R(5), vy = R(hop_y(d)) / R(5);
  const R zo = fma(c.X, vx, c.Y * vy);
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    const R z = h ? c.W - zo : c.W + zo;
    const R e1 = fma(c.kap, z, c.lam), e2 = z * fma(c.mu, z, c.D), e3 = (c.nu * z) * (z * z);
    R* v = h ? vn : vp;
#pragma unroll
    for (int j = 0; j < kShells; ++j) {
      const R p = qc.p0[j];
      v[j] = fma(fma(fma(e3, p, e2), p, e1), p, c.e0);
    }
  }
}

// Stored state := f^eq(n, u, T) - w (dense FP64 inputs).
template <typename S, class C>
__device__ __forceinline__ void init_body(S* __restrict__ fout, const DevSample& s,
                                          const double* n, const double* ux, const double* uy,
                                          const double* T, unsigned* err, const C& qc) {
  using R = typename Codec<S>::R;
  const int x = blockIdx.x * kBX + threadIdx.x;
  const int y = blockIdx.y;
  if (x >= s.nx) return;
  const long long k = (long long)y * s.nx + x;
  bool ok;
  const Macro<R> M = field_macro<R>(n, ux, uy, T, k, ok);
  if (!ok) atomicOr(err, kErrUnphysical);
  const EqCoeffs<R> c = stored_eq<S>(M, qc);
  const long long site = (long long)y * s.ldx + x;
  void* const dn0 = s.cur ? s.dn[1] : s.dn[0];
  if (dn0) static_cast<R*>(dn0)[site] = M.dn;     // the electric force's first step
#pragma unroll
  for (int d = 0; d < kDirs; d += 2) {
    R v[8];
    eq_pair<S>(c, d, qc, v, v + 4);
    Codec<S>::store4(fout + vec_index(s, d, site), v);
    Codec<S>::store4(fout + vec_index(s, d + 1, site), v + 4);
  }
}

// Stored state := the Chapman-Enskog seed of the fields (n, u, T): the state
// whose first pull-stream gives f^eq plus its first-order non-equilibrium part
// of a steady flow (steady Eq. discrete-rbe with f - f^eq small and slowly
// varying),
//     f_i(x) = f^eq_i(x) - (f^eq_i(x) - f^eq_i(x - n_i)) / omega_i(x),
// omega_i = gamma (1 - v_i.u) / tau, wherever the source x - n_i lies in the
// sample.  Stored per source site s with d = s + n_i (wrapped on periodic
// axes):  f*_i(s) = f^eq_i(d) - (f^eq_i(d) - f^eq_i(s)) / omega_i(d), and
// f^eq_i(s) where d lies outside (only the bounce-back at s reads it).  The
// relation is affine with unit weight on f^eq, so it holds for the stored
// relative deviations as well.  Each thread evaluates the equilibrium at its
// own site and, for each direction, at the arrival site.  For 16-bit storage
// only; FP64 and FP32 take two passes (ce_from_eq_body).
template <typename S, class C>
__device__ __forceinline__ void init_ce_body(S* __restrict__ fout, const DevSample& s,
                                             const double* n, const double* ux,
                                             const double* uy, const double* T, unsigned* err,
                                             const C& qc) {
  using R = typename Codec<S>::R;
  const int x = blockIdx.x * kBX + threadIdx.x;
  const int y = blockIdx.y;
  if (x >= s.nx) return;
  const long long k = (long long)y * s.nx + x;
  bool ok;
  const Macro<R> M = field_macro<R>(n, ux, uy, T, k, ok);
  if (!ok) atomicOr(err, kErrUnphysical);
  const EqCoeffs<R> c = stored_eq<S>(M, qc);
  const long long site = (long long)y * s.ldx + x;
  void* const dn0 = s.cur ? s.dn[1] : s.dn[0];
  if (dn0) static_cast<R*>(dn0)[site] = M.dn;     // the electric force's first step
#pragma unroll 1
  for (int d = 0; d < kDirs; d += 2) {
    R v[8];
    eq_pair<S>(c, d, qc, v, v + 4);
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const int dd = d + h;
      int tx = x + hop_x(dd), ty = y + hop_y(dd);
      if (s.periodic_x) tx = tx < 0 ? tx + s.nx : (tx >= s.nx ? tx - s.nx : tx);
      if (s.periodic_y) ty = ty < 0 ? ty + s.ny : (ty >= s.ny ? ty - s.ny : ty);
      if ((unsigned)tx < (unsigned)s.nx && (unsigned)ty < (unsigned)s.ny) {
        bool okd;
        const Macro<R> Md = field_macro<R>(n, ux, uy, T, (long long)ty * s.nx + tx, okd);
        R ed[8];
        eq_pair<S>(stored_eq<S>(Md, qc), d, qc, ed, ed + 4);
        const R vx = R(hop_x(dd)) / R(5), vy = R(hop_y(dd)) / R(5);
        const R om = Md.gamma * (R(1) - (vx * Md.ux + vy * Md.uy)) * R(s.inv_tau);
        const R iom = R(1) / om;
#pragma unroll
        for (int j = 0; j < kShells; ++j)
          v[4 * h + j] = ed[4 * h + j] - (ed[4 * h + j] - v[4 * h + j]) * iom;
      }
    }
    Codec<S>::store4(fout + vec_index(s, d, site), v);
    Codec<S>::store4(fout + vec_index(s, d + 1, site), v + 4);
  }
}

// The seed in two passes: `eq` holds the stored f^eq of every site (init_body
// into the other buffer), and each site d sends, for every direction,
//   f*_i(d - n_i) = f^eq_i(d) - (f^eq_i(d) - f^eq_i(d - n_i)) / omega_i(d)
// to the site it came from, and keeps f^eq_i(d) where its own arrival site
// d + n_i lies outside.  For FP64 and FP32 storage, where `eq` holds the
// values init_ce_body forms in registers (16-bit storage would round them
// twice).  init_ce_body evaluates the equilibrium coefficients at 13 sites per
// site, about 1,300 FP64 operations more than the two passes: FP64 1024 x 512
// about 1.7 ms -> 0.44 ms (0.28 + 0.16); FP32 4096 x 2048 0.89 ms, where FP16
// storage takes 4.6 ms.
template <typename S, class C>
__device__ __forceinline__ void ce_from_eq_body(const S* __restrict__ eq, S* __restrict__ fout,
                                                const DevSample& s, const double* ux,
                                                const double* uy, const C& qc) {
  using R = typename Codec<S>::R;
  const int x = blockIdx.x * kBX + threadIdx.x;
  const int y = blockIdx.y;
  if (x >= s.nx) return;
  const long long k = (long long)y * s.nx + x, site = (long long)y * s.ldx + x;
  const double vx = ux[k], vy = uy[k];
  const double g = qrsqrt(1.0 - fma(vx, vx, vy * vy));
  const R gt = R(g) * R(s.inv_tau), gx = gt * R(vx), gy = gt * R(vy);
#pragma unroll
  for (int d = 0; d < kDirs; ++d) {
    const int dx = hop_x(d), dy = hop_y(d);
    R own[4];
    Codec<S>::load4(eq + vec_index(s, d, site), pull_policy(false), own);
    int sx = x - dx, sy = y - dy;
    if (s.periodic_x) sx = sx < 0 ? sx + s.nx : (sx >= s.nx ? sx - s.nx : sx);
    if (s.periodic_y) sy = sy < 0 ? sy + s.ny : (sy >= s.ny ? sy - s.ny : sy);
    if ((unsigned)sx < (unsigned)s.nx && (unsigned)sy < (unsigned)s.ny) {
      const long long from = vec_index(s, d, (long long)sy * s.ldx + sx);
      R src[4];
      Codec<S>::load4(eq + from, pull_policy(false), src);
      const R om = fma(-gy, R(dy) / R(5), fma(-gx, R(dx) / R(5), gt));
      R iom;
      if constexpr (sizeof(R) == 8) iom = qrcp(om);
      else iom = R(1) / om;
#pragma unroll
      for (int j = 0; j < kShells; ++j) src[j] = fma(src[j] - own[j], iom, own[j]);
      Codec<S>::store4(fout + from, src);
    }
    int tx = x + dx, ty = y + dy;
    if (s.periodic_x) tx = tx < 0 ? tx + s.nx : (tx >= s.nx ? tx - s.nx : tx);
    if (s.periodic_y) ty = ty < 0 ? ty + s.ny : (ty >= s.ny ? ty - s.ny : ty);
    if (!((unsigned)tx < (unsigned)s.nx && (unsigned)ty < (unsigned)s.ny))
      Codec<S>::store4(fout + vec_index(s, d, site), own);
  }
}

// Dense FP64 deviations [48][ny][nx]  <->  stored vectors.
// Directions d0 .. d0 + gridDim.z - 1, one thread per site and direction (one
// vector access against four plane accesses, all coalesced); `out` / `in`
// point at population 4 d0 of the dense array.
template <typename S, class C>
__device__ __forceinline__ void get_state_body(const S* __restrict__ fin, const DevSample& s,
                                               int d0, double* out, const C& qc) {
  const int x = blockIdx.x * kBX + threadIdx.x;
  const int y = blockIdx.y;
  const int dd = blockIdx.z, d = d0 + dd;
  if (x >= s.nx) return;
  struct alignas(4 * sizeof(S) < 16 ? 4 * sizeof(S) : 16) Vec { S v[4]; };
  const Vec v = *reinterpret_cast<const Vec*>(fin + vec_index(s, d, (long long)y * s.ldx + x));
#pragma unroll
  for (int j = 0; j < kShells; ++j)
    out[((long long)(4 * dd + j) * s.ny + y) * s.nx + x] = Codec<S>::decode(v.v[j], dir_kind(d), j, qc);
}

template <typename S, class C>
__device__ __forceinline__ void set_state_body(S* __restrict__ fout, const DevSample& s, int d0,
                                               const double* in, const C& qc) {
  const int x = blockIdx.x * kBX + threadIdx.x;
  const int y = blockIdx.y;
  const int dd = blockIdx.z, d = d0 + dd;
  if (x >= s.nx) return;
  struct alignas(4 * sizeof(S) < 16 ? 4 * sizeof(S) : 16) Vec { S v[4]; };
  Vec v;
#pragma unroll
  for (int j = 0; j < kShells; ++j)
    v.v[j] = Codec<S>::encode(in[((long long)(4 * dd + j) * s.ny + y) * s.nx + x], dir_kind(d), j, qc);
  *reinterpret_cast<Vec*>(fout + vec_index(s, d, (long long)y * s.ldx + x)) = v;
}

}  // namespace rlbm
