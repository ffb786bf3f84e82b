// Kernel module for one storage type.  Included once per translation unit
// with RLBM_S (storage type) and RLBM_OPS (accessor name) defined; each unit
// owns its own copy of the quadrature constants in constant memory.
#include "kernels.cuh"
#include "ops.h"

#include <atomic>
#include <cmath>

namespace rlbm {
namespace {

using S = RLBM_S;
using R = typename Codec<S>::R;

__constant__ QuadConsts<R> c_qc;

// RLBM_STEP_MIN_BLOCKS: warps per SM sub-partition the register allocation
// aims for (blocks of 128 threads per SM), measured per storage type in us per
// step at 600 x 300 / 1024 x 512 / 4096 x 2048.  FP32 storage: 4: 11.0 / 27.5 /
// 458, 5: 10.5 / 26.5 / 458 (with the values parked in shared memory 5: 10.7 /
// 26.8 / 456, 6: 10.9 / 27.6 / 461, 7: 10.6 / 27.4 / 470); 5 is kept.  FP16
// storage at the two larger sizes: 6: 25.4 / 287, 7: 24.4 / 273, 8 (spills):
// 26.4 / 348; 7 is kept.  The FP64 kernels take all the registers they want
// (the FP64 pipe is busy with 8 warps).
#ifndef RLBM_STEP_MIN_BLOCKS
#define RLBM_STEP_MIN_BLOCKS 4
#endif
// Registers per thread of every step kernel of the module: one cap for all
// block widths (64 / 128 / 256 sites).  All launch shapes give bit-identical
// states: the module is compiled without contraction, every fused multiply-add
// of the per-site arithmetic is written out.
constexpr int kStepRegs = (65536 / (RLBM_STEP_MIN_BLOCKS * kBX)) > 255
                              ? 255 : ((65536 / (RLBM_STEP_MIN_BLOCKS * kBX)) & ~7);

// Threads per block of the single-sample step.  Us per step with blocks of
// 32 / 64 / 128: FP32 200 x 150 5.7 / 5.7 / 6.4, 1024 x 512 33.7 / 32.4 / 32.6,
// 4096 x 2048 481 / 460 / 460; FP16 4096 x 2048 290 / 294 / 299; FP64 64 x 64
// 22.8 / 22.7 / 25.6.
constexpr int kStepThreads = 64;

// Dynamic shared memory of the direct step kernels: the parking area
// (park_bytes: 12 x threads x 16 B with 16-bit storage, else none).
template <int FORCE, int RES, int BT>
__global__ void __maxnreg__(kStepRegs) k_step(const S* __restrict__ fin, S* __restrict__ fout,
                                              const __grid_constant__ DevSample s,
                                              const __grid_constant__ WarpTiles wt,
                                              const __grid_constant__ StepOffsets of,
                                              const R* __restrict__ ghost, StepAux<R> aux) {
  extern __shared__ __align__(128) unsigned char park_smem[];
  step_body<S, FORCE, RES, BT>(fin, fout, s, wt, of, ghost, aux, c_qc, park_smem);
}

// FP64 samples of few sites (split_body).
template <int FORCE, int RES>
__global__ void __launch_bounds__(96) k_step_split(const S* __restrict__ fin, S* __restrict__ fout,
                                                   const __grid_constant__ DevSample s,
                                                   const __grid_constant__ WarpTiles wt,
                                                   const __grid_constant__ StepOffsets of,
                                                   const R* __restrict__ ghost, StepAux<R> aux) {
  if constexpr (sizeof(S) == 8) {
    __shared__ GroupSums<double> part[3 * 32];
    split_body<S, FORCE, RES>(fin, fout, s, wt, of, ghost, aux, c_qc, part);
  }
}

template <int FORCE, int RES, int BX>
__global__ void __maxnreg__(kStepRegs)
k_step_batch(S* __restrict__ base, BatchArgs b, const R* __restrict__ ghost, StepAux<R> aux) {
  extern __shared__ __align__(128) unsigned char park_smem[];
  batch_body<S, FORCE, RES, BX>(base, b, ghost, aux, c_qc, park_smem);
}

// Staged pulls (persistent; dynamic shared memory: two slot-row buffers).
template <int FORCE, int RES, int BX>
__global__ void __maxnreg__(kStepRegs)
k_step_staged(S* __restrict__ base, BatchArgs b, const R* __restrict__ ghost, StepAux<R> aux) {
  extern __shared__ __align__(128) unsigned char stage_smem[];
  staged_batch_body<S, FORCE, RES, BX>(base, b, ghost, aux, c_qc, stage_smem);
}

// Shared-memory opt-in of the direct batched kernels: the parking area of a
// 256-thread block (12 x 256 x 16 B = 48 KiB with 16-bit storage) plus the
// residual reduction's static scratch exceed the default 48 KiB.
template <int BX>
cudaError_t allow_park_smem() {
  const int bytes = (int)park_bytes<S>(BX);
  cudaError_t e = cudaSuccess;
  if (bytes == 0) return e;
  auto set = [&](const void* fn) {
    if (e == cudaSuccess) e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
  };
  set((const void*)k_step_batch<0, 0, BX>);
  set((const void*)k_step_batch<0, 1, BX>);
  set((const void*)k_step_batch<0, 2, BX>);
  set((const void*)k_step_batch<1, 0, BX>);
  set((const void*)k_step_batch<1, 1, BX>);
  set((const void*)k_step_batch<1, 2, BX>);
  set((const void*)k_step_batch<2, 0, BX>);
  set((const void*)k_step_batch<2, 1, BX>);
  set((const void*)k_step_batch<2, 2, BX>);
  return e;
}

template <int BX>
cudaError_t allow_stage_smem() {
  const int bytes = (int)Stage<S>::template smem_bytes<BX>();
  cudaError_t e = cudaSuccess;
  auto set = [&](const void* fn) {
    if (e == cudaSuccess) e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
  };
  set((const void*)k_step_staged<0, 0, BX>);
  set((const void*)k_step_staged<0, 1, BX>);
  set((const void*)k_step_staged<0, 2, BX>);
  set((const void*)k_step_staged<1, 0, BX>);
  set((const void*)k_step_staged<1, 1, BX>);
  set((const void*)k_step_staged<1, 2, BX>);
  set((const void*)k_step_staged<2, 0, BX>);
  set((const void*)k_step_staged<2, 1, BX>);
  set((const void*)k_step_staged<2, 2, BX>);
  return e;
}

__global__ void __launch_bounds__(kBX) k_moments(const S* __restrict__ fin, DevSample s,
                                                 const R* __restrict__ ghost, double* n,
                                                 double* ux, double* uy, double* T,
                                                 unsigned* err, R* dn_out) {
  moments_body<S>(fin, s, ghost, n, ux, uy, T, err, c_qc, dn_out);
}

__global__ void __launch_bounds__(kBX) k_init(S* __restrict__ fout, DevSample s, const double* n,
                                              const double* ux, const double* uy,
                                              const double* T, unsigned* err) {
  init_body<S>(fout, s, n, ux, uy, T, err, c_qc);
}

// The two forms of the Chapman-Enskog seed: templates, so that a module holds
// only the one its storage type takes (seed).
template <typename E>
__global__ void __launch_bounds__(kBX) k_init_ce(E* __restrict__ fout, DevSample s,
                                                 const double* n, const double* ux,
                                                 const double* uy, const double* T,
                                                 unsigned* err) {
  init_ce_body<E>(fout, s, n, ux, uy, T, err, c_qc);
}

template <typename E>
__global__ void __launch_bounds__(kBX) k_ce_from_eq(const E* __restrict__ eq, E* __restrict__ fout,
                                                    DevSample s, const double* ux,
                                                    const double* uy) {
  ce_from_eq_body<E>(eq, fout, s, ux, uy, c_qc);
}

__global__ void __launch_bounds__(kBX) k_get(const S* __restrict__ fin, DevSample s, int d0,
                                             double* out) {
  get_state_body<S>(fin, s, d0, out, c_qc);
}

__global__ void __launch_bounds__(kBX) k_set(S* __restrict__ fout, DevSample s, int d0,
                                             const double* in) {
  set_state_body<S>(fout, s, d0, in, c_qc);
}

dim3 site_grid(const DevSample& s) { return dim3((s.nx + kBX - 1) / kBX, s.ny, 1); }

cudaError_t upload(const double p0[4], const double w[2][4], double scale) {
  QuadConsts<R> h;
  double K[4] = {0.0, 0.0, 0.0, 0.0};     // K_m = sum_j w_2j p0_j^m
  h.dec_s = R(1.0 / scale);
  h.enc_s = R(scale);
  for (int j = 0; j < kShells; ++j) {
    h.p0[j] = R(p0[j]);
    for (int k = 0; k < 2; ++k) {
      h.wd[k][j] = w[k][j];
      h.iwd[k][j] = 1.0 / w[k][j];
      h.iwl[k][j] = std::fma(-w[k][j], h.iwd[k][j], 1.0) / w[k][j];
      h.wp0[k][j] = R(w[k][j] * p0[j] / scale);
      h.wp0sq[k][j] = R(w[k][j] * p0[j] * p0[j] / scale);
    }
    for (int m = 1; m <= 3; ++m) K[m] += w[1][j] * std::pow(p0[j], m);
  }
  // operand pairs of the paired FP32 arithmetic (the values the kernels use)
  for (int q = 0; q < kDirs / 2; ++q) {
    const int d = 2 * q;
    const double vx = hop_x(d) / 5.0, vy = hop_y(d) / 5.0;
    h.vxo[q] = make_float2(float(vx), float(-vx));
    h.vyo[q] = make_float2(float(vy), float(-vy));
    h.vxy[q] = make_float2(float(vx), float(vy));
    h.vsq[q] = make_float2(float(vx * vx), float(vx * vy));
  }
  for (int k = 0; k < 2; ++k) {
    for (int j = 0; j < kShells; ++j)
      h.wab[k][j] = make_float2(float(w[k][j] * p0[j] / scale),
                                float(w[k][j] * p0[j] * p0[j] / scale));
  }
  h.p01 = make_float2(float(p0[0]), float(p0[1]));
  h.p23 = make_float2(float(p0[2]), float(p0[3]));
  // Conservation projection on the four (5,0)-type directions:
  //   [4K1 4K2; 4K2 4K3] (l0, l1) = -(rN, rE),   2 K3 lx = -rX,  2 K3 ly = -rY.
  const double det = 16.0 * (K[1] * K[3] - K[2] * K[2]);
  h.P00 = R(-4.0 * K[3] / det);
  h.P01 = R(4.0 * K[2] / det);
  h.P10 = R(4.0 * K[2] / det);
  h.P11 = R(-4.0 * K[1] / det);
  h.px = R(-1.0 / (2.0 * K[3]));
  cudaError_t e = cudaMemcpyToSymbol(c_qc, &h, sizeof(h));
  // shared-memory opt-in of the staged kernels (current device)
  if (e == cudaSuccess) e = allow_stage_smem<64>();
  if (e == cudaSuccess) e = allow_stage_smem<128>();
  if (e == cudaSuccess) e = allow_stage_smem<256>();
  if (e == cudaSuccess) e = allow_park_smem<256>();
  return e;
}

// Launch that may overlap its predecessor's end (chain_release / chain_wait):
// the blocks of the next step are placed while the last wave of this one
// drains.  FP32 600 x 300 (1.5 waves) 15.4 -> 11.0 us per step together with
// the warp tiles, FP16 1024 x 512 36 -> 26, FP32 1024 x 512 34.7 -> 32.6.
template <typename... P, typename... A>
void launch_chained(void (*k)(P...), unsigned grid, int block, size_t smem, cudaStream_t st,
                    A... args) {
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

// Attributes of the current device (looked up once per device; concurrent
// first calls store the same values).
int device_attr(cudaDeviceAttr attr, std::atomic<int> (&known)[64]) {
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return 0;
  int v = known[dev].load(std::memory_order_relaxed);
  if (v == 0 && cudaDeviceGetAttribute(&v, attr, dev) == cudaSuccess)
    known[dev].store(v, std::memory_order_relaxed);
  return v;
}
size_t l2_bytes() {
  static std::atomic<int> known[64];
  return (size_t)device_attr(cudaDevAttrL2CacheSize, known);
}
int sm_count() {
  static std::atomic<int> known[64];
  return device_attr(cudaDevAttrMultiProcessorCount, known);
}

template <int F, int BT>
void launch_single_bt(const S* a, S* b, const DevSample& s, const WarpTiles& wt,
                      const StepOffsets& of, const R* g, int res, const StepAux<R>& aux,
                      cudaStream_t st) {
  const unsigned grid = (wt.count + BT / 32 - 1) / (BT / 32);
  const size_t pk = park_bytes<S>(BT);
  if (res == 0) launch_chained(k_step<F, 0, BT>, grid, BT, pk, st, a, b, s, wt, of, g, aux);
  else if (res == 1) launch_chained(k_step<F, 1, BT>, grid, BT, pk, st, a, b, s, wt, of, g, aux);
  else launch_chained(k_step<F, 2, BT>, grid, BT, pk, st, a, b, s, wt, of, g, aux);
}

template <int F>
void launch_single(const S* a, S* b, const DevSample& s, const R* g, int res, const StepAux<R>& aux,
                   cudaStream_t st) {
  WarpTiles wt;
  wt.per_row = (unsigned)(s.nx + 31) / 32;
  wt.magic = wt.per_row > 1 ? (unsigned)((1ull << 32) / wt.per_row) : 0xffffffffu;
  wt.count = wt.per_row * (unsigned)s.ny;
  // Both rules were measured on FP32 storage, the only type whose loads take
  // the policy (us per step, neither / reversed /
  // reversed and evict-first): buffers of 48 MiB 14.7 / 14.7 / 14.0, 74 MiB
  // 24.6 / 23.2 / 20.9, 96 MiB (1024 x 512) 32.5 / 29.7 / 27.6, 144 MiB 46.6 /
  // 44.3 / 43.3, 192 MiB 60.9 / 58.3 / 57.8, 384 MiB 116.4 / 113.6 / 115.2,
  // 1.5 GiB 459 / 459 / 481 (L2: 129 MB); FP16 storage at 768 MiB loses 1.5 %
  // to the reversed order.
  const size_t bytes = (size_t)s.plane * kQ * sizeof(S), l2 = l2_bytes();
  wt.evict_first = bytes <= 2 * l2;
  wt.reverse = s.cur && bytes <= 4 * l2;
  // FP64, up to two blocks per SM (one warp per FP64 sub-partition): the next
  // step's blocks, placed while this one runs, would gather on the SMs it
  // leaves idle.  Us per step, early / not: 64 x 64 44 / 13.4, 150 x 77 52 / 29.
  // Room for one or two blocks per SM by a request for shared memory gives the
  // same times, but keeps several small solvers on their own streams apart
  // (eight of 64 x 64: 83 us per step of all, 58 so).
  wt.early = sizeof(S) != 8 || (wt.count + kStepThreads / 32 - 1) / (kStepThreads / 32) >
                                   2u * (unsigned)sm_count();
  StepOffsets of;
  for (int d = 0; d < kDirs; ++d) {
    of.pull_[d] = pull_offset<S>(d, s.plane, s.ldx);
    of.plane_[d] = plane_offset<S>(d, s.plane);
  }
  if constexpr (sizeof(S) == 8) {
    // up to one tile per SM: a second one would share sub-partitions, and two
    // split chains take as long as one whole chain
    if (wt.count <= (unsigned)sm_count()) {
      if (res == 0) launch_chained(k_step_split<F, 0>, wt.count, 96, 0, st, a, b, s, wt, of, g, aux);
      else if (res == 1) launch_chained(k_step_split<F, 1>, wt.count, 96, 0, st, a, b, s, wt, of, g, aux);
      else launch_chained(k_step_split<F, 2>, wt.count, 96, 0, st, a, b, s, wt, of, g, aux);
      return;
    }
  }
  launch_single_bt<F, kStepThreads>(a, b, s, wt, of, g, res, aux, st);
}

cudaError_t step(const void* fin, void* fout, const DevSample& s, const void* ghost, int force,
                 int res, void* uprev, double* acc, unsigned* err, cudaStream_t st) {
  StepAux<R> aux{static_cast<R*>(uprev), acc, err};
  const S* a = static_cast<const S*>(fin);
  S* b = static_cast<S*>(fout);
  const R* g = static_cast<const R*>(ghost);
  if (force == kForceLca) launch_single<kForceLca>(a, b, s, g, res, aux, st);
  else if (force == kForceUniform) launch_single<kForceUniform>(a, b, s, g, res, aux, st);
  else launch_single<kForceNone>(a, b, s, g, res, aux, st);
  return cudaGetLastError();
}

template <int F, int BX>
void launch_batch_f(S* base, const BatchArgs& b, const R* g, int res, int grid, int staged,
                    const StepAux<R>& aux, cudaStream_t st) {
  if (staged == 1) {
    const size_t sm = Stage<S>::template smem_bytes<BX>();
    if (res == 0) k_step_staged<F, 0, BX><<<grid, BX, sm, st>>>(base, b, g, aux);
    else if (res == 1) k_step_staged<F, 1, BX><<<grid, BX, sm, st>>>(base, b, g, aux);
    else k_step_staged<F, 2, BX><<<grid, BX, sm, st>>>(base, b, g, aux);
    return;
  }
  const size_t pk = park_bytes<S>(BX);
  if (res == 0) launch_chained(k_step_batch<F, 0, BX>, grid, BX, pk, st, base, b, g, aux);
  else if (res == 1) launch_chained(k_step_batch<F, 1, BX>, grid, BX, pk, st, base, b, g, aux);
  else launch_chained(k_step_batch<F, 2, BX>, grid, BX, pk, st, base, b, g, aux);
}

template <int BX>
void launch_batch(S* base, const BatchArgs& b, const R* g, int force, int res, int grid,
                  int staged, const StepAux<R>& aux, cudaStream_t st) {
  if (force == kForceLca) launch_batch_f<kForceLca, BX>(base, b, g, res, grid, staged, aux, st);
  else if (force == kForceUniform)
    launch_batch_f<kForceUniform, BX>(base, b, g, res, grid, staged, aux, st);
  else launch_batch_f<kForceNone, BX>(base, b, g, res, grid, staged, aux, st);
}

cudaError_t step_batch(void* base, const BatchArgs& b, const void* ghost, int force, int res,
                       int bx, int grid, int staged, void* uprev, double* acc, unsigned* err,
                       cudaStream_t st) {
  StepAux<R> aux{static_cast<R*>(uprev), acc, err};
  S* p = static_cast<S*>(base);
  const R* g = static_cast<const R*>(ghost);
  if (bx == 64) launch_batch<64>(p, b, g, force, res, grid, staged, aux, st);
  else if (bx == 256) launch_batch<256>(p, b, g, force, res, grid, staged, aux, st);
  else launch_batch<128>(p, b, g, force, res, grid, staged, aux, st);
  return cudaGetLastError();
}

cudaError_t moments(const void* fin, const DevSample& s, const void* ghost, double* n, double* ux,
                    double* uy, double* T, unsigned* err, void* dn_out, cudaStream_t st) {
  k_moments<<<site_grid(s), kBX, 0, st>>>(static_cast<const S*>(fin), s,
                                         static_cast<const R*>(ghost), n, ux, uy, T, err,
                                         static_cast<R*>(dn_out));
  return cudaGetLastError();
}

cudaError_t init(void* fout, const DevSample& s, const double* n, const double* ux,
                 const double* uy, const double* T, unsigned* err, cudaStream_t st) {
  k_init<<<site_grid(s), kBX, 0, st>>>(static_cast<S*>(fout), s, n, ux, uy, T, err);
  return cudaGetLastError();
}

template <typename E>
void seed(E* fout, E* scratch, const DevSample& s, const double* n, const double* ux,
          const double* uy, const double* T, unsigned* err, cudaStream_t st) {
  if constexpr (sizeof(E) >= sizeof(float)) {
    k_init<<<site_grid(s), kBX, 0, st>>>(scratch, s, n, ux, uy, T, err);
    k_ce_from_eq<E><<<site_grid(s), kBX, 0, st>>>(scratch, fout, s, ux, uy);
  } else {
    k_init_ce<E><<<site_grid(s), kBX, 0, st>>>(fout, s, n, ux, uy, T, err);
  }
}

cudaError_t init_ce(void* fout, void* scratch, const DevSample& s, const double* n,
                    const double* ux, const double* uy, const double* T, unsigned* err,
                    cudaStream_t st) {
  seed(static_cast<S*>(fout), static_cast<S*>(scratch), s, n, ux, uy, T, err, st);
  return cudaGetLastError();
}

cudaError_t get_state(const void* fin, const DevSample& s, int q0, int nq, double* out,
                      cudaStream_t st) {
  dim3 grid = site_grid(s);
  grid.z = nq / kShells;
  k_get<<<grid, kBX, 0, st>>>(static_cast<const S*>(fin), s, q0 / kShells, out);
  return cudaGetLastError();
}

cudaError_t set_state(void* fout, const DevSample& s, int q0, int nq, const double* in,
                      cudaStream_t st) {
  dim3 grid = site_grid(s);
  grid.z = nq / kShells;
  k_set<<<grid, kBX, 0, st>>>(static_cast<S*>(fout), s, q0 / kShells, in);
  return cudaGetLastError();
}

const PrecOps kOps = {
    RLBM_NAME, sizeof(S), sizeof(R), upload, step, step_batch, moments, init, init_ce, get_state,
    set_state, 1,
};

}  // namespace

const PrecOps* RLBM_OPS() { return &kOps; }

}  // namespace rlbm
