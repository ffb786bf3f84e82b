// Fused kernels of the neural operator for its default shape: width C = 32,
// projection width 128, 16 x 16 modes, 4 outputs, at most 16 inputs, canvas N
// a multiple of 8 from 32 to 512.  Included by fno_kernels.cu, whose tcgen05
// helpers they use.  Other shapes run the operator as a sequence of GEMMs.
//
// The contractions (60 GFLOP per training step at N = 256, batch 8) do not
// bound it.  The head kernels are bound by instruction issue (80 and 70 % of the
// slots: one erff, backward also one expf, for each of 67 M values), the row
// kernels by the latency of their phases (load, barrier, MMA, wait, epilogue,
// one after the other; issue 55 and 47 %, shared-memory pipe 41 and 30 %, a
// quarter to a third of the copy rate), k_spectral by one CTA's chain (issue
// 19 %, 14 - 17 us whatever the batch).  As a sequence of GEMMs a training step
// moved every activation through HBM two to four times (z as FP32 written,
// read, written; z1 and dz1, 268 MB each, three times) in 105 launches, 3.7 ms.
// Here a CTA keeps a canvas row in shared and tensor memory between the
// contractions:
//   k_fwd_rows     z_l = G Wm[b, x] + h W + b, h' = gelu(z_l), S1 = F1 h'
//                  (the first: h_0 = x P + bp, S1 = F1 h_0)
//   k_spectral     S2 = D S1[b], per-mode mixing, Wm[b] = Dinv U, one CTA per
//                  (ky, b); backward with the transposed matrices
//   k_head_fwd     y = gelu(h Q1 + bq1) Q2 + bq2 (nothing else stored)
//   k_head_bwd     z1 again from h, dz1, dh, and the gradients of Q1, bq1, Q2,
//                  bq2 and of the last layer's bias
//   k_bwd_rows     dh = dz W^T + F1^T dS1, dz' = dh gelu'(z), dWm = G^T dz',
//                  gradients of W and b (last: of P and bp)
//   k_mix_grad     gradient of the mixing matrices
// Every value that is rounded to BF16 is formed by the same FP32 operations
// in the same order as in the sequence of GEMMs (K in ascending steps of 16,
// then the additions of its epilogues), so outputs agree with it bit for bit;
// only the order of the FP32 sums of weight and bias gradients differs.
// Measured, GEMM sequence -> fused: training step 256 x 256, batch 8, 3.84 ->
// 0.90 ms, 64 x 64, batch 4, 1.70 -> 0.23 ms (105 launches from Python -> 27,
// the operator's 10 and 14 from one call per direction), inference 256 x 256,
// batch 1, 0.65 -> 0.106 ms.

namespace fused {

constexpr int kC = 32;            // width
constexpr int kQ = 128;           // projection width
constexpr int kM = 32;            // rows of the y transform (2 m2)
constexpr int kKy = 16;           // m2
constexpr int kModes = 64;        // rows of the x transform (2 KX)
constexpr int kTileRows = 128;    // sites per MMA tile (TMEM lanes)

// Shared-memory operands are K-major core matrices (8 rows x 16 bytes, no
// swizzle): element (r, k) at (k / 8) lbo + (r / 8) sbo + (r % 8) 16 + (k % 8) 2.
struct Op {
  uint32_t base, lbo, sbo;
  __device__ __forceinline__ uint32_t chunk(int r, int kg) const {
    return base + (uint32_t)kg * lbo + (uint32_t)(r >> 3) * sbo + (uint32_t)(r & 7) * 16;
  }
  __device__ __forceinline__ uint32_t elem(int r, int k) const {
    return chunk(r, k >> 3) + (uint32_t)(k & 7) * 2;
  }
};

__device__ __forceinline__ void sts16(uint32_t a, uint4 v) {
  asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};\n"
               :: "r"(a), "r"(v.x), "r"(v.y), "r"(v.z), "r"(v.w) : "memory");
}
__device__ __forceinline__ uint4 lds16(uint32_t a) {
  uint4 v;
  asm volatile("ld.shared.v4.b32 {%0, %1, %2, %3}, [%4];\n"
               : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "r"(a) : "memory");
  return v;
}
__device__ __forceinline__ void sts2(uint32_t a, uint16_t v) {
  asm volatile("st.shared.b16 [%0], %1;\n" :: "r"(a), "h"(v) : "memory");
}
__device__ __forceinline__ uint16_t bf16_bits(float v) {
  return __bfloat16_as_ushort(__float2bfloat16_rn(v));
}
__device__ __forceinline__ uint32_t pack_bits(uint16_t lo, uint16_t hi) {
  return (uint32_t)lo | ((uint32_t)hi << 16);
}
// the eight 16-bit values of a chunk to elements (r0 .. r0 + 7, k) of an operand
__device__ __forceinline__ void scatter8(const Op& o, int r0, int k, uint4 v) {
  const uint32_t w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
  for (int j = 0; j < 8; ++j)
    sts2(o.elem(r0 + j, k), (uint16_t)(w[j >> 1] >> (16 * (j & 1))));
}

__device__ __forceinline__ void proxy_fence() {
  asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");
}
__device__ __forceinline__ void tc_before() {
  asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
}
__device__ __forceinline__ void tc_after() {
  asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
}

// D (TMEM, 128 x n) (+)= A B^T over `steps` steps of 16 k; one thread.
__device__ __forceinline__ void mma(uint32_t d, const Op& a, uint32_t a_off, const Op& b,
                                    uint32_t b_off, int n, int steps, bool add) {
  const uint32_t idesc = tc_idesc(n);
  for (int s = 0; s < steps; ++s) {
    const uint64_t da = tc_desc(a.base + a_off + (uint32_t)s * 2 * a.lbo, a.lbo, a.sbo);
    const uint64_t db = tc_desc(b.base + b_off + (uint32_t)s * 2 * b.lbo, b.lbo, b.sbo);
    const uint32_t acc = (add || s > 0) ? 1u : 0u;
    asm volatile(
        "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
        " tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n"
        :: "r"(d), "l"(da), "l"(db), "r"(idesc), "r"(acc) : "memory");
  }
}
__device__ __forceinline__ void commit(uint32_t bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n"
               :: "r"(bar) : "memory");
}

// 16 FP32 columns of this warp's 32 accumulator rows (lane = row).
__device__ __forceinline__ void tmem_ld16(uint32_t addr, float (&v)[16]) {
  uint32_t r[16];
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,"
      "%15}, [%16];\n"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]),
        "=r"(r[7]), "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]),
        "=r"(r[14]), "=r"(r[15])
      : "r"(addr));
#pragma unroll
  for (int i = 0; i < 16; ++i) v[i] = __uint_as_float(r[i]);
}
__device__ __forceinline__ void tmem_wait() {
  asm volatile("tcgen05.wait::ld.sync.aligned;\n" ::: "memory");
  // uses of the loaded registers stay behind the wait
}

// TMEM columns and mbarriers of a CTA; warp 0 allocates.  Every wait is bounded:
// a warp whose wait gives up leaves out what depends on it, the CTA stops at its
// next sync() (at the latest in finish()), raises the error flag, waits
// (bounded by the default limit) for the MMAs it has committed and frees its
// TMEM.
template <int COLS, int BARS>
struct Cta {
  uint32_t tmem, bar0;
  uint32_t phases;      // bit i: parity of barrier i's next completion
  uint32_t open;        // bit i: committed to barrier i and not yet waited for
  long long limit;      // cycles a wait may take
  bool bad;             // a wait of this warp gave up
  __device__ __forceinline__ uint32_t bar(int i) const { return bar0 + 8u * (uint32_t)i; }
  __device__ __forceinline__ void start(uint64_t* bars, uint32_t* slot, long long cycles) {
    const int tid = threadIdx.x;
    if (tid < 32) {
      asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;\n"
                   :: "r"(smem_u32(slot)), "r"(COLS) : "memory");
      asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;\n" ::: "memory");
    }
    if (tid == 0) {
      for (int i = 0; i < BARS; ++i)
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;\n" :: "r"(smem_u32(bars + i)) : "memory");
      asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
    }
    tc_before();
    __syncthreads();
    tc_after();
    tmem = *slot;
    bar0 = smem_u32(bars);
    phases = open = 0;
    limit = cycles;
    bad = false;
  }
  // all threads, where thread 0 commits the MMAs it has issued to barrier i
  __device__ __forceinline__ void commit(int i) {
    if (threadIdx.x == 0) fused::commit(bar(i));
    open |= 1u << i;
  }
  // Waits (a warp) for the next completion of barrier i; false if any lane gave
  // up: the barrier's phase is then still the one to wait for.
  __device__ __forceinline__ bool wait(int i) {
    const bool ok = __all_sync(0xffffffffu, mbar_wait(bar(i), (phases >> i) & 1u, limit));
    tc_after();
    if (ok) {
      phases ^= 1u << i;
      open &= ~(1u << i);
    } else {
      bad = true;
    }
    return ok;
  }
  __device__ __forceinline__ bool waiting(int i) const { return (open >> i) & 1u; }
  // block barrier that makes shared-memory writes visible to the MMAs and
  // orders this thread's TMEM reads before them; true if a wait gave up
  __device__ __forceinline__ bool sync() {
    proxy_fence();
    tc_before();
    const bool stop = __syncthreads_or(bad);
    tc_after();
    return stop;
  }
  __device__ __forceinline__ void finish(bool stopped) {
    if (__syncthreads_or(stopped || bad)) {
      if (threadIdx.x == 0) atomicOr(&g_tc_error, 1u);
      // MMAs committed but not waited for end (bounded) before the TMEM and
      // the shared memory go
      for (int i = 0; i < BARS; ++i)
        if ((open >> i) & 1u) mbar_wait(bar(i), (phases >> i) & 1u);
    }
    tc_before();
    __syncthreads();
    if (threadIdx.x < 32)
      asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;\n" :: "r"(tmem), "r"(COLS)
                   : "memory");
  }
};

// The row kernels run 256 threads per 128 sites: a warp w owns the rows 32 (w %
// 4) .. of the tile (the TMEM lanes it may read) and the columns of half w / 4,
// so that twice as many warps hide the latency of the activations per byte of
// shared memory (training step 256 x 256, batch 8: 1,150 -> 972 us, with the
// wider slabs of k_spectral).
constexpr int kThreads = 256;

// Chained launches (programmatic dependent launch): a kernel loads its constant
// operands while its predecessor's last CTAs run, then waits for the
// predecessor's results, and only then lets its own successor start, so that
// whatever ran before the predecessor is complete too.  Before the wait a
// kernel reads nothing but weights and DFT matrices, which no kernel of a pass
// writes; the first kernel of a pass is launched without overlap.  Together
// with the prefetch of the next tile's rows: training step 256 x 256, batch 8,
// 972 -> 902 us, 64 x 64, batch 4, 285 -> 224, inference 139 -> 105.
__device__ __forceinline__ void chain() {
  asm volatile("griddepcontrol.wait;\n" ::: "memory");
  asm volatile("griddepcontrol.launch_dependents;\n" ::: "memory");
}
// Load that stays behind chain(): coherent, because a predecessor may still
// write the data when this kernel starts (and k_bwd_rows replaces dz in place).
// Weights and DFT matrices, which no kernel of a pass writes, and what an
// earlier pass has left are read with __ldg.
__device__ __forceinline__ uint4 ldg16(const void* p) {
  uint4 v;
  asm volatile("ld.global.v4.b32 {%0, %1, %2, %3}, [%4];\n"
               : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "l"(p) : "memory");
  return v;
}

// Per-warp staging of 32 rows x 32 bytes: row-owning lanes <-> 16-byte pieces
// in row order, so that global stores write whole sectors.
constexpr int kStagePitch = 48, kStageBytes = 32 * kStagePitch;

// Writes the warp's staged rows (32 bytes each, `sp` bytes apart) to rows of
// `pitch` bytes; nv rows are valid.
__device__ __forceinline__ void stage_out(uint32_t st, int sp, unsigned char* dst, long long pitch,
                                          int nv) {
  const int lane = threadIdx.x & 31;
  __syncwarp();
#pragma unroll
  for (int q = 0; q < 2; ++q) {
    const int i = lane + 32 * q, r = i >> 1, c = i & 1;
    const uint4 v = lds16(st + r * sp + c * 16);
    if (r < nv) *reinterpret_cast<uint4*>(dst + r * pitch + c * 16) = v;
  }
  __syncwarp();
}

// B operand (n = 32, k = 32) from a row-major [k][n] BF16 matrix, one 16-byte
// piece per thread of 128.
__device__ __forceinline__ uint4 fetch_kn32(const __nv_bfloat16* p) {
  return threadIdx.x < 128 ? ldg16(reinterpret_cast<const uint4*>(p) + threadIdx.x) : make_uint4(0, 0, 0, 0);
}
__device__ __forceinline__ void store_kn32(const Op& o, uint4 v) {
  const int i = threadIdx.x;
  if (i < 128) scatter8(o, (i & 3) * 8, i >> 2, v);
}
// Piece i of rows row0 .. of a [rows][32] BF16 array (nv rows valid).
__device__ __forceinline__ uint4 fetch_row(const __nv_bfloat16* p, long long row0, int i, int nv) {
  return (i >> 2) < nv ? ldg16(reinterpret_cast<const uint4*>(p + row0 * kC) + i) : make_uint4(0, 0, 0, 0);
}

// A operand (32 rows, k = sites) from a row-major [32][N] matrix, zero beyond N.
__device__ __forceinline__ void load_modes(const Op& o, const __nv_bfloat16* p, int N, int groups) {
  for (int i = threadIdx.x; i < 32 * groups; i += blockDim.x) {
    const int r = i / groups, kg = i - r * groups;
    uint4 v = make_uint4(0, 0, 0, 0);
    if (kg * 8 < N) v = __ldg(reinterpret_cast<const uint4*>(p + (long long)r * N + kg * 8));
    sts16(o.chunk(r, kg), v);
  }
}
// A operand (sites, k = 32) from a row-major [N][32] matrix, zero beyond N.
__device__ __forceinline__ void load_sites(const Op& o, const __nv_bfloat16* p, int N, int rows) {
  for (int i = threadIdx.x; i < rows * 4; i += blockDim.x) {
    uint4 v = make_uint4(0, 0, 0, 0);
    if ((i >> 2) < N) v = __ldg(reinterpret_cast<const uint4*>(p) + i);
    sts16(o.chunk(i >> 2, i & 3), v);
  }
}

// Strides.  Row tiles written in 16-byte pieces: k groups 128 B apart.
// Operands written element by element (a thread or lane per k): the strides
// put the 32 elements of one store on different banks.
constexpr uint32_t kRowLbo = 128, kRowSbo = 512;                // 128 rows x 32 k
constexpr uint32_t kColSbo = 144, kColLbo = 592;                // 32 rows, k = sites
constexpr uint32_t kSmallLbo = 576;                             // 32 rows x 32 k
constexpr uint32_t kColBytes = 16 * kColLbo;                    // 128 sites
// An operand with 32 of the MMA's 128 rows: the rest read (and ignore) what follows.
constexpr uint32_t kOverrun = 16 * kColSbo;

__host__ __device__ constexpr size_t modes_bytes(int tiles) { return (size_t)tiles * 16 * kColLbo; }
__host__ __device__ constexpr size_t sites_bytes(int tiles) { return (size_t)tiles * kTileRows * 64; }

// ---------------------------------------------------------------------------
// Forward, one canvas row (b, x) at a time; CTAs walk the rows with a grid
// stride and keep the constant matrices.  MODE 0: inputs (h_0 = x P + bp),
// 1: a layer, 2: the last layer (no activation, no transform).
// HBM bytes per row of N sites (layer): 64 N + 2 KiB in, 192 N + 2 KiB out.
// N = 256, batch 8: 143 MB, and one erff per value.
// ---------------------------------------------------------------------------
struct FwdRows {
  const __nv_bfloat16 *in, *Wm, *G, *F1, *W;
  const float* bias;
  float* z;
  __nv_bfloat16 *h, *S1, *xcopy;
  int N, items, cin;
  long long limit;
};

template <int MODE>
constexpr size_t fwd_smem(int tiles) {
  return (MODE != 0 ? sites_bytes(tiles) + 4 * kSmallLbo : 0) +
         (MODE != 2 ? modes_bytes(tiles) + kOverrun + kColBytes : 0) + 128 * 64 + 4 * kSmallLbo +
         8 * kStageBytes;
}

template <int MODE>
__global__ void __launch_bounds__(kThreads, 3) k_fwd_rows(FwdRows p) {
  extern __shared__ __align__(1024) uint8_t tc_smem[];
  __shared__ __align__(8) uint64_t bars[2];
  __shared__ uint32_t slot;
  __shared__ float bias[kC];
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int row = tid & 127, half = tid >> 7, quarter = warp & 3;
  const int tiles = (p.N + kTileRows - 1) / kTileRows;
  uint32_t at = smem_u32(tc_smem);
  auto take = [&](uint32_t bytes) { const uint32_t a = at; at += bytes; return a; };
  const Op F1{MODE != 2 ? take((uint32_t)modes_bytes(tiles)) : 0, kColLbo, kColSbo};
  const Op hT{MODE != 2 ? take(kColBytes + kOverrun) : 0, kColLbo, kColSbo};
  const Op G{MODE != 0 ? take((uint32_t)sites_bytes(tiles)) : 0, kRowLbo, kRowSbo};
  const Op Wm{MODE != 0 ? take(4 * kSmallLbo) : 0, kSmallLbo, kColSbo};
  const Op A{take(128 * 64), kRowLbo, kRowSbo};
  const Op W{take(4 * kSmallLbo), kSmallLbo, kColSbo};
  const uint32_t stage = take(8 * kStageBytes) + warp * kStageBytes;
  Cta<128, 2> cta;
  cta.start(bars, &slot, p.limit);
  const uint32_t dG = cta.tmem, dW = cta.tmem + 32, dS = cta.tmem + 64;
  const uint32_t lanes = (uint32_t)(quarter * 32) << 16;

  if (tid < kC) bias[tid] = p.bias[tid];
  if (MODE != 2) load_modes(F1, p.F1, p.N, tiles * 16);
  if (MODE != 0) {
    load_sites(G, p.G, p.N, tiles * kTileRows);
    store_kn32(W, fetch_kn32(p.W));
  } else {
    // x P: k = inputs, padded with zeros to 16
    for (int q = 0; q < 2; ++q) sts16(A.base + (tid + kThreads * q) * 16, make_uint4(0, 0, 0, 0));
    for (int i = tid; i < kC * 16; i += kThreads) {
      const int k = i / kC, c = i % kC;
      sts2(W.elem(c, k), k < p.cin ? __bfloat16_as_ushort(p.W[k * kC + c]) : (uint16_t)0);
    }
    __syncthreads();
  }
  chain();

  // the next tile's rows (and the next canvas row's Wm) are loaded while this
  // one is computed
  uint4 nextA[2] = {}, nextW = make_uint4(0, 0, 0, 0);
  auto prefetch = [&](int item, int t) {
    if (MODE == 0 || item >= p.items) return;
    const int nv = min(kTileRows, p.N - t * kTileRows);
#pragma unroll
    for (int q = 0; q < 2; ++q)
      nextA[q] = fetch_row(p.in, (long long)item * p.N + t * kTileRows, tid + kThreads * q, nv);
    if (t == 0) nextW = fetch_kn32(p.Wm + (long long)item * (kM * kC));
  };
  prefetch(blockIdx.x, 0);
  bool stop = false;
  for (int item = blockIdx.x; item < p.items && !stop; item += gridDim.x) {
    if (MODE != 0) store_kn32(Wm, nextW);
    for (int t = 0; t < tiles && !stop; ++t) {
      const int nv = min(kTileRows, p.N - t * kTileRows);
      const long long row0 = (long long)item * p.N + t * kTileRows;
      if (MODE != 0) {
#pragma unroll
        for (int q = 0; q < 2; ++q) {
          const int i = tid + kThreads * q;
          sts16(A.chunk(i >> 2, i & 3), nextA[q]);
        }
      } else {
        const uint4* src = reinterpret_cast<const uint4*>(p.in + row0 * p.cin);
        uint4* dst = reinterpret_cast<uint4*>(p.xcopy + row0 * p.cin);
        for (int i = tid; i < nv * p.cin / 8; i += kThreads) {
          const uint4 v = ldg16(src + i);      // src may be dst
          dst[i] = v;
          const uint32_t w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
          for (int j = 0; j < 8; ++j) {
            const int e = i * 8 + j, r = e / p.cin;
            sts2(A.elem(r, e - r * p.cin), (uint16_t)(w[j >> 1] >> (16 * (j & 1))));
          }
        }
      }
      if ((stop = cta.sync())) break;
      if (tid == 0) {
        if (MODE != 0) mma(dG, G, (uint32_t)t * 16 * kRowSbo, Wm, 0, kC, 2, false);
        mma(dW, A, 0, W, 0, kC, MODE != 0 ? 2 : 1, false);
      }
      cta.commit(0);
      if (t + 1 < tiles) prefetch(item, t + 1);
      else prefetch(item + (int)gridDim.x, 0);
      bool ok = cta.wait(0);
      if (MODE != 2 && t > 0) ok = cta.wait(1) && ok;      // the transform has read hT
      const int wv = max(0, min(32, nv - quarter * 32));   // valid rows of this warp
      const bool valid = lane < wv;
      const long long wrow = row0 + quarter * 32;
      if (ok) {
        float v[16], g[16];
        tmem_ld16(dW + lanes + half * 16, v);
        if (MODE != 0) tmem_ld16(dG + lanes + half * 16, g);
        tmem_wait();
#pragma unroll
        for (int j = 0; j < 16; ++j) {
          if (MODE != 0) v[j] = v[j] + g[j];
          v[j] += bias[half * 16 + j];
        }
        if (MODE != 0) {
#pragma unroll
          for (int q = 0; q < 2; ++q) {
#pragma unroll
            for (int c = 0; c < 2; ++c)
              sts16(stage + lane * kStagePitch + c * 16,
                    make_uint4(__float_as_uint(v[8 * q + 4 * c]), __float_as_uint(v[8 * q + 4 * c + 1]),
                               __float_as_uint(v[8 * q + 4 * c + 2]), __float_as_uint(v[8 * q + 4 * c + 3])));
            stage_out(stage, kStagePitch,
                      reinterpret_cast<unsigned char*>(p.z + wrow * kC + half * 16 + 8 * q), kC * 4, wv);
          }
        }
        uint32_t hp[8];
#pragma unroll
        for (int j = 0; j < 16; j += 2) {
          const uint16_t a = bf16_bits(MODE == 1 ? gelu(v[j]) : v[j]);
          const uint16_t b = bf16_bits(MODE == 1 ? gelu(v[j + 1]) : v[j + 1]);
          hp[j / 2] = pack_bits(a, b);
          if (MODE != 2) {
            sts2(hT.elem(half * 16 + j, row), valid ? a : (uint16_t)0);
            sts2(hT.elem(half * 16 + j + 1, row), valid ? b : (uint16_t)0);
          }
        }
#pragma unroll
        for (int c = 0; c < 2; ++c)
          sts16(stage + lane * kStagePitch + c * 16,
                make_uint4(hp[4 * c], hp[4 * c + 1], hp[4 * c + 2], hp[4 * c + 3]));
        stage_out(stage, kStagePitch, reinterpret_cast<unsigned char*>(p.h + wrow * kC + half * 16), kC * 2, wv);
      }
      if (MODE != 2) {
        if ((stop = cta.sync())) break;
        if (tid == 0) mma(dS, F1, (uint32_t)t * 16 * kColLbo, hT, 0, kC, 8, t > 0);
        cta.commit(1);
      }
    }
    if (MODE != 2 && !stop) {
      if (cta.wait(1) && quarter == 0) {
        uint32_t s[8];
        float v[16];
        tmem_ld16(dS + half * 16, v);
        tmem_wait();
#pragma unroll
        for (int j = 0; j < 16; j += 2) s[j / 2] = pack_bits(bf16_bits(v[j]), bf16_bits(v[j + 1]));
        uint4* o = reinterpret_cast<uint4*>(p.S1 + (long long)item * (kM * kC) + lane * kC + half * 16);
#pragma unroll
        for (int c = 0; c < 2; ++c) o[c] = make_uint4(s[4 * c], s[4 * c + 1], s[4 * c + 2], s[4 * c + 3]);
      }
    }
  }
  cta.finish(stop);
}

// ---------------------------------------------------------------------------
// x transform, mixing and inverse x transform of one (ky, b): the 32 channels
// of ky are 32 columns of every matrix.
//   S2 = A1 X (64 x 32, K = 2 N), kept in FP32;
//   mixing per kx (forward: U = S2 R; backward: dS = dU conj(R)^T);
//   out = A2 bf16(U) (2 N x 32, K = 64).
// Forward: A1 = D, X = S1, A2 = Dinv; backward: A1 = Dinv^T, X = dWm, A2 = D^T.
// Each CTA reads the 256 KiB of R that belong to its ky (shared by the batch
// in L2).  128 CTAs at batch 8: bound by latency and the 64 k complex FMAs.
// ---------------------------------------------------------------------------
struct Spectral {
  const __nv_bfloat16 *A1, *X, *A2;
  const float* R;
  float* S2;
  __nv_bfloat16* out;
  int N;
  long long limit;
};

constexpr int kSlabK = 256;                                        // k of one slab
constexpr uint32_t kSlabLbo = 144, kSlabSbo = 32 * 144;            // 64 rows x 256 k in 16-byte pieces
constexpr uint32_t kSlabA = 8 * kSlabSbo;
constexpr uint32_t kA2Sbo = 8 * 144, kTileA = 16 * kA2Sbo;         // 128 rows x 64 k
constexpr uint32_t kSlabB = 32 * kSmallLbo;                        // 32 rows x 256 k
constexpr int kMixPitch = 33;
// behind slab A: at least another slab's bytes, which its unused rows read
constexpr size_t kSpectralSmem = kSlabA + 2 * kTileA + kSlabB + kModes * kMixPitch * 4 +
                                 8 * 32 * kMixPitch * 8;

template <bool BWD>
__global__ void __launch_bounds__(256) k_spectral(Spectral p) {
  extern __shared__ __align__(1024) uint8_t tc_smem[];
  __shared__ __align__(8) uint64_t bars[1];
  __shared__ uint32_t slot;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int ky = blockIdx.x, b = blockIdx.y, K = 2 * p.N;
  const uint32_t base = smem_u32(tc_smem);
  const uint32_t a2 = base + kSlabA, bb = a2 + 2 * kTileA;
  const Op A1{base, kSlabLbo, kSlabSbo}, B{bb, kSmallLbo, kColSbo};
  auto A2 = [&](int w) { return Op{a2 + (uint32_t)w * kTileA, kSlabLbo, kA2Sbo}; };
  float* s2 = reinterpret_cast<float*>(tc_smem + kSlabA + 2 * kTileA + kSlabB);
  float2* rt = reinterpret_cast<float2*>(s2 + kModes * kMixPitch) + warp * 32 * kMixPitch;
  Cta<128, 1> cta;
  cta.start(bars, &slot, p.limit);
  const __nv_bfloat16* X = p.X + (long long)b * K * (kKy * kC) + ky * kC;

  // A2 tiles of round r (rows 256 r .. 256 r + 255), 16-byte pieces along k
  uint4 r2[8];
  auto load_a2 = [&](int r) {
#pragma unroll
    for (int q = 0; q < 8; ++q) {
      const int i = tid + 256 * q, g = r * 256 + (i >> 3);
      r2[q] = make_uint4(0, 0, 0, 0);
      if (g < K) r2[q] = __ldg(reinterpret_cast<const uint4*>(p.A2 + (long long)g * kModes) + (i & 7));
    }
  };
  auto store_a2 = [&]() {
#pragma unroll
    for (int q = 0; q < 8; ++q) {
      const int i = tid + 256 * q, row = i >> 3;
      sts16(A2(row >> 7).chunk(row & 127, i & 7), r2[q]);
    }
  };

  // first transform: slabs of 256 k, the next one loaded while one is multiplied
  const int slabs = (K + kSlabK - 1) / kSlabK;
  bool stop = false;
  uint4 ra[8], rb[4];
  auto load_a1 = [&](int s) {
#pragma unroll
    for (int q = 0; q < 8; ++q) {
      const int i = tid + 256 * q, k = s * kSlabK + (i & 31) * 8;
      ra[q] = make_uint4(0, 0, 0, 0);
      if (k < K) ra[q] = __ldg(reinterpret_cast<const uint4*>(p.A1 + (long long)(i >> 5) * K + k));
    }
  };
  auto load_x = [&](int s) {
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const int i = tid + 256 * q, k = s * kSlabK + (i >> 2);
      rb[q] = make_uint4(0, 0, 0, 0);
      if (k < K) rb[q] = ldg16(reinterpret_cast<const uint4*>(X + (long long)k * (kKy * kC)) + (i & 3));
    }
  };
  load_a1(0);
  chain();
  load_x(0);
  for (int s = 0; s < slabs; ++s) {
    if (s > 0) cta.wait(0);
#pragma unroll
    for (int q = 0; q < 8; ++q) {
      const int i = tid + 256 * q;
      sts16(A1.chunk(i >> 5, i & 31), ra[q]);
    }
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const int i = tid + 256 * q;
      scatter8(B, (i & 3) * 8, i >> 2, rb[q]);
    }
    if ((stop = cta.sync())) break;
    if (tid == 0)
      mma(cta.tmem, A1, 0, B, 0, kC, min(kSlabK, ((K - s * kSlabK) + 15) / 16 * 16) / 16, s > 0);
    cta.commit(0);
    if (s + 1 < slabs) { load_a1(s + 1); load_x(s + 1); }
    else load_a2(0);
  }
  // mixing: a warp takes kx = warp, warp + 8, ..; lane = output channel.  The
  // matrix of one kx is in flight while the one before is used.
  float2 c[kC];
  auto load_mix = [&](int kx) {
    const float2* w = reinterpret_cast<const float2*>(p.R) + (long long)(kx * kKy + ky) * kC * kC;
#pragma unroll
    for (int i = 0; i < kC; ++i) c[i] = __ldg(w + i * kC + lane);
  };
  if (!stop) {
    load_mix(warp);
    const bool ok = cta.wait(0);
    store_a2();
    if (ok && warp < 2) {
      float* g = p.S2 + ((long long)b * kModes + warp * 32 + lane) * (kKy * kC) + ky * kC;
#pragma unroll
      for (int half = 0; half < 2; ++half) {
        float v[16];
        tmem_ld16(cta.tmem + ((uint32_t)(warp * 32) << 16) + half * 16, v);
        tmem_wait();
#pragma unroll
        for (int j = 0; j < 16; ++j) s2[(warp * 32 + lane) * kMixPitch + half * 16 + j] = v[j];
#pragma unroll
        for (int q = 0; q < 4; ++q)
          reinterpret_cast<float4*>(g + half * 16)[q] = make_float4(v[4 * q], v[4 * q + 1], v[4 * q + 2], v[4 * q + 3]);
      }
    }
    stop = cta.sync();
  }
  if (!stop) {
#pragma unroll 1
    for (int kx = warp; kx < kModes / 2; kx += 8) {
      const float* re = s2 + (2 * kx) * kMixPitch;
      const float* im = re + kMixPitch;
      float ure = 0.f, uim = 0.f;
      if (!BWD) {
#pragma unroll
        for (int i = 0; i < kC; ++i) {
          ure = fmaf(re[i], c[i].x, fmaf(-im[i], c[i].y, ure));
          uim = fmaf(re[i], c[i].y, fmaf(im[i], c[i].x, uim));
        }
        if (kx + 8 < kModes / 2) load_mix(kx + 8);
      } else {
#pragma unroll
        for (int i = 0; i < kC; ++i) rt[i * kMixPitch + lane] = c[i];
        __syncwarp();
        if (kx + 8 < kModes / 2) load_mix(kx + 8);
#pragma unroll 8
        for (int o = 0; o < kC; ++o) {
          const float2 w = rt[lane * kMixPitch + o];
          ure = fmaf(re[o], w.x, fmaf(im[o], w.y, ure));
          uim = fmaf(im[o], w.x, fmaf(-re[o], w.y, uim));
        }
        __syncwarp();
      }
      sts2(B.elem(lane, 2 * kx), bf16_bits(ure));
      sts2(B.elem(lane, 2 * kx + 1), bf16_bits(uim));
    }
    const int rounds = (K + 255) / 256;
    for (int r = 0; r < rounds; ++r) {
      if (r > 0) store_a2();
      if ((stop = cta.sync())) break;
      if (tid == 0) {
        mma(cta.tmem + 32, A2(0), 0, B, 0, kC, 4, false);
        mma(cta.tmem + 64, A2(1), 0, B, 0, kC, 4, false);
      }
      cta.commit(0);
      if (r + 1 < rounds) load_a2(r + 1);
      if (!cta.wait(0)) continue;          // the next sync stops the CTA
      const int tile = warp >> 2;          // warps 0-3: first tile, 4-7: second
      const int row = r * 256 + tile * 128 + (warp & 3) * 32 + lane;
      uint32_t s[16];
#pragma unroll
      for (int half = 0; half < 2; ++half) {
        float v[16];
        tmem_ld16(cta.tmem + 32 + tile * 32 + ((uint32_t)((warp & 3) * 32) << 16) + half * 16, v);
        tmem_wait();
#pragma unroll
        for (int j = 0; j < 16; j += 2)
          s[half * 8 + j / 2] = pack_bits(bf16_bits(v[j]), bf16_bits(v[j + 1]));
      }
      if (row < K) {
        uint4* o = reinterpret_cast<uint4*>(p.out + ((long long)b * K + row) * (kKy * kC) + ky * kC);
#pragma unroll
        for (int q = 0; q < 4; ++q) o[q] = make_uint4(s[4 * q], s[4 * q + 1], s[4 * q + 2], s[4 * q + 3]);
      }
    }
  }
  cta.finish(stop);
}

// dR(kx, ky, i, o) += sum_b conj(S(b, kx, ky, i)) dU(b, kx, ky, o); one block
// per (kx, ky), the batch's modes in shared memory, 8-byte accesses of dR.
struct MixGrad {
  const float *S, *dU;
  float2* dR;
  int batch;
};

__global__ void __launch_bounds__(256) k_mix_grad(MixGrad p) {
  const float* const S = p.S;
  const float* const dU = p.dU;
  float2* const dR = p.dR;
  const int batch = p.batch;
  __shared__ float s[16][2][kC], g[16][2][kC];
  const int kx = blockIdx.x / kKy, ky = blockIdx.x % kKy, o = threadIdx.x & 31, warp = threadIdx.x >> 5;
  float rre[4] = {}, rim[4] = {};
  chain();
  for (int b0 = 0; b0 < batch; b0 += 16) {
    const int nb = min(16, batch - b0);
    __syncthreads();
    for (int i = threadIdx.x; i < nb * 64; i += 256) {
      const int b = i >> 6, ri = (i >> 5) & 1, c = i & 31;
      const long long at = ((long long)(b0 + b) * kModes + 2 * kx + ri) * (kKy * kC) + ky * kC + c;
      s[b][ri][c] = S[at];
      g[b][ri][c] = dU[at];
    }
    __syncthreads();
    for (int b = 0; b < nb; ++b) {
      const float gr = g[b][0][o], gi = g[b][1][o];
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const float sr = s[b][0][warp + 8 * q], si = s[b][1][warp + 8 * q];
        rre[q] = fmaf(sr, gr, fmaf(si, gi, rre[q]));
        rim[q] = fmaf(sr, gi, fmaf(-si, gr, rim[q]));
      }
    }
  }
  float2* d = dR + (long long)blockIdx.x * kC * kC;
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    float2 v = d[(warp + 8 * q) * kC + o];
    v.x += rre[q];
    v.y += rim[q];
    d[(warp + 8 * q) * kC + o] = v;
  }
}

// ---------------------------------------------------------------------------
// Head, forward: tiles of 128 sites; 64 B in and 16 B out per site, 128 erff.
// ---------------------------------------------------------------------------
struct Head {
  const __nv_bfloat16 *h, *Q1, *Q2;
  const float *bq1, *bq2;
  float* y;
  const float* dy;                      // backward from here
  __nv_bfloat16* dz;
  float *gQ1, *gb1, *gQ2, *gb2, *gb;    // gradients (accumulated)
  long long rows, limit;
};

constexpr uint32_t kQ1Lbo = 16 * 144;                    // B: n = 128, k = 32
constexpr uint32_t kY1Lbo = 128, kY1Sbo = 16 * 128;      // A: 128 rows, k = 128
constexpr uint32_t kQ2Lbo = 2 * 144;                     // B: n = 16, k = 128
constexpr size_t kHeadFwdSmem = 128 * 64 + 4 * kQ1Lbo + 16 * kY1Sbo + 16 * kQ2Lbo;

__device__ __forceinline__ void load_q1(const Op& o, const __nv_bfloat16* Q1) {
  for (int i = threadIdx.x; i < kC * kQ / 8; i += kThreads)
    scatter8(o, (i % (kQ / 8)) * 8, i / (kQ / 8), __ldg(reinterpret_cast<const uint4*>(Q1) + i));
}

__global__ void __launch_bounds__(kThreads, 4) k_head_fwd(Head p) {
  extern __shared__ __align__(1024) uint8_t tc_smem[];
  __shared__ __align__(8) uint64_t bars[1];
  __shared__ uint32_t slot;
  __shared__ float bq1[kQ];
  const int tid = threadIdx.x, row = tid & 127, half = tid >> 7, quarter = (tid >> 5) & 3;
  const uint32_t base = smem_u32(tc_smem);
  const Op A{base, kRowLbo, kRowSbo};
  const Op Q1{base + 128 * 64, kQ1Lbo, 144};
  const Op Y{Q1.base + 4 * kQ1Lbo, kY1Lbo, kY1Sbo};
  const Op Q2{Y.base + 16 * kY1Sbo, kQ2Lbo, 144};
  Cta<128, 1> cta;
  cta.start(bars, &slot, p.limit);
  if (tid < kQ) bq1[tid] = p.bq1[tid];
  load_q1(Q1, p.Q1);
  for (int i = tid; i < 16 * kQ; i += kThreads) {
    const int n = i / kQ, k = i % kQ;
    sts2(Q2.elem(n, k), n < 4 ? __bfloat16_as_ushort(p.Q2[k * 4 + n]) : (uint16_t)0);
  }
  const float4 b2 = make_float4(p.bq2[0], p.bq2[1], p.bq2[2], p.bq2[3]);
  const uint32_t lanes = (uint32_t)(quarter * 32) << 16;
  const long long tiles = (p.rows + 127) / 128;
  chain();
  uint4 next[2];
  auto prefetch = [&](long long t) {
    if (t >= tiles) return;
#pragma unroll
    for (int q = 0; q < 2; ++q)
      next[q] = fetch_row(p.h, t * 128, tid + kThreads * q, (int)min(128LL, p.rows - t * 128));
  };
  prefetch(blockIdx.x);
  bool stop = false;
  for (long long t = blockIdx.x; t < tiles && !stop; t += gridDim.x) {
    const long long row0 = t * 128;
    const int nv = (int)min(128LL, p.rows - row0);
#pragma unroll
    for (int q = 0; q < 2; ++q) {
      const int i = tid + kThreads * q;
      sts16(A.chunk(i >> 2, i & 3), next[q]);
    }
    if ((stop = cta.sync())) break;
    if (tid == 0) mma(cta.tmem, A, 0, Q1, 0, kQ, 2, false);
    cta.commit(0);
    prefetch(t + gridDim.x);
    const int cols = cta.wait(0) ? 64 : 0;
#pragma unroll 1
    for (int c0 = half * 64; c0 < half * 64 + cols; c0 += 16) {
      float v[16];
      tmem_ld16(cta.tmem + lanes + c0, v);
      tmem_wait();
      uint32_t s[8];
#pragma unroll
      for (int j = 0; j < 16; j += 2)
        s[j / 2] = pack_bits(bf16_bits(gelu(v[j] + bq1[c0 + j])), bf16_bits(gelu(v[j + 1] + bq1[c0 + j + 1])));
      sts16(Y.chunk(row, c0 / 8), make_uint4(s[0], s[1], s[2], s[3]));
      sts16(Y.chunk(row, c0 / 8 + 1), make_uint4(s[4], s[5], s[6], s[7]));
    }
    if ((stop = cta.sync())) break;
    if (tid == 0) mma(cta.tmem, Y, 0, Q2, 0, 16, 8, false);     // z1 is read: its columns are free
    cta.commit(0);
    if (cta.wait(0) && half == 0) {
      float v[16];
      tmem_ld16(cta.tmem + lanes, v);
      tmem_wait();
      if (row < nv)
        reinterpret_cast<float4*>(p.y)[row0 + row] = make_float4(v[0] + b2.x, v[1] + b2.y, v[2] + b2.z, v[3] + b2.w);
    }
  }
  cta.finish(stop);
}

// ---------------------------------------------------------------------------
// Head, backward: 128 sites per tile, the 128 projected channels in two
// halves.  Per half: z1 = h Q1 + bq1 and dy1 = dy Q2^T (MMA), then per value
// one erff and one expf for y1 = gelu(z1) and dz1 = dy1 gelu'(z1); dz1 and y1
// transposed into shared memory give the weight gradients: [dz1; y1]^T [h, dy]
// in one MMA whose accumulators stay in TMEM for all tiles of the CTA.  Bound by
// instruction issue (67 M values at N = 256, batch 8, 62 instructions each: 70 %
// of the slots, 163 us).
// ---------------------------------------------------------------------------
constexpr uint32_t kDyLbo = 128, kDySbo = 256;           // A: 128 rows, k = 16
constexpr uint32_t kQ2tLbo = 16 * 144;                   // B: n = 128, k = 16
constexpr uint32_t kDzLbo = 128, kDzSbo = 8 * 128;       // A: 128 rows, k = 64
constexpr uint32_t kQ1tLbo = 576;                        // B: n = 32, k = 128
constexpr uint32_t kTLbo = 16 * 144 + 16;                // A: 128 rows (64 dz1, 64 y1), k = 128 sites
constexpr uint32_t kBwLbo = 6 * 144;                     // B: n = 48 (32 h, 4 dy, 12 zero), k = 128 sites
constexpr size_t kHeadBwdSmem = 128 * 64 + 4 * kQ1Lbo + 16 * kDySbo + 2 * kQ2tLbo + 16 * kDzSbo +
                                16 * kQ1tLbo + 16 * kTLbo + 16 * kBwLbo;

// Sums over the 32 lanes of 16 values each: lane l gets the sum of value
// l / 2 (16 + 8 + 4 + 2 + 1 shuffles; both lanes of a pair hold it).
__device__ __forceinline__ float lane_sums16(float (&v)[16]) {
  const int lane = threadIdx.x & 31;
#pragma unroll
  for (int w = 8; w >= 1; w >>= 1) {
    const bool up = lane & (w * 2);
#pragma unroll
    for (int j = 0; j < w; ++j) {
      const float send = up ? v[j] : v[j + w];
      const float keep = up ? v[j + w] : v[j];
      v[j] = keep + __shfl_xor_sync(0xffffffffu, send, w * 2);
    }
  }
  return v[0] + __shfl_xor_sync(0xffffffffu, v[0], 1);
}

__global__ void __launch_bounds__(kThreads, 2) k_head_bwd(Head p) {
  extern __shared__ __align__(1024) uint8_t tc_smem[];
  __shared__ __align__(8) uint64_t bars[1];
  __shared__ uint32_t slot;
  __shared__ float bq1[kQ], sb1[4][kQ];     // sb1: this CTA's sums of dz1, per 32 rows
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int row = tid & 127, part = tid >> 7, quarter = warp & 3;
  uint32_t at = smem_u32(tc_smem);
  auto take = [&](uint32_t bytes) { const uint32_t a = at; at += bytes; return a; };
  const Op A{take(128 * 64), kRowLbo, kRowSbo};
  const Op Q1{take(4 * kQ1Lbo), kQ1Lbo, 144};
  const Op DY{take(16 * kDySbo), kDyLbo, kDySbo};
  const Op Q2t{take(2 * kQ2tLbo), kQ2tLbo, 144};
  const Op DZ{take(16 * kDzSbo), kDzLbo, kDzSbo};
  const Op Q1t{take(16 * kQ1tLbo), kQ1tLbo, 144};
  const Op T{take(16 * kTLbo), kTLbo, 144};
  const Op Bw{take(16 * kBwLbo), kBwLbo, 144};
  const uint32_t stage = DZ.base + warp * kStageBytes;     // free when dh is read
  Cta<256, 1> cta;
  cta.start(bars, &slot, p.limit);
  const uint32_t dZ = cta.tmem, dY = cta.tmem + 64, dH = cta.tmem + 128, dAcc = cta.tmem + 160;
  const uint32_t lanes = (uint32_t)(quarter * 32) << 16;
  if (tid < kQ) bq1[tid] = p.bq1[tid];
  load_q1(Q1, p.Q1);
  for (int i = tid; i < 16 * (int)kDySbo / 16; i += kThreads) sts16(DY.base + i * 16, make_uint4(0, 0, 0, 0));
  for (int i = tid; i < 16 * (int)kBwLbo / 16; i += kThreads) sts16(Bw.base + i * 16, make_uint4(0, 0, 0, 0));
  for (int i = tid; i < kQ * 16; i += kThreads) {
    const int n = i >> 4, k = i & 15;
    sts2(Q2t.elem(n, k), k < 4 ? __bfloat16_as_ushort(p.Q2[n * 4 + k]) : (uint16_t)0);
  }
  for (int i = tid; i < kC * kQ / 8; i += kThreads)
    sts16(Q1t.chunk(i / (kQ / 8), i % (kQ / 8)), __ldg(reinterpret_cast<const uint4*>(p.Q1) + i));
  __syncthreads();
  float sb2[4], sb[16];
  for (int i = part; i < 4; i += 2) sb1[i][row] = 0.f;
#pragma unroll
  for (int i = 0; i < 4; ++i) sb2[i] = 0.f;
#pragma unroll
  for (int i = 0; i < 16; ++i) sb[i] = 0.f;

  const long long tiles = (p.rows + 127) / 128;
  chain();
  uint4 nextA[2], nextD = make_uint4(0, 0, 0, 0);
  auto prefetch = [&](long long t) {
    if (t >= tiles) return;
    const int nv = (int)min(128LL, p.rows - t * 128);
#pragma unroll
    for (int q = 0; q < 2; ++q) nextA[q] = fetch_row(p.h, t * 128, tid + kThreads * q, nv);
    if (part == 0)
      nextD = row < nv ? ldg16(reinterpret_cast<const uint4*>(p.dy) + t * 128 + row) : make_uint4(0, 0, 0, 0);
  };
  prefetch(blockIdx.x);
  bool stop = false, first = true;
  for (long long t = blockIdx.x; t < tiles && !stop; t += gridDim.x, first = false) {
    const long long row0 = t * 128;
    const int nv = (int)min(128LL, p.rows - row0);
#pragma unroll
    for (int q = 0; q < 2; ++q) {
      const int i = tid + kThreads * q;
      sts16(A.chunk(i >> 2, i & 3), nextA[q]);
      scatter8(Bw, (i & 3) * 8, i >> 2, nextA[q]);
    }
    if (part == 0) {
      const float4 d = make_float4(__uint_as_float(nextD.x), __uint_as_float(nextD.y),
                                   __uint_as_float(nextD.z), __uint_as_float(nextD.w));
      sb2[0] += d.x; sb2[1] += d.y; sb2[2] += d.z; sb2[3] += d.w;
      const uint16_t e[4] = {bf16_bits(d.x), bf16_bits(d.y), bf16_bits(d.z), bf16_bits(d.w)};
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        sts2(DY.elem(row, j), e[j]);
        sts2(Bw.elem(kC + j, row), e[j]);
      }
    }
    if ((stop = cta.sync())) break;
    if (tid == 0) {
      mma(dZ, A, 0, Q1, 0, 64, 2, false);
      mma(dY, DY, 0, Q2t, 0, 64, 1, false);
    }
    cta.commit(0);
    prefetch(t + gridDim.x);
#pragma unroll 1
    for (int half = 0; half < 2; ++half) {
      const int chunks = cta.wait(0) ? 2 : 0;
#pragma unroll 1
      for (int c = 2 * part; c < 2 * part + chunks; ++c) {
        float z[16], g[16];
        tmem_ld16(dZ + lanes + c * 16, z);
        tmem_ld16(dY + lanes + c * 16, g);
        tmem_wait();
        uint32_t s[8];
#pragma unroll
        for (int j = 0; j < 16; j += 2) {
          uint16_t dz2[2], y2[2];
#pragma unroll
          for (int i = 0; i < 2; ++i) {
            const float x = z[j + i] + bq1[half * 64 + c * 16 + j + i];
            y2[i] = bf16_bits(gelu(x));
            g[j + i] = g[j + i] * gelu_grad(x);
            dz2[i] = bf16_bits(g[j + i]);
          }
          s[j / 2] = pack_bits(dz2[0], dz2[1]);
#pragma unroll
          for (int i = 0; i < 2; ++i) {
            sts2(T.elem(c * 16 + j + i, row), dz2[i]);
            sts2(T.elem(64 + c * 16 + j + i, row), y2[i]);
          }
        }
        sts16(DZ.chunk(row, c * 2), make_uint4(s[0], s[1], s[2], s[3]));
        sts16(DZ.chunk(row, c * 2 + 1), make_uint4(s[4], s[5], s[6], s[7]));
        const float col = lane_sums16(g);
        if ((lane & 1) == 0) sb1[quarter][half * 64 + c * 16 + (lane >> 1)] += col;
      }
      if ((stop = cta.sync())) break;
      if (tid == 0) {
        mma(dH, DZ, 0, Q1t, (uint32_t)half * 8 * kQ1tLbo, kC, 4, half > 0);
        mma(dAcc + half * 48, T, 0, Bw, 0, 48, 8, !first);
        if (half == 0) {
          mma(dZ, A, 0, Q1, 8 * 144, 64, 2, false);
          mma(dY, DY, 0, Q2t, 8 * 144, 64, 1, false);
        }
      }
      cta.commit(0);
    }
    if (stop) break;
    if (!cta.wait(0)) continue;            // the next sync stops the CTA
    const int wv = max(0, min(32, nv - quarter * 32));
    {
      float v[16];
      tmem_ld16(dH + lanes + part * 16, v);
      tmem_wait();
#pragma unroll
      for (int j = 0; j < 16; ++j) sb[j] += v[j];
#pragma unroll
      for (int c = 0; c < 2; ++c)
        sts16(stage + lane * kStagePitch + c * 16,
              make_uint4(pack_bits(bf16_bits(v[8 * c]), bf16_bits(v[8 * c + 1])),
                         pack_bits(bf16_bits(v[8 * c + 2]), bf16_bits(v[8 * c + 3])),
                         pack_bits(bf16_bits(v[8 * c + 4]), bf16_bits(v[8 * c + 5])),
                         pack_bits(bf16_bits(v[8 * c + 6]), bf16_bits(v[8 * c + 7]))));
    }
    stage_out(stage, kStagePitch,
              reinterpret_cast<unsigned char*>(p.dz + (row0 + quarter * 32) * kC + part * 16), kC * 2, wv);
  }
  if (!stop) stop = cta.sync();
  if (!stop && !first) {
    // accumulators: rows 0 .. 63 dz1 channels (columns: h), 64 .. 127 y1 channels (columns 32 ..: dy)
    {
      const int q = part * 64 + (row & 63);          // part: the half of the projected channels
      if (quarter < 2) {
#pragma unroll
        for (int c0 = 0; c0 < kC; c0 += 16) {
          float v[16];
          tmem_ld16(dAcc + part * 48 + lanes + c0, v);
          tmem_wait();
#pragma unroll
          for (int j = 0; j < 16; ++j) atomicAdd(p.gQ1 + (c0 + j) * kQ + q, v[j]);
        }
      } else {
        float v[16];
        tmem_ld16(dAcc + part * 48 + lanes + kC, v);
        tmem_wait();
#pragma unroll
        for (int j = 0; j < 4; ++j) atomicAdd(p.gQ2 + q * 4 + j, v[j]);
      }
    }
    if (tid < kQ) atomicAdd(p.gb1 + tid, (sb1[0][tid] + sb1[1][tid]) + (sb1[2][tid] + sb1[3][tid]));
    const float s = lane_sums16(sb);
    if ((lane & 1) == 0) atomicAdd(p.gb + part * 16 + (lane >> 1), s);
    if (part == 0) {
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        float d = sb2[j];
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) d += __shfl_xor_sync(0xffffffffu, d, o);
        if (lane == 0) atomicAdd(p.gb2 + j, d);
      }
    }
  }
  cta.finish(stop);
}

// ---------------------------------------------------------------------------
// Backward, one canvas row (b, x) at a time.  MODE 0: the last layer (dz given;
// its bias gradient came from the head), 1: from layer l + 1 to layer l, 2: to
// the inputs.  dz is replaced in place, row by row.
// HBM bytes per row of N sites (MODE 1): 256 N + 2 KiB in, 64 N + 2 KiB out.
// ---------------------------------------------------------------------------
struct BwdRows {
  __nv_bfloat16* dz;                       // [rows][32]: of layer l + 1 in, of layer l out
  const __nv_bfloat16 *dS1, *F1T, *W, *GT, *left;   // left: h_l, or the inputs (MODE 2)
  const float* z;
  __nv_bfloat16* dWm;
  float *gW, *gb;
  int N, items, cin;
  long long limit;
};

constexpr uint32_t kZPitch = 144;          // FP32 row of 32 in shared memory

template <int MODE>
constexpr size_t bwd_smem(int tiles) {
  return (MODE != 0 ? sites_bytes(tiles) + 8 * kSmallLbo + 128 * 64 : 0) +
         (MODE != 2 ? modes_bytes(tiles) + kOverrun : 0) + 2 * kColBytes + kOverrun +
         (MODE == 1 ? 128 * kZPitch : 0);
}

template <int MODE>
__global__ void __launch_bounds__(kThreads, 2) k_bwd_rows(BwdRows p) {
  extern __shared__ __align__(1024) uint8_t tc_smem[];
  __shared__ __align__(8) uint64_t bars[2];
  __shared__ uint32_t slot;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int row = tid & 127, half = tid >> 7, quarter = warp & 3;
  const int tiles = (p.N + kTileRows - 1) / kTileRows;
  uint32_t at = smem_u32(tc_smem);
  auto take = [&](uint32_t bytes) { const uint32_t a = at; at += bytes; return a; };
  const Op GT{MODE != 2 ? take((uint32_t)modes_bytes(tiles) + kOverrun) : 0, kColLbo, kColSbo};
  const Op L{take(kColBytes + kOverrun), kColLbo, kColSbo};       // left^T: channels x sites
  const Op dzT{take(kColBytes), kColLbo, kColSbo};                // B: channels x sites
  const Op F1T{MODE != 0 ? take((uint32_t)sites_bytes(tiles)) : 0, kRowLbo, kRowSbo};
  const Op A{MODE != 0 ? take(128 * 64) : 0, kRowLbo, kRowSbo};
  const Op W{MODE != 0 ? take(4 * kSmallLbo) : 0, kSmallLbo, kColSbo};
  const Op dS{MODE != 0 ? take(4 * kSmallLbo) : 0, kSmallLbo, kColSbo};
  const uint32_t zs = MODE == 1 ? take(128 * kZPitch) : 0;
  Cta<128, 2> cta;
  cta.start(bars, &slot, p.limit);
  const uint32_t tW = cta.tmem, tF = cta.tmem + 32, tM = cta.tmem + 64, tG = cta.tmem + 96;
  const uint32_t lanes = (uint32_t)(quarter * 32) << 16;
  if (MODE != 2) load_modes(GT, p.GT, p.N, tiles * 16);
  if (MODE != 0) {
    load_sites(F1T, p.F1T, p.N, tiles * kTileRows);
    if (tid < 128) sts16(W.chunk(tid >> 2, tid & 3), __ldg(reinterpret_cast<const uint4*>(p.W) + tid));
  }
  if (MODE == 2) {      // rows of left^T beyond the inputs stay zero
    for (int i = tid; i < (int)kColBytes / 16; i += kThreads) sts16(L.base + i * 16, make_uint4(0, 0, 0, 0));
    __syncthreads();
  }
  float sb[16];
#pragma unroll
  for (int i = 0; i < 16; ++i) sb[i] = 0.f;

  chain();
  // the next tile's dz and left operand (and the next canvas row's dS1) are
  // loaded while this one is computed
  uint4 nextD[2] = {}, nextL[2] = {}, nextS = make_uint4(0, 0, 0, 0);
  auto prefetch = [&](int item, int t) {
    if (item >= p.items) return;
    const int nv = min(kTileRows, p.N - t * kTileRows);
    const long long row0 = (long long)item * p.N + t * kTileRows;
#pragma unroll
    for (int q = 0; q < 2; ++q) {
      nextD[q] = fetch_row(p.dz, row0, tid + kThreads * q, nv);
      if (MODE != 2) nextL[q] = fetch_row(p.left, row0, tid + kThreads * q, nv);
    }
    if (MODE != 0 && t == 0) nextS = fetch_kn32(p.dS1 + (long long)item * (kM * kC));
  };
  prefetch(blockIdx.x, 0);
  bool stop = false, first = true;
  for (int item = blockIdx.x; item < p.items && !stop; item += gridDim.x) {
    if (MODE != 0) store_kn32(dS, nextS);
    for (int t = 0; t < tiles && !stop; ++t) {
      const int nv = min(kTileRows, p.N - t * kTileRows);
      const long long row0 = (long long)item * p.N + t * kTileRows;
      const int wv = max(0, min(32, nv - quarter * 32));
      if (MODE != 0) {
#pragma unroll
        for (int q = 0; q < 2; ++q) {
          const int i = tid + kThreads * q;
          sts16(A.chunk(i >> 2, i & 3), nextD[q]);
        }
        if ((stop = cta.sync())) break;
        if (tid == 0) {
          mma(tW, A, 0, W, 0, kC, 2, false);
          mma(tF, F1T, (uint32_t)t * 16 * kRowSbo, dS, 0, kC, 2, false);
        }
        cta.commit(0);
      }
      // the previous tile's gradient products have read L and dzT
      if (cta.waiting(1)) cta.wait(1);
      if (MODE != 2) {
#pragma unroll
        for (int q = 0; q < 2; ++q) {
          const int i = tid + kThreads * q;
          scatter8(L, (i & 3) * 8, i >> 2, nextL[q]);
          if (MODE == 0) scatter8(dzT, (i & 3) * 8, i >> 2, nextD[q]);
        }
      } else {
        const uint4* src = reinterpret_cast<const uint4*>(p.left + row0 * p.cin);
        for (int i = tid; i < kTileRows * p.cin / 8; i += kThreads) {
          uint4 v = make_uint4(0, 0, 0, 0);
          if (i < nv * p.cin / 8) v = ldg16(src + i);
          const uint32_t w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
          for (int j = 0; j < 8; ++j) {
            const int e = i * 8 + j, r = e / p.cin;
            sts2(L.elem(e - r * p.cin, r), (uint16_t)(w[j >> 1] >> (16 * (j & 1))));
          }
        }
      }
      if (t + 1 < tiles) prefetch(item, t + 1);
      else prefetch(item + (int)gridDim.x, 0);
      const uint32_t zw = zs + quarter * 32 * kZPitch + half * 64;   // this warp's rows and columns
      if (MODE == 1) {
        // z, coalesced into shared memory
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          const int i = lane + 32 * q, r = i >> 2, c = i & 3;
          uint4 v = make_uint4(0, 0, 0, 0);
          if (r < wv) v = __ldg(reinterpret_cast<const uint4*>(p.z + (row0 + quarter * 32 + r) * kC + half * 16) + c);
          sts16(zw + r * kZPitch + c * 16, v);
        }
        __syncwarp();
      }
      if (MODE != 0 && cta.wait(0)) {
        uint32_t hp[8];
        float v[16], f[16];
        tmem_ld16(tW + lanes + half * 16, v);
        tmem_ld16(tF + lanes + half * 16, f);
        tmem_wait();
        if (MODE == 1) {
          float z[16];
#pragma unroll
          for (int c = 0; c < 4; ++c) {
            const uint4 u = lds16(zw + lane * kZPitch + c * 16);
            z[4 * c] = __uint_as_float(u.x); z[4 * c + 1] = __uint_as_float(u.y);
            z[4 * c + 2] = __uint_as_float(u.z); z[4 * c + 3] = __uint_as_float(u.w);
          }
#pragma unroll
          for (int j = 0; j < 16; ++j) v[j] = (f[j] + v[j]) * gelu_grad(z[j]);
        } else {
#pragma unroll
          for (int j = 0; j < 16; ++j) v[j] = f[j] + v[j];
        }
#pragma unroll
        for (int j = 0; j < 16; j += 2) {
          if (lane >= wv) v[j] = v[j + 1] = 0.f;
          sb[j] += v[j];
          sb[j + 1] += v[j + 1];
          const uint16_t a = bf16_bits(v[j]), b = bf16_bits(v[j + 1]);
          hp[j / 2] = pack_bits(a, b);
          sts2(dzT.elem(half * 16 + j, row), a);
          sts2(dzT.elem(half * 16 + j + 1, row), b);
        }
        if (MODE == 1) {
          // staged in this warp's part of z (read above)
          __syncwarp();
#pragma unroll
          for (int c = 0; c < 2; ++c)
            sts16(zw + lane * kZPitch + c * 16,
                  make_uint4(hp[4 * c], hp[4 * c + 1], hp[4 * c + 2], hp[4 * c + 3]));
          stage_out(zw, kZPitch,
                    reinterpret_cast<unsigned char*>(p.dz + (row0 + quarter * 32) * kC + half * 16), kC * 2, wv);
        }
      }
      if ((stop = cta.sync())) break;
      if (tid == 0) {
        if (MODE != 2) mma(tM, GT, (uint32_t)t * 16 * kColLbo, dzT, 0, kC, 8, t > 0);
        mma(tG, L, 0, dzT, 0, kC, 8, !first);
      }
      cta.commit(1);
      first = false;
    }
    if (MODE != 2 && !stop) {
      if (cta.wait(1) && quarter == 0) {
        uint32_t s[8];
        float v[16];
        tmem_ld16(tM + half * 16, v);
        tmem_wait();
#pragma unroll
        for (int j = 0; j < 16; j += 2) s[j / 2] = pack_bits(bf16_bits(v[j]), bf16_bits(v[j + 1]));
        uint4* o = reinterpret_cast<uint4*>(p.dWm + (long long)item * (kM * kC) + lane * kC + half * 16);
#pragma unroll
        for (int c = 0; c < 2; ++c) o[c] = make_uint4(s[4 * c], s[4 * c + 1], s[4 * c + 2], s[4 * c + 3]);
      }
    }
  }
  if (cta.waiting(1) && !stop) cta.wait(1);
  if (!stop) stop = cta.sync();
  if (!first && !stop) {
    if (quarter == 0) {
      const int rows = MODE == 2 ? p.cin : kC;
      float v[16];
      tmem_ld16(tG + half * 16, v);
      tmem_wait();
      if (lane < rows) {
#pragma unroll
        for (int c = 0; c < 4; ++c)
          atomicAdd(reinterpret_cast<float4*>(p.gW + lane * kC + half * 16 + 4 * c),
                    make_float4(v[4 * c], v[4 * c + 1], v[4 * c + 2], v[4 * c + 3]));
      }
    }
    if (MODE != 0) {
      const float s = lane_sums16(sb);
      if ((lane & 1) == 0) atomicAdd(p.gb + half * 16 + (lane >> 1), s);
    }
  }
  cta.finish(stop);
}

}  // namespace fused
