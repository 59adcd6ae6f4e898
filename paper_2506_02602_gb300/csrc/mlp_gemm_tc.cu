// mlp_gemm_tc.cu -- the surrogate's training GEMM on the 5th-generation tensor cores:
// C[m, n] = alpha * sum_k A(m, k) B(n, k) (+ bias[n]) with A(m, k) = A[m*sam + k*sak] and
// B(n, k) = B[n*sbn + k*sbk] in BF16, FP32 accumulation in tensor memory (GemmArgs,
// mlp.cuh).  One kernel serves the forward layer (H W^T), the input gradient (G W) and
// the weight gradient (G^T H, split over the batch) through the strides.
//
// A CTA computes a 128 x Nt tile (Nt = 16, or 64 for wider outputs, which run as several
// tiles so a batch of 4096 rows spreads over 128 CTAs): 16 warps, one elected thread
// issues tcgen05.mma (M = 128, N = Nt, K = 16) into a 128-lane x Nt-column
// FP32 accumulator in tensor memory.  What bounds it is latency: 128 CTAs of 0.5 GFLOP in all
// run each once, so a K of up to 256 (every product of a training step on 4096 rows) is staged
// whole, all its loads in flight together, in the canonical K-major core-matrix layout of
// tc.cuh; a longer K goes 256 at a time.  Operands whose unit stride runs along k come by
// 16-byte cp.async copies; those whose unit stride runs along m or n by 16-byte loads that
// groups of eight lanes transpose through shuffles, so that they are stored 16 bytes at a
// time too (2-byte stores met 16-way bank conflicts).  Epilogue: each warp reads 32
// accumulator lanes (its lane quarter, tcgen05.ld 32x32b) for a half of the columns and
// applies alpha, bias, accumulation into Cf, GELU (or the product with GELU' of a given Z)
// and the FP32 / BF16 stores to half of the rows.  Its loops over rows are rolled: code that
// runs once per launch comes from the L2, and unrolled the GELU products took 30 us instead of
// 19 (4096 x 256 x 256, caches cold, with Z's product; 26 to 31 with two stages and half the
// warps in the epilogue).
//
// Every mbarrier wait is bounded; a wait that runs out sets *err (when given), the CTA
// issues nothing more, and still frees its tensor memory.
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <cstdint>

#include "internal.cuh"
#include "mlp.cuh"
#include "mma.cuh"
#include "tc.cuh"

namespace chem {

namespace {

constexpr int GM = 128;      // rows per CTA tile (MMA M)
constexpr int GKC = 64;      // K of a staged chunk
constexpr int GNMAX = 64;    // widest N tile (MMA N): 256-wide outputs run as 4 tiles, 4x the CTAs
constexpr int GTHR = 512;    // 16 warps: 4 per accumulator lane quarter, each half of the columns and of the rows
constexpr uint32_t kStageA = GM * GKC * 2;            // 16 KB
constexpr uint32_t kStageB = GNMAX * GKC * 2;         // 8 KB
constexpr uint32_t kStage = kStageA + kStageB;
constexpr int GKG = 4;                                // chunks staged together
// the epilogue's 16 tiles of 32 x 33 fp32 and, behind them, 16 x 32 of Z per warp
constexpr uint32_t SMG_Z = 16 * 32 * 33 * 4;
constexpr uint32_t kZBytes = 16 * 16 * 32 * 4;
constexpr uint32_t SMG_BAR = SMG_Z + kZBytes > GKG * kStage ? SMG_Z + kZBytes : GKG * kStage;  // mbarrier
constexpr uint32_t SMG_MISC = SMG_BAR + 16;           // tmem address, abort flag
constexpr uint32_t kGemmSmem = SMG_MISC + 16 + 1024;  // + alignment slack

// Operand staging modes (uniform per launch): 0 unit stride along k (16-byte rows of 8
// k), 1 unit stride along the row index (16-byte runs of 8 rows, transposed), 2 scalar.
__host__ inline int stage_mode(const __nv_bfloat16 *p, int64_t srow, int64_t sk) {
  const bool al = (reinterpret_cast<uintptr_t>(p) & 15u) == 0;
  if (sk == 1 && srow % 8 == 0 && al) return 0;
  if (srow == 1 && sk % 8 == 0 && al) return 1;
  return 2;
}

// 16-byte asynchronous copy global -> shared; src_bytes 0 fills the 16 bytes with zeros
// (the address is then not read).
__device__ __forceinline__ void cp_async16_zfill(uint32_t dst, const void *src, uint32_t src_bytes) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;\n" ::"r"(dst), "l"(src), "r"(src_bytes)
               : "memory");
}

// Rows [r0, r0 + ROWS) x k [k0, k0 + 64) of an operand with unit stride along k into the
// core-matrix tile at `tile` (zeros outside [0, rmax) x [k0, kend)) by 16-byte asynchronous
// copies (completed by the caller's cp.async.wait_all).
template <int ROWS>
__device__ __forceinline__ void stage_rows(unsigned char *tile, const __nv_bfloat16 *G, int64_t r0,
                                           int64_t rmax, int64_t sr, int64_t k0, int64_t kend) {
  constexpr int UNITS = ROWS * (GKC / 8);              // 16-byte units of the tile
  constexpr int NU = (UNITS + GTHR - 1) / GTHR;        // per thread
  const int tid = threadIdx.x;
  const __nv_bfloat16 z = __float2bfloat16(0.0f);
#pragma unroll
  for (int q = 0; q < NU; ++q) {
    const int u = tid + q * GTHR;
    if (UNITS % GTHR != 0 && u >= UNITS) break;
    const int r = u / (GKC / 8), j = u % (GKC / 8);
    const int64_t row = r0 + r, k = k0 + 8 * j;
    const uint32_t dst = smem_u32(tile + core_off(r, 8 * j, GKC));
    if (__builtin_expect(row < rmax && k + 8 <= kend, 1)) {
      cp_async16_zfill(dst, G + row * sr + k, 16u);
    } else if (row < rmax && k < kend) {
      __align__(16) __nv_bfloat16 h[8];
#pragma unroll
      for (int i = 0; i < 8; ++i) h[i] = (k + i < kend) ? G[row * sr + k + i] : z;
      *reinterpret_cast<uint4 *>(tile + core_off(r, 8 * j, GKC)) = *reinterpret_cast<const uint4 *>(h);
    } else {
      cp_async16_zfill(dst, G, 0u);
    }
  }
}

// The transposing modes: a warp's tile is RG groups of 8 rows x KO octets of k; lanes 8 g .. 8 g + 7
// hold one k each of an octet (8 rows in 16 bytes), and after the transposition one row each.
template <int ROWS>
struct TransTile {
  static constexpr int RG = ROWS / 8 < 4 ? ROWS / 8 : 4, KO = 4 / RG;
  static constexpr int RT = ROWS / 8 / RG, WT = RT * (GKC / 8 / KO);  // warp tiles of a chunk
  static constexpr int NU = (WT + GTHR / 32 - 1) / (GTHR / 32);       // per warp
  // row group and k octet of this lane in the warp's tile q; false beyond the chunk
  static __device__ __forceinline__ bool at(int q, int &rg, int &ko) {
    const int wt = (int)(threadIdx.x >> 5) + q * (GTHR / 32), g = (threadIdx.x & 31) >> 3;
    rg = (wt % RT) * RG + g % RG;
    ko = (wt / RT) * KO + g / RG;
    return wt < WT;
  }
  static __device__ __forceinline__ void load(uint4 (&h)[NU], const __nv_bfloat16 *G, int64_t r0, int64_t rmax,
                                              int64_t sr, int64_t k0, int64_t kend, int64_t sk, int mode) {
    const __nv_bfloat16 z = __float2bfloat16(0.0f);
#pragma unroll
    for (int q = 0; q < NU; ++q) {
      int rg, ko;
      if (!at(q, rg, ko)) break;
      const int64_t row = r0 + 8 * rg, k = k0 + 8 * ko + (threadIdx.x & 7);
      if (__builtin_expect(k < kend && mode == 1 && row + 8 <= rmax, 1)) {
        h[q] = *reinterpret_cast<const uint4 *>(G + k * sk + row);
      } else {
        __align__(16) __nv_bfloat16 t[8];
#pragma unroll
        for (int i = 0; i < 8; ++i) t[i] = (k < kend && row + i < rmax) ? G[(row + i) * sr + k * sk] : z;
        h[q] = *reinterpret_cast<const uint4 *>(t);
      }
    }
  }
  static __device__ __forceinline__ void store(unsigned char *tile, const uint4 (&h)[NU]) {
    const unsigned full = 0xffffffffu;
    const int l = threadIdx.x & 7;
#pragma unroll
    for (int q = 0; q < NU; ++q) {
      int rg, ko;
      if (!at(q, rg, ko)) break;  // the same for the warp's lanes
      uint32_t x0 = h[q].x, x1 = h[q].y, x2 = h[q].z, x3 = h[q].w;
      // 8 x 8 transposition, one index bit at a time
      uint32_t t0 = __shfl_xor_sync(full, (l & 4) ? x0 : x2, 4), t1 = __shfl_xor_sync(full, (l & 4) ? x1 : x3, 4);
      if (l & 4) { x0 = t0; x1 = t1; } else { x2 = t0; x3 = t1; }
      t0 = __shfl_xor_sync(full, (l & 2) ? x0 : x1, 2);
      t1 = __shfl_xor_sync(full, (l & 2) ? x2 : x3, 2);
      if (l & 2) { x0 = t0; x2 = t1; } else { x1 = t0; x3 = t1; }
      auto half = [&](uint32_t x) {
        const uint32_t y = __shfl_xor_sync(full, x, 1);
        return (l & 1) ? __byte_perm(y, x, 0x7632) : __byte_perm(x, y, 0x5410);
      };
      x0 = half(x0); x1 = half(x1); x2 = half(x2); x3 = half(x3);
      *reinterpret_cast<uint4 *>(tile + core_off(8 * rg + l, 8 * ko, GKC)) = make_uint4(x0, x1, x2, x3);
    }
  }
};

// The group's chunks c0 .. of an operand in a transposing mode into the stages from `tiles` on:
// all loads first, then the stores.
template <int ROWS>
__device__ __forceinline__ void stage_transposed(unsigned char *tiles, const __nv_bfloat16 *G, int64_t r0, int64_t rmax,
                                                 int64_t sr, int64_t kbeg, int c0, int nch, int64_t kend, int64_t sk,
                                                 int mode) {
  using T = TransTile<ROWS>;
  uint4 h[GKG][T::NU];
#pragma unroll
  for (int c = 0; c < GKG; ++c)
    if (c0 + c < nch) T::load(h[c], G, r0, rmax, sr, kbeg + (int64_t)(c0 + c) * GKC, kend, sk, mode);
#pragma unroll
  for (int c = 0; c < GKG; ++c)
    if (c0 + c < nch) T::store(tiles + (uint32_t)c * kStage, h[c]);
}

struct GemmTc {
  GemmArgs g;
  int mode_a, mode_b;
  int nt;         // N tile width (multiple of 16, <= 256)
  uint32_t cols;  // tensor-memory columns allocated (power of two >= 32, >= nt)
  int *err;
};

template <int NT>
__device__ __forceinline__ void gemm_body(const GemmTc &p, unsigned char *sm, uint32_t sbase) {
  const GemmArgs &g = p.g;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  volatile uint32_t *s_tmem = reinterpret_cast<volatile uint32_t *>(sm + SMG_MISC);
  volatile int *s_abort = reinterpret_cast<volatile int *>(sm + SMG_MISC + 4);
  const uint32_t bar0 = sbase + SMG_BAR;
  if (tid == 0) {
    *s_abort = 0;
    mbar_init(bar0, 1);
    asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
  }
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;\n" ::"r"(sbase + SMG_MISC),
                 "r"(p.cols)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;\n" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *s_tmem;

  const int64_t m0 = (int64_t)blockIdx.y * GM, n0 = (int64_t)blockIdx.x * NT;
  int64_t kbeg = 0, kend = g.K;
  if (g.split > 1) {
    const int64_t steps = (g.K + GKC - 1) / GKC, per = (steps + g.split - 1) / g.split;
    kbeg = (int64_t)blockIdx.z * per * GKC;
    kend = kbeg + per * GKC < g.K ? kbeg + per * GKC : g.K;
  }
  const int nch = kend > kbeg ? (int)((kend - kbeg + GKC - 1) / GKC) : 0;
  const uint32_t idesc = idesc_bf16(GM, NT);
  uint32_t ngroup = 0;  // groups whose MMAs were committed
  for (int c0 = 0; c0 < nch; c0 += GKG) {
    // the MMAs of the group before read these stages
    if (ngroup && !mbar_wait(bar0, (ngroup - 1) & 1)) *s_abort = 1;
    if (__all_sync(0xffffffffu, !*s_abort)) {  // the transposing shuffles need whole warps
#pragma unroll 1
      for (int c = 0; c < GKG && c0 + c < nch; ++c) {
        const int64_t k0 = kbeg + (int64_t)(c0 + c) * GKC;
        unsigned char *sa = sm + (uint32_t)c * kStage;
        if (p.mode_a == 0) stage_rows<GM>(sa, g.A, m0, g.M, g.sam, k0, kend);
        if (p.mode_b == 0) stage_rows<NT>(sa + kStageA, g.B, n0, g.N, g.sbn, k0, kend);
      }
      if (p.mode_a != 0) stage_transposed<GM>(sm, g.A, m0, g.M, g.sam, kbeg, c0, nch, kend, g.sak, p.mode_a);
      if (p.mode_b != 0) stage_transposed<NT>(sm + kStageA, g.B, n0, g.N, g.sbn, kbeg, c0, nch, kend, g.sbk, p.mode_b);
    }
    asm volatile("cp.async.wait_all;\n" ::: "memory");
    fence_async_smem();
    tc_fence_before();
    __syncthreads();
    if (*s_abort) break;
    if (tid == 0) {
      tc_fence_after();
      for (int c = c0; c < nch && c < c0 + GKG; ++c) {
        const int64_t k0 = kbeg + (int64_t)c * GKC;
        const int nk = (int)((kend - k0 + 15) / 16) < GKC / 16 ? (int)((kend - k0 + 15) / 16) : GKC / 16;
        const uint32_t a0 = sbase + (uint32_t)(c - c0) * kStage, b0 = a0 + kStageA;
        for (int kk = 0; kk < nk; ++kk)
          mma_bf16_tc(tmem, smem_desc(a0 + (uint32_t)(kk * 2) * 128, 128, (GKC / 8) * 128),
                      smem_desc(b0 + (uint32_t)(kk * 2) * 128, 128, (GKC / 8) * 128), idesc,
                      (c > 0 || kk > 0) ? 1u : 0u);
      }
      mma_commit(bar0);
    }
    ++ngroup;
  }
  // the last commit covers every MMA of the tile
  bool have = ngroup > 0 && !*s_abort;
  if (have && !mbar_wait(bar0, (ngroup - 1) & 1)) {
    have = false;
    *s_abort = 1;
  }
  tc_fence_after();
  __syncthreads();
  if (*s_abort) {
    if (p.err && tid == 0) atomicExch(p.err, 1);
  } else {
    // epilogue: warp w reads accumulator lanes (rows) m0 + 32 (w % 4) .. + 31, the lane
    // quarter tcgen05.ld lets it reach, of a column group of 32 (16 in the 16-wide tile) and
    // finishes its share of the 32 rows; they go through a padded 32 x 33 shared-memory
    // tile (the stages are idle: the last commit covered every MMA), so the global stores
    // run along rows, coalesced
    const int q = warp & 3, grp = warp >> 2;
    constexpr int NG = NT >= 32 ? NT / 32 : 1;  // column groups
    static_assert(NG == 1 || NG == 2 || NG == 4, "the four warps of a lane quarter share them evenly");
    constexpr int CW = NT / NG < 32 ? NT / NG : 32;  // columns of a group
    constexpr int RW = 32 * NG / 4;                  // rows a warp finishes
    const int cb = (grp % NG) * CW, r0 = (grp / NG) * RW;
    float *tp = reinterpret_cast<float *>(sm) + warp * (32 * 33);
    const uint32_t t_lane = tmem + ((uint32_t)(32 * q) << 16);
    if constexpr (CW == 32) {
      uint32_t r[32];
      tmem_ld32_async(t_lane + (uint32_t)cb, r);
      tmem_wait32(r);
#pragma unroll
      for (int i = 0; i < 32; ++i) tp[lane * 33 + i] = have ? __uint_as_float(r[i]) : 0.0f;
    } else {
      float w[16];
      tmem_ld16(t_lane + (uint32_t)cb, w);
#pragma unroll
      for (int i = 0; i < 16; ++i) tp[lane * 33 + i] = have ? w[i] : 0.0f;
    }
    __syncwarp();
    const int64_t n = n0 + cb + lane, mq = m0 + 32 * q + r0;
    if (lane < CW && n < g.N) {
      const int rows = (int)(g.M - mq < RW ? g.M - mq : RW);  // of this warp, may be negative
      const float *tr = tp + r0 * 33 + lane;
      // the loops over rows stay rolled: unrolled, GELU's code came cold from the L2 in every launch
      if (g.split > 1) {
        float *c = g.Cf + (int64_t)blockIdx.z * g.split_ld + mq * g.ldc + n;
#pragma unroll 4
        for (int rr = 0; rr < rows; ++rr) c[rr * g.ldc] = tr[rr * 33] * g.alpha;
      } else {
        const float bn = g.bias ? g.bias[n] : 0.0f;
        float *zs = reinterpret_cast<float *>(sm + SMG_Z) + warp * (16 * 32) + lane;
        static_assert(RW <= 16, "rows of Z a warp keeps");
        if (g.dgelu_z) {  // the rows' Z, all loads in flight together, into this lane's own words
          float z[RW];
#pragma unroll
          for (int rr = 0; rr < RW; ++rr) z[rr] = rr < rows ? __ldg(g.dgelu_z + (mq + rr) * g.ldz + n) : 0.0f;
#pragma unroll
          for (int rr = 0; rr < RW; ++rr) zs[rr * 32] = z[rr];
        }
        float *cf = g.Cf ? g.Cf + mq * g.ldc + n : nullptr;
        __nv_bfloat16 *cb = g.Cb ? g.Cb + mq * g.ldcb + n : nullptr;
        const int ldc = (int)g.ldc, ldcb = (int)g.ldcb;
        const float alpha = g.alpha;
        const bool dg = g.dgelu_z != nullptr, ge = g.gelu != 0, acc = g.accumulate != 0;
#pragma unroll 2
        for (int rr = 0; rr < rows; ++rr) {
          float x = tr[rr * 33] * alpha;
          x += bn;
          if (acc) x += cf[rr * ldc];
          if (cf) cf[rr * ldc] = x;
          if (cb) cb[rr * ldcb] = __float2bfloat16(dg ? x * gelu_grad_f(zs[rr * 32]) : ge ? gelu_f(x) : x);
        }
      }
    }
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  if (warp == 0)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;\n" ::"r"(tmem), "r"(p.cols) : "memory");
}

__global__ void __launch_bounds__(GTHR) k_gemm_tc(const __grid_constant__ GemmTc p) {
  extern __shared__ __align__(1024) unsigned char gsm_raw[];
  unsigned char *sm = reinterpret_cast<unsigned char *>(
      (reinterpret_cast<uintptr_t>(gsm_raw) + 1023) & ~static_cast<uintptr_t>(1023));
  const uint32_t sbase = smem_u32(sm);
  // the tile widths: 16 (the padded input and output layers) and 64 (the hidden layers'
  // 256 outputs as four tiles); a column beyond N is zero-filled and not stored
  if (p.nt == 16) gemm_body<16>(p, sm, sbase);
  else gemm_body<GNMAX>(p, sm, sbase);
}

}  // namespace

cudaError_t gemm_prepare() {
  static bool attr_set[64] = {};
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (dev < 0 || dev >= 64 || !attr_set[dev]) {
    e = cudaFuncSetAttribute(k_gemm_tc, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kGemmSmem);
    if (e != cudaSuccess) return e;
    if (dev >= 0 && dev < 64) attr_set[dev] = true;
  }
  return cudaSuccess;
}

cudaError_t launch_gemm(const GemmArgs &g, cudaStream_t s) {
  if (g.M <= 0 || g.N <= 0) return cudaSuccess;
  if (g.split > 1 && (!g.Cf || g.Cb || g.bias || g.accumulate)) return cudaErrorInvalidValue;
  cudaError_t e = gemm_prepare();
  if (e != cudaSuccess) return e;
  GemmTc p{};
  p.g = g;
  p.mode_a = stage_mode(g.A, g.sam, g.sak);
  p.mode_b = stage_mode(g.B, g.sbn, g.sbk);
  p.nt = g.N <= 16 ? 16 : GNMAX;
  p.cols = p.nt <= 32 ? 32u : (uint32_t)GNMAX;
  p.err = g.err;
  dim3 grid((unsigned)((g.N + p.nt - 1) / p.nt), (unsigned)((g.M + GM - 1) / GM),
            (unsigned)(g.split > 1 ? g.split : 1));
  k_gemm_tc<<<grid, GTHR, kGemmSmem, s>>>(p);
  return cudaGetLastError();
}

}  // namespace chem
