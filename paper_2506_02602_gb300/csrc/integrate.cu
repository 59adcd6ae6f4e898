// integrate.cu -- the one-pass integration kernel (one thread per cell, Sec. 4.1.2) and
// the (rho, e) from (T, p, Y) kernel.  The per-cell arithmetic is in cell.cuh.
#include <cuda_runtime.h>

#include "cell.cuh"
#include "internal.cuh"

namespace chem {

// BLOCK threads per block; the registers are capped for MINB resident blocks per SM, which shared memory
// (per-thread columns and tables) may not hold.  The register file is split
// between the SM's four sub-partitions, so 12 warps per SM allow 170 registers a thread
// (128 x 3), 16 warps 128 (64 x 8, 32 x 16, 128 x 4) and 32 warps 64 (64 x 16, 32 x 32);
// anything between rounds down; 8 warps (256 x 1) leave the 255-register maximum.
// SCH: CHEM_SCHEME_LSRK (the two-register scheme of Eq. 21) or one of the full-storage
// comparators (cell_attempt_full).
template <int V, int BLOCK, int MINB, int SCH = CHEM_SCHEME_LSRK>
__global__ void __launch_bounds__(BLOCK, MINB) k_lsrk(const __grid_constant__ MechTables mt,
                                                      const CellArgs a, const StepParams p) {
  if constexpr (V == CHEM_VARIANT_MIXED) {
    load_mixed_tables<BLOCK>(mt);
    init_mixed_cols<BLOCK>(mixed_cols<BLOCK>());
  } else {
    load_fixed_tables(mt);
    load_math_tables();
  }
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  const bool live = i < a.n;
  CellState c;
  c.nacc = c.nrej = c.nrhs = 0;
  c.status = CHEM_CELL_OK;
  if (live) {
#pragma unroll
    for (int k = 0; k < NSP; ++k) c.X[k] = a.Y[k * a.ld + i];
    c.T = a.T[i];
    c.h = a.h ? a.h[i] : CUDART_NAN;
    cell_begin(c, a.rho[i], a.e[i], p.dt);
    if constexpr (SCH == CHEM_SCHEME_LSRK) {
      while (!c.done) cell_attempt<V, BLOCK>(mt, c, p);
    } else {
      while (!c.done) cell_attempt_full<V, SCH, BLOCK>(mt, c, p);
    }
    cell_finish<V, BLOCK>(mt, c);
#pragma unroll
    for (int k = 0; k < NSP; ++k) a.Y[k * a.ld + i] = c.X[k];
    a.T[i] = c.T;
    if (a.h) a.h[i] = c.h;
    if (a.status) a.status[i] = c.status;
    if (a.nsteps) a.nsteps[i] = c.nacc + c.nrej;
  }
  if (a.stats) {
    int hist[6];
#pragma unroll
    for (int s = 0; s < 6; ++s) hist[s] = live && c.status == s;
    accumulate_stats(a.stats, live ? 1 : 0, c.nacc, c.nrej, c.nrhs, c.nacc + c.nrej, hist);
  }
}

__global__ void k_state_from_TPY(const __grid_constant__ MechTables mt, int64_t n,
                                 const double *__restrict__ T, const double *__restrict__ p,
                                 const double *__restrict__ Y, int64_t ld, double *__restrict__ rho,
                                 double *__restrict__ e) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const double Ti = T[i];
  double y[NSP], inv_w = 0.0;
#pragma unroll
  for (int k = 0; k < NSP; ++k) {
    y[k] = Y[k * ld + i];
    inv_w += y[k] * mt.invW[k];
  }
  double m[6];
  mix_ecoef(mt, Ti >= mt.T_mid, y, 0.0, m);
  rho[i] = p[i] / (R_U * Ti * inv_w);
  e[i] = R_U * e_over_R(m, Ti);
}

// Launch with the variant's dynamic shared memory (the per-thread columns).
template <int V, int BLOCK, int MINB, int SCH>
static cudaError_t launch_one(const MechTables &mt, const CellArgs &a, const StepParams &p, cudaStream_t s) {
  const size_t smem = cols_bytes(V, BLOCK);
  const cudaError_t e = allow_smem(reinterpret_cast<const void *>(k_lsrk<V, BLOCK, MINB, SCH>), smem);
  if (e != cudaSuccess) return e;
  k_lsrk<V, BLOCK, MINB, SCH><<<(unsigned)((a.n + BLOCK - 1) / BLOCK), BLOCK, smem, s>>>(mt, a, p);
  return cudaGetLastError();
}

// The compiled shapes.  fp64: 12 warps per SM (128 x 3, 146 registers, no spills) run the
// 1M-cell detonation slice in 24.9 ms, 64 threads (128 registers; the columns and the 23 KB of
// tables leave 10 warps) in 26.2, 32 threads in 33.7 and 8 warps (256) in 30.6.  With 13 species the
// columns leave 8 warps at 128 and at 64 threads: 6.9 and 6.4 ms on 401 x 379 cells.  The mixed
// two-register kernel's per-thread columns allow 16 warps
// per SM (12 with 13 species): 128 x 4 at 128 registers, 8.0 ms on the 1M-cell detonation slice;
// its 32- and 64-thread shapes keep 64 registers (14 warps of 64 threads, spilling): 9.4 ms at
// 64, 11.2 at 32, and 13.2 at 256 (8 warps).
template <int V, int SCH>
static cudaError_t launch_shape(const MechTables &mt, const CellArgs &a, const StepParams &p, int block,
                                cudaStream_t s) {
  constexpr bool dense = V == CHEM_VARIANT_MIXED && SCH == CHEM_SCHEME_LSRK;
  if (block == 32) return launch_one<V, 32, dense ? 32 : 16, SCH>(mt, a, p, s);
  if (block == 64) return launch_one<V, 64, dense ? 16 : 8, SCH>(mt, a, p, s);
  if (block == 256) return launch_one<V, 256, 1, SCH>(mt, a, p, s);
  return launch_one<V, 128, dense && NSP <= 9 ? 4 : 3, SCH>(mt, a, p, s);
}

template <int SCH>
static cudaError_t launch_variant(int variant, const MechTables &mt, const CellArgs &a,
                                  const StepParams &p, int block, cudaStream_t s) {
  if (variant == CHEM_VARIANT_MIXED) return launch_shape<CHEM_VARIANT_MIXED, SCH>(mt, a, p, block, s);
  return launch_shape<CHEM_VARIANT_FP64, SCH>(mt, a, p, block, s);
}

cudaError_t launch_lsrk(int variant, int scheme, const MechTables &mt, const CellArgs &a,
                        const StepParams &p, int block, cudaStream_t s) {
  if (a.n <= 0) return cudaSuccess;
  if (scheme == CHEM_SCHEME_FULL_STORAGE)
    return launch_variant<CHEM_SCHEME_FULL_STORAGE>(variant, mt, a, p, block, s);
  if (scheme == CHEM_SCHEME_RKF45) return launch_variant<CHEM_SCHEME_RKF45>(variant, mt, a, p, block, s);
  return launch_variant<CHEM_SCHEME_LSRK>(variant, mt, a, p, block, s);
}

cudaError_t launch_state_from_TPY(const MechTables &mt, int64_t n, const double *T,
                                  const double *p, const double *Y, int64_t ld, double *rho,
                                  double *e, cudaStream_t s) {
  if (n <= 0) return cudaSuccess;
  const int block = 256;
  const int64_t grid = (n + block - 1) / block;
  k_state_from_TPY<<<(unsigned)grid, block, 0, s>>>(mt, n, T, p, Y, ld, rho, e);
  return cudaGetLastError();
}

}  // namespace chem
