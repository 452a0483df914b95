// kernels.cu -- the fused cell-centred finite-volume step on sm_103a.
//
// One thread updates one triangle T (cell-centric, so no atomics on the
// state): it gathers its own state, its three neighbours' states (or builds
// ghost states at boundary faces), evaluates the Lax-Friedrichs flux of each
// face, sums them into the residual of Eq. 4 and applies the update of
// Sec. 6.2.2 (forward Euler, Eq. 6, or the second stage of Heun's scheme).
// The same thread then evaluates the CFL bound of its new state; a warp
// shuffle and shared-memory block minimum feed one 64-bit atomicMin per
// block, which gives the next step's dt without another pass over memory.
//
// The flux is evaluated without rotating into the face frame: with the
// unnormalised normal n (|n| = face length) and q = u.n,
//   |n| F(U).n-hat = (rho q, rho u q + p n_x, rho v q + p n_y, (E + p) q)
// and |n| (|u-bar_n| + c-bar) = (|q_L + q_R| + |n| (c_L + c_R)) / 2,
// which is algebraically the rotated form of Eq. 7a-7d (rotation R_n of the
// update equation), with the dissipation sign of Eq. 5.
//
// Data layout (all device arrays, one record per cell in the current order):
//   U     4 values per cell (rho, rho u, rho v, E), float4 or 32-byte doubles
//   nbr   int4 per cell: neighbour across faces 0..2, negative = ghost kind
//   geom  8 values per cell: n0x n0y n1x n1y n2x n2y 1/V 2V/P
#include <cuda_runtime.h>

#include <cstdint>

#include "cell_math.cuh"
#include "kernels.h"
#include "launch_util.cuh"

namespace fv {

namespace {

template <typename R, int WAVE = kWaveAverage>
__device__ __forceinline__ R sum_fluxes(const StepArgs& a, const rec_t<R>* __restrict__ U,
                                        const CellIn<R>& c, const R* uinf, R acc[4]) {
  const rec_t<R>& UL = c.U;
  const Prim<R> L = primitive<R>(UL);
  R perim = add_face_flux<R, WAVE>(UL, L, c.n0, c.g0.x, c.g0.y, U, uinf, acc, a.n, a.err, true);
  perim = add(perim, add_face_flux<R, WAVE>(UL, L, c.n1, c.g0.z, c.g0.w, U, uinf, acc, a.n, a.err));
  return add(perim,
             add_face_flux<R, WAVE>(UL, L, c.n2, c.g1.x, c.g1.y, U, uinf, acc, a.n, a.err));
}

template <typename R, int MODE, bool COMP, int WAVE = kWaveAverage>
__device__ __forceinline__ void update_cell(const StepArgs& a, const rec_t<R>* __restrict__ U,
                                            rec_t<R>* out, int64_t i, const CellIn<R>& c, R dt,
                                            const R* uinf, R& bmin, bool& ok) {
  R acc[4];
  const R perim = sum_fluxes<R, WAVE>(a, U, c, uinf, acc);
  finish_cell<R, MODE, COMP>(a, out, i, c, acc, perim, dt, bmin, ok);
}

// The fused step.  Shape variants (chosen per mesh by the autotuner):
//   VAR 0: one thread per cell, a grid covering all cells;
//   VAR 1: a persistent grid (resident blocks only) walks the cells with a
//          grid stride; the own-cell loads of the next cell are issued before
//          the current cell gathers its neighbours and computes, so each
//          thread keeps two cells' worth of loads in flight;
//   VAR 2: VAR 1 limited to 64 registers (4 blocks of 256 per SM);
//   VAR 3: VAR 0 limited to 40 registers (6 blocks per SM);
//   VAR 4: VAR 0 limited to 32 registers (8 blocks per SM, full occupancy).
// One block minimum per block at the end feeds the next dt.
constexpr bool var_persistent(int v) { return v == 1 || v == 2; }
constexpr int var_min_blocks(int v) { return v == 2 ? 4 : v == 3 ? 6 : v == 4 ? 8 : 1; }

template <typename R, int MODE, bool COMP, int VAR, int WAVE>
__global__ void __launch_bounds__(kBlock, var_min_blocks(VAR)) k_step(StepArgs a) {
  const rec_t<R>* __restrict__ U = static_cast<const rec_t<R>*>(a.U);
  const rec_t<R>* __restrict__ geom = static_cast<const rec_t<R>*>(a.geom);
  rec_t<R>* out = static_cast<rec_t<R>*>(a.out);
  __shared__ double s_t, s_dt;
  R bmin = R(INFINITY);
  bool ok = true;
  // cell ids are 32-bit (a mesh holds fewer than 2^31 / 3 cells): 32-bit
  // index arithmetic, one wide multiply-add per address
  const int n = (int)a.n;
  int i = blockIdx.x * blockDim.x + threadIdx.x;
  const int stride = gridDim.x * blockDim.x;
  CellIn<R> cur, nxt;
  // the first cell's tables are read while the previous step still runs
  if (i < n) load_tables<R>(a, geom, i, cur);
  chain_entry();
  if (i < n) load_values<R, MODE, COMP>(a, U, i, cur);
  if (var_persistent(VAR) && i + stride < n) load_cell<R, MODE, COMP>(a, U, geom, i + stride, nxt);
  // dt is formed once per block, while the others sum fluxes.  Formed in every
  // warp (nine FP64 instructions of 16 clocks each on the SM's one FP64 pipe)
  // it took most of shape 0's time: 1M cells, plain, 18.8 -> 14.0 us per step;
  // shape 1, with fewer warps, 12.8 -> 12.2
  if (MODE != kModeResidual && threadIdx.x == 0) block_dt(a, s_t, s_dt);
  R acc[4], perim = R(0);
  if (i < n) perim = sum_fluxes<R, WAVE>(a, U, cur, far_field<R>(a), acc);
  if (MODE != kModeResidual) __syncthreads();
  const double t = MODE != kModeResidual ? s_t : 0.0, dt = MODE != kModeResidual ? s_dt : 0.0;
  const R dtR = R(dt);
  if (i < n) finish_cell<R, MODE, COMP>(a, out, i, cur, acc, perim, dtR, bmin, ok);
  if (var_persistent(VAR)) {
    for (i += stride; i < n; i += stride) {
      cur = nxt;
      const int j = i + stride;
      if (j < n) load_cell<R, MODE, COMP>(a, U, geom, j, nxt);
      update_cell<R, MODE, COMP, WAVE>(a, U, out, i, cur, dtR, far_field<R>(a), bmin, ok);
    }
  }
  if (MODE == kModeFE || MODE == kModeRK2b) {
    if (!ok) atomicOr(a.err, 1);
    const double m = (double)block_min<R>(bmin);
    if (threadIdx.x == 0) {
      atomicMin(a.bmin_write, (unsigned long long)__double_as_longlong(m));
      if (blockIdx.x == 0) {
        *a.t_write = t + dt;
        *a.bmin_reset = kInfBits;
      }
    }
  }
}

// ---------------------------------------------------------------------------
// Many meshes in one launch.  The meshes are concatenated into one cell range,
// each padded to a multiple of the block size, so every block belongs to one
// mesh; the block looks its mesh up, uses that mesh's dt, time and free
// stream, and feeds that mesh's minimum.  The per-cell work is the same
// load_cell / update_cell as the single-mesh kernel, so each mesh advances
// bit for bit as it would alone.
// ---------------------------------------------------------------------------
template <typename R, int MODE, bool COMP>
__global__ void __launch_bounds__(kBlock, sizeof(R) == 4 ? 6 : 1) k_step_batch(BatchArgs b) {
  const StepArgs& a = b.s;
  const rec_t<R>* __restrict__ U = static_cast<const rec_t<R>*>(a.U);
  const rec_t<R>* __restrict__ geom = static_cast<const rec_t<R>*>(a.geom);
  rec_t<R>* out = static_cast<rec_t<R>*>(a.out);
  const int m = __ldg(b.block_mesh + blockIdx.x);
  const int i = blockIdx.x * blockDim.x + threadIdx.x;  // cell ids are 32-bit
  const bool has = i < __ldg(b.mesh_end + m);
  __shared__ double s_t, s_dt;
  CellIn<R> c;
  // as k_step: tables before the grid wait, dt once per block
  if (has) load_tables<R>(a, geom, i, c);
  chain_entry();
  if (has) load_values<R, MODE, COMP>(a, U, i, c);
  if (threadIdx.x == 0) batch_dt(b, m, s_t, s_dt);
  R acc[4], perim = R(0);
  if (has) perim = sum_fluxes<R>(a, U, c, batch_far_field<R>(b, m), acc);
  __syncthreads();
  R bmin = R(INFINITY);
  bool ok = true;
  if (has) finish_cell<R, MODE, COMP>(a, out, i, c, acc, perim, R(s_dt), bmin, ok);
  if (MODE == kModeFE || MODE == kModeRK2b) {
    if (!ok) atomicOr(a.err, 1);
    const double mn = (double)block_min<R>(bmin);
    if (threadIdx.x == 0) {
      atomicMin(&b.bmin[b.slot_write * b.n_meshes + m], (unsigned long long)__double_as_longlong(mn));
      if (blockIdx.x == 0 || __ldg(b.block_mesh + blockIdx.x - 1) != m) {  // first block of m
        b.t[b.t_write * b.n_meshes + m] = s_t + s_dt;
        b.bmin[b.slot_reset * b.n_meshes + m] = kInfBits;
      }
    }
  }
}

__global__ void k_batch_init(unsigned long long* bmin, double* t, int n_meshes, int* err) {
  const int j = blockIdx.x * blockDim.x + threadIdx.x;
  if (j < 3 * n_meshes) bmin[j] = kInfBits;
  if (j < 2 * n_meshes) t[j] = 0.0;
  if (j == 0) *err = 0;
}

template <typename R>
__global__ void __launch_bounds__(kBlock) k_batch_bound(const rec_t<R>* __restrict__ U,
                                                        const rec_t<R>* __restrict__ geom,
                                                        const int* block_mesh,
                                                        const int64_t* mesh_end, int n_meshes,
                                                        unsigned long long* bmin, int* err) {
  const int m = __ldg(block_mesh + blockIdx.x);
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  R bnd = R(INFINITY);
  bool ok = true;
  if (i < __ldg(mesh_end + m)) bnd = cell_bound<R>(Rec<R>::ld(U + i), geom_inradius<R>(geom, i), ok);
  if (!ok) atomicOr(err, 1);
  const double mn = (double)block_min<R>(bnd);
  if (threadIdx.x == 0) atomicMin(&bmin[m], (unsigned long long)__double_as_longlong(mn));
}

// per-mesh totals: one partial per block (blocks never span meshes), then one
// block per mesh adds its blocks' partials in a fixed order
template <typename R>
__global__ void __launch_bounds__(kBlock) k_batch_totals_partial(const rec_t<R>* __restrict__ U,
                                                                 const double* __restrict__ vol,
                                                                 const int* block_mesh,
                                                                 const int64_t* mesh_end,
                                                                 double* partials) {
  const int m = __ldg(block_mesh + blockIdx.x);
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  double s[4] = {0.0, 0.0, 0.0, 0.0};
  if (i < __ldg(mesh_end + m)) {
    const rec_t<R> u = Rec<R>::ld(U + i);
    const double v = __ldg(vol + i);
    s[0] = v * (double)u.x;
    s[1] = v * (double)u.y;
    s[2] = v * (double)u.z;
    s[3] = v * (double)u.w;
  }
  __shared__ double sm[4][kBlock / 32];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    for (int o = 16; o > 0; o >>= 1) s[q] += __shfl_xor_sync(0xffffffffu, s[q], o);
    if (lane == 0) sm[q][warp] = s[q];
  }
  __syncthreads();
  if (threadIdx.x < 4) {
    double acc = 0.0;
    for (int w = 0; w < kBlock / 32; ++w) acc += sm[threadIdx.x][w];
    partials[4 * blockIdx.x + threadIdx.x] = acc;
  }
}

__global__ void __launch_bounds__(kBlock) k_batch_totals_final(const double* partials,
                                                               const int* mesh_first_block,
                                                               double* out) {
  const int m = blockIdx.x;
  const int b0 = mesh_first_block[m], b1 = mesh_first_block[m + 1];
  double s[4] = {0.0, 0.0, 0.0, 0.0};
  for (int j = b0 + threadIdx.x; j < b1; j += blockDim.x)
#pragma unroll
    for (int q = 0; q < 4; ++q) s[q] += partials[4 * j + q];
  __shared__ double sm[4][kBlock / 32];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    for (int o = 16; o > 0; o >>= 1) s[q] += __shfl_xor_sync(0xffffffffu, s[q], o);
    if (lane == 0) sm[q][warp] = s[q];
  }
  __syncthreads();
  if (threadIdx.x < 4) {
    double acc = 0.0;
    for (int w = 0; w < kBlock / 32; ++w) acc += sm[threadIdx.x][w];
    out[4 * m + threadIdx.x] = acc;
  }
}

__global__ void k_init_scalars(LoopScalars* d) {
  d->bmin[0] = d->bmin[1] = d->bmin[2] = kInfBits;
  d->t[0] = d->t[1] = 0.0;
  d->err = 0;
}

template <typename R>
__global__ void __launch_bounds__(kBlock) k_bound(const rec_t<R>* __restrict__ U,
                                                  const rec_t<R>* __restrict__ geom, int64_t n,
                                                  unsigned long long* bmin, int* err) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  R b = R(INFINITY);
  bool ok = true;
  if (i < n) b = cell_bound<R>(Rec<R>::ld(U + i), geom_inradius<R>(geom, i), ok);
  if (!ok) atomicOr(err, 1);
  const double m = (double)block_min<R>(b);
  if (threadIdx.x == 0) atomicMin(bmin, (unsigned long long)__double_as_longlong(m));
}

// fv_compute_dt in one launch: the blocks' minima and error meet in the aux
// scalars (at rest +inf and 0), the last block to finish forms dt and puts the
// scalars back.
template <typename R>
__global__ void __launch_bounds__(kBlock) k_compute_dt(const rec_t<R>* __restrict__ U,
                                                       const rec_t<R>* __restrict__ geom, int64_t n,
                                                       double cfl, LoopScalars* sc) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  R b = R(INFINITY);
  bool ok = true;
  if (i < n) b = cell_bound<R>(Rec<R>::ld(U + i), geom_inradius<R>(geom, i), ok);
  const bool bad = __syncthreads_or(!ok);
  const R m = block_min<R>(b);
  if (threadIdx.x != 0) return;
  if (bad) atomicOr(&sc->aux_err, 1);
  atomicMin(&sc->aux_bmin, (unsigned long long)__double_as_longlong((double)m));
  __threadfence();
  if (atomicInc(&sc->aux_ticket, gridDim.x - 1) != gridDim.x - 1) return;
  __threadfence();
  const unsigned long long bits = atomicExch(&sc->aux_bmin, kInfBits);
  sc->dt_out = cfl * __longlong_as_double((long long)bits);
  sc->dt_err = atomicExch(&sc->aux_err, 0);
}

__global__ void k_init_aux(LoopScalars* sc) {
  sc->aux_bmin = kInfBits;
  sc->aux_err = sc->dt_err = 0;
  sc->aux_ticket = sc->totals_ticket = 0u;
}

// Deterministic totals sum_T V_T U_T in FP64: a thread-to-cell assignment
// fixed by the number of cells (kTotalsBlocks blocks at most) and fixed
// reduction trees; the last block to finish adds the partials, in block order.
// Warps without cells leave the tree out (their sums are zero): on 41,410
// cells, seven of eight warps of the full grid, whose additions alone held the
// FP64 pipe for some 10 us.
template <typename R>
__global__ void __launch_bounds__(kBlock) k_totals(const rec_t<R>* __restrict__ U,
                                                   const double* __restrict__ vol, int64_t n,
                                                   double* partials, unsigned* ticket,
                                                   double* out) {
  __shared__ double sm[4][kBlock / 32];
  __shared__ bool last;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  double s[4] = {0.0, 0.0, 0.0, 0.0};
  auto block_sum = [&](bool any, double* to) {  // any: uniform in the warp
    if (any) {
#pragma unroll
      for (int q = 0; q < 4; ++q)
        for (int o = 16; o > 0; o >>= 1) s[q] += __shfl_xor_sync(0xffffffffu, s[q], o);
    }
    if (lane == 0)
#pragma unroll
      for (int q = 0; q < 4; ++q) sm[q][warp] = s[q];
    __syncthreads();
    if (threadIdx.x < 4) {
      double acc = 0.0;
      for (int w = 0; w < kBlock / 32; ++w) acc += sm[threadIdx.x][w];
      to[threadIdx.x] = acc;
    }
  };
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  const int64_t first = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  for (int64_t i = first; i < n; i += stride) {
    const rec_t<R> u = Rec<R>::ld(U + i);
    const double v = __ldg(vol + i);
    s[0] += v * (double)u.x;
    s[1] += v * (double)u.y;
    s[2] += v * (double)u.z;
    s[3] += v * (double)u.w;
  }
  block_sum(first - lane < n, partials + 4 * blockIdx.x);
  if (threadIdx.x < 4) __threadfence();
  __syncthreads();
  if (threadIdx.x == 0) last = atomicInc(ticket, gridDim.x - 1) == gridDim.x - 1;
  __syncthreads();
  if (!last) return;
  __threadfence();
  s[0] = s[1] = s[2] = s[3] = 0.0;
  for (int j = threadIdx.x; j < (int)gridDim.x; j += blockDim.x)
#pragma unroll
    for (int q = 0; q < 4; ++q) s[q] += __ldcg(partials + 4 * j + q);
  block_sum((threadIdx.x & ~31u) < gridDim.x, out);
}

inline unsigned grid_for(int64_t n) { return (unsigned)((n + kBlock - 1) / kBlock); }

// Resident blocks of a kernel on the current device (cached per kernel).
template <typename K>
unsigned resident_blocks(K kernel) {
  static int cached = 0;
  if (cached == 0) {
    int dev = 0, sms = 0, per_sm = 0;
    if (cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess ||
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kernel, kBlock, 0) != cudaSuccess ||
        per_sm < 1)
      return 1024;
    cached = sms * per_sm;
  }
  return (unsigned)cached;
}

template <typename R, int MODE, bool COMP, int VAR, int WAVE = kWaveAverage>
cudaError_t launch_one(const StepArgs& a, cudaStream_t s) {
  auto kernel = k_step<R, MODE, COMP, VAR, WAVE>;
  const int64_t want = a.n > 0 ? (a.n + kBlock - 1) / kBlock : 1;  // a time step always runs its scalars
  unsigned g = (unsigned)want;
  if (var_persistent(VAR)) {
    const unsigned cap = resident_blocks(kernel);
    g = (unsigned)(want < (int64_t)cap ? want : cap);
  }
  return launch_chained(kernel, g, kBlock, 0, s, a.chained, a);
}

template <typename R, int MODE, bool COMP>
cudaError_t launch_var(int var, const StepArgs& a, cudaStream_t s) {
  if (a.wave == kWaveMax)  // the Rusanov wave speed is built for shapes 0 and 1
    return var == 0 ? launch_one<R, MODE, COMP, 0, kWaveMax>(a, s)
                    : launch_one<R, MODE, COMP, 1, kWaveMax>(a, s);
  switch (var) {
    case 0: return launch_one<R, MODE, COMP, 0>(a, s);
    case 1: return launch_one<R, MODE, COMP, 1>(a, s);
    case 2: return launch_one<R, MODE, COMP, 2>(a, s);
    case 3: return launch_one<R, MODE, COMP, 3>(a, s);
    case 4: return launch_one<R, MODE, COMP, 4>(a, s);
    default: return cudaErrorInvalidValue;
  }
}

template <typename R, bool COMP>
cudaError_t launch_step_t(int mode, int var, const StepArgs& a, cudaStream_t s) {
  if (a.n <= 0 && mode == kModeResidual) return cudaSuccess;
  switch (mode) {
    case kModeFE: return launch_var<R, kModeFE, COMP>(var, a, s);
    case kModeRK2a: return launch_var<R, kModeRK2a, COMP>(var, a, s);
    case kModeRK2b: return launch_var<R, kModeRK2b, COMP>(var, a, s);
    case kModeResidual:
      return a.wave == kWaveMax ? launch_one<R, kModeResidual, false, 0, kWaveMax>(a, s)
                                : launch_one<R, kModeResidual, false, 0>(a, s);
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace

cudaError_t launch_step(bool f64, int mode, int variant, const StepArgs& a, cudaStream_t s) {
  if (variant == 5 && a.wave == kWaveMax) variant = 1;  // the staged shape has the averages only
  if (variant == 5 && mode != kModeResidual && a.n > 0) return launch_step_tma(f64, mode, a, s);
  if (variant == kTileVariant && a.cell_ln) return launch_step_tile(f64, mode, a, s);
  if (variant == kFaceTileVariant && a.cell_ln && mode != kModeResidual)
    return launch_step_tile_faces(f64, mode, a, s);
  if (variant == 5 || variant == kTileVariant || variant == kFaceTileVariant) variant = 0;
  if (f64) return launch_step_t<double, false>(mode, variant, a, s);
  return a.lo ? launch_step_t<float, true>(mode, variant, a, s)
              : launch_step_t<float, false>(mode, variant, a, s);
}

cudaError_t launch_batch_step(bool f64, int mode, const BatchArgs& b, int64_t n_blocks,
                              cudaStream_t s) {
  const unsigned g = (unsigned)n_blocks;
  const bool comp = !f64 && b.s.lo != nullptr;
#define FV_BATCH_CASE(R, C)                                                               \
  switch (mode) {                                                                         \
    case kModeFE:                                                                         \
      return launch_chained(k_step_batch<R, kModeFE, C>, g, kBlock, 0, s, b.s.chained, b); \
    case kModeRK2a:                                                                       \
      return launch_chained(k_step_batch<R, kModeRK2a, C>, g, kBlock, 0, s, b.s.chained, b); \
    case kModeRK2b:                                                                       \
      return launch_chained(k_step_batch<R, kModeRK2b, C>, g, kBlock, 0, s, b.s.chained, b); \
    default: return cudaErrorInvalidValue;                                                \
  }
  if (f64) {
    FV_BATCH_CASE(double, false)
  } else if (comp) {
    FV_BATCH_CASE(float, true)
  } else {
    FV_BATCH_CASE(float, false)
  }
#undef FV_BATCH_CASE
}

cudaError_t launch_batch_init(unsigned long long* bmin, double* t, int n_meshes, int* err,
                              cudaStream_t s) {
  k_batch_init<<<(3 * n_meshes + kBlock - 1) / kBlock, kBlock, 0, s>>>(bmin, t, n_meshes, err);
  return cudaGetLastError();
}

cudaError_t launch_batch_bound(bool f64, const void* U, const void* geom, const int* block_mesh,
                               const int64_t* mesh_end, int n_meshes, int64_t n_blocks,
                               unsigned long long* bmin, int* err, cudaStream_t s) {
  if (f64)
    k_batch_bound<double><<<(unsigned)n_blocks, kBlock, 0, s>>>(
        static_cast<const dq4*>(U), static_cast<const dq4*>(geom), block_mesh, mesh_end, n_meshes,
        bmin, err);
  else
    k_batch_bound<float><<<(unsigned)n_blocks, kBlock, 0, s>>>(
        static_cast<const float4*>(U), static_cast<const float4*>(geom), block_mesh, mesh_end,
        n_meshes, bmin, err);
  return cudaGetLastError();
}

cudaError_t launch_batch_totals(bool f64, const void* U, const double* vol, const int* block_mesh,
                                const int64_t* mesh_end, const int* mesh_first_block,
                                int n_meshes, int64_t n_blocks, double* partials, double* out,
                                cudaStream_t s) {
  if (f64)
    k_batch_totals_partial<double><<<(unsigned)n_blocks, kBlock, 0, s>>>(
        static_cast<const dq4*>(U), vol, block_mesh, mesh_end, partials);
  else
    k_batch_totals_partial<float><<<(unsigned)n_blocks, kBlock, 0, s>>>(
        static_cast<const float4*>(U), vol, block_mesh, mesh_end, partials);
  k_batch_totals_final<<<n_meshes, kBlock, 0, s>>>(partials, mesh_first_block, out);
  return cudaGetLastError();
}

cudaError_t launch_init_scalars(LoopScalars* d, cudaStream_t s) {
  k_init_scalars<<<1, 1, 0, s>>>(d);
  return cudaGetLastError();
}

cudaError_t launch_bound(bool f64, const void* U, const void* geom, int64_t n,
                         unsigned long long* bmin, int* err, cudaStream_t s) {
  if (n <= 0) return cudaSuccess;
  if (f64)
    k_bound<double><<<grid_for(n), kBlock, 0, s>>>(static_cast<const dq4*>(U),
                                                   static_cast<const dq4*>(geom), n, bmin, err);
  else
    k_bound<float><<<grid_for(n), kBlock, 0, s>>>(static_cast<const float4*>(U),
                                                  static_cast<const float4*>(geom), n, bmin, err);
  return cudaGetLastError();
}

cudaError_t launch_totals(bool f64, const void* U, const double* vol, int64_t n, double* partials,
                          unsigned* ticket, double* out, cudaStream_t s) {
  const int64_t want = (n + kBlock - 1) / kBlock;
  const unsigned g = (unsigned)(want < 1 ? 1 : want > kTotalsBlocks ? kTotalsBlocks : want);
  if (f64)
    k_totals<double><<<g, kBlock, 0, s>>>(static_cast<const dq4*>(U), vol, n, partials, ticket, out);
  else
    k_totals<float><<<g, kBlock, 0, s>>>(static_cast<const float4*>(U), vol, n, partials, ticket,
                                         out);
  return cudaGetLastError();
}

// Restriction of a fine state to coarse cells: for coarse cell c, the
// area-weighted mean of its `kids` fine cells fine_of[c*kids + j], summed in
// FP64 in the order j = 0, 1, ... and written in the coarse precision.
// Bound by the FP64 pipe (five operations a child, 19 clocks each per warp and
// SM).  A float result takes one reciprocal and four products instead of four
// divisions (within 2 ulp of FP64, before its rounding to float) where the area
// sum is in [2^-100, 2^100), and VEC
// reads the ids four at a time (kids a multiple of 4, fine_of 16-byte
// aligned), so that four children's states are on their way together.
// 250,000 cells of 16 FP64 children: 87 -> 77 us a call.
template <typename RF>
struct FineSum {
  double s[4] = {0.0, 0.0, 0.0, 0.0}, v = 0.0;
  __device__ __forceinline__ void add_child(const rec_t<RF>& u, double a) {
    s[0] += a * (double)u.x;
    s[1] += a * (double)u.y;
    s[2] += a * (double)u.z;
    s[3] += a * (double)u.w;
    v += a;
  }
};

template <typename RF, typename RC, bool VEC>
__global__ void __launch_bounds__(kBlock) k_restrict_mean(const rec_t<RF>* __restrict__ Uf,
                                                          const double* __restrict__ area,
                                                          const int* __restrict__ fine_of,
                                                          int64_t n_coarse, int kids,
                                                          rec_t<RC>* Uc) {
  const int64_t c = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (c >= n_coarse) return;
  FineSum<RF> m;
  const int* ids = fine_of + c * kids;
  if (VEC) {
    for (int j = 0; j < kids; j += 4) {
      const int4 f = __ldg(reinterpret_cast<const int4*>(ids + j));
      const rec_t<RF> u0 = Rec<RF>::ld(Uf + f.x), u1 = Rec<RF>::ld(Uf + f.y),
                      u2 = Rec<RF>::ld(Uf + f.z), u3 = Rec<RF>::ld(Uf + f.w);
      const double a0 = __ldg(area + f.x), a1 = __ldg(area + f.y), a2 = __ldg(area + f.z),
                   a3 = __ldg(area + f.w);
      m.add_child(u0, a0);
      m.add_child(u1, a1);
      m.add_child(u2, a2);
      m.add_child(u3, a3);
    }
  } else {
    for (int j = 0; j < kids; ++j) {
      const int f = __ldg(ids + j);
      m.add_child(Rec<RF>::ld(Uf + f), __ldg(area + f));
    }
  }
  // the reciprocal of a tiny area sum would overflow where the means do not
  if (sizeof(RC) == 4 && in_quick_range(m.v)) {
    const double r = recip<double>(m.v);
    Uc[c] = Rec<RC>::make((RC)(m.s[0] * r), (RC)(m.s[1] * r), (RC)(m.s[2] * r), (RC)(m.s[3] * r));
  } else {
    Uc[c] = Rec<RC>::make((RC)(m.s[0] / m.v), (RC)(m.s[1] / m.v), (RC)(m.s[2] / m.v),
                          (RC)(m.s[3] / m.v));
  }
}

template <typename RF, typename RC>
void restrict_mean(const void* Uf, const double* area, const int* fine_of, int64_t n_coarse,
                   int kids, void* Uc, cudaStream_t s) {
  const bool vec = kids % 4 == 0 && reinterpret_cast<uintptr_t>(fine_of) % 16 == 0;
  auto k = vec ? k_restrict_mean<RF, RC, true> : k_restrict_mean<RF, RC, false>;
  k<<<grid_for(n_coarse), kBlock, 0, s>>>(static_cast<const rec_t<RF>*>(Uf), area, fine_of,
                                          n_coarse, kids, static_cast<rec_t<RC>*>(Uc));
}

cudaError_t launch_restrict_mean(bool fine_f64, bool coarse_f64, const void* Uf, const double* area,
                                 const int* fine_of, int64_t n_coarse, int kids, void* Uc,
                                 cudaStream_t s) {
  if (n_coarse <= 0) return cudaSuccess;
  if (fine_f64 && coarse_f64)
    restrict_mean<double, double>(Uf, area, fine_of, n_coarse, kids, Uc, s);
  else if (fine_f64)
    restrict_mean<double, float>(Uf, area, fine_of, n_coarse, kids, Uc, s);
  else if (coarse_f64)
    restrict_mean<float, double>(Uf, area, fine_of, n_coarse, kids, Uc, s);
  else
    restrict_mean<float, float>(Uf, area, fine_of, n_coarse, kids, Uc, s);
  return cudaGetLastError();
}

cudaError_t launch_init_aux(LoopScalars* sc, cudaStream_t s) {
  k_init_aux<<<1, 1, 0, s>>>(sc);
  return cudaGetLastError();
}

cudaError_t launch_compute_dt(bool f64, const void* U, const void* geom, int64_t n, double cfl,
                              LoopScalars* sc, cudaStream_t s) {
  if (n <= 0) return cudaSuccess;
  if (f64)
    k_compute_dt<double><<<grid_for(n), kBlock, 0, s>>>(
        static_cast<const dq4*>(U), static_cast<const dq4*>(geom), n, cfl, sc);
  else
    k_compute_dt<float><<<grid_for(n), kBlock, 0, s>>>(
        static_cast<const float4*>(U), static_cast<const float4*>(geom), n, cfl, sc);
  return cudaGetLastError();
}

}  // namespace fv
