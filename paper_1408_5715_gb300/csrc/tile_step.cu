// tile_step.cu -- one step per launch on tiles staged in shared memory (shape
// variant 6 of the step kernel).
//
// A block owns a tile of consecutive cells.  It loads the states of the tile
// and of its first halo ring (the cells outside the tile adjacent to it,
// tiles.cpp) into shared memory and forms their primitive variables (Eq. 2)
// once per cell; the one-thread-per-cell kernels form them once per face,
// i.e. four times per cell.  Each tile cell then sums its three face fluxes
// from the shared-memory neighbours and finishes exactly as the other shapes
// do (finish_cell: forward Euler, Heun's stages or the residual, plain or
// compensated), so all shapes give the same bits.  The FP64 step, bound by
// its division and square-root sequences, gains most.
#include <cuda_runtime.h>

#include <cstdint>

#include "cell_math.cuh"
#include "kernels.h"
#include "launch_util.cuh"
#include "tile_math.cuh"

namespace fv {

namespace {

// Barrier of a block's compute threads alone (without the warp of dt).
__device__ __forceinline__ void compute_sync(int threads) {
  asm volatile("bar.sync 1, %0;" ::"r"(threads) : "memory");
}

// VTX (FP32 only): normals from the grid coordinates of the tile's nodes,
// staged in shared memory after the states (vertex_geom.cpp), and 1/V from a
// 4-byte array, instead of each cell's 32-byte geometry record.
// FP32 keeps 1280 threads per SM resident (five blocks of 256: at most 48
// registers); FP64 needs its registers.
template <typename R, int MODE, bool COMP, int THREADS, int KMAX, int WAVE, bool VTX>
__global__ void __launch_bounds__(THREADS, sizeof(R) == 4 ? 1280 / THREADS : 1)
    k_step_tile(StepArgs a) {
  extern __shared__ __align__(128) unsigned char smem_raw[];
  rec_t<R>* sU = reinterpret_cast<rec_t<R>*>(smem_raw);  // [t1_cap] states
  rec_t<R>* sP = sU + a.t1_cap;                            // [t1_cap] (u, v, p, c)
  int2* sQ = reinterpret_cast<int2*>(sP + a.t1_cap);       // [v_cap] node grid coordinates
  const rec_t<R>* __restrict__ U = static_cast<const rec_t<R>*>(a.U);
  const rec_t<R>* __restrict__ geom = static_cast<const rec_t<R>*>(a.geom);
  rec_t<R>* out = static_cast<rec_t<R>*>(a.out);
  const int t0 = blockIdx.x * a.tile;  // cell ids are 32-bit
  const int nt = min(a.tile, (int)a.n - t0);
  const int hs = __ldg(a.tile_info + 2 * blockIdx.x);
  const int h1 = __ldg(a.tile_info + 2 * blockIdx.x + 1);
  chain_entry();
  // dt formed once per block (FP64 scalar work), read after the barrier
  __shared__ double s_t, s_dt;
  if (threadIdx.x == 0 && MODE != kModeResidual) block_dt(a, s_t, s_dt);
  // the tile's node coordinates: loads issued with the states', stored after
  constexpr int VA = KMAX / 2 + 1;  // per thread: 3 x 256 for the ~600 nodes of 1024 cells
  int2 qv[VTX ? VA : 1];
  int vb = 0, nv = 0;
  if constexpr (VTX) {
    vb = __ldg(a.tile_voff + blockIdx.x);
    nv = __ldg(a.tile_voff + blockIdx.x + 1) - vb;
#pragma unroll
    for (int k = 0; k < VA; ++k) {
      const int e = threadIdx.x + k * THREADS;
      if (e < nv) qv[k] = __ldg(a.tile_vq + vb + e);
    }
  }
  stage_states<R, THREADS, kStageBatch<R, KMAX>>(U, t0, nt, h1, a.halo_id + hs, sU, sP, a.n,
                                                 a.err);
  if constexpr (VTX) {
#pragma unroll
    for (int k = 0; k < VA; ++k) {
      const int e = threadIdx.x + k * THREADS;
      if (e < nv) sQ[e] = qv[k];
    }
    for (int e = threadIdx.x + VA * THREADS; e < nv; e += THREADS) sQ[e] = __ldg(a.tile_vq + vb + e);
  }
  __syncthreads();
  const double t = MODE != kModeResidual ? s_t : 0.0, dt = MODE != kModeResidual ? s_dt : 0.0;
  const R dtR = R(dt);
  R bmin = R(INFINITY);
  bool ok = true;
#pragma unroll
  for (int k = 0; k < KMAX; ++k) {
    const int e = threadIdx.x + k * THREADS;
    if (e < nt) {
      const int i = t0 + e;
      CellIn<R> c;
      const uint2 ln = __ldg(a.cell_ln + i);
      if constexpr (VTX) {
        const unsigned vl = __ldg(a.cell_vl + i);
        // node ids index the nv staged nodes (checked in the bounds-checked build)
        auto node = [&](unsigned q) { return index_ok(q, nv, a.err) ? sQ[q] : make_int2(0, 0); };
        vertex_geometry(node(ln.y >> 16), node(vl & 0xffffu), node(vl >> 16), a.vscale,
                        __ldg(a.inv_vol + i), c.g0, c.g1);
      } else {
        c.g0 = Rec<R>::ld(geom + 2 * i);
        c.g1 = Rec<R>::ld(geom + 2 * i + 1);
      }
      c.U = sU[e];
      if (MODE == kModeRK2b) c.base = static_cast<const rec_t<R>*>(a.Ubase)[i];
      if (COMP && MODE != kModeResidual) c.lo = a.lo[i];
      if (COMP && MODE == kModeRK2b) c.lo_stage = a.lo_stage[i];
      R acc[4] = {R(0), R(0), R(0), R(0)};
      const R perim = cell_fluxes<R, WAVE>(c.g0, c.g1, ln, c.U, rec_prim<R>(sP[e]), sU, sP,
                                           far_field<R>(a), acc, nt + h1, a.err);
      finish_cell<R, MODE, COMP>(a, out, i, c, acc, perim, dtR, bmin, ok);
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

// The tile shape for tiles that are all resident at a time, one cell per
// thread (FP32, up to kQuickTile cells).  A step of such a mesh (some 12,000 to
// 150,000 cells) is a chain of latencies, so what does not depend on the
// previous step is done while that still runs: the kernel lets its successor
// start at once (griddepcontrol.launch_dependents; the successor's blocks fit
// beside it), which loads the tile's tables and its threads' geometry and then
// waits for this grid's end.  One warp forms dt (FP64, some 400 clocks) while
// the others load states, form primitives and sum fluxes.
// Measured (us per step, compensated, tiles of 128; k_step_tile -> this):
// 16,384 cells 2.67 -> 2.08, 41,410 2.98 -> 2.30, 65,536 3.23 -> 2.47.
template <int MODE, bool COMP, int WAVE>
__global__ void __launch_bounds__(kQuickTile + 32, 4) k_step_tile_quick(StepArgs a) {
  extern __shared__ __align__(128) unsigned char smem_raw[];
  float4* sU = reinterpret_cast<float4*>(smem_raw);  // [t1_cap] states
  float4* sP = sU + a.t1_cap;                          // [t1_cap] (u, v, p, c)
  __shared__ float s_dt, s_min[kQuickTile / 32];
  const int threads = blockDim.x - 32, tid = threadIdx.x, lane = tid & 31;
  constexpr bool kBound = MODE != kModeRK2a;
  if (tid >= threads) {  // the warp of dt
    chain_entry();
    chain_next();
    double t, dt;
    block_dt(a, t, dt);
    if (lane == 0) s_dt = (float)dt;
    __syncthreads();
    if (!kBound) return;
    if (blockIdx.x == 0 && lane == 0) {
      *a.t_write = t + dt;
      *a.bmin_reset = kInfBits;
    }
    __syncthreads();  // the warps' minima are there
    float m = lane < threads / 32 ? s_min[lane] : INFINITY;
    m = __uint_as_float(__reduce_min_sync(0xffffffffu, __float_as_uint(m)));  // positive or inf
    if (lane == 0) atomicMin(a.bmin_write, (unsigned long long)__double_as_longlong((double)m));
    return;
  }
  const float4* __restrict__ geom = static_cast<const float4*>(a.geom);
  const float4* U = static_cast<const float4*>(a.U);  // written by the previous grid
  float4* out = static_cast<float4*>(a.out);
  const int t0 = blockIdx.x * a.tile;
  const int nt = min(a.tile, (int)a.n - t0);
  const int hs = __ldg(a.tile_info + 2 * blockIdx.x);
  const int h1 = __ldg(a.tile_info + 2 * blockIdx.x + 1);
  const int i = t0 + tid;
  const bool has = tid < nt;
  CellIn<float> c{};
  uint2 ln = make_uint2(0u, 0u);
  if (has) {
    c.g0 = __ldg(geom + 2 * i);
    c.g1 = __ldg(geom + 2 * i + 1);
    ln = __ldg(a.cell_ln + i);
  }
  int g = tid < h1 ? __ldg(a.halo_id + hs + tid) : 0;
  if (!index_ok(g, a.n, a.err)) g = t0;
  chain_entry();
  chain_next();
  if (has) {
    c.U = U[i];
    if (MODE == kModeRK2b) c.base = static_cast<const float4*>(a.Ubase)[i];
    if (COMP) c.lo = a.lo[i];
    if (COMP && MODE == kModeRK2b) c.lo_stage = a.lo_stage[i];
  }
  float4 halo = make_float4(1.f, 0.f, 0.f, 1.f);
  if (tid < h1) halo = U[g];
  Prim<float> L{};
  if (has) {
    L = primitive<float>(c.U);
    sU[tid] = c.U;
    sP[tid] = prim_rec<float>(L);
  }
  if (tid < h1) {
    sU[nt + tid] = halo;
    sP[nt + tid] = prim_rec<float>(primitive<float>(halo));
  }
  for (int e = tid + threads; e < h1; e += threads) {  // a ring larger than the tile
    const float4 u = U[staged_id<float>(t0, nt, nt + e, a.halo_id + hs, a.n, a.err)];
    sU[nt + e] = u;
    sP[nt + e] = prim_rec<float>(primitive<float>(u));
  }
  compute_sync(threads);
  float acc[4] = {0.f, 0.f, 0.f, 0.f}, perim = 0.f;
  if (has)
    perim = cell_fluxes<float, WAVE>(c.g0, c.g1, ln, c.U, L, sU, sP, a.uinf_f, acc, nt + h1, a.err);
  __syncthreads();  // dt is there
  bool ok = true;
  float bmin = INFINITY;
  if (has) finish_cell<float, MODE, COMP>(a, out, i, c, acc, perim, s_dt, bmin, ok);
  if (!kBound) return;
  if (!ok) atomicOr(a.err, 1);
  bmin = __uint_as_float(__reduce_min_sync(0xffffffffu, __float_as_uint(bmin)));
  if (lane == 0) s_min[tid >> 5] = bmin;
  __syncthreads();
}

// Shape 7: the tile shape with each face evaluated once.  Phase 1: the
// threads share the tile's face list (tiles.cpp): every face of a tile cell
// except those whose other side is a tile cell of lower local id (for a cell
// bordering itself across a periodic seam, its lower face); each writes the
// flux value to the slot sF[3e + q] of its cell and, across an inner face,
// the negation to the slot of the face pointing back.  The face
// fluxes are exactly antisymmetric (face_flux_value), so every slot holds the
// bits the cell would compute itself.  Phase 2: every tile cell adds its three
// slots in face order and finishes as the other shapes do: the same bits, with
// about half the face arithmetic.  sF costs 3 records per tile cell of shared
// memory.  It pays where the arithmetic is the bottleneck, in FP64, which has a
// kernel of its own (k_step_faces64); this one is FP32's.
template <typename R, int MODE, bool COMP, int THREADS, int KMAX, int WAVE>
__global__ void __launch_bounds__(THREADS, 1) k_step_tile_faces(StepArgs a) {
  static_assert(sizeof(R) == 4);
  extern __shared__ __align__(128) unsigned char smem_raw[];
  rec_t<R>* sU = reinterpret_cast<rec_t<R>*>(smem_raw);  // [t1_cap] states
  rec_t<R>* sP = sU + a.t1_cap;                            // [t1_cap] (u, v, p, c)
  rec_t<R>* sF = sP + a.t1_cap;                            // [3 tile] face flux values
  const rec_t<R>* __restrict__ U = static_cast<const rec_t<R>*>(a.U);
  const rec_t<R>* __restrict__ geom = static_cast<const rec_t<R>*>(a.geom);
  rec_t<R>* out = static_cast<rec_t<R>*>(a.out);
  const int t0 = blockIdx.x * a.tile;  // cell ids are 32-bit
  const int nt = min(a.tile, (int)a.n - t0);
  const int hs = __ldg(a.tile_info + 2 * blockIdx.x);
  const int h1 = __ldg(a.tile_info + 2 * blockIdx.x + 1);
  chain_entry();
  __shared__ double s_t, s_dt;
  if (threadIdx.x == 0 && MODE != kModeResidual) block_dt(a, s_t, s_dt);
  stage_states<R, THREADS, kStageBatch<R, KMAX>>(U, t0, nt, h1, a.halo_id + hs, sU, sP, a.n,
                                                 a.err);
  __syncthreads();
  const R* uinf = far_field<R>(a);
  // phase 1: the tile's faces, each once, spread evenly over the threads
  const int f1 = __ldg(a.tile_face_off + blockIdx.x + 1);
  for (int f = __ldg(a.tile_face_off + blockIdx.x) + threadIdx.x; f < f1; f += THREADS) {
    const uint2 r = __ldg(a.tile_face + f);
    const unsigned e = r.x & 0xffffu, q = (r.x >> 16) & 3u, kv = (r.x >> 18) & 3u, v = r.y;
    if (!index_ok(e, nt, a.err)) continue;
    const int i = t0 + (int)e;
    R nx, ny;
    face_normal<R>(geom, i, q, nx, ny);
    const rec_t<R> UL = sU[e];
    const Prim<R> L = rec_prim<R>(sP[e]);
    const bool inner = v < (unsigned)nt;
    rec_t<R> UR;
    Prim<R> W;
    if (v < kGhostCodes) {
      if (index_ok(v, nt + h1, a.err)) {
        UR = sU[v];
        W = rec_prim<R>(sP[v]);
      } else {
        UR = UL;
        W = L;
      }
    } else {
      UR = ghost<R>((int)v - 0x10000, UL, nx, ny, uinf);
      W = primitive<R>(UR);
    }
    R X[4];
    face_flux_value<R, false, WAVE>(UL, L, UR, W, nx, ny, face_len<R>(nx, ny), R(1), X);
    sF[3 * e + q] = Rec<R>::make(X[0], X[1], X[2], X[3]);
    if (inner) sF[3 * v + kv] = Rec<R>::make(-X[0], -X[1], -X[2], -X[3]);
  }
  __syncthreads();
  const double t = MODE != kModeResidual ? s_t : 0.0, dt = MODE != kModeResidual ? s_dt : 0.0;
  const R dtR = R(dt);
  R bmin = R(INFINITY);
  bool ok = true;
  // phase 2: the three face values in face order, then the cell's update
#pragma unroll
  for (int k = 0; k < KMAX; ++k) {
    const int e = threadIdx.x + k * THREADS;
    if (e < nt) {
      const int i = t0 + e;
      CellIn<R> c;
      c.g0 = Rec<R>::ld(geom + 2 * i);
      c.g1 = Rec<R>::ld(geom + 2 * i + 1);
      c.U = sU[e];
      if (MODE == kModeRK2b) c.base = static_cast<const rec_t<R>*>(a.Ubase)[i];
      if (COMP && MODE != kModeResidual) c.lo = a.lo[i];
      if (COMP && MODE == kModeRK2b) c.lo_stage = a.lo_stage[i];
      R acc[4] = {R(0), R(0), R(0), R(0)};
#pragma unroll
      for (int q = 0; q < 3; ++q) {
        const rec_t<R> X = sF[3 * e + q];
        acc[0] = add(acc[0], X.x);
        acc[1] = add(acc[1], X.y);
        acc[2] = add(acc[2], X.z);
        acc[3] = add(acc[3], X.w);
      }
      // the perimeter (FP32 forms 2V/P from it; FP64 stores 2V/P)
      R perim = R(0);
      if constexpr (sizeof(R) == 4)
        perim = add(add(face_len<R>(c.g0.x, c.g0.y), face_len<R>(c.g0.z, c.g0.w)),
                    face_len<R>(c.g1.x, c.g1.y));
      finish_cell<R, MODE, COMP>(a, out, i, c, acc, perim, dtR, bmin, ok);
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

// x with its sign bit changed by `sign` (0 or 0x80000000), without the FP64 pipe.
__device__ __forceinline__ double flip(double x, unsigned sign) {
  return __hiloint2double(__double2hiint(x) ^ (int)sign, __double2loint(x));
}

// A CFL bound in FP32 that rules most cells out of the FP64 minimum: within
// kBoundSlack of the exact bound of a cell whose state is plainly good (true),
// else the cell has to be evaluated exactly.
constexpr float kBoundSlack = 1e-4f;

// x to float by integer shifts (a conversion takes the FP64 pipe as long as an
// addition): rounded toward zero, 0 below 2^-100; big is set from 2^100 on.
__device__ __forceinline__ float rough_float(double x, bool& big) {
  const unsigned hi = (unsigned)__double2hiint(x), mag = hi & 0x7fffffffu;
  const unsigned w = __funnelshift_l((unsigned)__double2loint(x), hi, 3);
  big = big || mag >= (1123u << 20);
  const unsigned f = ((w ^ 0x40000000u) & 0x7fffffffu) | (hi & 0x80000000u);
  return mag < (923u << 20) ? 0.0f : __uint_as_float(f);
}

__device__ __forceinline__ bool rough_bound(const dq4& U, double inradius, float& b) {
  bool big = false;
  const float rho = rough_float(U.x, big), mx = rough_float(U.y, big), my = rough_float(U.z, big),
              E = rough_float(U.w, big), r = rough_float(inradius, big);
  const float ir = recip<float>(rho), u = mx * ir, v = my * ir;
  const float pe = E - 0.5f * (mx * u + my * v);  // p / (gamma - 1)
  const float vv = u * u + v * v, cc = (float)(kGamma * kGammaM1) * pe * ir;
  b = r * recip<float>(root<float>(vv) + root<float>(cc));
  // rounding moves pe by at most a few 2^-23 E: at pe > E / 100 the sound
  // speed is good to 4e-5, and the exact pressure is positive too.  The squares
  // and the bound have limits of their own: speeds of ordinary rho and pe can
  // leave the floats' range (then b would be 0 or infinite), and at cc > 1e-24
  // what vv loses below the normal floats is nothing beside c
  return !big && rho > 1e-20f && rho < 1e20f && E < 1e20f && pe > 0.01f * E && pe > 1e-20f &&
         r > 1e-20f && vv < 1e30f && cc > 1e-24f && cc < 1e30f && b < 1e38f;
}

// Shape 7 in FP64, bound by the FP64 pipe (two lanes a clock and SM): 84 % of
// it busy with 173 FP64 instructions per cell in the form above, of which the
// fluxes are a third.  What is not the fluxes' is taken out:
//   - a face's record carries its normal and length (32 bytes, read in order),
//     so no square root per face; boundary faces come last in a tile's list,
//     so that few warps evaluate ghost states; a face's flux is stored once and
//     the cells find theirs by reference (51 bytes of shared memory a cell
//     instead of 96 for a slot per side: one more block per SM);
//   - the CFL bound (two square roots, two divisions) is evaluated only for
//     cells that may be the minimum: an FP32 bound of every cell, the block's
//     minimum of those, and FP64 for the cells within the FP32 error of it --
//     unless the minimum so far already rules the block out.  The minimum is
//     that of the exact bounds, whatever the order;
//   - reciprocals and square roots start from FP32 (recip, root).
// A small mesh is bound by latency instead (a dependent FP64 operation takes
// 64 clocks): the tile's tables and each thread's first face are read before
// the previous step ends, the blocks have about a thread per face, and one more
// warp forms dt.
// Measured (us per step): channel of 250,000 cells, autotuned, 89 -> 46;
// square of 12,800 cells 18.3 (shape 1) -> 6.3.
template <int MODE, int THREADS, int KMAX, int WAVE>
__global__ void __launch_bounds__(THREADS + 32) k_step_faces64(StepArgs a) {
  extern __shared__ __align__(128) unsigned char smem_raw[];
  // 16-byte halves of the records in arrays of their own (no bank conflicts):
  // states and (u, v, p, c) of tile and ring, flux values of the tile's faces
  double2* sU[2];
  double2* sP[2];
  double2* sF[2];
  sU[0] = reinterpret_cast<double2*>(smem_raw);
  sU[1] = sU[0] + a.t1_cap;
  sP[0] = sU[1] + a.t1_cap;
  sP[1] = sP[0] + a.t1_cap;
  sF[0] = sP[1] + a.t1_cap;
  sF[1] = sF[0] + a.f_cap;
  auto get = [](double2* const h[2], unsigned e) {
    const double2 x = h[0][e], y = h[1][e];
    return dq4{x.x, x.y, y.x, y.y};
  };
  auto put = [](double2* const h[2], unsigned e, const dq4& r) {
    h[0][e] = make_double2(r.x, r.y);
    h[1][e] = make_double2(r.z, r.w);
  };
  __shared__ double s_dt;
  __shared__ float s_so_far, s_min[THREADS / 32];
  constexpr bool kBound = MODE != kModeRK2a;
  const int tid = threadIdx.x;
  if (tid >= THREADS) {  // the warp of dt
    chain_entry();
    double t, dt;
    block_dt(a, t, dt);
    if (tid == THREADS) {
      s_dt = dt;
      if (kBound)  // the minimum already found by other blocks
        s_so_far = (float)__longlong_as_double(
            (long long)*static_cast<volatile unsigned long long*>(a.bmin_write));
    }
    __syncthreads();
    if (kBound && blockIdx.x == 0 && tid == THREADS) {
      *a.t_write = t + dt;
      *a.bmin_reset = kInfBits;
    }
    if (kBound) __syncthreads();
    return;
  }
  const dq4* U = static_cast<const dq4*>(a.U);  // written by the previous grid
  const double2* __restrict__ geom = static_cast<const double2*>(a.geom);
  const double2* __restrict__ faces = reinterpret_cast<const double2*>(a.tile_face);
  dq4* out = static_cast<dq4*>(a.out);
  const int t0 = blockIdx.x * a.tile;  // cell ids are 32-bit
  const int nt = min(a.tile, (int)a.n - t0);
  const int hs = __ldg(a.tile_info + 2 * blockIdx.x);
  const int h1 = __ldg(a.tile_info + 2 * blockIdx.x + 1);
  const int f0 = __ldg(a.tile_face_off + blockIdx.x);
  int f = f0 + tid;
  const int f1 = __ldg(a.tile_face_off + blockIdx.x + 1);
  const int first = tid < nt + h1 ? (int)staged_id<double>(t0, nt, tid, a.halo_id + hs, a.n, a.err) : 0;
  double2 nrm{}, lr{}, g_first{};
  if (f < f1) nrm = __ldg(faces + 2 * (int64_t)f), lr = __ldg(faces + 2 * (int64_t)f + 1);
  uint2 ref_first = make_uint2(0u, 0u);
  if (tid < nt) {
    g_first = __ldg(geom + 4 * (int64_t)(t0 + tid) + 3);  // 1/V, 2V/P
    ref_first = __ldg(a.cell_ref + t0 + tid);
  }
  chain_entry();
  for (int e = tid; e < nt + h1; e += THREADS) {
    const int64_t i =
        e == tid ? first : staged_id<double>(t0, nt, e, a.halo_id + hs, a.n, a.err);
    const double2 x = reinterpret_cast<const double2*>(U + i)[0],
                  y = reinterpret_cast<const double2*>(U + i)[1];
    const dq4 u{x.x, x.y, y.x, y.y};
    put(sU, e, u);
    put(sP, e, prim_rec<double>(primitive<double>(u)));
  }
  compute_sync(THREADS);
  // phase 1: the tile's faces, each once, spread evenly over the threads, the
  // next record read ahead
  while (f < f1) {
    const double2 n_cur = nrm, l_cur = lr;
    const int slot = f - f0;
    f += THREADS;
    if (f < f1) nrm = __ldg(faces + 2 * (int64_t)f), lr = __ldg(faces + 2 * (int64_t)f + 1);
    const unsigned rx = (unsigned)__double2loint(l_cur.y), v = (unsigned)__double2hiint(l_cur.y);
    const unsigned e = rx & 0xffffu;
    if (!index_ok(e, nt, a.err)) continue;
    const dq4 UL = get(sU, e);
    const Prim<double> L = rec_prim<double>(get(sP, e));
    dq4 UR = UL;
    Prim<double> W = L;
    if (v < kGhostCodes) {
      if (index_ok(v, nt + h1, a.err)) {
        UR = get(sU, v);
        W = rec_prim<double>(get(sP, v));
      }
    } else {
      UR = ghost<double>((int)v - 0x10000, UL, n_cur.x, n_cur.y, a.uinf);
      W = primitive<double>(UR);
    }
    double X[4];
    face_flux_value<double, false, WAVE>(UL, L, UR, W, n_cur.x, n_cur.y, l_cur.x, 1.0, X);
    put(sF, slot, dq4{X[0], X[1], X[2], X[3]});
  }
  __syncthreads();
  const double dt = s_dt;
  bool ok = true;
  double2 g[KMAX];
  uint2 ref[KMAX];
  float rough[KMAX];
  float least = INFINITY;
  unsigned exact = 0u;  // cells (bit k) to be evaluated in FP64 whatever the minimum
#pragma unroll
  for (int k = 0; k < KMAX; ++k) {
    const int e = tid + k * THREADS;
    g[k] = g_first;
    ref[k] = ref_first;
    if (k > 0 && e < nt) {
      g[k] = __ldg(geom + 4 * (int64_t)(t0 + e) + 3);
      ref[k] = __ldg(a.cell_ref + t0 + e);
    }
  }
  // phase 2: the three face values in face order, then the cell's update
#pragma unroll
  for (int k = 0; k < KMAX; ++k) {
    const int e = tid + k * THREADS;
    rough[k] = INFINITY;
    if (e < nt) {
      const int i = t0 + e;
      dq4 base{};
      if (MODE == kModeRK2b) base = static_cast<const dq4*>(a.Ubase)[i];
      // the faces in order, as every shape adds them
      auto flux = [&](unsigned r) {  // bit 15: the face was evaluated from the other side
        const unsigned at = r & 0x7fffu, sign = (r & 0x8000u) << 16;
        const dq4 x = get(sF, index_ok(at, a.f_cap, a.err) ? at : 0u);
        return dq4{flip(x.x, sign), flip(x.y, sign), flip(x.z, sign), flip(x.w, sign)};
      };
      const dq4 X0 = flux(ref[k].x & 0xffffu), X1 = flux(ref[k].x >> 16),
                X2 = flux(ref[k].y & 0xffffu);
      const double acc[4] = {add(add(X0.x, X1.x), X2.x), add(add(X0.y, X1.y), X2.y),
                             add(add(X0.z, X1.z), X2.z), add(add(X0.w, X1.w), X2.w)};
      uint2 none;
      const dq4 Un =
          advance_state<double, MODE, false>(get(sU, e), base, acc, g[k].x, dt, none, none, none);
      out[i] = Un;
      if (kBound) {
        put(sU, e, Un);  // this thread's own entry from here on
        if (rough_bound(Un, g[k].y, rough[k]))
          least = fminf(least, rough[k]);
        else
          exact |= 1u << k;
      }
    }
  }
  if (!kBound) return;
  least = __uint_as_float(__reduce_min_sync(0xffffffffu, __float_as_uint(least)));  // positive
  if ((tid & 31) == 0) s_min[tid >> 5] = least;
  __syncthreads();
  least = s_so_far;
#pragma unroll
  for (int w = 0; w < THREADS / 32; ++w) least = fminf(least, s_min[w]);
  const float limit = least * (1.0f + 4.0f * kBoundSlack);
  double bmin = INFINITY;
#pragma unroll
  for (int k = 0; k < KMAX; ++k) {
    const int e = tid + k * THREADS;
    if (e < nt && (((exact >> k) & 1u) || rough[k] <= limit)) {
      bool c_ok;
      bmin = fmin(bmin, cell_bound<double>(get(sU, e), g[k].y, c_ok));
      ok = ok && c_ok;
    }
  }
  if (!ok) atomicOr(a.err, 1);
  if (__any_sync(0xffffffffu, bmin < INFINITY)) {
    for (int o = 16; o > 0; o >>= 1) bmin = fmin(bmin, __shfl_xor_sync(0xffffffffu, bmin, o));
    if ((tid & 31) == 0) atomicMin(a.bmin_write, (unsigned long long)__double_as_longlong(bmin));
  }
}

// The face records of k_step_faces64, a block per tile (once per mesh and tile
// size); the length is face_len's, as every other kernel forms it.
__global__ void k_face_records(const dq4* __restrict__ geom, const int* __restrict__ face_off,
                               const uint2* __restrict__ words, int tile, dq4* records) {
  const int f1 = face_off[blockIdx.x + 1];
  for (int f = face_off[blockIdx.x] + threadIdx.x; f < f1; f += blockDim.x) {
    const uint2 w = words[f];
    double nx, ny;
    face_normal<double>(geom, (int)blockIdx.x * tile + (int)(w.x & 0xffffu), (w.x >> 16) & 3u, nx,
                        ny);
    records[f] = dq4{nx, ny, face_len<double>(nx, ny), __hiloint2double((int)w.y, (int)w.x)};
  }
}

// Many meshes: each block is one tile of one mesh (tiles never span meshes)
// and uses that mesh's dt, time, far field and CFL-minimum slot; the mesh's
// first tile advances its time and clears its next slot.
template <typename R, int MODE, bool COMP, int THREADS, int KMAX>
__global__ void __launch_bounds__(THREADS) k_step_tile_batch(BatchArgs b) {
  const StepArgs& a = b.s;
  extern __shared__ __align__(128) unsigned char smem_raw[];
  rec_t<R>* sU = reinterpret_cast<rec_t<R>*>(smem_raw);  // [t1_cap] states
  rec_t<R>* sP = sU + a.t1_cap;                            // [t1_cap] (u, v, p, c)
  const rec_t<R>* __restrict__ U = static_cast<const rec_t<R>*>(a.U);
  const rec_t<R>* __restrict__ geom = static_cast<const rec_t<R>*>(a.geom);
  rec_t<R>* out = static_cast<rec_t<R>*>(a.out);
  const int tile = blockIdx.x;
  const int m = __ldg(b.tile_mesh + tile);
  const int64_t t0 = __ldg(b.tile_start + tile);
  const int nt = __ldg(b.tile_cells + tile);
  const int hs = __ldg(a.tile_info + 2 * tile);
  const int h1 = __ldg(a.tile_info + 2 * tile + 1);
  chain_entry();
  __shared__ double s_t, s_dt;
  if (threadIdx.x == 0) batch_dt(b, m, s_t, s_dt);
  stage_states<R, THREADS, kStageBatch<R, KMAX>>(U, t0, nt, h1, a.halo_id + hs, sU, sP, a.n,
                                                 a.err);
  __syncthreads();
  const double t = MODE != kModeResidual ? s_t : 0.0, dt = MODE != kModeResidual ? s_dt : 0.0;
  const R dtR = R(dt);
  const R* uinf = batch_far_field<R>(b, m);
  R bmin = R(INFINITY);
  bool ok = true;
#pragma unroll
  for (int k = 0; k < KMAX; ++k) {
    const int e = threadIdx.x + k * THREADS;
    if (e < nt) {
      const int64_t i = t0 + e;
      CellIn<R> c;
      c.g0 = Rec<R>::ld(geom + 2 * i);
      c.g1 = Rec<R>::ld(geom + 2 * i + 1);
      c.U = sU[e];
      if (MODE == kModeRK2b) c.base = static_cast<const rec_t<R>*>(a.Ubase)[i];
      if (COMP && MODE != kModeResidual) c.lo = a.lo[i];
      if (COMP && MODE == kModeRK2b) c.lo_stage = a.lo_stage[i];
      const uint2 ln = __ldg(a.cell_ln + i);
      R acc[4] = {R(0), R(0), R(0), R(0)};
      const R perim =
          cell_fluxes<R>(c.g0, c.g1, ln, c.U, rec_prim<R>(sP[e]), sU, sP, uinf, acc, nt + h1, a.err);
      finish_cell<R, MODE, COMP>(a, out, i, c, acc, perim, dtR, bmin, ok);
    }
  }
  if (MODE == kModeFE || MODE == kModeRK2b) {
    if (!ok) atomicOr(a.err, 1);
    const double mn = (double)block_min<R>(bmin);
    if (threadIdx.x == 0) {
      atomicMin(&b.bmin[b.slot_write * b.n_meshes + m], (unsigned long long)__double_as_longlong(mn));
      if (tile == __ldg(b.mesh_first_tile + m)) {
        b.t[b.t_write * b.n_meshes + m] = t + dt;
        b.bmin[b.slot_reset * b.n_meshes + m] = kInfBits;
      }
    }
  }
}

template <typename R, int MODE, bool COMP, int THREADS, int KMAX>
cudaError_t launch_tile_batch_t(const BatchArgs& b, cudaStream_t s) {
  auto k = k_step_tile_batch<R, MODE, COMP, THREADS, KMAX>;
  const size_t smem = tile_smem_bytes(sizeof(R) == 8, b.s.t1_cap);
  cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  return launch_chained(k, (unsigned)b.n_tiles, THREADS, smem, s, b.s.chained, b);
}

template <typename R, bool COMP>
cudaError_t launch_tile_batch_mode(int mode, const BatchArgs& b, cudaStream_t s) {
  if (b.s.tile != 1024) return cudaErrorInvalidValue;
  switch (mode) {
    case kModeFE: return launch_tile_batch_t<R, kModeFE, COMP, 256, 4>(b, s);
    case kModeRK2a: return launch_tile_batch_t<R, kModeRK2a, COMP, 256, 4>(b, s);
    case kModeRK2b: return launch_tile_batch_t<R, kModeRK2b, COMP, 256, 4>(b, s);
    default: return cudaErrorInvalidValue;
  }
}

template <typename R, int MODE, bool COMP, int THREADS, int KMAX, bool VTX>
cudaError_t launch_tile_t(const StepArgs& a, cudaStream_t s) {
  auto k = a.wave == kWaveMax ? k_step_tile<R, MODE, COMP, THREADS, KMAX, kWaveMax, VTX>
                              : k_step_tile<R, MODE, COMP, THREADS, KMAX, kWaveAverage, VTX>;
  const size_t smem = tile_smem_bytes(sizeof(R) == 8, a.t1_cap, VTX ? a.v_cap : 0);
  cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  const int64_t tiles = (a.n + a.tile - 1) / a.tile;
  return launch_chained(k, (unsigned)tiles, THREADS, smem, s, a.chained, a);
}

template <typename R, int MODE, bool COMP, int THREADS, int KMAX>
cudaError_t launch_faces_t(const StepArgs& a, cudaStream_t s) {
  void (*k)(StepArgs);
  if constexpr (sizeof(R) == 8)
    k = a.wave == kWaveMax ? k_step_faces64<MODE, THREADS, KMAX, kWaveMax>
                           : k_step_faces64<MODE, THREADS, KMAX, kWaveAverage>;
  else
    k = a.wave == kWaveMax ? k_step_tile_faces<R, MODE, COMP, THREADS, KMAX, kWaveMax>
                           : k_step_tile_faces<R, MODE, COMP, THREADS, KMAX, kWaveAverage>;
  const size_t smem = tile_faces_smem_bytes(sizeof(R) == 8, a.t1_cap, a.tile, a.f_cap);
  cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  const int64_t tiles = (a.n + a.tile - 1) / a.tile;
  return launch_chained(k, (unsigned)tiles, sizeof(R) == 8 ? THREADS + 32 : THREADS, smem, s,
                        a.chained, a);
}

template <typename R, int MODE, bool COMP>
cudaError_t launch_faces_size(const StepArgs& a, cudaStream_t s) {
  if (a.tile < 1 || a.tile > kMaxTileCells) return cudaErrorInvalidValue;
  if constexpr (sizeof(R) == 8) {
    // small tiles: about a thread per face
    if (a.tile <= 32) return launch_faces_t<R, MODE, COMP, 64, 1>(a, s);
    if (a.tile <= 64) return launch_faces_t<R, MODE, COMP, 128, 1>(a, s);
    if (a.tile <= 112) return launch_faces_t<R, MODE, COMP, 192, 1>(a, s);
    if (a.tile <= 256) return launch_faces_t<R, MODE, COMP, 256, 1>(a, s);
  }
  if (a.tile <= 512) return launch_faces_t<R, MODE, COMP, 256, 2>(a, s);
  if (a.tile <= 768) return launch_faces_t<R, MODE, COMP, 256, 3>(a, s);
  if (a.tile <= 1024) return launch_faces_t<R, MODE, COMP, 256, 4>(a, s);
  return launch_faces_t<R, MODE, COMP, 512, 4>(a, s);
}

template <typename R, bool COMP>
cudaError_t launch_faces_mode(int mode, const StepArgs& a, cudaStream_t s) {
  switch (mode) {
    case kModeFE: return launch_faces_size<R, kModeFE, COMP>(a, s);
    case kModeRK2a: return launch_faces_size<R, kModeRK2a, COMP>(a, s);
    case kModeRK2b: return launch_faces_size<R, kModeRK2b, COMP>(a, s);
    default: return cudaErrorInvalidValue;
  }
}

template <int MODE, bool COMP>
cudaError_t launch_quick(const StepArgs& a, cudaStream_t s) {
  auto k = a.wave == kWaveMax ? k_step_tile_quick<MODE, COMP, kWaveMax>
                              : k_step_tile_quick<MODE, COMP, kWaveAverage>;
  const unsigned tiles = (unsigned)((a.n + a.tile - 1) / a.tile);
  return launch_chained(k, tiles, (unsigned)((a.tile + 31) / 32 * 32 + 32),
                        tile_smem_bytes(false, a.t1_cap), s, a.chained, a);
}

// Any tile size up to 2048 cells: the block shape whose KMAX x THREADS cells
// cover it (the cells of a tile beyond nt are skipped).
template <typename R, int MODE, bool COMP, bool VTX>
cudaError_t launch_tile_size(const StepArgs& a, cudaStream_t s) {
  if (a.tile < 1 || a.tile > kMaxTileCells) return cudaErrorInvalidValue;
  if constexpr (sizeof(R) == 4 && !VTX && MODE != kModeResidual)
    if (a.quick) return launch_quick<MODE, COMP>(a, s);
  if (a.tile <= 512) return launch_tile_t<R, MODE, COMP, 256, 2, VTX>(a, s);
  if (a.tile <= 768) return launch_tile_t<R, MODE, COMP, 256, 3, VTX>(a, s);
  if (a.tile <= 1024) return launch_tile_t<R, MODE, COMP, 256, 4, VTX>(a, s);
  return launch_tile_t<R, MODE, COMP, 512, 4, VTX>(a, s);
}

template <typename R, bool COMP, bool VTX = false>
cudaError_t launch_tile_mode(int mode, const StepArgs& a, cudaStream_t s) {
  switch (mode) {
    case kModeFE: return launch_tile_size<R, kModeFE, COMP, VTX>(a, s);
    case kModeRK2a: return launch_tile_size<R, kModeRK2a, COMP, VTX>(a, s);
    case kModeRK2b: return launch_tile_size<R, kModeRK2b, COMP, VTX>(a, s);
    case kModeResidual: return launch_tile_size<R, kModeResidual, false, VTX>(a, s);
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace

// Whether all tiles are resident at a time in the one-cell-per-thread form
// (with the most registers its kernels take, and shared memory without opting
// in to more).
bool tile_quick_fits(int64_t n, int tile, int t1_cap) {
  if (tile > kQuickTile) return false;
  const int threads = (tile + 31) / 32 * 32 + 32;
  const size_t smem = tile_smem_bytes(false, t1_cap);
  int dev = 0, sms = 0, per_sm = 0;
  if (smem > 48 * 1024 - 512 || cudaGetDevice(&dev) != cudaSuccess ||
      cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess ||
      cudaOccupancyMaxActiveBlocksPerMultiprocessor(
          &per_sm, k_step_tile_quick<kModeRK2b, true, kWaveAverage>, threads, smem) != cudaSuccess)
    return false;
  return (n + tile - 1) / tile <= (int64_t)sms * per_sm;
}

cudaError_t launch_batch_step_tile(bool f64, int mode, const BatchArgs& b, cudaStream_t s) {
  if (b.n_tiles <= 0) return cudaSuccess;
  if (!b.s.cell_ln || !b.s.tile_info || !b.s.halo_id || !b.tile_mesh) return cudaErrorInvalidValue;
  if (f64) return launch_tile_batch_mode<double, false>(mode, b, s);
  if (b.s.lo) return launch_tile_batch_mode<float, true>(mode, b, s);
  return launch_tile_batch_mode<float, false>(mode, b, s);
}

cudaError_t launch_face_records(const void* geom, const int* face_off, const uint2* words,
                                int n_tiles, int tile, void* records, cudaStream_t s) {
  if (n_tiles <= 0) return cudaSuccess;
  k_face_records<<<(unsigned)n_tiles, 128, 0, s>>>(static_cast<const dq4*>(geom), face_off, words,
                                                   tile, static_cast<dq4*>(records));
  return cudaGetLastError();
}

cudaError_t launch_step_tile_faces(bool f64, int mode, const StepArgs& a, cudaStream_t s) {
  if (a.n <= 0) return cudaSuccess;
  if (!a.cell_ln || !a.tile_info || !a.halo_id || a.tile_vq || !a.tile_face_off || !a.tile_face)
    return cudaErrorInvalidValue;
  if (f64) {
    if (!a.cell_ref) return cudaErrorInvalidValue;
    return launch_faces_mode<double, false>(mode, a, s);
  }
  if (a.lo) return launch_faces_mode<float, true>(mode, a, s);
  return launch_faces_mode<float, false>(mode, a, s);
}

cudaError_t launch_step_tile(bool f64, int mode, const StepArgs& a, cudaStream_t s) {
  if (a.n <= 0) return cudaSuccess;
  if (!a.cell_ln || !a.tile_info || !a.halo_id) return cudaErrorInvalidValue;
  if (a.tile_vq) {
    if (f64 || !a.cell_vl || !a.tile_voff || !a.inv_vol) return cudaErrorInvalidValue;
    if (a.lo) return launch_tile_mode<float, true, true>(mode, a, s);
    return launch_tile_mode<float, false, true>(mode, a, s);
  }
  if (f64) return launch_tile_mode<double, false>(mode, a, s);
  if (a.lo) return launch_tile_mode<float, true>(mode, a, s);
  return launch_tile_mode<float, false>(mode, a, s);
}

}  // namespace fv
