// loop_step.cu -- a whole time loop in one launch for small FP32 meshes: the
// resident loop.
//
// A step of a small mesh is all launch and memory latency: 2.9 us at 4,096
// cells, of which the arithmetic is a third.  Here one thread-block cluster of
// up to 16 SMs keeps the mesh on chip for the whole loop: each block a tile of
// consecutive cells and its ring, whose states sit in two shared-memory arrays
// that swap roles every stage, the remainders of the compensated update beside
// them.  A cell that borders another tile pushes its new state into that
// block's ring, and every warp pushes its minimum CFL bound into all blocks,
// by asynchronous stores to distributed shared memory that complete on the
// receiver's mbarriers: no fence, no cluster barrier (its release and acquire
// took 1,700 clocks per step and emptied the L1 of the geometry) and no trip
// through the L2 (2,000 clocks and more for the quickest exchange of all SMs).
// One warp of each block forms the next dt while the others sum the fluxes,
// which need no dt.  A cell finishes with the helpers of the one-step kernels
// (face_flux_acc, advance_state, cell_bound), so every state is bit for bit
// that of a launch per step.
//
// Each mbarrier has a twin: stages of even and odd number (epoch) use their
// own, so what a quick neighbour sends ahead never counts for the stage still
// awaited; it cannot be two stages ahead, since its stage needs this block's
// last one.
//
// Waits are bounded.  A block in which one gives up (error bit 2) stops as a
// whole at the next barrier of dt, so it has pushed its stages whole or not at
// all, and the blocks that wait for it give up in turn.  Every block leaves the
// number of stages it pushed with all others before the closing cluster
// barrier; one that gave up then knows which stores are still on their way to
// it and awaits those (drain) before it leaves.  (Stopping at a vote behind the
// wait for RK2's first stage too cost 3-7 % of a step.)
#include <cuda_runtime.h>

#include <algorithm>
#include <cstdint>
#include <type_traits>

#include "cell_math.cuh"
#include "kernels.h"
#include "tile_math.cuh"
#include "tma_util.cuh"

namespace fv {

namespace {

__device__ __forceinline__ void cluster_sync() {
  asm volatile("barrier.cluster.arrive.release;\nbarrier.cluster.wait.acquire;" ::: "memory");
}

// Address in block `rank`'s shared memory of what lies at p in this block's.
__device__ __forceinline__ unsigned remote(const void* p, unsigned rank) {
  unsigned r;
  asm("mapa.shared::cluster.u32 %0, %1, %2;"
      : "=r"(r)
      : "r"((unsigned)__cvta_generic_to_shared(p)), "r"(rank));
  return r;
}
// Asynchronous stores to cluster addresses; their bytes complete on the
// mbarrier (also a cluster address, in the same block).
__device__ __forceinline__ void push_state(unsigned to, const float4& u, unsigned bar) {
  asm volatile(
      "st.async.weak.shared::cluster.mbarrier::complete_tx::bytes.v4.f32 [%0], {%1, %2, %3, %4}, "
      "[%5];" ::"r"(to), "f"(u.x), "f"(u.y), "f"(u.z), "f"(u.w), "r"(bar)
      : "memory");
}
__device__ __forceinline__ void push_value(unsigned to, float v, unsigned bar) {
  asm volatile("st.async.weak.shared::cluster.mbarrier::complete_tx::bytes.f32 [%0], %1, [%2];" ::"r"(
                   to),
               "f"(v), "r"(bar)
               : "memory");
}

__device__ __forceinline__ void store_remote(unsigned to, unsigned x, unsigned y) {
  asm volatile("st.shared::cluster.v2.u32 [%0], {%1, %2};" ::"r"(to), "r"(x), "r"(y) : "memory");
}
// Takes bytes that will not come off what an mbarrier of this block expects
// (in the pieces they would have come in, so that no sum jumps over zero).
__device__ __forceinline__ void forgo_tx(uint64_t* bar, unsigned bytes) {
  asm volatile("mbarrier.complete_tx.relaxed.cta.shared::cta.b64 [%0], %1;" ::"r"(smem_addr(bar)),
               "r"(bytes)
               : "memory");
}

// Waits for an mbarrier that other blocks' stores complete; false after `limit` tries.
__device__ __forceinline__ bool await(uint64_t* bar, unsigned parity, unsigned limit) {
  for (unsigned k = 0; k < limit; ++k) {
    unsigned ok;
    asm volatile(
        "{\n.reg .pred p;\n"
        "mbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\n"
        "selp.u32 %0, 1, 0, p;\n}"
        : "=r"(ok)
        : "r"(smem_addr(bar)), "r"(parity)
        : "memory");
    if (ok) return true;
  }
  return false;
}

// Minimum over the warp of values that are positive or +inf (in every lane).
__device__ __forceinline__ float warp_min_positive(float v) {
  return __uint_as_float(__reduce_min_sync(0xffffffffu, __float_as_uint(v)));
}

constexpr unsigned kNoPush = 0xFFFFFFFFu;

// A cell's records: geometry, the
// neighbours' positions in the block (or ghost codes) and, for a cell that
// borders other tiles, where its state goes in their s0 (cluster addresses,
// kNoPush for none) and on which mbarriers.
struct LoopCell {
  float4 g0, g1;
  unsigned v[3];
  unsigned to[3], bar[3];
};

// Barrier of the compute threads alone.
template <int THREADS>
__device__ __forceinline__ void compute_sync() {
  asm volatile("bar.sync 1, %0;" ::"n"(THREADS) : "memory");
}

// THREADS compute threads, each with at most one cell, whose records stay in
// registers, and one warp for dt.
template <int THREADS, bool RK2, bool COMP, int WAVE>
__global__ void __launch_bounds__(THREADS + 32, 1) k_loop(LoopArgs a) {
  constexpr int kWarps = THREADS / 32;
  constexpr int kRow = kLoopMaxTiles * kWarps;  // the warps' minima of all blocks
  extern __shared__ __align__(128) unsigned char smem_raw[];
  float4* s0 = reinterpret_cast<float4*>(smem_raw);  // [cap] tile, then its ring
  float4* s1 = s0 + a.cap;                             // [cap]
  // remainders of the tile's cells: U^n's, then (RK2) the stage's
  uint2* lo = reinterpret_cast<uint2*>(s1 + a.cap);
  uint2* lo_stage = lo + a.tile;
  __shared__ __align__(16) float s_min[2][kRow];
  __shared__ float s_dt;
  __shared__ __align__(8) uint64_t ring_bar[2], min_bar[2];  // of even and odd epochs
  // by block: the last ring epoch and the number of minima it has pushed
  __shared__ uint2 s_sent[kLoopMaxTiles];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int rank = blockIdx.x, blocks = gridDim.x;  // the grid is one cluster
  const int4 info = __ldg(a.info + rank);           // ring offset, ring size, edge cells, pushes
  const unsigned ring_bytes = (unsigned)info.y * 16u;
  const unsigned min_bytes = (unsigned)(blocks * kWarps) * 4u;
  const int t0 = rank * a.tile;
  const int nt = max(0, min(a.tile, a.n - t0));
  bool fail = false;

  if (tid == 0) {
    for (int p = 0; p < 2; ++p) {
      mbar_init(&ring_bar[p], 1);
      mbar_init(&min_bar[p], 1);
    }
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  for (int k = tid; k < 2 * kRow; k += THREADS + 32) (&s_min[0][0])[k] = INFINITY;
  // read here: block 0 may write the time at the end of a launch of one bound
  // before another block's warp of dt has begun
  double t = warp == kWarps ? *a.t : 0.0;
  cluster_sync();  // every block's mbarriers are ready

  if (warp == kWarps) {
    // ring epochs 1, 2, ... (states after each stage), minima 0, 1, ...: the
    // last one armed of each (and with it the one before)
    unsigned armed_ring = 2u, armed_min = 1u;
    if (lane == 0) {
      mbar_expect_tx(&ring_bar[1], ring_bytes);
      mbar_expect_tx(&ring_bar[0], ring_bytes);
      mbar_expect_tx(&min_bar[0], min_bytes);
      mbar_expect_tx(&min_bar[1], min_bytes);
    }
    double dt_raw = 0.0;
    unsigned epoch = 0u, minima = 0u;
    // Behind the barrier of dt every thread has been through the waits before
    // it: their mbarriers are armed for the epoch after next (what a quick block
    // has already sent of that one only counts the bytes below zero meanwhile).
    auto rearm = [&](bool due) {
      if (lane == 0) {
        if (due) mbar_expect_tx(&min_bar[(minima + 1u) & 1u], min_bytes);
        if (epoch > 0u && RK2) mbar_expect_tx(&ring_bar[1], ring_bytes);
        if (epoch > 0u) mbar_expect_tx(&ring_bar[RK2 ? 0u : epoch & 1u], ring_bytes);
      }
      if (due) armed_min = minima + 1u;
      if (epoch > 0u) armed_ring = epoch + 2u;
    };
    bool due = true;
    for (int j = 0; j < a.nsteps; ++j) {
      if (due) {
        const unsigned p = minima & 1u;
        if (!await(&min_bar[p], (minima >> 1) & 1u, a.polls)) fail = true;
        float m = INFINITY;
#pragma unroll
        for (int k = 0; k < kRow / 128; ++k) {
          const float4 x = reinterpret_cast<const float4*>(s_min[p])[lane + 32 * k];
          m = fminf(m, fminf(fminf(x.x, x.y), fminf(x.z, x.w)));
        }
        m = warp_min_positive(m);
        dt_raw = a.fixed_dt ? -a.cfl : a.cfl * (double)m;
        ++minima;
      }
      // dt of step j, clamped so the time never passes t_stop
      double dt = dt_raw;
      if (a.clamp) {
        const double rem = a.t_stop - t;
        if (rem < dt) dt = rem;
        if (!(dt > 0.0)) dt = 0.0;
      }
      if (lane == 0) s_dt = (float)dt;
      if (__syncthreads_or(fail)) break;  // C: dt is there, the ring was awaited
      t += dt;
      rearm(due);
      due = a.steps_per_bound == 1 || !due;
      epoch += RK2 ? 2u : 1u;
      if (RK2) __syncthreads();  // B
      if (j + 1 == a.nsteps) break;
      __syncthreads();  // A
    }
    const bool failed = __syncthreads_or(fail);
    if (!failed && rank == 0 && lane == 0) *a.t = t;
    cluster_sync();  // no block pushes any more, and s_sent is complete
    if (failed) {
      // What may be on its way: of the last two epochs armed, and of a ring's
      // one after those when the wait that gave up was for RK2's first stage
      // (the block then still pushed that step, which its neighbours answer).
      bool drained = true;
      for (unsigned b = 0; b < 2; ++b) {
        const unsigned e = armed_ring - b, m = armed_min - b;
        unsigned ahead = 0u;  // bytes of epoch e + 2
        for (int r = lane; r < info.y; r += 32) {
          const int i = __ldg(a.ring_id + info.x + r);
          const unsigned sent = s_sent[index_ok(i, a.n, a.err) ? i / a.tile : rank].x;
          if (sent < e) forgo_tx(&ring_bar[e & 1u], 16u);
          if (sent >= e + 2u) ahead += 16u;
        }
        ahead = __reduce_add_sync(0xffffffffu, ahead);
        if (lane < blocks && s_sent[lane].y <= m)
          for (int k = 0; k < kWarps; ++k) forgo_tx(&min_bar[m & 1u], 4u);
        __syncwarp();
        drained = __all_sync(0xffffffffu,
                             await(&min_bar[m & 1u], (m >> 1) & 1u, a.drain_polls) && drained);
        if (__all_sync(0xffffffffu,
                       await(&ring_bar[e & 1u], ((e - 1u) >> 1) & 1u, a.drain_polls))) {
          if (lane == 0) mbar_expect_tx(&ring_bar[e & 1u], ahead);
          __syncwarp();
          drained = await(&ring_bar[e & 1u], ((e + 1u) >> 1) & 1u, a.drain_polls) && drained;
        } else {
          drained = false;
        }
      }
      if (!drained) atomicOr(a.err, 4);
    }
    return;
  }

  const float4* __restrict__ geom = a.geom + 2 * (int64_t)t0;
  const int* __restrict__ ord = a.ord + t0;
  const int edges = info.z;
  float4* const base = s0;
  unsigned epoch = 0u;  // of the states now read
  unsigned pushed = 0u;  // the last epoch this block's edge cells were pushed of

  LoopCell c{};
  const bool has = tid < nt;
  if (has) {
    c.g0 = __ldg(geom + 2 * tid);
    c.g1 = __ldg(geom + 2 * tid + 1);
    const uint2 l = __ldg(a.ln + t0 + tid);
    c.v[0] = l.x & 0xffffu;
    c.v[1] = l.x >> 16;
    c.v[2] = l.y & 0xffffu;
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      c.to[k] = kNoPush;
      if (tid < edges) {
        const unsigned at = __ldg(a.push + 3 * (info.w + tid) + k);  // tile << 16 | ring entry
        if (at != kNoPush) {
          c.to[k] = remote(base + a.tile + (at & 0xffffu), at >> 16);
          c.bar[k] = remote(&ring_bar[0], at >> 16);
        }
      }
    }
  }
  bool ok = true;
  float bmin = INFINITY;

  // The flux sum of the thread's cell in src (twice it, face_flux_acc) and
  // its perimeter.
  float acc[4], perim = 0.f;
  auto fluxes = [&](const float4* src) {
    const float4 UL = src[tid];
    const Prim<float> L = primitive<float>(UL);
    const float nx[3] = {c.g0.x, c.g0.z, c.g1.x}, ny[3] = {c.g0.y, c.g0.w, c.g1.y};
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      float4 UR;
      if (c.v[k] < kGhostCodes)
        UR = index_ok(c.v[k], a.cap, a.err) ? src[c.v[k]] : UL;
      else
        UR = ghost<float>((int)c.v[k] - 0x10000, UL, nx[k], ny[k], a.uinf);
      const float len = face_len<float>(nx[k], ny[k]);
      face_flux_acc<float, false, WAVE>(UL, L, UR, primitive<float>(UR), nx[k], ny[k], len, 1.f,
                                        acc, k == 0);
      perim = k == 0 ? len : add(perim, len);
    }
  };
  // The update of the cell from its flux sum: src -> dst (the second stage of
  // RK2 finds U^n in dst), pushed to the rings it belongs to.
  auto finish = [&](auto mode_tag, const float4* src, float4* dst, float dt, bool send) {
    constexpr int MODE = decltype(mode_tag)::value;
    uint2 lo_in = make_uint2(0u, 0u), lo_st = lo_in, lo_out;
    if (COMP) {
      lo_in = lo[tid];
      if (MODE == kModeRK2b) lo_st = lo_stage[tid];
    }
    const float4 UL = src[tid];
    const float4 b = MODE == kModeRK2b ? dst[tid] : UL;
    const float4 Un =
        advance_state<float, MODE, COMP>(UL, b, acc, c.g1.z, dt, lo_in, lo_st, lo_out);
    if (send && tid < edges) {
      const unsigned shift = dst == base ? 0u : (unsigned)(a.cap * sizeof(float4));
      const unsigned twin = ((epoch + 1u) & 1u) * (unsigned)sizeof(uint64_t);
#pragma unroll
      for (int k = 0; k < 3; ++k)
        if (c.to[k] != kNoPush) push_state(c.to[k] + shift, Un, c.bar[k] + twin);
    }
    dst[tid] = Un;
    if (COMP) (MODE == kModeRK2a ? lo_stage : lo)[tid] = lo_out;
    if (MODE != kModeRK2a) {
      bool c_ok;
      bmin = cell_bound<float>(Un, inradius<float>(c.g1, perim), c_ok);
      ok = ok && c_ok;
    }
  };
  // the warp's minimum of a state's bounds, to every block
  unsigned minima = 0u;
  auto send_min = [&]() {
    const float m = warp_min_positive(bmin);
    const unsigned p = minima & 1u;
    if (lane < blocks)
      push_value(remote(&s_min[p][rank * kWarps + warp], lane), m, remote(&min_bar[p], lane));
    ++minima;
    bmin = INFINITY;
  };
  // the ring of the epoch now read has arrived (epoch 0 came with the start)
  auto await_ring = [&]() {
    if (epoch == 0u) return;
    if (!await(&ring_bar[epoch & 1u], ((epoch - 1u) >> 1) & 1u, fail ? 0u : a.polls))
      fail = true;
  };

  // U^0 of the tile and its ring, the remainders and the bound
  for (int e = tid; e < nt + info.y; e += THREADS) {  // nt <= THREADS
    const int i = e < nt ? __ldg(ord + e) : __ldg(a.ring_id + info.x + (e - nt));
    const float4 u = index_ok(i, a.n, a.err) ? a.U[i] : make_float4(1.f, 0.f, 0.f, 1.f);
    s0[e < nt ? e : a.tile + (e - nt)] = u;
    if (e >= nt) continue;
    if (COMP) lo[e] = a.lo_in ? a.lo_in[i] : make_uint2(0u, 0u);
    if (!a.fixed_dt) {
      bool c_ok;
      bmin = fmin(bmin, cell_bound<float>(u, geom_inradius<float>(geom, e), c_ok));
      ok = ok && c_ok;
    }
  }
  compute_sync<THREADS>();
  send_min();
  bool stop = false, due = true;
  for (int j = 0; j < a.nsteps && !stop; ++j) {
    const bool last = j + 1 == a.nsteps;
    // the fluxes do not depend on dt: they are summed while it is formed
    await_ring();
    if (has) fluxes(s0);
    stop = __syncthreads_or(fail);  // C
    if (stop) break;
    const float dt = s_dt;
    constexpr int kFirst = RK2 ? kModeRK2a : kModeFE;
    if (has) finish(std::integral_constant<int, kFirst>{}, s0, s1, dt, RK2 || !last);
    ++epoch;
    if (RK2 || !last) pushed = epoch;
    if (RK2) {
      __syncthreads();  // B: U* of the tile is complete
      await_ring();
      if (has) {
        fluxes(s1);
        finish(std::integral_constant<int, kModeRK2b>{}, s1, s0, dt, !last);
      }
      ++epoch;
      if (!last) pushed = epoch;
    } else {
      float4* s = s0;
      s0 = s1;
      s1 = s;
    }
    due = a.steps_per_bound == 1 || !due;  // whether the next step has a bound of its own
    if (!last && due) send_min();
    bmin = INFINITY;
    if (!last) __syncthreads();  // A: U^{j+1} of the tile is complete
  }
  if (__syncthreads_or(fail)) {
    if (tid == 0) atomicOr(a.err, 2);
  } else {
    const int i = has ? __ldg(ord + tid) : 0;
    if (has && index_ok(i, a.n, a.err)) {
      a.U[i] = s0[tid];
      if (COMP) a.lo_out[i] = lo[tid];
    }
    if (!ok) atomicOr(a.err, 1);
  }
  if (warp == 0 && lane < blocks) store_remote(remote(&s_sent[rank], lane), pushed, minima);
  cluster_sync();  // no block leaves while another may still write to it
}

// The geometry records in the loop's order (a copy made once per mesh).
__global__ void k_loop_geometry(const float4* __restrict__ geom, const int* __restrict__ ord, int n,
                                float4* out) {
  const int p = blockIdx.x * blockDim.x + threadIdx.x;
  if (p < 2 * n) out[p] = __ldg(geom + 2 * (int64_t)__ldg(ord + (p >> 1)) + (p & 1));
}

template <int THREADS, bool RK2, bool COMP, int WAVE>
cudaError_t launch_loop_t(const LoopArgs& a, cudaStream_t s, int* clusters) {
  auto k = k_loop<THREADS, RK2, COMP, WAVE>;
  const size_t smem = loop_smem_bytes(a.cap, a.tile, COMP, RK2);
  cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e == cudaSuccess) e = cudaFuncSetAttribute(k, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
  if (e != cudaSuccess) return e;
  unsigned blocks = 1;
  while ((int)blocks < a.n_tiles) blocks *= 2;
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3(blocks);
  cfg.blockDim = dim3(THREADS + 32);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = blocks;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  if (clusters) return cudaOccupancyMaxActiveClusters(clusters, k, &cfg);
  return cudaLaunchKernelEx(&cfg, k, a);
}

template <int THREADS>
cudaError_t launch_loop_r(const LoopArgs& a, bool rk2, bool comp, int wave, cudaStream_t s,
                          int* clusters) {
  switch ((rk2 ? 4 : 0) | (comp ? 2 : 0) | (wave == kWaveMax ? 1 : 0)) {
    case 0: return launch_loop_t<THREADS, false, false, kWaveAverage>(a, s, clusters);
    case 1: return launch_loop_t<THREADS, false, false, kWaveMax>(a, s, clusters);
    case 2: return launch_loop_t<THREADS, false, true, kWaveAverage>(a, s, clusters);
    case 3: return launch_loop_t<THREADS, false, true, kWaveMax>(a, s, clusters);
    case 4: return launch_loop_t<THREADS, true, false, kWaveAverage>(a, s, clusters);
    case 5: return launch_loop_t<THREADS, true, false, kWaveMax>(a, s, clusters);
    case 6: return launch_loop_t<THREADS, true, true, kWaveAverage>(a, s, clusters);
    default: return launch_loop_t<THREADS, true, true, kWaveMax>(a, s, clusters);
  }
}

// the block shape for a tile size: one cell per thread
cudaError_t dispatch_loop(const LoopArgs& a, bool rk2, bool comp, int wave, cudaStream_t s,
                          int* clusters) {
  if (a.n_tiles > kLoopMaxTiles || a.tile > kLoopMaxTile) return cudaErrorInvalidValue;
  if (a.tile <= 256) return launch_loop_r<256>(a, rk2, comp, wave, s, clusters);
  if (a.tile <= 512) return launch_loop_r<512>(a, rk2, comp, wave, s, clusters);
  return launch_loop_r<kLoopMaxTile>(a, rk2, comp, wave, s, clusters);
}

}  // namespace

cudaError_t launch_loop(const LoopArgs& a, bool rk2, bool comp, int wave, cudaStream_t s) {
  if (a.n <= 0 || a.nsteps <= 0) return cudaSuccess;
  return dispatch_loop(a, rk2, comp, wave, s, nullptr);
}

cudaError_t loop_clusters(const LoopArgs& a, bool rk2, bool comp, int* clusters) {
  return dispatch_loop(a, rk2, comp, kWaveAverage, nullptr, clusters);
}

cudaError_t launch_loop_geometry(const float4* geom, const int* ord, int n, float4* out,
                                 cudaStream_t s) {
  if (n <= 0) return cudaSuccess;
  k_loop_geometry<<<(unsigned)((2 * (int64_t)n + 255) / 256), 256, 0, s>>>(geom, ord, n, out);
  return cudaGetLastError();
}

}  // namespace fv
