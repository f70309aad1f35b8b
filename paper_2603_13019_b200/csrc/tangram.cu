// Host side of the C ABI declared in include/tangram.h, and the per-pool round kernel.
#include <cuda_runtime.h>
#include <stdint.h>
#include <stdio.h>
#include <string.h>
#include <limits.h>
#include <new>

#include "../../include/tangram.h"
#include "common.cuh"
#include "prefix_stream.cuh"
#include "order_pin.cuh"
#include "arrange.cuh"
#include "evict.cuh"
#include "place.cuh"

#define K2_THREADS 256
#define TG_PROF_CALLS 256   // calls whose kernels can be timed between two queries
#define TG_FILL_BLOCKS_PER_SM 4   // k_fill is a trickle beside the sort, not a flood
#define TG_IO_CHUNKS 16
// Scenarios per SM up to which a round is one launch of k_round: as many blocks as an SM holds at once (128 registers
// x 256 threads), so that no block waits for another.  Beyond that the head walks of eight scenarios share a block, and
// pools that need a selection are handed out before the others.
#define TG_FUSED_PER_SM 2
#define TG_SMEM_PER_SM 233472   // shared memory an SM can split among resident blocks
#define TG_REPLAY_SMEM 114688    // a replay block takes at most that much (the rest of the SM's is L1)
#define TG_PROF_K 3         // timed intervals per call at most
#define TG_N_KERNELS 8

// ---------------------------------------------------------------------------------------
// Per-(scenario, pool) work of a round, one warp per task: gather the pool's candidates, decide
// them (arrange.cuh, evict.cuh), place what was granted, write the candidates' outputs (Eq. 2).
//   k_pool     the batched path, behind k_head / k_stream; pools that the head kernel certified
//              take a short way without any selection
//   k_round    small batches and the allocation-free entry point: the whole round, one block per scenario
// ---------------------------------------------------------------------------------------
// Tasks are handed out by a counter so that long tasks do not pile up on the same warps.
__device__ __forceinline__ int next_task(u64* counter, int lane) {
  u64 x = 0;
  if (lane == 0) x = atomicAdd(counter, 1ull);
  return (int)__shfl_sync(TG_FULL, x, 0);
}

struct CandArrays {
  i64* cs; i64* cp; u32* cmask; int* cidx; int* pnode; int* poff; int* rowcand;
  u8* cg; u8* rsel; u8* rkeep;
};

__device__ bool gather_candidates(const Params& P, int sc, int j, const PoolMeta& mt, Slab& slab, int lane,
                                  CandArrays& C) {
  const int m = mt.m;
  const PoolDev& pd = P.pool[j];
  const size_t row = (size_t)sc * P.N;
  // what the sequential loops read over and over goes to the warp's shared-memory window while
  // it lasts (most wanted first), the rest to the warp's slab in global memory
  C.cg = (u8*)slab.take_fast(m);
  C.rkeep = (u8*)slab.take_fast(m);
  C.rsel = (u8*)slab.take_fast(m);
  C.cmask = (u32*)slab.take_fast((u64)m * 4);
  C.rowcand = (int*)slab.take_fast((u64)m * 4);
  C.cp = (i64*)slab.take_fast((u64)m * 8);
  C.cs = (i64*)slab.take_fast((u64)m * 8);
  C.cidx = (int*)slab.take((u64)m * 4);
  C.pnode = (int*)slab.take((u64)m * 4);
  C.poff = (int*)slab.take((u64)m * 4);
  if (!C.cg || !C.rkeep || !C.rsel || !C.cmask || !C.rowcand || !C.cp || !C.cs || !C.cidx || !C.pnode || !C.poff) return false;
  // four candidates per lane at a time: first all their indices, then all their records, so that a
  // pool of up to 128 candidates costs two rounds of loads instead of two per 32 candidates
#pragma unroll 1
  for (int i0 = lane; i0 < m; i0 += 128) {
    int idx[4]; u8 un[4]; u32 mk[4]; i64 sv[4], pv[4];
#pragma unroll
    for (int x = 0; x < 4; ++x) idx[x] = i0 + 32 * x < m ? P.order[row + mt.cbase + i0 + 32 * x] : 0;
#pragma unroll
    for (int x = 0; x < 4; ++x) {
      const bool on = i0 + 32 * x < m;
      un[x] = on ? P.a_unit[row + idx[x]] : 1; mk[x] = on ? P.a_mask[row + idx[x]] : 1;
      sv[x] = on ? P.a_s[row + idx[x]] : 0; pv[x] = on ? P.a_p[row + idx[x]] : 0;
    }
#pragma unroll
    for (int x = 0; x < 4; ++x) {
      const int i = i0 + 32 * x;
      if (i >= m) break;
      const int g = un[x] & 0x7f, gang = (un[x] >> 7) && pd.type == TG_POOL_GPU;
      const u32 eff = mk[x] & usable_levels(P, j, un[x]);
      C.cidx[i] = idx[x]; C.cmask[i] = eff; C.cg[i] = (u8)(g | (gang << 7));
      C.cs[i] = clamp_param(sv[x]); C.cp[i] = clamp_param(pv[x]);
      C.rkeep[i] = (u8)__ffs(eff);
      C.pnode[i] = -1; C.poff[i] = -1;
    }
  }
  __syncwarp();
  return true;
}

// the calling warp's scratch: work area and window in shared memory, slab in global memory
#define WARP_WORK_BYTES 7424
#define WARP_FAST_BYTES 2048
#define WARP_TASK_BYTES 384
#define WARP_SMEM_BYTES (WARP_WORK_BYTES + WARP_FAST_BYTES + WARP_TASK_BYTES)
static_assert(sizeof(PoolTask) <= WARP_TASK_BYTES, "");
// the choices of a small table in the work area (solve_prefix): behind the staged levels and all that ev_run_regs<8> uses
static_assert((64 * 8 + 2 * EV_BLOCK + 4) * 4 <= 32 * CELL_LEVELS * 16 && 32 * CELL_LEVELS * 16 + CELL_SHARED_ROWS * 64 <= WARP_WORK_BYTES, "");
#define K2_DYN_SMEM ((K2_THREADS / 32) * WARP_SMEM_BYTES + 16)
__device__ __forceinline__ char* warp_smem() {
  extern __shared__ __align__(16) unsigned char k2_smem[];
  return (char*)(((u64)k2_smem + 15u) & ~(u64)15) + (threadIdx.x >> 5) * WARP_SMEM_BYTES;
}
__device__ __forceinline__ PoolTask& warp_task() { return *(PoolTask*)(warp_smem() + WARP_WORK_BYTES + WARP_FAST_BYTES); }
__device__ __forceinline__ Slab warp_slab(const Params& P, int gw) {
  Slab s;
  s.base = P.slabs + (u64)gw * P.slab_bytes; s.cap = P.slab_bytes; s.used = 0;
  s.fbase = warp_smem() + WARP_WORK_BYTES;
  s.fcap = WARP_FAST_BYTES; s.fused = 0;
  return s;
}

__device__ PoolTask& make_task(const Params& P, int sc, int ws, int j, const PoolMeta& mt, const CandArrays& C, int lane) {
  const PoolDev& pd = P.pool[j];
  const size_t row = (size_t)sc * P.N;
  const u8* busy_row = P.gpu_busy ? P.gpu_busy + (size_t)sc * P.n_nodes_total : nullptr;
  int cap[4] = {pd.capacity, 0, 0, 0};
  if (pd.type == TG_POOL_GPU) gpu_caps(pd, busy_row, lane, cap);
  if (P.n_side > 0 && pd.type == TG_POOL_API) cap[0] -= P.side_res[(size_t)ws * P.P + j];   // set aside for the other pools' candidates
  Act first;
  first.s = first.p = 0; first.mask = 1; first.g = 1; first.gang = 0;
  const int n_ac = mt.count - mt.m;
  if (n_ac > 0) {
    const size_t o = row + mt.first_wait;
    decode_levels(pd, P.a_unit[o], P.a_mask[o], first.g, first.gang, first.mask);
    first.s = clamp_param(P.a_s[o]); first.p = clamp_param(P.a_p[o]);
  }
  PoolTask& T = warp_task();
  __syncwarp();
  if (lane == 0) {
    T.type = pd.type; T.group = pd.group;
#pragma unroll 1
    for (int l = 0; l < 4; ++l) T.cap[l] = cap[l];
    T.m = mt.m; T.cs = C.cs; T.cp = C.cp; T.cmask = C.cmask; T.cg = C.cg;
    T.n_ac = n_ac; T.ac_tmin = P.tmin + row + mt.base + mt.m; T.ac_first = first;
    T.seeds = nullptr; T.n_seeds = 0;
    T.depth = P.depth;
    T.rsel = C.rsel; T.rkeep = C.rkeep; T.rowcand = C.rowcand;
    T.wk = warp_smem(); T.wk_bytes = WARP_WORK_BYTES;
  }
  __syncwarp();
  return T;
}

// placement on a fresh copy of the pool's topology state, then the candidates' outputs.  CACHE: GPU pools have a service
// cache; instances of their own, since the others are slower with its code in them (16384 x 4096 1555 us a call against 1510)
template <bool CACHE>
__device__ __forceinline__ void place_and_write(const Params& P, int sc, int j, const PoolMeta& mt, const CandArrays& C,
                                int keep, Slab slab, int lane) {
  const int m = mt.m;
  const PoolDev& pd = P.pool[j];
  const size_t row = (size_t)sc * P.N;
  const u8* busy_row = P.gpu_busy ? P.gpu_busy + (size_t)sc * P.n_nodes_total : nullptr;
  const u8* missed = nullptr;                            // candidates whose chunk did not cache their service
  if (CACHE && pd.type == TG_POOL_GPU) {
    // with a service cache: the chunk that caches the instance first, entries updated, misses noted in C.rsel
    u8* nm = (u8*)slab.take_fast(pd.n_nodes);
    if (!nm) { if (lane == 0) atomicOr(&P.o_status[sc], TG_ST_WORKSPACE); keep = 0; }
    else {
#pragma unroll 1
      for (int v = lane; v < pd.n_nodes; v += 32) nm[v] = busy_row ? busy_row[pd.node0 + v] : 0;
      __syncwarp();
      const size_t cbase = ((size_t)sc * P.n_nodes_total + pd.node0) * 8 * P.cache_slots;
      place_gpu_cache(pd, BusyNodes{nm}, keep, C.cg, C.rkeep, C.cidx, C.pnode, C.poff, C.rsel, C.rowcand,
                      P.a_service ? P.a_service + row : nullptr, P.cache_tag + cbase, P.cache_use + cbase, P.cache_slots, P.now, lane,
                      warp_smem(), WARP_WORK_BYTES);   // (the selection is done with its work area)
      missed = C.rsel;
    }
  } else if (pd.type == TG_POOL_GPU) {
    const u8* br = busy_row ? busy_row + pd.node0 : nullptr;
    int R[4];
    gpu_requests(keep, C.cg, C.rkeep, C.pnode, C.poff, R, lane);
    const u64 bytes = (u64)(R[0] + R[1] + R[2] + R[3]) * 4;
    u8* nm = pd.n_nodes > 32 ? (u8*)slab.take_fast(pd.n_nodes) : nullptr;   // (before the list, which can be done without)
    u32* list = bytes <= WARP_WORK_BYTES ? (u32*)warp_smem() : (u32*)slab.take(bytes);   // (the selection is done with its work area)
    __syncwarp();
    if (pd.n_nodes > 32 && !nm) { if (lane == 0) atomicOr(&P.o_status[sc], TG_ST_WORKSPACE); keep = 0; }
    else if (list && pd.n_nodes <= 32) place_gpu_lists<true>(pd, br, nullptr, list, R, keep, C.pnode, C.poff, lane);
    else if (list) place_gpu_lists<false>(pd, br, nm, list, R, keep, C.pnode, C.poff, lane);
    else {
#pragma unroll 1
      for (int v = lane; v < pd.n_nodes; v += 32) nm[v] = br ? br[v] : 0;
      __syncwarp();
      place_gpu(pd, nm, keep, C.cg, C.rkeep, C.pnode, C.poff, lane);
    }
  } else if (pd.type == TG_POOL_CPU && pd.capacity / pd.group <= 128 && pd.group < 65536) {
    CpuFresh<4> F(pd, lane);
#pragma unroll 1
    for (int i0 = 0; i0 < keep; i0 += 32) {
      const int i = i0 + lane;
      int node = -1, off = -1;
      F.place(pd, i < keep ? (C.cg[i] & 0x7f) * C.rkeep[i] : 0, min(32, keep - i0), lane, node, off);
      if (i < keep) { C.pnode[i] = node; C.poff[i] = off; }
    }
  } else if (pd.type == TG_POOL_CPU) {
    const int D = pd.capacity / pd.group;
    int* dfree = (int*)slab.take_fast((u64)D * 4);
    if (!dfree) { if (lane == 0) atomicOr(&P.o_status[sc], TG_ST_WORKSPACE); keep = 0; }
    else place_cpu_fresh(pd, dfree, keep, C.cg, C.rkeep, C.pnode, C.poff, lane);
  } else {
    int used = 0;                                        // Section 5.1: offset = units consumed before
#pragma unroll 1
    for (int i0 = 0; i0 < keep; i0 += 32) {
      const int i = i0 + lane, u = i < keep ? (C.cg[i] & 0x7f) * C.rkeep[i] : 0;
      const int incl = warp_incl_scan32(u, lane);
      if (i < keep) { C.pnode[i] = 0; C.poff[i] = used + incl - u; }
      used += __shfl_sync(TG_FULL, incl, 31);
    }
  }
  __syncwarp();
  i64 tot = 0; int cnt = 0;
#pragma unroll 1
  for (int i = lane; i < m; i += 32) {
    const size_t o = row + C.cidx[i];
    if (i < keep) {
      int r = C.rkeep[i];
      i64 arr = P.a_arrival ? P.a_arrival[o] : 0;
      i64 act = (P.now - arr) + duration(C.cs[i], C.cp[i], r);
      if (CACHE && missed && missed[i] && P.a_restore) act += clamp_param(P.a_restore[o]);   // restoration precedes execution
      P.o_alloc[o] = (C.cg[i] & 0x7f) * r; P.o_act[o] = act;
      P.o_node[o] = C.pnode[i]; P.o_off[o] = C.poff[i];
      tot += act; ++cnt;
    } else {
      P.o_alloc[o] = 0; P.o_node[o] = -1; P.o_off[o] = -1; P.o_act[o] = -1;
    }
  }
  tot = warp_sum64(tot); cnt = warp_sum32(cnt);
  if (lane == 0 && cnt) {
    atomicAdd((u64*)&P.o_total[sc], (u64)tot);
    atomicAdd(&P.o_nsel[sc], cnt);
  }
}

// A pool whose every candidate takes its best level (no elastic candidate, or all largest levels fit: the smallest
// level that reaches the lowest duration, and no eviction can pay), of a type whose placement goes by queue order:
// 32 candidates at a time through registers.  Bound by the chain of placements on a core pool (one warp
// minimum per candidate).
template <int NS>
__device__ __forceinline__ void pool_best_levels(const Params& P, int sc, int j, const PoolMeta& mt, int lane) {
  const PoolDev& pd = P.pool[j];
  const size_t row = (size_t)sc * P.N;
  const int* ord = P.order + row + mt.cbase;
  const bool cpu = pd.type == TG_POOL_CPU;
  CpuFresh<NS> F(pd, lane);
  i64 tot = 0; int used = 0;
#pragma unroll 1
  for (int i0 = 0; i0 < mt.m; i0 += 32) {
    const int i = i0 + lane;
    const bool on = i < mt.m;
    size_t o = row; int u = 0; i64 act = 0;
    if (on) {
      o += ord[i];
      const int unit = P.a_unit[o], g = unit & 0x7f;
      const u32 eff = P.a_mask[o] & usable_levels(P, j, unit);
      const i64 s = clamp_param(P.a_s[o]), p = clamp_param(P.a_p[o]);
      const int r = best_level(p, eff);
      act = (P.now - (P.a_arrival ? P.a_arrival[o] : 0)) + duration(s, p, r);
      u = g * r;
      tot += act;
    }
    int node = 0, off = 0;
    if (cpu) F.place(pd, u, min(32, mt.m - i0), lane, node, off);
    else {
      const int incl = warp_incl_scan32(u, lane);
      off = used + incl - u;
      used += __shfl_sync(TG_FULL, incl, 31);
    }
    if (on) { P.o_alloc[o] = u; P.o_act[o] = act; P.o_node[o] = node; P.o_off[o] = off; }
  }
  tot = warp_sum64(tot);                                 // (exact modulo 2^64, so also where an arrival lies behind now)
  if (lane == 0) {
    atomicAdd((u64*)&P.o_total[sc], (u64)tot);
    atomicAdd(&P.o_nsel[sc], mt.m);
  }
}

// ws: whose rows of the workspace the pool's facts are in
template <bool CACHE, int U>
__device__ __forceinline__ void run_pool_task(const Params& P, int sc, int ws, int j, const PoolMeta& mt, Slab slab, int lane) {
  CandArrays C;
  if (!gather_candidates(P, sc, j, mt, slab, lane, C)) {
    if (lane == 0) atomicOr(&P.o_status[sc], TG_ST_WORKSPACE);
    return;
  }
  int keep = mt.m;
  if (mt.elastic) {
    keep = evict_loop<U>(P, make_task(P, sc, ws, j, mt, C, lane), slab, lane);
    if (keep < 0) { if (lane == 0) atomicOr(&P.o_status[sc], TG_ST_WORKSPACE); keep = 0; }
  }
  place_and_write<CACHE>(P, sc, j, mt, C, keep, slab, lane);
}

template <bool CACHE, int U>
__device__ __forceinline__ void decide_pool(const Params& P, int sc, int ws, int j, u32 need, int slab, int lane) {
  PoolMeta mt = P.meta[(size_t)ws * P.P + j];            // (a scenario with an invalid record has no candidates)
  mt.m = uniform(mt.m); mt.count = uniform(mt.count); mt.elastic = uniform(mt.elastic);
  if (mt.m == 0) return;
  if (!((need >> j) & 1u) && P.pool[j].queue_place) {
    if (P.pool[j].type == TG_POOL_API || P.pool[j].capacity <= 64 * P.pool[j].group) pool_best_levels<2>(P, sc, j, mt, lane);
    else pool_best_levels<4>(P, sc, j, mt, lane);
  } else run_pool_task<CACHE, U>(P, sc, ws, j, mt, warp_slab(P, slab), lane);
}

// All pools of a batched round, pool-major, the pools that may need a selection first.  The rows that stay queued are
// written beside the first pool's tasks, which are most of the work and leave the memory alone, or, where a warp has no
// second one of those, as tasks behind all others, which idle warps find while the longest pools are decided.  Spread
// over all pools, or with the second ones on, they meet the short tasks, which wait for memory themselves: 16384 x 4096 k_pool
// 1188 us against 1109 (1014 without the rows).  Bulk copies of constant blocks in shared memory instead of stores: 1110.
template <bool CACHE>
__global__ void __launch_bounds__(K2_THREADS, 2) k_pool(const __grid_constant__ Params P, const HeadState* hst) {
  const int lane = threadIdx.x & 31;
  const int gw = (blockIdx.x * K2_THREADS + threadIdx.x) >> 5;
  const int n_pool_tasks = P.S * P.P, warps = gridDim.x * (K2_THREADS / 32);
  const bool with_first = P.S > warps, fill = !P.perm;     // (k_fill wrote the rows of an ordered round)
  const int n_tasks = n_pool_tasks + (fill && !with_first ? P.S : 0);
#pragma unroll 1
  for (;;) {
    const int x = next_task(P.arena_top + 1, lane);
    if (x >= n_tasks) break;
    const int sc = x % P.S, k = x / P.S;
    if (fill && k == (with_first ? 0 : P.P)) fill_rows(P, sc, hst[sc].n, lane);
    if (k < P.P) decide_pool<CACHE, 2>(P, sc, sc, P.pool_order[k], hst[sc].need, gw, lane);
  }
}

// The whole round of a small batch in one launch, one block per scenario: the first warp walks the head of the queue
// while the others write "not scheduled" everywhere, all of them stream the rest of the queue, then every pool
// gets a warp (wpb < n_pools of them where memory is short: the static entry).  A block's scratch is its own, so nothing depends on the number of scenarios.  What bounds a small
// batch is latency, and one launch instead of three and a memset saves the gaps: 1 x 64 38.6 -> 26.8 us a call, 16 x 500
// (static) 110 -> 84 us when it took the place of four.  The last block to finish resets the bump pointer of the arena for
// the next call.
#define TG_DONE_COUNTER 4           // word of arena_top that counts finished blocks
template <bool SIDE, bool SORTED, bool CACHE>
__global__ void __launch_bounds__(K2_THREADS, 2) k_round(const __grid_constant__ Params P, int wpb) {
  __shared__ StreamShared X;
  __shared__ HeadState H;
  __shared__ int s_side_bad;
  const int t = threadIdx.x, lane = t & 31, warp = t >> 5, ws = blockIdx.x;
#pragma unroll 1
  for (int sc = blockIdx.x; sc < P.S; sc += gridDim.x) {
    const size_t row = (size_t)sc * P.N;
    if (SIDE) {
      if (t == 0) s_side_bad = 0;
      __syncthreads();
      const int n = min(max(P.n_actions[sc], 0), P.N);
      bool bad = false;
#pragma unroll 1
      for (int i = t; i < n; i += K2_THREADS)
        for (int e = 0; e < P.n_side; ++e) bad |= side_entry_bad(P, e, row + i);
      if (bad) s_side_bad = 1;
      __syncthreads();
    }
    if (warp == 0) head_walk<SIDE>(P, sc, ws, H, SIDE && s_side_bad, lane);
    else if (outputs_aligned(P)) {
      const size_t lo = (row + 3) / 4 * 4, hi = (row + P.N) / 4 * 4;       // groups of four of the whole array
      const size_t mid = lo < hi ? hi : lo;
      for (size_t o = lo + (size_t)(t - 32) * 4; o < hi; o += (size_t)(K2_THREADS - 32) * 4) write_unscheduled4(P, o);
      const size_t end = row + P.N;
      if (t < 40) { const size_t o = row + (t - 32); if (t < 36 && o < lo && o < end) write_unscheduled(P, o); }
      if (t >= 64 && t < 68) { const size_t o = mid + (t - 64); if (o < end) write_unscheduled(P, o); }
    } else
      for (int i = t - 32; i < P.N; i += K2_THREADS - 32) write_unscheduled(P, row + i);
    __syncthreads();
    stream_queue<SORTED>(P, sc, ws, H, X, t);
    __syncthreads();
#pragma unroll 1
    for (int x = warp; x < P.P && warp < wpb; x += wpb) decide_pool<CACHE, 4>(P, sc, ws, P.pool_order[x], H.need, ws * wpb + warp, lane);
    __syncthreads();
  }
  if (t == 0) {
    __threadfence();
    if (atomicAdd(P.arena_top + TG_DONE_COUNTER, 1ull) + 1 == gridDim.x) { P.arena_top[0] = 0; P.arena_top[TG_DONE_COUNTER] = 0; }
  }
}

#include "replay.cuh"

// ---------------------------------------------------------------------------------------
// host
// ---------------------------------------------------------------------------------------
static thread_local char g_cuda_err[256] = "";

static int cuda_fail(cudaError_t e, const char* what) {
  snprintf(g_cuda_err, sizeof(g_cuda_err), "%s: %s", what, cudaGetErrorString(e));
  return TANGRAM_ECUDA;
}
#define CK(call) do { cudaError_t e_ = (call); if (e_ != cudaSuccess) return cuda_fail(e_, #call); } while (0)

struct tangram_round {
  tangram_round_desc desc;
  tangram_pool_desc pools[TANGRAM_MAX_POOLS];
  Params P;                 // template: pools, sizes, workspace pointers
  int device;
  int64_t launches;
  // workspace
  void* d_order; void* d_tmin; void* d_meta; void* d_slabs; void* d_arena; void* d_arena_top;
  HeadState* hst; u32* d_ok_table; int* d_side_bad; int* d_side_res;
  int n_sm;
  ReplayWs R; int replay_smem;
  // host-buffer mode: copy-in, kernels and copy-out of successive chunks on streams of their own
  cudaStream_t io_in, io_comp, io_out;
  cudaEvent_t io_begin, io_end, io_in_done[TG_IO_CHUNKS], io_comp_done[TG_IO_CHUNKS];
  // the output fill of an ordered round runs beside its sort
  cudaStream_t side; cudaEvent_t side_fork, side_join;
  // the sorted order of tangram_schedule_batch_ordered, allocated at its first call
  int* d_perm; u64* d_wkey;
  // staging for host-buffer mode
  char* d_stage; size_t stage_bytes;
  size_t in_off[8], out_off[9];
  // optional per-kernel timing: events recorded around every kernel of a call
  cudaEvent_t* ev; int ev_calls, ev_used; int ev_kernel[TG_PROF_CALLS][TG_PROF_K];
};

static const char* const g_kernel_names[TG_N_KERNELS] = {"k_head", "k_round", "k_replay", "k_pool",
                                                          "k_stream", "k_order", "k_pin", "k_fill"};

static cudaError_t fill_tables() {
  u64 recip[33];
  recip[0] = recip[1] = 0;
  // ceil(2^64 / r) = floor((2^64 - 1) / r) + 1 for every r >= 2
  for (int r = 2; r <= 32; ++r) recip[r] = 0xffffffffffffffffull / (u64)r + 1ull;
  return cudaMemcpyToSymbol(c_recip, recip, sizeof(recip));
}

extern "C" const char* tangram_strerror(int code) {
  switch (code) {
    case TANGRAM_OK: return "ok";
    case TANGRAM_EINVAL: return "invalid argument";
    case TANGRAM_ENOMEM: return "out of device memory";
    case TANGRAM_ECUDA: return "CUDA runtime error";
    case TANGRAM_ETOOBIG: return "problem too large for the static scratch array";
    default: return "unknown error";
  }
}

extern "C" const char* tangram_last_cuda_error(void) { return g_cuda_err; }

extern "C" int64_t tangram_kernel_launches(const tangram_round* r) { return r ? r->launches : 0; }

static size_t align_up(size_t v, size_t a) { return (v + a - 1) / a * a; }

// GPU pools first (their tasks may go on evicting), then CPU pools, then API pools
static void fill_pool_order(Params& P) {
  int k = 0;
  const int rank[3] = {TG_POOL_GPU, TG_POOL_CPU, TG_POOL_API};
  for (int r = 0; r < 3; ++r)
    for (int j = 0; j < P.P; ++j)
      if (P.pool[j].type == rank[r]) P.pool_order[k++] = j;
}

// a pool has at most min(max_actions, capacity) candidates
static void fill_candidate_rows(Params& P) {
  P.cand_off[0] = 0;
  for (int j = 0; j < P.P; ++j)
    P.cand_off[j + 1] = P.cand_off[j] + (int)align_up((size_t)(P.pool[j].capacity < P.N ? P.pool[j].capacity : P.N), 8);
  P.cand_stride = P.cand_off[P.P];
}

// pools whose grants are placed one after the other in queue order with their state in registers
static int queue_place_ok(const PoolDev& d) {
  return d.type == TG_POOL_API || (d.type == TG_POOL_CPU && d.capacity / d.group <= 128 && d.group < 65536);
}

static bool has_cache(const Params& P) { return P.cache_slots > 0 && P.n_nodes_total > 0; }
static const void* round_kernel(bool cache, bool side, bool sorted) {
  if (cache) return side ? (const void*)k_round<true, false, true> : (const void*)k_round<false, false, true>;
  return side ? (const void*)k_round<true, false, false> : sorted ? (const void*)k_round<false, true, false> : (const void*)k_round<false, false, false>;
}

// The replay's instance: with the code of the extensions or not, for a round whose running actions and live state are in
// shared memory or not.  Plain replays take a plain one in either case: 1024 traces of 2000 actions on 256 cores and 8 GPUs,
// whose running actions do not fit, 9.9 ms against 12.3 with the extensions' code, 2048 on 512 cores and 64 GPUs 14.8
// against 18.5.
static const void* replay_kernel(const ReplayWs& R, bool ext) {
  if (R.rcap == 0 || R.state_bytes == 0) return ext ? (const void*)k_replay<true, false> : (const void*)k_replay<false, false>;
  return ext ? (const void*)k_replay<true, true> : (const void*)k_replay<false, true>;
}

extern "C" int tangram_round_create(const tangram_round_desc* desc, tangram_round** out) {
  if (!desc || !out || !desc->pools) return TANGRAM_EINVAL;
  if (desc->n_scenarios < 1 || desc->max_actions < 1 || desc->n_pools < 1 ||
      desc->n_pools > TANGRAM_MAX_POOLS || desc->depth < 1 || desc->depth > 32 || desc->max_rounds < 0 ||
      desc->round_us < 0 || desc->workspace_bytes < 0 || desc->slot_wait_us < 0 || desc->cache_slots < 0 ||
      desc->cache_slots > 4 || (desc->cache_slots > 0 && desc->host_buffers) || desc->side_costs < 0 ||
      desc->side_costs > 2 || (desc->side_costs > 0 && desc->host_buffers))
    return TANGRAM_EINVAL;
  if ((int64_t)desc->n_scenarios * desc->max_actions > (int64_t)1 << 31) return TANGRAM_EINVAL;
  tangram_round* r = new (std::nothrow) tangram_round();
  if (!r) return TANGRAM_ENOMEM;
  memset(r, 0, sizeof(*r));
  r->desc = *desc;
  Params& P = r->P;
  P.S = desc->n_scenarios; P.N = desc->max_actions; P.P = desc->n_pools; P.depth = desc->depth;
  P.cache_slots = desc->cache_slots;
  int node0 = 0, slot0 = 0;
  for (int j = 0; j < desc->n_pools; ++j) {
    const tangram_pool_desc& pd = desc->pools[j];
    r->pools[j] = pd;
    bool ok = pd.capacity >= 1 && pd.capacity <= (1 << 20) && pd.window_us >= 0;
    if (pd.type == TANGRAM_POOL_GPU)
      ok = ok && (pd.group == 1 || pd.group == 2 || pd.group == 4 || pd.group == 8) && pd.capacity % pd.group == 0;
    else if (pd.type == TANGRAM_POOL_CPU) ok = ok && pd.group >= 1 && pd.capacity % pd.group == 0;
    else if (pd.type != TANGRAM_POOL_API) ok = false;
    if (!ok) { delete r; return TANGRAM_EINVAL; }
    PoolDev& d = P.pool[j];
    d.type = pd.type; d.capacity = pd.capacity; d.group = pd.type == TANGRAM_POOL_API ? 1 : pd.group;
    d.window_us = pd.type == TANGRAM_POOL_API ? pd.window_us : 0;
    d.node0 = node0; d.n_nodes = pd.type == TANGRAM_POOL_GPU ? pd.capacity / pd.group : 0;
    node0 += d.n_nodes;
    d.slot0 = slot0; d.n_slots = pd.type == TANGRAM_POOL_GPU ? 4 : 1;
    slot0 += d.n_slots;
    d.queue_place = queue_place_ok(d);
  }
  r->desc.pools = r->pools;
  P.n_nodes_total = node0;
  P.V = slot0 + desc->n_pools;
  fill_pool_order(P);
  fill_candidate_rows(P);

  cudaError_t e = cudaGetDevice(&r->device);
  cudaDeviceProp prop;
  if (e == cudaSuccess) e = cudaGetDeviceProperties(&prop, r->device);
  if (e == cudaSuccess) e = fill_tables();
  if (e != cudaSuccess) { delete r; return cuda_fail(e, "device set-up"); }

  const size_t SN = (size_t)P.S * P.N, SC = (size_t)P.S * P.cand_stride;
  P.n_workers = prop.multiProcessorCount * 2 * (K2_THREADS / 32);   // what k_pool keeps resident
  if ((int64_t)P.n_workers > (int64_t)P.S * P.P) P.n_workers = (int)align_up((size_t)P.S * P.P, K2_THREADS / 32);
  // every worker warp owns a slab that holds the candidate arrays, heaps and small DP tables of
  // the pool it is working on; larger DP tables come from the shared arena
  size_t per_cand = 8 + 8 + 4 + 4 + 4 + 4 + 4 + 3 + 16 * (size_t)desc->depth;
  size_t slab = align_up((size_t)P.N * per_cand + 64 * 1024 + (1 << 20) / 4 + 4096, 256);
  P.slab_bytes = slab;
  P.arena_bytes = desc->workspace_bytes ? (u64)desc->workspace_bytes : (2ull << 30);
  {
    const int64_t us = desc->slot_wait_us ? desc->slot_wait_us : 100000;
    P.slot_tries = (int)(us / 2 > 0x3fffffff ? 0x3fffffff : (us / 2 < 1 ? 1 : us / 2));
  }
  bool bad = false;
  bad |= cudaMalloc(&r->d_order, SC * sizeof(int)) != cudaSuccess;
  bad |= cudaMalloc(&r->d_tmin, SN * sizeof(i64) * P.P) != cudaSuccess;
  bad |= cudaMalloc(&r->d_meta, (size_t)P.S * P.P * sizeof(PoolMeta)) != cudaSuccess;
  bad |= cudaMalloc((void**)&r->hst, (size_t)P.S * sizeof(HeadState)) != cudaSuccess;
  bad |= cudaMalloc(&r->d_slabs, (size_t)P.n_workers * slab) != cudaSuccess;
  bad |= cudaMalloc(&r->d_arena, P.arena_bytes) != cudaSuccess;
  bad |= cudaMalloc(&r->d_arena_top, 256) != cudaSuccess;
  if (desc->side_costs > 0) {                              // cost vectors: flags and set-aside amounts
    bad |= cudaMalloc((void**)&r->d_side_bad, (size_t)P.S * sizeof(int)) != cudaSuccess;
    bad |= cudaMalloc((void**)&r->d_side_res, (size_t)P.S * P.P * sizeof(int)) != cudaSuccess;
  }
  r->n_sm = prop.multiProcessorCount;
  if (desc->max_rounds > 0) {                              // state of the trace replay
    ReplayWs& R = r->R;
    int u = 0, d = 0, w = 0;
    for (int j = 0; j < P.P; ++j) {
      R.unit0[j] = u; R.dom0[j] = d; R.word0[j] = w;
      if (P.pool[j].type != TG_POOL_API) u += P.pool[j].capacity;
      if (P.pool[j].type == TG_POOL_GPU) w += P.pool[j].n_nodes;
      if (P.pool[j].type != TG_POOL_CPU) continue;
      R.n_dom[j] = P.pool[j].capacity / P.pool[j].group; R.wpd[j] = (P.pool[j].group + 63) / 64;
      d += R.n_dom[j]; w += 2 * R.n_dom[j] * R.wpd[j];
    }
    R.U = u ? u : 1; R.Dtot = d; R.W = w;
    R.round_us = desc->round_us > 0 ? desc->round_us : 1; R.max_rounds = desc->max_rounds;
    R.round_recip = R.round_us > 1 && R.round_us < (1 << 22) ? ~0ull / (u64)R.round_us + 1ull : 0;
    bad |= cudaMalloc((void**)&R.wait, SN * sizeof(int)) != cudaSuccess;
    // what a block (one scenario at a time) keeps in shared memory: live state, running actions, waiting records
    {
      size_t running = 0;                                  // a running action holds a unit at least, quota calls aside
      for (int j = 0; j < P.P; ++j) running += P.pool[j].type == TG_POOL_API && P.pool[j].window_us > 0 ? (size_t)P.N : (size_t)P.pool[j].capacity;
      running = align_up(running < (size_t)P.N ? running : (size_t)P.N, 8);
      // Resident blocks of an SM: all of its scenarios, or as many at a time as turns of KR_PER_SM take, so that the last turn is
      // as full as the others.  With six at most, 1024 traces of 2000 actions on 256 cores and 8 GPUs took two turns, 9.9 ms,
      // against 7.3 in one of seven (2048: 17.6 and 14.3; pinned to three nodes 17.2 and 12.3).
      size_t per_sm = ((size_t)P.S + r->n_sm - 1) / r->n_sm;
      const size_t turns = (per_sm + KR_PER_SM - 1) / KR_PER_SM;
      per_sm = (per_sm + turns - 1) / turns;
      size_t room = (size_t)TG_SMEM_PER_SM / per_sm - 1024;
      if (room > TG_REPLAY_SMEM) room = TG_REPLAY_SMEM;
      size_t left = room - KR_BASE_BYTES;
      // The live state goes to global memory where it leaves no room for KR_MIN_WAIT waiting records, each of which would be
      // decoded from scattered columns whenever it is looked at: 1024 traces on 3712 cores, state of 16 KB beside none 28.3 ms,
      // beside 128 26.0, in global memory 23.5 (seven blocks).  On 1024 cores 5 KB beside 96 records 5.5 ms, in global
      // memory 5.7.
      const size_t state = replay_state_bytes(R);
      R.state_bytes = state <= KR_STATE_MAX && state + KR_MIN_WAIT * KR_WAIT_BYTES <= left ? (int)state : 0;
      left -= (size_t)R.state_bytes;
      R.rcap = running * KR_RUN_BYTES <= left / 2 ? (int)running : 0;
      left -= (size_t)R.rcap * KR_RUN_BYTES;
      size_t wc = left / KR_WAIT_BYTES;
      if (wc > 2048) wc = 2048;
      if (wc > align_up((size_t)P.N, 32)) wc = align_up((size_t)P.N, 32);
      R.wcap = (int)(wc / 32 * 32);
      r->replay_smem = KR_BASE_BYTES + R.state_bytes + (int)align16((size_t)R.rcap * KR_RUN_BYTES) + (int)align16((size_t)R.wcap * KR_WAIT_BYTES);
      if (R.rcap == 0) {
        bad |= cudaMalloc((void**)&R.run_at, SN * sizeof(uint4)) != cudaSuccess;
        bad |= cudaMalloc((void**)&R.run_fin, SN * sizeof(i64)) != cudaSuccess;
        bad |= cudaMalloc((void**)&R.run_end, SN * sizeof(int)) != cudaSuccess;
        bad |= cudaMalloc((void**)&R.run_pu, SN * sizeof(u32)) != cudaSuccess;
        bad |= cudaMalloc((void**)&R.run_idx, SN * sizeof(int)) != cudaSuccess;
      }
    }
    bad |= cudaMalloc((void**)&R.rounds_used, (size_t)P.S * sizeof(int)) != cudaSuccess;
    if (R.state_bytes == 0) {
      bad |= cudaMalloc((void**)&R.words, (size_t)P.S * (R.W + 2) * sizeof(u32)) != cudaSuccess;
      bad |= cudaMalloc((void**)&R.dfree, (size_t)P.S * (R.Dtot + 1) * sizeof(int)) != cudaSuccess;
      bad |= cudaMalloc((void**)&R.owner, (size_t)P.S * R.U * sizeof(int)) != cudaSuccess;
    }
  }
  {
    // the fill's stream: highest priority, so that its few blocks get in between those of the sort
    int lo = 0, hi = 0;
    bad |= cudaDeviceGetStreamPriorityRange(&lo, &hi) != cudaSuccess;
    bad |= cudaStreamCreateWithPriority(&r->side, cudaStreamNonBlocking, hi) != cudaSuccess;
    bad |= cudaEventCreateWithFlags(&r->side_fork, cudaEventDisableTiming) != cudaSuccess;
    bad |= cudaEventCreateWithFlags(&r->side_join, cudaEventDisableTiming) != cudaSuccess;
  }
  if (!bad && desc->host_buffers) {
    bad |= cudaStreamCreateWithFlags(&r->io_in, cudaStreamNonBlocking) != cudaSuccess;
    bad |= cudaStreamCreateWithFlags(&r->io_comp, cudaStreamNonBlocking) != cudaSuccess;
    bad |= cudaStreamCreateWithFlags(&r->io_out, cudaStreamNonBlocking) != cudaSuccess;
    bad |= cudaEventCreateWithFlags(&r->io_begin, cudaEventDisableTiming) != cudaSuccess;
    bad |= cudaEventCreateWithFlags(&r->io_end, cudaEventDisableTiming) != cudaSuccess;
    for (int c = 0; c < TG_IO_CHUNKS; ++c) {
      bad |= cudaEventCreateWithFlags(&r->io_in_done[c], cudaEventDisableTiming) != cudaSuccess;
      bad |= cudaEventCreateWithFlags(&r->io_comp_done[c], cudaEventDisableTiming) != cudaSuccess;
    }
    size_t off = 0;
    size_t in_sz[8] = {SN, SN, SN * 4, SN * 8, SN * 8, SN * 8, (size_t)P.S * 4, (size_t)P.S * (node0 ? node0 : 1)};
    for (int k = 0; k < 8; ++k) { r->in_off[k] = off; off = align_up(off + in_sz[k], 256); }
    size_t occ = (size_t)P.S * (desc->max_rounds > 0 ? desc->max_rounds : 0) * P.P * 4;
    size_t out_sz[9] = {SN * 4, SN * 4, SN * 4, SN * 8, (size_t)P.S * 8, (size_t)P.S * 4, (size_t)P.S * 4,
                        occ ? occ : 4, (size_t)P.S * 4};
    for (int k = 0; k < 9; ++k) { r->out_off[k] = off; off = align_up(off + out_sz[k], 256); }
    r->stage_bytes = off;
    bad |= cudaMalloc((void**)&r->d_stage, off) != cudaSuccess;
  }
  if (bad) { cudaGetLastError(); tangram_round_destroy(r); return TANGRAM_ENOMEM; }
  {
    // usable multiplicities by (pool, unit byte), as decode_levels computes them
    static_assert(sizeof(u32) == 4, "");
    u32* tab = new (std::nothrow) u32[TG_MAX_POOLS * 256]();
    cudaError_t ce = tab ? cudaMalloc((void**)&r->d_ok_table, TG_MAX_POOLS * 256 * sizeof(u32)) : cudaErrorMemoryAllocation;
    if (ce == cudaSuccess) {
      for (int j = 0; j < P.P; ++j)
        for (int un = 0; un < 256; ++un) {
          const int g = un & 0x7f;
          const bool gpu = P.pool[j].type == TG_POOL_GPU, gang = (un >> 7) && gpu;
          u32 ok = g == 0 ? 0u : 0xffffffffu;
          if (g != 0 && gpu) {
            const bool p2 = (g & (g - 1)) == 0;
            if (gang) {
              ok = 0;
              if (p2) {
                if (g <= P.pool[j].group) ok |= 1u;
                if (2 * g <= P.pool[j].group) ok |= 2u;
                if (4 * g <= P.pool[j].group) ok |= 8u;
                if (8 * g <= P.pool[j].group) ok |= 128u;
              }
            } else if (!(p2 && g <= P.pool[j].group)) ok = 0;
          }
          tab[j * 256 + un] = ok;
        }
      ce = cudaMemcpy(r->d_ok_table, tab, TG_MAX_POOLS * 256 * sizeof(u32), cudaMemcpyHostToDevice);
    }
    delete[] tab;
    if (ce != cudaSuccess) { cudaGetLastError(); tangram_round_destroy(r); return TANGRAM_ENOMEM; }
    P.ok_table = r->d_ok_table;
  }
  P.order = (int*)r->d_order; P.tmin = (i64*)r->d_tmin; P.meta = (PoolMeta*)r->d_meta;
  P.n_side = desc->side_costs; P.side_plane = (u64)P.S * P.N;
  P.side_bad = r->d_side_bad; P.side_res = r->d_side_res;
  P.slabs = (char*)r->d_slabs; P.arena = (char*)r->d_arena; P.arena_top = (u64*)r->d_arena_top;
  e = cudaMemset(r->d_arena_top, 0, 256);
  // the instances that this round's calls can take (a sorted queue has no cache and no further costs)
  const bool cache = has_cache(P);
  const void* kern[3] = {cache ? (const void*)k_pool<true> : (const void*)k_pool<false>, round_kernel(cache, false, false),
                         cache || desc->side_costs > 0 ? round_kernel(cache, true, false) : round_kernel(false, false, true)};
  for (int k = 0; k < 3 && e == cudaSuccess; ++k) e = cudaFuncSetAttribute(kern[k], cudaFuncAttributeMaxDynamicSharedMemorySize, K2_DYN_SMEM);
  if (desc->max_rounds > 0) {
    // Here and not at the call, which may be captured; the same limit for every round, as it is the kernel's and not the
    // round's: another thread's round must not lower it between a call's two steps.
    for (int k = 0; k < 2 && e == cudaSuccess; ++k)
      e = cudaFuncSetAttribute(replay_kernel(r->R, k != 0), cudaFuncAttributeMaxDynamicSharedMemorySize, TG_REPLAY_SMEM);
    cudaFuncAttributes fa;
    if (e == cudaSuccess) e = cudaFuncGetAttributes(&fa, k_occupancy);      // (loads it)
  }
  if (e != cudaSuccess) { tangram_round_destroy(r); return cuda_fail(e, "cudaFuncSetAttribute"); }
  *out = r;
  return TANGRAM_OK;
}

extern "C" int tangram_set_profiling(tangram_round* r, int enable) {
  if (!r) return TANGRAM_EINVAL;
  if (enable && !r->ev) {
    const int n = TG_PROF_CALLS * (TG_PROF_K + 1);
    r->ev = new (std::nothrow) cudaEvent_t[n];
    if (!r->ev) return TANGRAM_ENOMEM;
    for (int i = 0; i < n; ++i) {
      cudaError_t e = cudaEventCreate(&r->ev[i]);
      if (e != cudaSuccess) {
        for (int k = 0; k < i; ++k) cudaEventDestroy(r->ev[k]);
        delete[] r->ev; r->ev = nullptr;
        return cuda_fail(e, "cudaEventCreate");
      }
    }
  }
  if (!enable && r->ev) {
    for (int i = 0; i < TG_PROF_CALLS * (TG_PROF_K + 1); ++i) cudaEventDestroy(r->ev[i]);
    delete[] r->ev; r->ev = nullptr;
  }
  r->ev_used = 0;
  return TANGRAM_OK;
}

extern "C" const char* tangram_kernel_name(int kernel) {
  return kernel >= 0 && kernel < TG_N_KERNELS ? g_kernel_names[kernel] : "";
}

extern "C" int tangram_kernel_time_ms(tangram_round* r, int kernel, double* total_ms, int64_t* launches) {
  if (!r || !total_ms || !launches || kernel < 0 || kernel >= TG_N_KERNELS) return TANGRAM_EINVAL;
  *total_ms = 0.0; *launches = 0;
  if (!r->ev) return TANGRAM_OK;
  for (int c = 0; c < r->ev_used; ++c)
    for (int k = 0; k < TG_PROF_K; ++k) {
      if (r->ev_kernel[c][k] != kernel) continue;
      float ms = 0.f;
      cudaEvent_t* e = r->ev + c * (TG_PROF_K + 1);
      CK(cudaEventElapsedTime(&ms, e[k], e[k + 1]));
      *total_ms += ms; *launches += 1;
    }
  return TANGRAM_OK;
}

// events of the current call, or null when timing is off or the event pool is used up
static cudaEvent_t* prof_begin(tangram_round* r, int k0, int k1, int k2) {
  if (!r->ev || r->ev_used >= TG_PROF_CALLS) return nullptr;
  int c = r->ev_used++;
  r->ev_kernel[c][0] = k0; r->ev_kernel[c][1] = k1; r->ev_kernel[c][2] = k2;
  return r->ev + c * (TG_PROF_K + 1);
}

extern "C" void tangram_round_destroy(tangram_round* r) {
  if (!r) return;
  if (r->ev) tangram_set_profiling(r, 0);
  cudaFree(r->d_order); cudaFree(r->d_tmin); cudaFree(r->d_meta); cudaFree(r->d_slabs);
  cudaFree(r->d_ok_table); cudaFree(r->d_arena); cudaFree(r->d_arena_top); cudaFree(r->d_stage); cudaFree(r->hst); cudaFree(r->d_side_bad); cudaFree(r->d_side_res); cudaFree(r->d_perm); cudaFree(r->d_wkey);
  cudaFree(r->R.wait); cudaFree(r->R.run_at); cudaFree(r->R.run_fin); cudaFree(r->R.run_end); cudaFree(r->R.run_pu); cudaFree(r->R.run_idx);
  cudaFree(r->R.words); cudaFree(r->R.dfree); cudaFree(r->R.owner); cudaFree(r->R.rounds_used);
  if (r->io_in) cudaStreamDestroy(r->io_in);
  if (r->io_comp) cudaStreamDestroy(r->io_comp);
  if (r->io_out) cudaStreamDestroy(r->io_out);
  if (r->io_begin) cudaEventDestroy(r->io_begin);
  if (r->io_end) cudaEventDestroy(r->io_end);
  for (int c = 0; c < TG_IO_CHUNKS; ++c) {
    if (r->io_in_done[c]) cudaEventDestroy(r->io_in_done[c]);
    if (r->io_comp_done[c]) cudaEventDestroy(r->io_comp_done[c]);
  }
  if (r->side) cudaStreamDestroy(r->side);
  if (r->side_fork) cudaEventDestroy(r->side_fork);
  if (r->side_join) cudaEventDestroy(r->side_join);
  delete r;
}

// Host-buffer mode: the staging area holds device copies of the caller's arrays.
static void bind_stage(tangram_round* r, const tangram_actions* a, Params& P) {
  char* d = r->d_stage;
  P.a_pool = (const u8*)(d + r->in_off[0]); P.a_unit = (const u8*)(d + r->in_off[1]);
  P.a_mask = (const u32*)(d + r->in_off[2]); P.a_s = (const i64*)(d + r->in_off[3]);
  P.a_p = (const i64*)(d + r->in_off[4]);
  P.a_arrival = a->arrival_us ? (const i64*)(d + r->in_off[5]) : nullptr;
  P.n_actions = (const int*)(d + r->in_off[6]);
  P.gpu_busy = (a->gpu_busy && P.n_nodes_total) ? (const u8*)(d + r->in_off[7]) : nullptr;
  P.o_alloc = (int*)(d + r->out_off[0]); P.o_node = (int*)(d + r->out_off[1]); P.o_off = (int*)(d + r->out_off[2]);
  P.o_act = (i64*)(d + r->out_off[3]); P.o_total = (i64*)(d + r->out_off[4]); P.o_nsel = (int*)(d + r->out_off[5]);
  P.o_status = (int*)(d + r->out_off[6]);
}

#define IO_IN 8          // input columns, the per-action ones first
#define IO_IN_ROWS 6
#define IO_OUT 7         // output columns, the per-action ones first
#define IO_OUT_ROWS 4
// inputs of scenarios [s0, s1) host -> staging
static int copy_in(tangram_round* r, const tangram_actions* a, const Params& P, int s0, int s1, cudaStream_t st, int k0 = 0, int k1 = IO_IN) {
  char* d = r->d_stage;
  const void* src[8] = {a->pool, a->unit, a->level_mask, a->s_us, a->p_us, a->arrival_us, a->n_actions, a->gpu_busy};
  const size_t per[8] = {(size_t)P.N, (size_t)P.N, (size_t)P.N * 4, (size_t)P.N * 8, (size_t)P.N * 8, (size_t)P.N * 8,
                         4, (size_t)P.n_nodes_total};
  for (int k = k0; k < k1; ++k)
    if (src[k] && per[k])
      CK(cudaMemcpyAsync(d + r->in_off[k] + per[k] * s0, (const char*)src[k] + per[k] * s0, per[k] * (s1 - s0),
                         cudaMemcpyHostToDevice, st));
  return TANGRAM_OK;
}

// results of scenarios [s0, s1) staging -> host
static int copy_out(tangram_round* r, const tangram_result* res, const Params& P, int s0, int s1, cudaStream_t st, int k0 = 0, int k1 = IO_OUT) {
  char* d = r->d_stage;
  void* dst[7] = {res->alloc_units, res->place_node, res->place_off, res->act_us, res->total_act_us,
                  res->n_selected, res->status};
  const size_t per[7] = {(size_t)P.N * 4, (size_t)P.N * 4, (size_t)P.N * 4, (size_t)P.N * 8, 8, 4, 4};
  for (int k = k0; k < k1; ++k)
    CK(cudaMemcpyAsync((char*)dst[k] + per[k] * s0, d + r->out_off[k] + per[k] * s0, per[k] * (s1 - s0),
                       cudaMemcpyDeviceToHost, st));
  return TANGRAM_OK;
}

static bool check_io(const tangram_actions* a, const tangram_result* res) {
  return a && res && a->pool && a->unit && a->level_mask && a->s_us && a->p_us && a->n_actions &&
         res->alloc_units && res->place_node && res->place_off && res->act_us && res->total_act_us &&
         res->n_selected && res->status;
}

static void bind_device_io(Params& P, const tangram_actions* a, const tangram_result* res) {
  P.a_pool = a->pool; P.a_unit = a->unit; P.a_mask = a->level_mask;
  P.a_s = (const i64*)a->s_us; P.a_p = (const i64*)a->p_us; P.a_arrival = (const i64*)a->arrival_us;
  P.n_actions = a->n_actions;
  P.gpu_busy = P.n_nodes_total ? a->gpu_busy : nullptr;
  P.a_service = a->service; P.a_restore = (const i64*)a->restore_us;
  P.cache_tag = a->gpu_cache_tag; P.cache_use = (i64*)a->gpu_cache_use;
  P.a_side_pool = a->side_pool; P.a_side_units = a->side_units;
  if (!a->side_pool) P.n_side = 0;                         // no entries handed over: the key resource only
  P.o_alloc = res->alloc_units; P.o_node = res->place_node; P.o_off = res->place_off;
  P.o_act = (i64*)res->act_us; P.o_total = (i64*)res->total_act_us;
  P.o_nsel = res->n_selected; P.o_status = res->status;
}

// The kernels of one round for the scenarios that P describes, on stream st.
static bool one_launch(const tangram_round* r) {           // all blocks of k_round are resident at once
  return r->P.S <= TG_FUSED_PER_SM * r->n_sm && r->P.S * r->P.P <= r->P.n_workers;
}

static int launch_fill(tangram_round* r, const Params& P, cudaStream_t st) {
  CK(cudaEventRecord(r->side_fork, st));
  CK(cudaStreamWaitEvent(r->side, r->side_fork, 0));
  size_t blocks = ((size_t)P.S * P.N / 4 + 256) / 256;
  if (blocks > (size_t)r->n_sm * TG_FILL_BLOCKS_PER_SM) blocks = (size_t)r->n_sm * TG_FILL_BLOCKS_PER_SM;
  k_fill<<<(unsigned)blocks, 256, 0, r->side>>>(P);
  CK(cudaEventRecord(r->side_join, r->side));
  r->launches += 1;
  return TANGRAM_OK;
}

static int run_pipeline(tangram_round* r, const Params& P, cudaStream_t st, bool timed) {
  if (one_launch(r)) {
    cudaEvent_t* ev = timed ? prof_begin(r, 1, -1, -1) : nullptr;
    if (ev) CK(cudaEventRecord(ev[0], st));
    const int smem = P.P * WARP_SMEM_BYTES + 16;
    void (*kern)(Params, int) = (void (*)(Params, int))round_kernel(has_cache(P), P.n_side > 0, P.perm != nullptr);
    kern<<<P.S, K2_THREADS, smem, st>>>(P, P.P);
    if (ev) CK(cudaEventRecord(ev[1], st));
    r->launches += 1;
    CK(cudaGetLastError());
    return TANGRAM_OK;
  }
  cudaEvent_t* ev = timed ? prof_begin(r, 0, 4, 3) : nullptr;
  CK(cudaMemsetAsync(P.arena_top, 0, 256, st));          // arena top and the task counters
  if (ev) CK(cudaEventRecord(ev[0], st));
  if (P.n_side > 0) {
    CK(cudaMemsetAsync(P.side_bad, 0, (size_t)P.S * sizeof(int), st));
    size_t blocks = ((size_t)P.S * P.N + 255) / 256;
    if (blocks > (size_t)r->n_sm * 16) blocks = (size_t)r->n_sm * 16;
    k_side_check<<<(unsigned)blocks, 256, 0, st>>>(P);
    r->launches += 1;
  }
  if (P.n_side > 0) k_head<true><<<(P.S + 7) / 8, 256, 0, st>>>(P, r->hst);
  else k_head<false><<<(P.S + 7) / 8, 256, 0, st>>>(P, r->hst);
  if (ev) CK(cudaEventRecord(ev[1], st));
  if (P.perm) k_stream<true><<<P.S, KS_THREADS, 0, st>>>(P, r->hst);
  else k_stream<false><<<P.S, KS_THREADS, 0, st>>>(P, r->hst);
  if (ev) CK(cudaEventRecord(ev[2], st));
  if (P.perm) CK(cudaStreamWaitEvent(st, r->side_join, 0));   // it wrote the candidates' rows as well
  if (has_cache(P)) k_pool<true><<<P.n_workers / (K2_THREADS / 32), K2_THREADS, K2_DYN_SMEM, st>>>(P, r->hst);
  else k_pool<false><<<P.n_workers / (K2_THREADS / 32), K2_THREADS, K2_DYN_SMEM, st>>>(P, r->hst);
  if (ev) CK(cudaEventRecord(ev[3], st));
  r->launches += 3;
  CK(cudaGetLastError());
  return TANGRAM_OK;
}

extern "C" int tangram_schedule_batch(tangram_round* r, const tangram_actions* a, int64_t now_us,
                                      tangram_result* res, void* cuda_stream) {
  if (!r || !check_io(a, res)) return TANGRAM_EINVAL;
  if (r->desc.cache_slots > 0 && r->P.n_nodes_total > 0 && (!a->gpu_cache_tag || !a->gpu_cache_use)) return TANGRAM_EINVAL;
  if (r->desc.side_costs > 0 && (!a->side_pool) != (!a->side_units)) return TANGRAM_EINVAL;
  cudaStream_t st = (cudaStream_t)cuda_stream;
  Params P = r->P;
  P.now = now_us;
  if (!r->desc.host_buffers) {
    bind_device_io(P, a, res);
    return run_pipeline(r, P, st, true);
  }
  bind_stage(r, a, P);
  // Host buffers: scenarios go through in chunks, so that the copy-in of a chunk, the kernels
  // of the one before and the copy-out of the one before that overlap (three internal streams).
  const size_t bytes = (size_t)P.S * P.N * 42;
  // A chunk costs about 80 us of calls and start-up.  On PCIe 5 two chunks pay from 16 MB on (67 MB: 1735 -> 1458 us), three
  // at 189 MB (two 3846, three 3693, eight 4078 us), six or seven at 688 MB (ten 9867, six 9565 us).
  int C = bytes < ((size_t)16 << 20) ? 1 : 2 + (int)(bytes >> 27);
  if (C > TG_IO_CHUNKS) C = TG_IO_CHUNKS;
  if (C > P.S) C = P.S;
  if (C <= 1 || r->ev) {                                   // small batch, or per-kernel timing wanted
    int rc = copy_in(r, a, P, 0, P.S, st);
    if (!rc) rc = run_pipeline(r, P, st, true);
    if (!rc) rc = copy_out(r, res, P, 0, P.S, st);
    return rc;
  }
  CK(cudaEventRecord(r->io_begin, st));
  CK(cudaStreamWaitEvent(r->io_in, r->io_begin, 0));
  CK(cudaStreamWaitEvent(r->io_comp, r->io_begin, 0));
  CK(cudaStreamWaitEvent(r->io_out, r->io_begin, 0));
  int rc = copy_in(r, a, P, 0, P.S, r->io_in, IO_IN_ROWS, IO_IN);   // what is per scenario, for all chunks
  if (rc) return rc;
  for (int c = 0; c < C; ++c) {
    const int s0 = (int)((long long)P.S * c / C), s1 = (int)((long long)P.S * (c + 1) / C);
    const size_t o = (size_t)s0 * P.N;
    rc = copy_in(r, a, P, s0, s1, r->io_in, 0, IO_IN_ROWS);
    if (rc) return rc;
    CK(cudaEventRecord(r->io_in_done[c], r->io_in));
    Params Q = P;                                          // this chunk's view of everything per scenario
    Q.S = s1 - s0;
    Q.a_pool += o; Q.a_unit += o; Q.a_mask += o; Q.a_s += o; Q.a_p += o;
    if (Q.a_arrival) Q.a_arrival += o;
    Q.n_actions += s0;
    if (Q.gpu_busy) Q.gpu_busy += (size_t)s0 * P.n_nodes_total;
    Q.o_alloc += o; Q.o_node += o; Q.o_off += o; Q.o_act += o;
    Q.o_total += s0; Q.o_nsel += s0; Q.o_status += s0;
    if ((int64_t)Q.n_workers > (int64_t)Q.S * P.P) Q.n_workers = (int)align_up((size_t)Q.S * P.P, K2_THREADS / 32);
    CK(cudaStreamWaitEvent(r->io_comp, r->io_in_done[c], 0));
    rc = run_pipeline(r, Q, r->io_comp, false);   // the workspace is reused chunk after chunk
    if (rc) return rc;
    CK(cudaEventRecord(r->io_comp_done[c], r->io_comp));
    CK(cudaStreamWaitEvent(r->io_out, r->io_comp_done[c], 0));
    rc = copy_out(r, res, P, s0, s1, r->io_out, 0, IO_OUT_ROWS);
    if (rc) return rc;
  }
  rc = copy_out(r, res, P, 0, P.S, r->io_out, IO_OUT_ROWS, IO_OUT);
  if (rc) return rc;
  CK(cudaEventRecord(r->io_end, r->io_out));
  CK(cudaStreamWaitEvent(st, r->io_end, 0));
  return TANGRAM_OK;
}

static int replay_impl(tangram_round* r, const tangram_actions* a, tangram_result* res, void* cuda_stream, int policy,
                       const tangram_pinning* pin = nullptr);

extern "C" int tangram_replay_trace(tangram_round* r, const tangram_actions* a, tangram_result* res,
                                    void* cuda_stream) {
  return replay_impl(r, a, res, cuda_stream, 0);
}

extern "C" int tangram_replay_trace_ordered(tangram_round* r, const tangram_actions* a, int policy, tangram_result* res,
                                            void* cuda_stream) {
  if (policy < 0 || policy > 3) return TANGRAM_EINVAL;
  return replay_impl(r, a, res, cuda_stream, policy == 3 ? 0 : policy);   // a trace is sorted by arrival already
}

extern "C" int tangram_replay_trace_pinned(tangram_round* r, const tangram_actions* a, int policy,
                                           const tangram_pinning* pin, tangram_result* res, void* cuda_stream) {
  if (policy < 0 || policy > 3 || !r || !pin || r->desc.host_buffers || !pin->trajectory || !pin->traj_mem ||
      pin->max_trajectories < 1 || !pin->traj_node || !pin->node_mem_free || !pin->pool_out)
    return TANGRAM_EINVAL;
  return replay_impl(r, a, res, cuda_stream, policy == 3 ? 0 : policy, pin);
}

static int replay_impl(tangram_round* r, const tangram_actions* a, tangram_result* res, void* cuda_stream, int policy,
                       const tangram_pinning* pin) {
  if (!r || !check_io(a, res) || r->desc.max_rounds <= 0 || !a->arrival_us) return TANGRAM_EINVAL;
  if (policy && !r->d_wkey) {                              // sort keys of the waiting actions, kept by the round
    if (cudaMalloc((void**)&r->d_wkey, (size_t)r->P.S * r->P.N * sizeof(u64)) != cudaSuccess) {
      cudaGetLastError(); r->d_wkey = nullptr;
      return TANGRAM_ENOMEM;
    }
  }
  if (r->desc.cache_slots > 0 && r->P.n_nodes_total > 0 && (!a->gpu_cache_tag || !a->gpu_cache_use)) return TANGRAM_EINVAL;
  if (r->desc.side_costs > 0 && (!a->side_pool) != (!a->side_units)) return TANGRAM_EINVAL;
  cudaStream_t st = (cudaStream_t)cuda_stream;
  Params P = r->P;
  P.now = 0;
  ReplayWs R = r->R;
  R.policy = policy; R.wkey = policy ? r->d_wkey : nullptr;
  R.trajectory = nullptr; R.traj_mem = nullptr; R.traj_last = nullptr; R.max_traj = 0;
  R.traj_node = nullptr; R.mem_free = nullptr; R.pool_rw = nullptr;
  if (r->desc.host_buffers) {
    bind_stage(r, a, P);
    int rc = copy_in(r, a, P, 0, P.S, st);
    if (rc) return rc;
    R.occupancy = res->occupancy ? (int*)(r->d_stage + r->out_off[7]) : nullptr;
    if (res->rounds_used) R.rounds_used = (int*)(r->d_stage + r->out_off[8]);
  } else {
    bind_device_io(P, a, res);
    R.occupancy = res->occupancy;
    if (res->rounds_used) R.rounds_used = res->rounds_used;
  }
  CK(cudaMemsetAsync(P.arena_top, 0, 256, st));
  const int blocks = P.n_workers < P.S ? P.n_workers : P.S;
  cudaEvent_t* ev = prof_begin(r, 2, -1, -1);
  if (ev) CK(cudaEventRecord(ev[0], st));
  if (R.occupancy) CK(cudaMemsetAsync(R.occupancy, 0, (size_t)P.S * R.max_rounds * P.P * sizeof(int), st));
  if (pin) {
    // the kernel reads and rewrites the caller's pool_out: it starts as a copy of the pool column
    CK(cudaMemcpyAsync(pin->pool_out, a->pool, (size_t)P.S * P.N, cudaMemcpyDeviceToDevice, st));
    P.a_pool = pin->pool_out;
    R.trajectory = pin->trajectory; R.traj_mem = pin->traj_mem; R.traj_last = pin->traj_last;
    R.max_traj = pin->max_trajectories; R.traj_node = pin->traj_node; R.mem_free = (i64*)pin->node_mem_free;
    R.pool_rw = pin->pool_out;
  }
  void (*kern)(Params, ReplayWs) = (void (*)(Params, ReplayWs))replay_kernel(R, policy || pin || P.n_side > 0 || has_cache(P));
  kern<<<blocks, KR_THREADS, r->replay_smem, st>>>(P, R);
  if (R.occupancy) { k_occupancy<<<P.S, 256, 0, st>>>(P.P, R.max_rounds, R.rounds_used, P.o_status, R.occupancy); r->launches += 1; }
  if (ev) CK(cudaEventRecord(ev[1], st));
  CK(cudaMemsetAsync(P.arena_top, 0, 256, st));            // k_round starts from counters at zero
  r->launches += 1;
  CK(cudaGetLastError());
  if (r->desc.host_buffers) {
    int rc = copy_out(r, res, P, 0, P.S, st);
    if (rc) return rc;
    if (res->occupancy)
      CK(cudaMemcpyAsync(res->occupancy, r->d_stage + r->out_off[7],
                         (size_t)P.S * r->desc.max_rounds * P.P * sizeof(int), cudaMemcpyDeviceToHost, st));
    if (res->rounds_used)
      CK(cudaMemcpyAsync(res->rounds_used, r->d_stage + r->out_off[8], (size_t)P.S * sizeof(int), cudaMemcpyDeviceToHost, st));
  }
  return TANGRAM_OK;
}

// ---------------------------------------------------------------------------------------
// Other queue orders (Section 4.2) and trajectories pinned to CPU nodes (Section 5.2)
// ---------------------------------------------------------------------------------------
// Threads and actions per thread of the sort: enough blocks on an SM to hide its barriers, and few idle threads on short queues.
static int launch_order(tangram_round* r, const Params& P, int policy, int* perm, cudaStream_t st) {
  OrderIo O;
  O.policy = policy; O.perm = perm;
  const int threads = P.N <= 512 ? 128 : P.N <= 1024 ? 256 : KO_MAX_THREADS;
  int ept = 1;
  while (ept * threads < P.N) ept <<= 1;
  const size_t sm = (size_t)ept * threads * 8 + ko_counter_bytes(ept, threads);
  void (*kern)(Params, OrderIo) = ept == 1 ? k_order<1> : ept == 2 ? k_order<2> : ept == 4 ? k_order<4> :
                                  ept == 8 ? k_order<8> : ept == 16 ? k_order<16> : k_order<32>;
  if (sm > 40 * 1024) CK(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm));
  kern<<<P.S, threads, sm, st>>>(P, O);
  r->launches += 1;
  CK(cudaGetLastError());
  return TANGRAM_OK;
}

static bool order_args_ok(const tangram_round* r, const tangram_actions* a, int policy) {
  return r && a && a->pool && a->unit && a->level_mask && a->s_us && a->p_us && a->n_actions &&
         policy >= 1 && policy <= 3 && !r->desc.host_buffers;
}

extern "C" int tangram_order_queue(tangram_round* r, const tangram_actions* a, int policy, int32_t* perm,
                                   void* cuda_stream) {
  if (!order_args_ok(r, a, policy) || !perm) return TANGRAM_EINVAL;
  if (r->P.N > KO_MAX_N) return TANGRAM_ETOOBIG;
  Params P = r->P;
  P.a_pool = a->pool; P.a_unit = a->unit; P.a_mask = a->level_mask;
  P.a_s = (const i64*)a->s_us; P.a_p = (const i64*)a->p_us; P.a_arrival = (const i64*)a->arrival_us;
  P.n_actions = a->n_actions;
  return launch_order(r, P, policy, perm, (cudaStream_t)cuda_stream);
}

extern "C" int tangram_schedule_batch_ordered(tangram_round* r, const tangram_actions* a, int policy, int64_t now_us,
                                              tangram_result* res, void* cuda_stream) {
  if (!r || !check_io(a, res)) return TANGRAM_EINVAL;
  if (policy == 0) return tangram_schedule_batch(r, a, now_us, res, cuda_stream);
  if (!order_args_ok(r, a, policy) || r->desc.cache_slots > 0 || r->desc.side_costs > 0) return TANGRAM_EINVAL;
  if (r->P.N > KO_MAX_N) return TANGRAM_ETOOBIG;
  cudaStream_t st = (cudaStream_t)cuda_stream;
  Params P = r->P;
  P.now = now_us;
  bind_device_io(P, a, res);
  if (!r->d_perm && cudaMalloc((void**)&r->d_perm, (size_t)P.S * P.N * sizeof(int)) != cudaSuccess) {
    cudaGetLastError(); r->d_perm = nullptr;
    return TANGRAM_ENOMEM;
  }
  P.perm = r->d_perm;
  if (!one_launch(r)) { const int rc = launch_fill(r, P, st); if (rc) return rc; }   // beside the sort
  const int rc = launch_order(r, P, policy, r->d_perm, st);
  return rc ? rc : run_pipeline(r, P, st, false);
}

extern "C" int tangram_pin_trajectories(tangram_round* r, const tangram_actions* a, const tangram_pinning* pin,
                                        void* cuda_stream) {
  if (!r || !a || !pin || !a->pool || !a->unit || !a->level_mask || !a->n_actions || r->desc.host_buffers ||
      !pin->trajectory || !pin->traj_mem || pin->max_trajectories < 1 || !pin->traj_node || !pin->node_mem_free ||
      !pin->pool_out || !pin->n_admitted)
    return TANGRAM_EINVAL;
  Params P = r->P;
  P.a_pool = a->pool; P.a_unit = a->unit; P.a_mask = a->level_mask; P.n_actions = a->n_actions;
  PinIo X;
  X.trajectory = pin->trajectory; X.traj_mem = pin->traj_mem; X.max_traj = pin->max_trajectories;
  X.traj_node = pin->traj_node; X.mem_free = (i64*)pin->node_mem_free; X.pool_out = pin->pool_out;
  X.n_admitted = pin->n_admitted;
  k_pin<<<(P.S + 7) / 8, 256, 0, (cudaStream_t)cuda_stream>>>(P, X);
  r->launches += 1;
  CK(cudaGetLastError());
  return TANGRAM_OK;
}

// ---------------------------------------------------------------------------------------
// tangram_schedule_batch_static: the same round for callers that must not allocate.
// All scratch (partition order, least-level durations, per-pool facts, worker slabs, DP arena)
// is carved out of one file-scope device array that every GPU loading this library holds
// until the process exits.
// ---------------------------------------------------------------------------------------
static __device__ __align__(256) unsigned char g_static_scratch[TANGRAM_STATIC_SCRATCH_BYTES];

#define TG_MAX_DEVICES 64
static unsigned char* g_static_ptr[TG_MAX_DEVICES];   // device address of the array, per device
static bool g_static_ready[TG_MAX_DEVICES];

// Once per device, with that device current: resolve the array's device address (its name is
// only a host-side handle here and must not be handed to a kernel) and load the constant tables.
static int static_setup(int* dev_out) {
  int dev = -1;
  CK(cudaGetDevice(&dev));
  if (dev < 0 || dev >= TG_MAX_DEVICES) return TANGRAM_EINVAL;
  if (!g_static_ready[dev]) {
    unsigned char* ptr = nullptr;
    CK(cudaGetSymbolAddress((void**)&ptr, g_static_scratch));
    CK(fill_tables());
    CK(cudaFuncSetAttribute(k_round<false, false, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, K2_DYN_SMEM));
    g_static_ptr[dev] = ptr;
    g_static_ready[dev] = true;
  }
  *dev_out = dev;
  return TANGRAM_OK;
}

extern "C" int tangram_schedule_batch_static(const tangram_round_desc* desc, const tangram_actions* a,
                                             int64_t now_us, tangram_result* res, void* cuda_stream) {
  if (!desc || !desc->pools || !check_io(a, res)) return TANGRAM_EINVAL;
  if (desc->n_scenarios < 1 || desc->max_actions < 1 || desc->n_pools < 1 ||
      desc->n_pools > TANGRAM_MAX_POOLS || desc->depth < 1 || desc->depth > 32 || desc->host_buffers ||
      desc->cache_slots != 0 || desc->side_costs != 0)
    return TANGRAM_EINVAL;
  if ((int64_t)desc->n_scenarios * desc->max_actions > (int64_t)1 << 31) return TANGRAM_ETOOBIG;
  Params P;
  memset(&P, 0, sizeof(P));
  P.S = desc->n_scenarios; P.N = desc->max_actions; P.P = desc->n_pools; P.depth = desc->depth;
  int node0 = 0, slot0 = 0;
  for (int j = 0; j < desc->n_pools; ++j) {
    const tangram_pool_desc& pd = desc->pools[j];
    bool ok = pd.capacity >= 1 && pd.capacity <= (1 << 20) && pd.window_us >= 0;
    if (pd.type == TANGRAM_POOL_GPU)
      ok = ok && (pd.group == 1 || pd.group == 2 || pd.group == 4 || pd.group == 8) && pd.capacity % pd.group == 0;
    else if (pd.type == TANGRAM_POOL_CPU) ok = ok && pd.group >= 1 && pd.capacity % pd.group == 0;
    else if (pd.type != TANGRAM_POOL_API) ok = false;
    if (!ok) return TANGRAM_EINVAL;
    PoolDev& d = P.pool[j];
    d.type = pd.type; d.capacity = pd.capacity; d.group = pd.type == TANGRAM_POOL_API ? 1 : pd.group;
    d.window_us = pd.type == TANGRAM_POOL_API ? pd.window_us : 0;
    d.node0 = node0; d.n_nodes = pd.type == TANGRAM_POOL_GPU ? pd.capacity / pd.group : 0;
    node0 += d.n_nodes;
    d.slot0 = slot0; d.n_slots = pd.type == TANGRAM_POOL_GPU ? 4 : 1;
    slot0 += d.n_slots;
    d.queue_place = queue_place_ok(d);
  }
  P.n_nodes_total = node0;
  P.V = slot0 + desc->n_pools;
  fill_pool_order(P);
  fill_candidate_rows(P);
  P.now = now_us;

  // what a batch may need at most is fixed by the header; the scratch itself is per block, as many as fit
  const size_t SN = (size_t)P.S * P.N;
  const size_t budget = TANGRAM_STATIC_SCRATCH_BYTES, arena_min = (size_t)4 << 20;
  const size_t per_cand = 8 + 8 + 4 + 4 + 4 + 4 + 4 + 3 + 16 * (size_t)desc->depth;
  const size_t slab = align_up((size_t)P.N * per_cand + 64 * 1024 + (1 << 20) / 4 + 4096, 256);
  if (256 + align_up((size_t)P.S * P.P * sizeof(PoolMeta), 256) + align_up(SN * sizeof(int), 256) + align_up(SN * sizeof(i64), 256) +
      arena_min + slab * (K2_THREADS / 32) > budget) return TANGRAM_ETOOBIG;
  const size_t b_meta = align_up((size_t)P.P * sizeof(PoolMeta), 256), b_order = align_up((size_t)P.cand_stride * sizeof(int), 256),
               b_tmin = align_up((size_t)P.P * P.N * sizeof(i64), 256), room = budget - arena_min - 256;
  int wpb = P.P;                                           // the rows of one block are per pool: with many pools of long queues
  while (wpb > 1 && b_meta + b_order + b_tmin + slab * wpb > room) --wpb;   // a block has fewer slabs than pools
  const size_t per_block = b_meta + b_order + b_tmin + slab * wpb;
  size_t blocks = room / per_block;
  if (blocks > (size_t)P.S) blocks = (size_t)P.S;
  if (blocks < 1) return TANGRAM_ETOOBIG;
  const size_t o_meta = 256, o_order = o_meta + blocks * b_meta, o_tmin = o_order + blocks * b_order, o_slabs = o_tmin + blocks * b_tmin,
               o_arena = o_slabs + blocks * slab * wpb;

  int dev = -1;
  int rc = static_setup(&dev);
  if (rc) return rc;
  unsigned char* base = g_static_ptr[dev];
  P.arena_top = (u64*)base; P.meta = (PoolMeta*)(base + o_meta);
  P.order = (int*)(base + o_order); P.tmin = (i64*)(base + o_tmin);
  P.slabs = (char*)(base + o_slabs); P.slab_bytes = slab; P.n_workers = (int)blocks * wpb;
  P.arena = (char*)(base + o_arena); P.arena_bytes = budget - o_arena;
  P.slot_tries = 50000;
  bind_device_io(P, a, res);

  cudaStream_t st = (cudaStream_t)cuda_stream;
  CK(cudaMemsetAsync(P.arena_top, 0, 256, st));           // whatever an overlapping call may have left
  k_round<false, false, false><<<(unsigned)blocks, K2_THREADS, wpb * WARP_SMEM_BYTES + 16, st>>>(P, wpb);
  CK(cudaGetLastError());
  return TANGRAM_OK;
}
