// Device-resident trace replay (workflow of Section 3: submit, queue, schedule, execute,
// return), one warp per scenario, no host round trips.  Every round at now = r * round_us
//   1. refills quota pools whose window changed (Section 5.1),
//   2. releases what has finished (cores, chunks, concurrency slots),
//   3. admits the actions that have arrived to the waiting queue,
//   4. runs the scheduler of Algorithm 1 on the queue with the running actions of a pool in
//      its completion heap (Algorithm 2), using the same per-pool routines as a single round,
//   5. starts what was selected and records the occupancy.
// Rounds in which nothing can change are jumped over (their occupancy rows are still written).
//
// A scenario is one long chain of dependent rounds, each of which handles one or two actions, so what
// counts is the latency of a round: the records of the waiting actions (decoded once, on arrival), the
// running actions with their completion times, the owner of every core and GPU and the free counts sit in
// the warp's shared memory, arrivals are read 32 at a time into lane registers, the demand of every pool
// and chunk level is one lane's register, and pools without a choice to make (one candidate, or
// none elastic) never build the arrays of the selection.  What was spent per worked round before: about
// 15000 cycles, most of them dependent loads of scattered records and instruction fetch.
#pragma once
#include "common.cuh"
#include "arrange.cuh"
#include "evict.cuh"
#include "place.cuh"
#include "order_pin.cuh"

struct ReplayWs {
  int* wait;        // [S][N] waiting actions behind the first wcap, by queue position
  u64* wkey;        // [S][N] their sort keys (policy 1 / 2 only)
  int* owner;       // [S][U]  action holding each core / GPU (-1 free, -2 occupied beforehand)
  u8* nm;           // [S][nodes] GPU busy masks
  int* dfree;       // [S][Dtot] free cores per NUMA domain
  int* pst;         // [S][P][2] quota used in the window / concurrency slots in use
  i64* win;         // [S][P] current quota window
  // running actions where they do not fit shared memory: completion, action, pool << 24 | units, lowest core, domain
  i64* run_fin; int* run_idx; u32* run_pu; int* run_off; int* run_dom;
  int unit0[TG_MAX_POOLS], dom0[TG_MAX_POOLS];   // first unit / domain of every pool in a row
  int U, Dtot;
  i64 round_us; int max_rounds;
  int* occupancy; int* rounds_used;
  int policy;       // 0: first come first served; 1 / 2: the queue is kept in shortest / longest least-level duration order
  // trajectories pinned to CPU nodes as their actions arrive (Section 5.2); trajectory == nullptr: none of it
  const int* trajectory; const u32* traj_mem; const u8* traj_last; int max_traj;
  int* traj_node; i64* mem_free; u8* pool_rw;   // pool_rw: the pool column the kernel reads (P.a_pool) and rewrites
  int state_bytes;  // > 0: a scenario's live state (owner .. win) takes that many bytes of the warp's shared memory
  int wcap, rcap;   // waiting records / running actions in shared memory (rcap 0: running actions in global memory)
};

__host__ __device__ __forceinline__ size_t align16(size_t v) { return (v + 15) & ~(size_t)15; }

#define KR_THREADS 32
#define KR_FAST_BYTES 8192        // shared-memory window of the selection's arrays
#define KR_WAIT_BYTES 58          // per waiting record: s, p, least duration, arrival, key, action, packed meta, mask, queue, free list, unit
#define KR_RUN_BYTES 24
#define KR_STATE_MAX 16384
// shared memory of a block (one warp) without the parts sized by the round
#define KR_BASE_BYTES (WARP_SMEM_BYTES + KR_FAST_BYTES + 64)

// Waiting records: slots that do not move, and the queue as slot numbers.  meta: pool (4 bits), first demand slot
// (6), chunk class of the least level (2), units of the least level (13); bit 31: started in this round.
struct ReplayQueue {
  i64* s; i64* p; i64* tl; i64* arr; u64* key; int* idx; u32* meta; u32* mask; u8* cg; unsigned short* q; unsigned short* free;
  int cap;
};
#define RQ_POOL(m) ((int)((m) & 15u))
#define RQ_SLOT(m) ((int)(((m) >> 4) & 63u))
#define RQ_CLASS(m) ((int)(((m) >> 10) & 3u))
#define RQ_UNITS(m) ((int)(((m) >> 12) & 0x1fffu))
#define RQ_STARTED 0x80000000u
struct ReplayRun { i64* fin; int* idx; u32* pu; int* off; int* dom; };   // dom: NUMA domain of a core grant, -1 where it spans several

// A decoded record
struct ReplayRec { i64 s, p, tl, arr; u32 meta, mask; u8 cg; };
__device__ __forceinline__ ReplayRec replay_decode(const Params& P, int j, u32 unit, u32 mk, i64 s, i64 p) {
  ReplayRec r;
  const PoolDev& pd = P.pool[j];
  int g, gang; u32 eff;
  decode_levels(pd, (u8)unit, mk, g, gang, eff);
  const int rmin = __ffs(eff), c = pd.type == TG_POOL_GPU ? level_of(g, gang, rmin) : 0;
  r.s = clamp_param(s); r.p = clamp_param(p); r.tl = duration(r.s, r.p, rmin);
  r.mask = eff; r.cg = (u8)(g | (gang << 7));
  r.meta = (u32)j | ((u32)pd.slot0 << 4) | ((u32)c << 10) | ((u32)(g * rmin) << 12);
  return r;
}
// the waiting record at a queue position (any lane's own)
__device__ __forceinline__ ReplayRec replay_rec(const Params& P, const ReplayQueue& Q, const int* wait, size_t row, int i, int& a) {
  if (i < Q.cap) {
    const int x = Q.q[i];
    ReplayRec r;
    r.s = Q.s[x]; r.p = Q.p[x]; r.tl = Q.tl[x]; r.arr = Q.arr[x]; r.meta = Q.meta[x]; r.mask = Q.mask[x]; r.cg = Q.cg[x];
    a = Q.idx[x];
    return r;
  }
  a = wait[i];
  ReplayRec r = replay_decode(P, P.a_pool[row + a], P.a_unit[row + a], P.a_mask[row + a], P.a_s[row + a], P.a_p[row + a]);
  r.arr = P.a_arrival ? P.a_arrival[row + a] : 0;
  return r;
}
__device__ __forceinline__ u32 replay_meta(const Params& P, const ReplayQueue& Q, const int* wait, size_t row, int i) {
  if (i < Q.cap) return Q.meta[Q.q[i]];
  const int a = wait[i];
  return replay_decode(P, P.a_pool[row + a], P.a_unit[row + a], P.a_mask[row + a], 0, 0).meta;
}

// Live state of the scenario at hand: in the warp's shared memory, or in the arrays of ReplayWs where it is large.
struct ReplayState { int* owner; u8* nm; int* dfree; int* pst; i64* win; };

// One grant on a core pool with cores in use (fewest free cores that still fit, lowest domain,
// lowest cores first; else ascending domains).  fit: the domain, -1 where the grant spans several.
__device__ __forceinline__ void replay_place_cpu(const PoolDev& pd, int* owner, int* dfree, int k, int id, int lane, int& node, int& off, int& fit) {
  const int D = pd.capacity / pd.group;
  u32 best = 0xffffffffu; int dom = -1;
#pragma unroll 1
  for (int d = lane; d < D; d += 32) { const int f = dfree[d]; if (f >= k && (u32)f < best) { best = (u32)f; dom = d; } }
  const u32 mn = __reduce_min_sync(TG_FULL, best);
  int lo = 0, hi = pd.capacity, d1 = -1;
  if (mn != 0xffffffffu) {
    d1 = (int)__reduce_min_sync(TG_FULL, best == mn ? (u32)dom : 0xffffffffu);
    lo = d1 * pd.group; hi = lo + pd.group;
  }
  int need = k, first = -1;
#pragma unroll 1
  for (int c0 = lo; c0 < hi && need > 0; c0 += 32) {
    const int c = c0 + lane;
    const u32 b = __ballot_sync(TG_FULL, c < hi && owner[c] < 0);
    const int rank = __popc(b & ((1u << lane) - 1u));
    const bool mine = ((b >> lane) & 1u) && rank < need;
    if (mine) owner[c] = id;
    if (b && first < 0) first = c0 + __ffs(b) - 1;
    const int got = min(need, __popc(b));
    if (d1 < 0 && mine) atomicSub(&dfree[c / pd.group], 1);
    need -= got;
  }
  if (d1 >= 0 && lane == 0) dfree[d1] -= k;
  node = d1 >= 0 ? d1 : (first >= 0 ? first / pd.group : -1); off = first; fit = d1;
  __syncwarp();
}

// One candidate alone on a GPU pool: nreq chunks of 2^lz GPUs (Section 5.3: smallest sufficient maximal free block,
// lowest node, lowest start); node / off: the first chunk.
__device__ __forceinline__ void replay_place_gpu(const PoolDev& pd, u8* nm, int* owner, int lz, int nreq, int id, int lane, int& node, int& off) {
  const int top = ilog2(pd.group), z = 1 << lz;
  const u32 pad = (~((1u << pd.group) - 1u)) & 0xffu;
  node = -1; off = -1;
#pragma unroll 1
  for (int rep = 0; rep < nreq; ++rep) {
    int at = -1, level = 4;
#pragma unroll 1
    for (int v0 = 0; v0 < pd.n_nodes; v0 += 32) {
      const u32 lev = v0 + lane < pd.n_nodes ? node_levels(nm[v0 + lane] | pad) & (~0u << lz) : 0u;
      const int mine = lev ? __ffs(lev) - 1 : 4;           // the smallest sufficient block of the lane's node
      const int best = __reduce_min_sync(TG_FULL, mine);
      if (best < level) { level = best; at = v0 + __ffs(__ballot_sync(TG_FULL, mine == best)) - 1; }
      if (level == lz) break;
    }
    if (at < 0 || level > top) continue;                  // cannot happen: the selection fits
    const u32 busy = nm[at] | pad;
    const int start = node_block_start(busy, level);
    __syncwarp();
    if (lane == 0) nm[at] |= (u8)(((1u << z) - 1u) << start);
    if (lane < z) owner[at * pd.group + start + lane] = id;
    if (rep == 0) { node = at; off = start; }
    __syncwarp();
  }
}

// The selection of a pool with a choice to make: its candidates (among the first n positions) and, where an eviction
// step can look at them, the waiting actions behind and the running ones are gathered into arrays.
template <bool EXT>
__device__ __forceinline__ bool replay_select(const Params& P, const ReplayQueue Q, const ReplayRun run, const int* wait, int sc, int j,
                                           int n, int nw, int nr, int m, i64 now, int cap0, int cap1, int cap2, int cap3, Slab& slab,
                                           CandArrays& C, int& keep, int lane) {
  const size_t row = (size_t)sc * P.N;
  const PoolDev& pd = P.pool[j];
  C.cg = (u8*)slab.take_fast(m); C.rsel = (u8*)slab.take_fast(m); C.rkeep = (u8*)slab.take_fast(m);
  C.cmask = (u32*)slab.take_fast((u64)m * 4); C.rowcand = (int*)slab.take_fast((u64)m * 4);
  C.cs = (i64*)slab.take_fast((u64)m * 8); C.cp = (i64*)slab.take_fast((u64)m * 8);
  C.cidx = (int*)slab.take_fast((u64)m * 4); C.pnode = (int*)slab.take_fast((u64)m * 4); C.poff = (int*)slab.take_fast((u64)m * 4);
  if (!C.cg || !C.rsel || !C.rkeep || !C.cmask || !C.rowcand || !C.cs || !C.cp || !C.cidx || !C.pnode || !C.poff) return false;
  int cm = 0;
  bool elastic = false;
#pragma unroll 1
  for (int i0 = 0; i0 < n; i0 += 32) {
    const int i = i0 + lane;
    int a = 0; ReplayRec r; r.meta = 15u;
    if (i < n) r = replay_rec(P, Q, wait, row, i, a);
    const bool mine = i < n && RQ_POOL(r.meta) == j;
    const u32 b = __ballot_sync(TG_FULL, mine);
    if (mine) {
      const int k = cm + __popc(b & ((1u << lane) - 1u));
      C.cidx[k] = a; C.cmask[k] = r.mask; C.cg[k] = r.cg; C.cs[k] = r.s; C.cp[k] = r.p;
      C.rkeep[k] = (u8)__ffs(r.mask); C.pnode[k] = -1; C.poff[k] = -1;
      elastic |= (r.mask & (r.mask - 1)) != 0;
    }
    cm += __popc(b);
  }
  elastic = __any_sync(TG_FULL, elastic);
  __syncwarp();
  keep = m;
  if (!elastic) return true;
  PoolTask& T = warp_task();
  i64* ac = nullptr; i64* seeds = nullptr;
  int n_ac = 0, ns = 0, first = -1;
  if (m >= 2) {                                           // (a single candidate is never evicted)
    ac = (i64*)slab.take_fast((u64)(nw - n + 1) * 8);
    seeds = (i64*)slab.take_fast((u64)(nr + 1) * 8);
    if (!ac || !seeds) return false;
#pragma unroll 1
    for (int i0 = n; i0 < nw; i0 += 32) {
      const int i = i0 + lane;
      int a; ReplayRec r; r.meta = 15u;
      if (i < nw) r = replay_rec(P, Q, wait, row, i, a);
      const u32 b = __ballot_sync(TG_FULL, i < nw && RQ_POOL(r.meta) == j);
      if ((b >> lane) & 1u) ac[n_ac + __popc(b & ((1u << lane) - 1u))] = r.tl;
      if (first < 0 && b) first = i0 + __ffs(b) - 1;
      n_ac += __popc(b);
    }
    // completion times (relative to now) of what runs on this pool seed the heap
#pragma unroll 1
    for (int i0 = 0; i0 < nr; i0 += 32) {
      const int i = i0 + lane;
      const u32 b = __ballot_sync(TG_FULL, i < nr && (int)(run.pu[i] >> 24) == j);
      if ((b >> lane) & 1u) { const i64 f = run.fin[i]; seeds[ns + __popc(b & ((1u << lane) - 1u))] = f > now ? f - now : 0; }
      ns += __popc(b);
    }
  }
  __syncwarp();
  if (lane == 0) {
    T.type = pd.type; T.group = pd.group;
    T.cap[0] = cap0; T.cap[1] = cap1; T.cap[2] = cap2; T.cap[3] = cap3;
    T.m = m; T.cs = C.cs; T.cp = C.cp; T.cmask = C.cmask; T.cg = C.cg;
    T.n_ac = n_ac; T.ac_tmin = ac;
    T.ac_first.s = T.ac_first.p = 0; T.ac_first.mask = 1; T.ac_first.g = 1; T.ac_first.gang = 0;
    if (first >= 0) {
      int a;
      const ReplayRec r = replay_rec(P, Q, wait, row, first, a);
      T.ac_first.s = r.s; T.ac_first.p = r.p; T.ac_first.mask = r.mask; T.ac_first.g = r.cg & 0x7f; T.ac_first.gang = r.cg >> 7;
    }
    T.seeds = seeds; T.n_seeds = ns;
    T.depth = P.depth;
    T.rsel = C.rsel; T.rkeep = C.rkeep; T.rowcand = C.rowcand;
    T.wk = warp_smem(); T.wk_bytes = WARP_WORK_BYTES;
  }
  __syncwarp();
  keep = evict_loop(P, T, slab, lane);
  return keep >= 0;
}

// EXT: the queue may be kept sorted by R.policy's key, trajectories pinned on arrival (R.trajectory), further cost-vector
// entries (n_side) and a service cache; the plain instance carries none of their code.
template <bool EXT>
__global__ void __launch_bounds__(KR_THREADS, 1) k_replay(const __grid_constant__ Params P, const __grid_constant__ ReplayWs R) {
  extern __shared__ __align__(16) unsigned char k2_smem[];
  const int lane = threadIdx.x;
  const u32 below = (1u << lane) - 1u;
  char* const sm = (char*)(((u64)k2_smem + 15u) & ~(u64)15);
  char* const fast = sm + WARP_SMEM_BYTES;
  // per-warp arrays behind the selection's work area
  ReplayQueue Q;
  Q.cap = R.wcap;
  {
    char* at = fast + KR_FAST_BYTES;
    Q.s = (i64*)at; Q.p = Q.s + Q.cap; Q.tl = Q.p + Q.cap; Q.arr = Q.tl + Q.cap; Q.key = (u64*)(Q.arr + Q.cap);
    at = (char*)(Q.key + (EXT ? Q.cap : 0));
    Q.idx = (int*)at; Q.meta = (u32*)(Q.idx + Q.cap); Q.mask = Q.meta + Q.cap;
    Q.q = (unsigned short*)(Q.mask + Q.cap); Q.free = Q.q + Q.cap; Q.cg = (u8*)(Q.free + Q.cap);
  }
  char* const run_at = fast + KR_FAST_BYTES + align16((size_t)Q.cap * KR_WAIT_BYTES);
  char* const state_at = run_at + align16((size_t)R.rcap * KR_RUN_BYTES);
#pragma unroll 1
  for (int sc = blockIdx.x; sc < P.S; sc += gridDim.x) {
    const size_t row = (size_t)sc * P.N;
    const int n_act = uniform(min(max(P.n_actions[sc], 0), P.N));
    int* wait = R.wait + row; u64* wkey = EXT && R.wkey ? R.wkey + row : nullptr;
    ReplayRun run;
    if (R.rcap > 0) { run.fin = (i64*)run_at; run.idx = (int*)(run.fin + R.rcap); run.pu = (u32*)(run.idx + R.rcap); run.off = (int*)(run.pu + R.rcap); run.dom = run.off + R.rcap; }
    else { run.fin = R.run_fin + row; run.idx = R.run_idx + row; run.pu = R.run_pu + row; run.off = R.run_off + row; run.dom = R.run_dom + row; }
    ReplayState Z;
    if (R.state_bytes > 0) {
      const size_t o_nm = align16((size_t)R.U * 4), o_df = o_nm + align16((size_t)P.n_nodes_total + 1),
                   o_ps = o_df + align16((size_t)R.Dtot * 4), o_wn = o_ps + align16((size_t)P.P * 8);
      Z.owner = (int*)state_at; Z.nm = (u8*)(state_at + o_nm); Z.dfree = (int*)(state_at + o_df);
      Z.pst = (int*)(state_at + o_ps); Z.win = (i64*)(state_at + o_wn);
    } else {
      Z.owner = R.owner + (size_t)sc * R.U; Z.nm = R.nm + (size_t)sc * P.n_nodes_total; Z.dfree = R.dfree + (size_t)sc * R.Dtot;
      Z.pst = R.pst + (size_t)sc * P.P * 2; Z.win = R.win + (size_t)sc * P.P;
    }
    int* occ = R.occupancy ? R.occupancy + (size_t)sc * R.max_rounds * P.P : nullptr;
    // outputs and state start empty
#pragma unroll 4
    for (int i = lane; i < P.N; i += 32) { P.o_alloc[row + i] = 0; P.o_node[row + i] = -1; P.o_off[row + i] = -1; P.o_act[row + i] = -1; }
    int status = 0;
#pragma unroll 1
    for (int i = lane; i < n_act; i += 32) {
      const int j = P.a_pool[row + i];
      int g, gang; u32 eff;
      if (j >= P.P || !decode_levels(P.pool[j], P.a_unit[row + i], P.a_mask[row + i], g, gang, eff)) status |= TG_ST_BAD_ACTION;
      if (EXT)
#pragma unroll 1
        for (int e = 0; e < P.n_side; ++e) {                // further entries: a quota / concurrency pool other than j, 1 .. capacity
          const int k = P.a_side_pool[e * P.side_plane + row + i];
          if (k == 0xff) continue;
          const int c = P.a_side_units[e * P.side_plane + row + i];
          if (k >= P.P || P.pool[k < P.P ? k : 0].type != TG_POOL_API || k == j || c < 1 || c > P.pool[k < P.P ? k : 0].capacity)
            status |= TG_ST_BAD_ACTION;
        }
      if (i > 0 && P.a_arrival && P.a_arrival[row + i - 1] > P.a_arrival[row + i]) status |= TG_ST_UNSORTED;
    }
    status = __reduce_or_sync(TG_FULL, status);
    if (status & TG_ST_BAD_ACTION) status = TG_ST_BAD_ACTION;
    int busy = 0;                                          // lane j: units in use of core / GPU pool j
#pragma unroll 1
    for (int j = 0; j < P.P; ++j) {
      const PoolDev& pd = P.pool[j];
      if (pd.type == TG_POOL_API) { if (lane < 2) Z.pst[j * 2 + lane] = 0; if (lane == 0) Z.win[j] = 0; continue; }
      int taken = 0;
#pragma unroll 1
      for (int c = lane; c < pd.capacity; c += 32) {
        int v = -1;
        if (pd.type == TG_POOL_GPU && P.gpu_busy && (P.gpu_busy[(size_t)sc * P.n_nodes_total + pd.node0 + c / pd.group] >> (c % pd.group) & 1)) { v = -2; ++taken; }
        Z.owner[R.unit0[j] + c] = v;
      }
      taken = warp_sum32(taken);
      if (lane == j) busy = taken;
      if (pd.type == TG_POOL_GPU)
#pragma unroll 1
        for (int v = lane; v < pd.n_nodes; v += 32)
          Z.nm[pd.node0 + v] = (P.gpu_busy ? P.gpu_busy[(size_t)sc * P.n_nodes_total + pd.node0 + v] : 0) & ((1u << pd.group) - 1u);
      if (pd.type == TG_POOL_CPU)
#pragma unroll 1
        for (int d = lane; d < pd.capacity / pd.group; d += 32) Z.dfree[R.dom0[j] + d] = pd.group;
    }
#pragma unroll 1
    for (int i = lane; i < Q.cap; i += 32) Q.free[i] = (unsigned short)i;
    if (occ)
#pragma unroll 4
      for (int i = lane; i < R.max_rounds * P.P; i += 32) occ[i] = 0;
    __syncwarp();
    int rounds = 0;
    if (status == 0) {
      int next = 0, nw = 0, nr = 0, r = 0, free_slots = Q.cap;
      bool drained = false, gated = false;                 // gated: an arrival waits for a node (Section 5.2)
      i64 total = 0; int selected = 0;
      i64 min_fin = TG_INF;                                // earliest completion among what runs
      // first round at or after time t > now_t, the time of round r_t (a 32-bit division where the distance allows)
      auto round_after = [&](i64 t, i64 now_t, int r_t) -> i64 {
        const i64 d = max(t - now_t, 1ll);
        return d <= 0xffffffffll && R.round_us <= 0xffffffffll ? (i64)r_t + (i64)(((u32)d - 1u) / (u32)R.round_us + 1u) : (i64)r_t + (d - 1) / R.round_us + 1;
      };
      // arrivals, 32 at a time: lane k holds record base + k
      int base = -32;
      i64 b_arr = TG_INF; ReplayRec b_rec; b_rec.s = b_rec.p = b_rec.tl = b_rec.arr = 0; b_rec.meta = 0; b_rec.mask = 1; b_rec.cg = 1;
      i64 next_arr = TG_INF;
      auto refill = [&]() {                                // the records from `next` on
        base = next;
        const int i = base + lane;
        b_arr = TG_INF;
        if (i < n_act) {
          const int j = P.a_pool[row + i];
          const u32 un = P.a_unit[row + i], mk = P.a_mask[row + i];
          const i64 s = P.a_s[row + i], p = P.a_p[row + i];
          b_arr = P.a_arrival ? P.a_arrival[row + i] : 0;
          b_rec = replay_decode(P, j, un, mk, s, p);
        }
        next_arr = __shfl_sync(TG_FULL, b_arr, 0);
      };
      if (n_act > 0) refill();
      int capreg = 0;                                      // lane v: free capacity of demand slot v
      u32 stale = ~0u;                                     // pools whose slots have to be worked out again
      bool windows = false;
      // lane j: where pool j's units in use are counted if it is a quota / concurrency pool, else -1
      const int api_at = lane < P.P && P.pool[lane].type == TG_POOL_API ? lane * 2 + (P.pool[lane].window_us > 0 ? 0 : 1) : -1;
#pragma unroll 1
      for (int j = 0; j < P.P; ++j) windows |= P.pool[j].type == TG_POOL_API && P.pool[j].window_us > 0;
      while (r < R.max_rounds) {
        const i64 now = (i64)r * R.round_us;
        // 1. quota refill
        if (windows)
#pragma unroll 1
          for (int j = 0; j < P.P; ++j) {
            const PoolDev& pd = P.pool[j];
            if (pd.type != TG_POOL_API || pd.window_us <= 0) continue;
            const i64 w0 = Z.win[j];
            if (now >= w0 * pd.window_us && now < (w0 + 1) * pd.window_us) continue;
            __syncwarp();
            if (lane == 0) { Z.win[j] = now / pd.window_us; Z.pst[j * 2] = 0; }
            __syncwarp();
            stale |= 1u << j;
          }
        // 2. release what has finished; the running list is compacted in place
        if (min_fin <= now) {
          int kept = 0;
          i64 mf = TG_INF;
#pragma unroll 1
          for (int i0 = 0; i0 < nr; i0 += 32) {
            const int i = i0 + lane;
            i64 fin = TG_INF; int a = 0, of = 0, dm = -1; u32 pu = 0;
            if (i < nr) { fin = run.fin[i]; a = run.idx[i]; pu = run.pu[i]; of = run.off[i]; dm = run.dom[i]; }
            const bool done = fin <= now, stay = i < nr && !done;
            if (stay) mf = min(mf, fin);
            const u32 bk = __ballot_sync(TG_FULL, stay);
            u32 rest = __ballot_sync(TG_FULL, done);
            if (rest || kept != i0) {
              if (stay) { const int k = kept + __popc(bk & below); run.fin[k] = fin; run.idx[k] = a; run.pu[k] = pu; run.off[k] = of; run.dom[k] = dm; }
            }
            kept += __popc(bk);
            __syncwarp();
#pragma unroll 1
            for (; rest; rest &= rest - 1) {
              const int b = __ffs(rest) - 1;
              const int fa = __shfl_sync(TG_FULL, a, b), fo = __shfl_sync(TG_FULL, of, b), fd = __shfl_sync(TG_FULL, dm, b);
              const u32 fpu = __shfl_sync(TG_FULL, pu, b);
              const int j = (int)(fpu >> 24), units = (int)(fpu & 0xffffffu);
              const PoolDev& pd = P.pool[j];
              stale |= 1u << j;
              if (EXT && R.trajectory && R.traj_last && lane == 0 && pd.type == TG_POOL_CPU && R.traj_last[row + fa]) {
                // the trajectory's last action has ended: its memory goes back to its node
                const int t = R.trajectory[row + fa];
                if (t >= 0 && t < R.max_traj) {
                  int* tn = R.traj_node + (size_t)sc * R.max_traj;
                  if (tn[t] >= 0) { R.mem_free[(size_t)sc * P.P + tn[t]] += (i64)R.traj_mem[row + fa]; tn[t] = -1; }
                }
              }
              if (EXT && P.n_side > 0) stale = ~0u;
              if (EXT && P.n_side > 0 && lane == 0)        // a concurrency pool held the action's further amounts until now
#pragma unroll 1
                for (int e = 0; e < P.n_side; ++e) {
                  const int k = P.a_side_pool[e * P.side_plane + row + fa];
                  if (k != 0xff && P.pool[k].window_us == 0) Z.pst[k * 2 + 1] -= P.a_side_units[e * P.side_plane + row + fa];
                }
              if (pd.type == TG_POOL_API) { if (pd.window_us == 0 && lane == 0) Z.pst[j * 2 + 1] -= units; }
              else {
                if (lane == j) busy -= units;
                int* ow = Z.owner + R.unit0[j];
                int left = units;
                // (a core pool's grant starts at its lowest core; chunks of replicas can lie anywhere)
#pragma unroll 1
                for (int c0 = pd.type == TG_POOL_CPU ? fo & ~31 : 0; c0 < pd.capacity && left > 0; c0 += 32) {
                  const int c = c0 + lane;
                  const bool mine = c < pd.capacity && ow[c] == fa;
                  const u32 mb = __ballot_sync(TG_FULL, mine);
                  if (!mb) continue;
                  if (mine) ow[c] = -1;
                  left -= __popc(mb);
                  if (pd.type == TG_POOL_CPU) {
                    if (fd < 0) { if (mine) atomicAdd(&Z.dfree[R.dom0[j] + c / pd.group], 1); }
                    else if (lane == 0) Z.dfree[R.dom0[j] + fd] += __popc(mb);
                  }
                  else if (lane < 32 / pd.group) {
                    const u32 bits = (mb >> (lane * pd.group)) & ((1u << pd.group) - 1u);
                    if (bits) Z.nm[pd.node0 + c0 / pd.group + lane] &= (u8)~bits;
                  }
                }
              }
              __syncwarp();
            }
          }
          nr = kept;
          min_fin = warp_min64(mf);
          gated = false;
        }
        // 3. admit arrivals
        bool was_gated = gated;
#pragma unroll 1
        while (next_arr <= now && !was_gated) {
          int cnt = __popc(__ballot_sync(TG_FULL, base + lane >= next && b_arr <= now));   // sorted: the lanes from next - base on
          const int k0 = next - base;
          if (EXT && R.trajectory) {
            // per-node CPU scheduling: an arrival joins the queue once its trajectory has a node; the first one
            // that finds none waits outside, with everything that arrived after it
            __syncwarp();
            i64 mf = 0; int cores = -1;
            if (lane < P.P && P.pool[lane].type == TG_POOL_CPU) { mf = R.mem_free[(size_t)sc * P.P + lane]; cores = P.pool[lane].capacity; }
            int pool_of = 0xff;
            const bool have = lane >= k0 && lane < k0 + cnt;
            const int out = pin_chunk(P, R.pool_rw, row + base + lane, have, R.trajectory, R.traj_mem, R.max_traj,
                                      R.traj_node + (size_t)sc * R.max_traj, mf, cores, lane, pool_of);
            if (lane < P.P && cores >= 0) R.mem_free[(size_t)sc * P.P + lane] = mf;
            if (have && lane < out) {
              R.pool_rw[row + base + lane] = (u8)pool_of;
              b_rec.meta = (b_rec.meta & ~0x3ffu) | (u32)pool_of | ((u32)P.pool[pool_of].slot0 << 4);
            }
            __syncwarp();
            if (out < k0 + cnt) { cnt = out - k0; was_gated = true; gated = true; }   // the gate
          }
          const bool in = lane >= k0 && lane < k0 + cnt;
          const int pos = nw + lane - k0;                  // queue position of this lane's arrival
          const bool fits = in && pos < Q.cap;
          if (EXT && R.policy) {
            // Other queue orders (Section 4.2): the queue stays sorted by the policy's key, equal keys in arrival order.
            // Each arrival goes behind the last entry whose key is not larger; the tail moves up by one.
#pragma unroll 1
            for (int b = k0; b < k0 + cnt; ++b) {
              const i64 tl = __shfl_sync(TG_FULL, b_rec.tl, b);
              const u64 key = R.policy == 2 ? (u64)((1ll << 42) - tl) : (u64)tl;
              int p = 0;
#pragma unroll 1
              for (int i0 = 0; i0 < nw; i0 += 32) {
                const int i = i0 + lane;
                const u64 ki = i >= nw ? ~0ull : (i < Q.cap ? Q.key[Q.q[i]] : wkey[i]);
                const u32 le = __ballot_sync(TG_FULL, i < nw && ki <= key);
                p += __popc(le);
                if (le != TG_FULL) break;                  // (sorted)
              }
              // what lies in global memory moves up first; the last record in shared memory follows it there
              if (nw >= Q.cap) {
#pragma unroll 1
                for (int hi = nw; hi > max(p, Q.cap);) {
                  const int lo = max(max(p, Q.cap), hi - 32), i = lo + lane;
                  int va = 0; u64 vk = 0;
                  if (i < hi) { va = wait[i]; vk = wkey[i]; }
                  __syncwarp();
                  if (i < hi) { wait[i + 1] = va; wkey[i + 1] = vk; }
                  __syncwarp();
                  hi = lo;
                }
                if (p < Q.cap) {
                  const int x = Q.q[Q.cap - 1];
                  if (lane == 0) { wait[Q.cap] = Q.idx[x]; wkey[Q.cap] = Q.key[x]; Q.free[free_slots] = (unsigned short)x; }
                  ++free_slots;
                  __syncwarp();
                }
              }
              if (p < Q.cap) {
#pragma unroll 1
                for (int hi = min(nw, Q.cap - 1); hi > p;) {
                  const int lo = max(p, hi - 32), i = lo + lane;
                  unsigned short v = 0;
                  if (i < hi) v = Q.q[i];
                  __syncwarp();
                  if (i < hi) Q.q[i + 1] = v;
                  __syncwarp();
                  hi = lo;
                }
                const int x = Q.free[--free_slots];
                __syncwarp();
                if (lane == b) {
                  Q.q[p] = (unsigned short)x; Q.s[x] = b_rec.s; Q.p[x] = b_rec.p; Q.tl[x] = b_rec.tl; Q.arr[x] = b_arr; Q.key[x] = key;
                  Q.idx[x] = base + b; Q.meta[x] = b_rec.meta; Q.mask[x] = b_rec.mask; Q.cg[x] = b_rec.cg;
                }
              } else if (lane == b) { wait[p] = base + b; wkey[p] = key; }
              __syncwarp();
              ++nw;
            }
          } else {
            if (fits) {
              const int x = Q.free[free_slots - 1 - (lane - k0)];
              Q.q[pos] = (unsigned short)x; Q.s[x] = b_rec.s; Q.p[x] = b_rec.p; Q.tl[x] = b_rec.tl; Q.arr[x] = b_arr;
              Q.idx[x] = base + lane; Q.meta[x] = b_rec.meta; Q.mask[x] = b_rec.mask; Q.cg[x] = b_rec.cg;
            } else if (in) wait[pos] = base + lane;
            free_slots -= __popc(__ballot_sync(TG_FULL, fits));
            nw += cnt;
          }
          next += cnt;
          __syncwarp();
          if (next == base + 32 || next == n_act) {
            next_arr = TG_INF;
            if (next < n_act) refill();
          } else next_arr = __shfl_sync(TG_FULL, b_arr, next - base);
        }
        // 4. schedule
        int blocked_pool = -1;                             // pool of a head-of-line action that does not fit
        bool any_started = false;
        if (nw > 0) {
#pragma unroll 1
          for (stale &= (1u << P.P) - 1u; stale; stale &= stale - 1u) {
            const int j = __ffs(stale) - 1;
            const PoolDev& pd = P.pool[j];
            if (pd.type == TG_POOL_GPU) {
              int c[4];
              gpu_caps(pd, Z.nm, lane, c);
              if (lane >= pd.slot0 && lane < pd.slot0 + 4) capreg = pick4(c, lane - pd.slot0);
            } else {
              const int used = pd.type == TG_POOL_CPU ? __shfl_sync(TG_FULL, busy, j) : Z.pst[j * 2 + (pd.window_us > 0 ? 0 : 1)];
              if (lane == pd.slot0) capreg = pd.capacity - used;
            }
          }
          // Candidate prefix (Algorithm 1, line 2): lane v adds up the demand on slot v, action by action; lane j counts
          // the candidates of pool j and (cost vectors) what is set aside of it for the others
          int n = 0, run_dem = 0, nc = 0, aside = 0;
          bool stop = false;
#pragma unroll 1
          for (int i0 = 0; i0 < nw && !stop; i0 += 32) {
            const int i = i0 + lane, nb = min(32, nw - i0);
            const u32 meta = i < nw ? replay_meta(P, Q, wait, row, i) : 0u;
            int k0 = 0xff, u0 = 0, k1 = 0xff, u1 = 0;      // further entries of the cost vector
            if (EXT && P.n_side > 0 && i < nw) {
              const int a = i < Q.cap ? Q.idx[Q.q[i]] : wait[i];
              k0 = P.a_side_pool[row + a]; u0 = P.a_side_units[row + a];
              if (P.n_side > 1) { k1 = P.a_side_pool[P.side_plane + row + a]; u1 = P.a_side_units[P.side_plane + row + a]; }
            }
#pragma unroll 1
            for (int b = 0; b < nb; ++b) {
              const u32 mb = __shfl_sync(TG_FULL, meta, b);
              int dem = 0, sa = 0, aj = 0;
              if (lane >= RQ_SLOT(mb) && lane <= RQ_SLOT(mb) + RQ_CLASS(mb)) dem = RQ_UNITS(mb);
              if (EXT && P.n_side > 0) {
                const int a0 = __shfl_sync(TG_FULL, k0, b), c0 = __shfl_sync(TG_FULL, u0, b);
                const int a1 = __shfl_sync(TG_FULL, k1, b), c1 = __shfl_sync(TG_FULL, u1, b);
                if (a0 != 0xff && lane == P.pool[a0].slot0) sa += c0;
                if (a1 != 0xff && lane == P.pool[a1].slot0) sa += c1;
                if (lane == a0) aj += c0;
                if (lane == a1) aj += c1;
              }
              if (__any_sync(TG_FULL, dem + sa > 0 && run_dem + dem + sa > capreg)) { stop = true; break; }
              run_dem += dem + sa; aside += aj;
              if (lane == RQ_POOL(mb)) ++nc;
              ++n;
            }
          }
          if (n == 0) blocked_pool = RQ_POOL(uniform((int)replay_meta(P, Q, wait, row, 0)));
          const int nr0 = nr;
          bool ok = true;
          // Algorithm 1, line 3: pool by pool
#pragma unroll 1
          for (u32 pools = __ballot_sync(TG_FULL, nc > 0); pools && ok; pools &= pools - 1) {
            const int j = __ffs(pools) - 1, m = __shfl_sync(TG_FULL, nc, j);
            const PoolDev& pd = P.pool[j];
            const int slot0 = pd.slot0, aside_j = EXT ? __shfl_sync(TG_FULL, aside, j) : 0;
            const int cap0 = __shfl_sync(TG_FULL, capreg, slot0) - aside_j;
            int* ow = Z.owner + R.unit0[j];
            int started_units = 0;
            // elastic candidates?
            bool el = false;
            if (m > 1) {
#pragma unroll 1
              for (int i = lane; i < n; i += 32) {
                int a;
                const ReplayRec x = replay_rec(P, Q, wait, row, i, a);
                el |= RQ_POOL(x.meta) == j && (x.mask & (x.mask - 1)) != 0;
              }
              el = __any_sync(TG_FULL, el);
            }
            const bool cached = EXT && pd.type == TG_POOL_GPU && P.cache_slots > 0;
            if ((m == 1 || (!el && pd.type != TG_POOL_GPU)) && !cached) {
              // Nothing to choose between candidates: each takes its level (a lone one DPArrange's answer in closed form: the
              // feasible level of least duration, the smallest among equals) and is placed in queue order.
              int seen = 0;
#pragma unroll 1
              for (int i0 = 0; i0 < n && seen < m; i0 += 32) {
                int a = 0; ReplayRec x; x.meta = 15u; x.s = x.p = 0; x.mask = 1; x.cg = 1;
                if (i0 + lane < n) x = replay_rec(P, Q, wait, row, i0 + lane, a);
                const bool mine = i0 + lane < n && RQ_POOL(x.meta) == j;
                const u32 mb = __ballot_sync(TG_FULL, mine);
                int rr = __ffs(x.mask), node = -1, off = -1, dom = -1;
                if (m == 1 && mb) {
                  const int b = __ffs(mb) - 1;
                  const u32 mk = __shfl_sync(TG_FULL, x.mask, b), cg = __shfl_sync(TG_FULL, (u32)x.cg, b);
                  if (mk & (mk - 1)) {
                    const i64 s = __shfl_sync(TG_FULL, x.s, b), p = __shfl_sync(TG_FULL, x.p, b);
                    const int g = cg & 0x7f, gang = cg >> 7, rl = lane + 1;
                    bool fit = (mk >> lane) & 1u;
                    const int c = fit && pd.type == TG_POOL_GPU ? level_of(g, gang, rl) : 0;
                    const int room = __shfl_sync(TG_FULL, capreg, slot0 + c) - (c == 0 ? aside_j : 0);
                    fit = fit && g * rl <= room;
                    const i64 best = warp_min64(fit ? ((duration(s, p, rl) << 6) | (i64)rl) : TG_INF);
                    if (lane == b && best != TG_INF) rr = (int)(best & 63);
                  }
                }
                const int units = mine ? (x.cg & 0x7f) * rr : 0;
#pragma unroll 1
                for (u32 todo = mb; todo; todo &= todo - 1) {
                  const int b = __ffs(todo) - 1;
                  const int k = __shfl_sync(TG_FULL, units, b), id = __shfl_sync(TG_FULL, a, b);
                  int nd = 0, of = 0, ft = -1;
                  if (pd.type == TG_POOL_CPU) replay_place_cpu(pd, ow, Z.dfree + R.dom0[j], k, id, lane, nd, of, ft);
                  else if (pd.type == TG_POOL_GPU) {
                    const u32 cg = __shfl_sync(TG_FULL, (u32)x.cg, b);
                    const int rb = __shfl_sync(TG_FULL, rr, b), g = cg & 0x7f, gang = cg >> 7;
                    replay_place_gpu(pd, Z.nm + pd.node0, ow, ilog2(gang ? g * rb : g), gang ? 1 : rb, id, lane, nd, of);
                  } else {
                    int* ps = Z.pst + j * 2 + (pd.window_us > 0 ? 0 : 1);
                    of = *ps;
                    __syncwarp();
                    if (lane == 0) *ps = of + k;
                    __syncwarp();
                  }
                  if (lane == b) { node = nd; off = of; dom = ft; }
                }
                // start (Eq. 2: completion - arrival = waited so far + execution)
                if (mine) {
                  const size_t o = row + a;
                  const i64 fin = now + duration(x.s, x.p, rr), act = fin - x.arr;
                  P.o_alloc[o] = units; P.o_node[o] = node; P.o_off[o] = off; P.o_act[o] = act;
                  const int k = nr + __popc(mb & below);
                  run.fin[k] = fin; run.idx[k] = a; run.pu[k] = ((u32)j << 24) | (u32)units; run.off[k] = off; run.dom[k] = dom;
                  if (i0 + lane < Q.cap) Q.meta[Q.q[i0 + lane]] = x.meta | RQ_STARTED;
                  total += act; min_fin = min(min_fin, fin);
                  started_units += units;
                }
                nr += __popc(mb); seen += __popc(mb); selected += __popc(mb);
              }
            } else {
              Slab slab;
              slab.base = P.slabs + (u64)blockIdx.x * P.slab_bytes; slab.cap = P.slab_bytes; slab.used = 0;
              slab.fbase = fast; slab.fcap = KR_FAST_BYTES; slab.fused = 0;
              CandArrays C; int keep = 0;
              ok = replay_select<EXT>(P, Q, run, wait, sc, j, n, nw, nr, m, now, cap0, __shfl_sync(TG_FULL, capreg, (slot0 + 1) & 31),
                                      __shfl_sync(TG_FULL, capreg, (slot0 + 2) & 31), __shfl_sync(TG_FULL, capreg, (slot0 + 3) & 31), slab, C, keep, lane);
              if (!ok) break;
              const u8* missed = nullptr;                  // candidates whose chunk did not cache their service
              if (cached) {
                const size_t cbase = ((size_t)sc * P.n_nodes_total + pd.node0) * 8 * P.cache_slots;
                place_gpu_cache(pd, Z.nm + pd.node0, keep, C.cg, C.rkeep, C.cidx, C.pnode, C.poff, C.rsel,
                                P.a_service ? P.a_service + row : nullptr, P.cache_tag + cbase, P.cache_use + cbase, P.cache_slots, now, lane, ow);
                missed = C.rsel;
              } else if (pd.type == TG_POOL_GPU) {
                place_gpu(pd, Z.nm + pd.node0, keep, C.cg, C.rkeep, C.pnode, C.poff, lane, ow, C.cidx);
              } else if (pd.type == TG_POOL_CPU) {
#pragma unroll 1
                for (int i = 0; i < keep; ++i) {
                  int nd, of, ft;
                  replay_place_cpu(pd, ow, Z.dfree + R.dom0[j], (C.cg[i] & 0x7f) * C.rkeep[i], C.cidx[i], lane, nd, of, ft);
                  if (lane == 0) { C.pnode[i] = nd; C.poff[i] = of; C.rowcand[i] = ft; }
                }
              } else if (lane == 0) {
                int* ps = Z.pst + j * 2 + (pd.window_us > 0 ? 0 : 1);
#pragma unroll 1
                for (int i = 0; i < keep; ++i) { C.pnode[i] = 0; C.poff[i] = *ps; *ps += (C.cg[i] & 0x7f) * C.rkeep[i]; }
              }
              __syncwarp();
#pragma unroll 1
              for (int i = lane; i < keep; i += 32) {
                const size_t o = row + C.cidx[i];
                const int rr = C.rkeep[i], units = (C.cg[i] & 0x7f) * rr;
                i64 fin = now + duration(C.cs[i], C.cp[i], rr);
                if (EXT && missed && missed[i] && P.a_restore) fin += clamp_param(P.a_restore[o]);   // restoration precedes execution
                const i64 act = fin - (P.a_arrival ? P.a_arrival[o] : 0);
                P.o_alloc[o] = units; P.o_node[o] = C.pnode[i]; P.o_off[o] = C.poff[i]; P.o_act[o] = act;
                run.fin[nr + i] = fin; run.idx[nr + i] = C.cidx[i]; run.pu[nr + i] = ((u32)j << 24) | (u32)units; run.off[nr + i] = C.poff[i]; run.dom[nr + i] = pd.type == TG_POOL_CPU ? C.rowcand[i] : -1;
                total += act; min_fin = min(min_fin, fin);
                started_units += units;
              }
              // the kept ones are the pool's first `keep` in queue order
              int seen = 0;
#pragma unroll 1
              for (int i0 = 0; i0 < n && seen < keep; i0 += 32) {
                const int i = i0 + lane;
                const u32 meta = i < n ? replay_meta(P, Q, wait, row, i) : 15u;
                const u32 mb = __ballot_sync(TG_FULL, i < n && RQ_POOL(meta) == j);
                if (((mb >> lane) & 1u) && seen + __popc(mb & below) < keep && i < Q.cap) Q.meta[Q.q[i]] = meta | RQ_STARTED;
                seen += __popc(mb);
              }
              nr += keep; selected += keep;
            }
            started_units = warp_sum32(started_units);
            if (lane == j && pd.type != TG_POOL_API) busy += started_units;
            stale |= 1u << j;
            __syncwarp();
          }
          if (!ok) { status = TG_ST_WORKSPACE; break; }
          any_started = nr > nr0;
          if (EXT && P.n_side > 0 && any_started) {         // the started actions consume their further amounts
            stale = ~0u;
#pragma unroll 1
            for (int i = nr0 + lane; i < nr; i += 32)
#pragma unroll 1
              for (int e = 0; e < P.n_side; ++e) {
                const int k = P.a_side_pool[e * P.side_plane + row + run.idx[i]];
                if (k != 0xff)
                  atomicAdd(&Z.pst[k * 2 + (P.pool[k].window_us > 0 ? 0 : 1)], (int)P.a_side_units[e * P.side_plane + row + run.idx[i]]);
              }
            __syncwarp();
          }
          if (any_started) {                                // drop the started actions from the queue
            int kw = 0;
#pragma unroll 1
            for (int i0 = 0; i0 < nw; i0 += 32) {
              const int i = i0 + lane;
              bool stay = false; int x = 0, a = 0; u64 kk = 0;
              if (i < min(nw, Q.cap)) { x = Q.q[i]; stay = !(Q.meta[x] & RQ_STARTED); }
              else if (i < nw) { a = wait[i]; stay = P.o_act[row + a] < 0; if (EXT && R.policy) kk = wkey[i]; }
              const u32 b = __ballot_sync(TG_FULL, stay), gone = __ballot_sync(TG_FULL, i < min(nw, Q.cap) && !stay);
              const int to = kw + __popc(b & below);
              __syncwarp();
              if (stay && i < Q.cap) Q.q[to] = (unsigned short)x;
              else if (stay && to >= Q.cap) { wait[to] = a; if (EXT && R.policy) wkey[to] = kk; }
              if ((gone >> lane) & 1u) Q.free[free_slots + __popc(gone & below)] = (unsigned short)x;
              free_slots += __popc(gone);
              __syncwarp();
              const u32 mv = __ballot_sync(TG_FULL, stay && i >= Q.cap && to < Q.cap);
              if ((mv >> lane) & 1u) {                      // a record moves up into shared memory
                const int y = Q.free[free_slots - 1 - __popc(mv & below)];
                const ReplayRec rec = replay_decode(P, P.a_pool[row + a], P.a_unit[row + a], P.a_mask[row + a], P.a_s[row + a], P.a_p[row + a]);
                Q.q[to] = (unsigned short)y; Q.s[y] = rec.s; Q.p[y] = rec.p; Q.tl[y] = rec.tl; Q.arr[y] = P.a_arrival ? P.a_arrival[row + a] : 0;
                if (EXT) Q.key[y] = kk;
                Q.idx[y] = a; Q.meta[y] = rec.meta; Q.mask[y] = rec.mask; Q.cg[y] = rec.cg;
              }
              free_slots -= __popc(mv);
              __syncwarp();
              kw += __popc(b);
            }
            nw = kw;
            min_fin = warp_min64(min_fin);
          }
        }
        // 5. occupancy of this round: lane j holds pool j's
        int in_use = busy;
        if (api_at >= 0) in_use = Z.pst[api_at];
        if (occ && lane < P.P) occ[(size_t)r * P.P + lane] = in_use;
        ++r;
        if (next == n_act && nw == 0 && nr == 0) { drained = true; break; }
        // Rounds in which nothing can change are jumped over, their rows repeat this occupancy (quota usage restarts
        // with its window).
        i64 t_next = TG_INF;
        bool jump = false, partial = false;
        if (nw == 0) {
          // with an empty queue: to the next arrival or completion (a gated arrival waits for a completion)
          jump = true;
          t_next = min(gated ? TG_INF : next_arr, min_fin);
        } else if (blocked_pool >= 0) {
          // The action at the head of the queue does not fit, so nothing can start until an action that runs ends, a quota
          // window turns or (in a sorted queue) an arrival becomes the head.
          jump = true;
          const PoolDev& hp = P.pool[blocked_pool];
          if (EXT && (P.n_side > 0 || R.trajectory)) {
            // (the head may wait for any pool's amounts; an arrival would be pinned against the memory free at its time)
            t_next = min(gated ? TG_INF : next_arr, min_fin);
#pragma unroll 1
            for (int j = 0; j < P.P; ++j)
              if (P.pool[j].type == TG_POOL_API && P.pool[j].window_us > 0) t_next = min(t_next, (Z.win[j] + 1) * (i64)P.pool[j].window_us);
          } else {
            // ... on its pool: arrivals join behind it, what ends on other pools leaves the rows from its round on
            partial = true;
            if (hp.type == TG_POOL_API && hp.window_us > 0) t_next = (Z.win[blocked_pool] + 1) * (i64)hp.window_us;
            if (EXT && R.policy) t_next = min(t_next, next_arr);
#pragma unroll 1
            for (int i = lane; i < nr; i += 32)
              if ((int)(run.pu[i] >> 24) == blocked_pool) t_next = min(t_next, run.fin[i]);
            t_next = warp_min64(t_next);
          }
        }
        if (jump) {
          int r_next = R.max_rounds;
          if (t_next <= now) r_next = r;
          else if (t_next < now + (i64)(R.max_rounds - r + 1) * R.round_us) r_next = min(r_next, (int)round_after(t_next, now, r - 1));
          if (r_next > r) {
            if (occ) {
              if (lane < P.P) {
                // (this lane's pool; its usage restarts with its window)
                int turn = r_next;
                if (windows && api_at >= 0 && !(api_at & 1)) {
                  const i64 tr = round_after((Z.win[lane] + 1) * (i64)P.pool[lane].window_us, now, r - 1);
                  if (tr < (i64)turn) turn = (int)tr;
                }
                int* at = occ + (size_t)r * P.P + lane;
#pragma unroll 1
                for (int rr = r; rr < r_next; ++rr, at += P.P) *at = rr < turn ? in_use : 0;
              }
              if (partial) {
                __syncwarp();
#pragma unroll 1
                for (int i = lane; i < nr; i += 32) {
                  const i64 fin = run.fin[i];
                  if (fin > (i64)(r_next - 1) * R.round_us) continue;
                  const u32 pu = run.pu[i];
                  const int j = (int)(pu >> 24);
                  if (P.pool[j].type == TG_POOL_API && P.pool[j].window_us > 0) continue;      // used quota is not given back
                  const int fr = max(r, (int)round_after(fin, now, r - 1));
#pragma unroll 1
                  for (int rr = fr; rr < r_next; ++rr) atomicSub(&occ[(size_t)rr * P.P + j], (int)(pu & 0xffffffu));
                }
                __syncwarp();
              }
            }
            r = r_next;
          }
        }
      }
      rounds = drained ? r : R.max_rounds;
      if (!drained && r < R.max_rounds) rounds = r;
      total = warp_sum64(total);
      if (lane == 0) { P.o_total[sc] = total; P.o_nsel[sc] = selected; P.o_status[sc] = status; }
    } else if (lane == 0) { P.o_total[sc] = 0; P.o_nsel[sc] = 0; P.o_status[sc] = status; }
    if (R.rounds_used && lane == 0) R.rounds_used[sc] = rounds;
    __syncwarp();
  }
}
