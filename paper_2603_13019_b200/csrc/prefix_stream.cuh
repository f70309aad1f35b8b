// First two kernels of a batched round.
//
// k_head, one warp per scenario, walks the queue 32 actions at a time until the candidate
// prefix ends (Algorithm 1, line 2): lane v keeps the running least-level demand of demand
// slot v (one slot per core / quota pool, four nested chunk levels per GPU pool), lane j the
// number of actions of pool j seen so far; a chunk's demand goes through one warp scan per
// slot and the first action that overflows a slot ends the prefix.  Candidates get their
// position inside their pool (Algorithm 1, line 4) and their index is written to the pool's
// part of `order`.  The same walk sums every slot's demand at the candidates' LARGEST levels:
// where that fits, every candidate gets its best level, no eviction can pay and nobody will
// read the pool's waiting list.
//
// k_stream, one CTA per scenario, streams everything behind the head 4096 actions at a time
// (16 per thread, 128-bit loads): records are validated, and only for the pools that may need
// an estimate the least-level durations (Eq. 1) of the waiting actions are appended, in queue
// order, to the pool's list in `tmin`.
//
// The output rows behind the candidate prefix get "not scheduled" from the selection kernel, which leaves the memory
// idle (fill_rows); of an ordered round k_fill writes all rows beside the sort, on a stream of its own.
//
// Partitioned arrays (order, tmin and the solver's arrays) give every (scenario, pool) its own
// row of max_actions entries, so a position never depends on another pool's count and the
// queue is read once.
#pragma once
#include "common.cuh"

#define KS_THREADS 256
#define KS_ITEMS 16
#define KS_TILE (KS_THREADS * KS_ITEMS)

// what k_head leaves for k_stream
struct HeadState {
  int hs;                     // first action the stream has to look at (a multiple of 32, or n_actions)
  u32 need;                   // pools whose waiting list may be read
  int bad;                    // an invalid record was seen
  int n;                      // length of the candidate prefix
  int cur[TG_MAX_POOLS];      // actions of every pool in [0, hs)
};

__device__ __forceinline__ int warp_incl_scan32(int x, int lane) {
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) { int y = __shfl_up_sync(TG_FULL, x, o); if (lane >= o) x += y; }
  return x;
}

// Further entries of the cost vectors (Section 4.1): an entry has to name a quota / concurrency pool other
// than the action's key pool and an amount of 1 .. its capacity.
__device__ __forceinline__ bool side_entry_bad(const Params& P, int e, size_t o) {
  const int k = P.a_side_pool[e * P.side_plane + o];
  if (k == 0xff) return false;
  const int c = P.a_side_units[e * P.side_plane + o];
  return k >= P.P || P.pool[k < P.P ? k : 0].type != TG_POOL_API || k == P.a_pool[o] || c < 1 || c > P.pool[k < P.P ? k : 0].capacity;
}
// One thread per action; a scenario with a bad entry is flagged for k_head, which then decides nothing of it.
__global__ void __launch_bounds__(256) k_side_check(const __grid_constant__ Params P) {
  // sixteen consecutive actions of one scenario per thread (128-bit loads) where the rows allow it
  const bool vec = (P.N % 16 == 0) && (P.side_plane % 16 == 0) &&
                   ((((size_t)P.a_pool | (size_t)P.a_side_pool) & 15) == 0) && (((size_t)P.a_side_units & 15) == 0);
  const size_t total = (size_t)P.S * P.N, step = (size_t)gridDim.x * blockDim.x;
  if (vec) {
    for (size_t q = (size_t)blockIdx.x * blockDim.x + threadIdx.x; q < total / 16; q += step) {
      const size_t o = q * 16;
      const int sc = (int)(o / P.N), i0 = (int)(o - (size_t)sc * P.N);
      const int n = min(max(P.n_actions[sc], 0), P.N) - i0;    // records of this group that exist
      if (n <= 0) continue;
      bool bad = false;
      for (int e = 0; e < P.n_side; ++e) {
        __align__(16) u8 k[16];
        *(uint4*)k = *(const uint4*)(P.a_side_pool + e * P.side_plane + o);
        const uint4 kk = *(const uint4*)k;
        if ((kk.x & kk.y & kk.z & kk.w) == 0xffffffffu) continue;   // no entry in the whole group
        __align__(16) unsigned short c[16];
        __align__(16) u8 kp[16];
        *(uint4*)c = *(const uint4*)(P.a_side_units + e * P.side_plane + o);
        *(uint4*)(c + 8) = *(const uint4*)(P.a_side_units + e * P.side_plane + o + 8);
        *(uint4*)kp = *(const uint4*)(P.a_pool + o);
#pragma unroll
        for (int x = 0; x < 16; ++x) {
          if (x >= n || k[x] == 0xff) continue;
          const int kx = k[x] < P.P ? k[x] : 0;
          bad |= k[x] >= P.P || P.pool[kx].type != TG_POOL_API || k[x] == kp[x] || c[x] < 1 || c[x] > P.pool[kx].capacity;
        }
      }
      if (bad) P.side_bad[sc] = 1;
    }
    return;
  }
  for (size_t o = (size_t)blockIdx.x * blockDim.x + threadIdx.x; o < total; o += step) {
    const int sc = (int)(o / P.N), i = (int)(o - (size_t)sc * P.N);
    if (i >= min(max(P.n_actions[sc], 0), P.N)) continue;
    bool bad = false;
    for (int e = 0; e < P.n_side; ++e) bad |= side_entry_bad(P, e, o);
    if (bad) P.side_bad[sc] = 1;
  }
}

// SIDE: the actions carry further cost-vector entries (Section 4.1); the plain instance keeps its registers.
// ws: whose rows of the workspace are used (the scenario's own; the block's, where a block works a scenario off alone).
template <bool SIDE>
__device__ __forceinline__ void head_walk(const Params& P, int sc, int ws, HeadState& hs_out, bool side_bad, int lane) {
  const size_t row = (size_t)sc * P.N;
  const size_t prow = (size_t)ws * P.P * P.N;       // pool j's part starts at prow + j * N
  const int n_act = min(max(P.n_actions[sc], 0), P.N);
  const int D = P.V - P.P;                          // demand slots

  // lane v < D: capacity, running least-level demand and candidates' largest-level demand of slot v
  // lane j < P: actions / candidates / first waiting action of pool j, and the pool's description
  int capreg = 0, run = 0, mxd = 0, cnt = 0, mreg = 0, fwreg = -1;
  int sres = 0;                                     // lane v: what the candidates ask of slot v beside their key resource
  u32 pinfo = 0;                                    // type | GPUs per node << 4 | slot0 << 8
  for (int j = 0; j < P.P; ++j) {
    const PoolDev& pd = P.pool[j];
    if (pd.type == TG_POOL_GPU) {
      int cap[4];
      gpu_caps(pd, P.gpu_busy ? P.gpu_busy + (size_t)sc * P.n_nodes_total : nullptr, lane, cap);
#pragma unroll
      for (int l = 0; l < 4; ++l) if (lane == pd.slot0 + l) capreg = cap[l];
    } else if (lane == pd.slot0) capreg = pd.capacity;
    if (lane == j) pinfo = (u32)pd.type | ((u32)(pd.type == TG_POOL_GPU ? pd.group : 0) << 4) | ((u32)pd.slot0 << 8);
  }

  u32 el = 0, need = 0;
  bool bad = false;
  int hs = n_act, n_pref = n_act;
  const u32 lt = (1u << lane) - 1u;
  // the records of the next chunk are loaded while this one is worked on
  int nj = 0; u32 nun = 0, nmk = 0; i64 ns = 0, np_ = 0;
  int nk0 = 0xff, nu0 = 0, nk1 = 0xff, nu1 = 0;    // further entries of the cost vectors
  if (SIDE && lane < n_act) {
    nk0 = P.a_side_pool[row + lane]; nu0 = P.a_side_units[row + lane];
    if (P.n_side > 1) { nk1 = P.a_side_pool[P.side_plane + row + lane]; nu1 = P.a_side_units[P.side_plane + row + lane]; }
  }
  int nsrc = lane;                                  // where in the row the queue's next action is
  if (lane < n_act) {
    if (P.perm) nsrc = P.perm[row + lane];
    nj = P.a_pool[row + nsrc]; nun = P.a_unit[row + nsrc]; nmk = P.a_mask[row + nsrc]; ns = P.a_s[row + nsrc]; np_ = P.a_p[row + nsrc];
  }
  for (int c0 = 0; c0 < n_act; c0 += 32) {
    const int i = c0 + lane;
    const bool present = i < n_act;
    const int j = nj, src = nsrc; const u32 un = nun, mk = nmk; const i64 s = ns, p = np_;
    const int k0 = nk0, k1 = nk1;
    int su0 = nu0, su1 = nu1;
    if (SIDE) {
      const int i2 = i + 32;
      nk0 = 0xff; nk1 = 0xff; nu0 = 0; nu1 = 0;
      if (i2 < n_act) {
        nk0 = P.a_side_pool[row + i2]; nu0 = P.a_side_units[row + i2];
        if (P.n_side > 1) { nk1 = P.a_side_pool[P.side_plane + row + i2]; nu1 = P.a_side_units[P.side_plane + row + i2]; }
      }
    }
    {
      const int i2 = i + 32;
      nj = 0; nun = 0; nmk = 0; ns = 0; np_ = 0; nsrc = i2;
      if (i2 < n_act) {
        if (P.perm) nsrc = P.perm[row + i2];
        nj = P.a_pool[row + nsrc]; nun = P.a_unit[row + nsrc]; nmk = P.a_mask[row + nsrc]; ns = P.a_s[row + nsrc]; np_ = P.a_p[row + nsrc];
      }
    }
    bool valid = present && j < P.P;
    const u32 pi = __shfl_sync(TG_FULL, pinfo, valid ? j : 0);
    PoolDev pd;
    pd.type = pi & 15; pd.group = (pi >> 4) & 15;
    const int slot0 = pi >> 8;
    int g = 1, gang = 0; u32 eff = 1;
    if (valid) valid = decode_levels(pd, (u8)un, mk, g, gang, eff);
    bad |= present && !valid;
    const bool gpu = pd.type == TG_POOL_GPU;
    const int rmin = __ffs(eff), rmax = 32 - __clz(eff);
    const int units = g * rmin, mxu = g * rmax;
    const int lz = gpu ? level_of(g, gang, rmin) : 0, lzx = gpu ? level_of(g, gang, rmax) : 0;
    // further entries of the cost vector: the slot they charge and the amount (slot -1: none)
    int ss0 = -1, ss1 = -1;
    if (SIDE) {
      const u32 p0 = __shfl_sync(TG_FULL, pinfo, k0 < P.P ? k0 : 0), p1 = __shfl_sync(TG_FULL, pinfo, k1 < P.P ? k1 : 0);
      if (valid && k0 < P.P) ss0 = p0 >> 8;
      if (valid && k1 < P.P) ss1 = p1 >> 8;
    }
    // least-level demand: one scan per slot; the first action that overflows a slot ends the prefix
    // First the chunk's total per slot (one warp reduction each): only the chunk in which a slot
    // overflows needs the scans that tell which action does it.
    int tot_mine = 0;                                  // lane v: the chunk's demand on slot v
    for (int v = 0; v < D; ++v) {
      const int c = ((valid && v >= slot0 && v <= slot0 + lz) ? units : 0) + (ss0 == v ? su0 : 0) + (ss1 == v ? su1 : 0);
      const int tot = __reduce_add_sync(TG_FULL, c);
      if (lane == v) tot_mine = tot;
    }
    bool over = false;
    if (__any_sync(TG_FULL, lane < D && run + tot_mine > capreg)) {
      for (int v = 0; v < D; ++v) {
        const int c = ((valid && v >= slot0 && v <= slot0 + lz) ? units : 0) + (ss0 == v ? su0 : 0) + (ss1 == v ? su1 : 0);
        const int incl = warp_incl_scan32(c, lane);
        const int rv = __shfl_sync(TG_FULL, run, v), cv = __shfl_sync(TG_FULL, capreg, v);
        over |= c > 0 && rv + incl > cv;
      }
    }
    run += tot_mine;                                   // beyond the prefix the totals are not used any more
    const u32 ob = __ballot_sync(TG_FULL, over);
    const int f = ob ? __ffs(ob) - 1 : 32;           // lanes >= f wait
    const bool cand = valid && lane < f;
    // position inside the pool
    int pos = __shfl_sync(TG_FULL, cnt, valid ? j : 0);  // the pool's count before this chunk
    const u32 below_f = f >= 32 ? TG_FULL : ((1u << f) - 1u);
    for (int jj = 0; jj < P.P; ++jj) {
      const u32 b = __ballot_sync(TG_FULL, valid && j == jj);
      if (valid && j == jj) pos += __popc(b & lt);
      if (lane == jj) { cnt += __popc(b); mreg += __popc(b & below_f); }
    }
    if (cand) {
      P.order[(size_t)ws * P.cand_stride + P.cand_off[j] + pos] = src;
      if (eff & (eff - 1)) el |= 1u << j;
    }
    for (int v = 0; v < D; ++v) {
      const int sd = cand ? (ss0 == v ? su0 : 0) + (ss1 == v ? su1 : 0) : 0;
      const int c = ((cand && v >= slot0 && v <= slot0 + lzx) ? mxu : 0) + sd;
      const int tot = __reduce_add_sync(TG_FULL, c);
      if (lane == v) mxd += tot;
      if (SIDE) { const int st = __reduce_add_sync(TG_FULL, sd); if (lane == v) sres += st; }
    }
    if (ob) {
      // The prefix is complete.  A pool may need its waiting list only if one of its candidates
      // is elastic and the candidates' largest levels do not all fit.
      const u32 unfit = __ballot_sync(TG_FULL, lane < D && mxd > capreg);
      const u32 elw = __reduce_or_sync(TG_FULL, el);
      for (int jj = 0; jj < P.P; ++jj) {
        const u32 slots = ((1u << P.pool[jj].n_slots) - 1u) << P.pool[jj].slot0;
        if (((elw >> jj) & 1u) && (unfit & slots)) need |= 1u << jj;
      }
      const int mj = __shfl_sync(TG_FULL, mreg, valid ? j : 0);
      const bool waits = valid && lane >= f;
      if (waits && ((need >> j) & 1u))
        P.tmin[prow + (size_t)j * P.N + pos] = duration(clamp_param(s), clamp_param(p), rmin);
      for (int jj = 0; jj < P.P; ++jj) {               // the pool's first waiting action
        const u32 b = __ballot_sync(TG_FULL, waits && j == jj && pos == mj);
        const int fw = __shfl_sync(TG_FULL, src, b ? __ffs(b) - 1 : 0);
        if (lane == jj && b) fwreg = fw;
      }
      hs = min(c0 + 32, n_act); n_pref = c0 + f;
      break;
    }
  }
  const u32 elw = __reduce_or_sync(TG_FULL, el);
  if (hs == n_act && n_pref == n_act) {
    // the whole queue is the candidate prefix: the same test tells which pools are certified
    const u32 unfit = __ballot_sync(TG_FULL, lane < D && mxd > capreg);
    for (int jj = 0; jj < P.P; ++jj) {
      const u32 slots = ((1u << P.pool[jj].n_slots) - 1u) << P.pool[jj].slot0;
      if (((elw >> jj) & 1u) && (unfit & slots)) need |= 1u << jj;
    }
  }
  const int anybad = (__any_sync(TG_FULL, bad) || (SIDE && side_bad)) ? 1 : 0;
  if (SIDE) {
    const int sr = __shfl_sync(TG_FULL, sres, lane < P.P ? P.pool[lane].slot0 : 0);
    if (lane < P.P) P.side_res[(size_t)ws * P.P + lane] = sr;
  }
  if (lane < P.P) {
    PoolMeta mt;
    mt.base = ((i64)ws * P.P + lane - sc) * P.N;      // row + base = prow + lane * N
    mt.cbase = (i64)ws * P.cand_stride + P.cand_off[lane] - (i64)sc * P.N;
    // an invalid record among the actions seen here: nothing of the scenario is decided
    mt.count = anybad ? 0 : cnt; mt.m = anybad ? 0 : mreg; mt.elastic = anybad ? 0 : ((elw >> lane) & 1u);
    mt.first_wait = anybad ? -1 : fwreg;
    P.meta[(size_t)ws * P.P + lane] = mt;
    hs_out.cur[lane] = cnt;
  }
  if (lane == 0) {
    hs_out.hs = hs; hs_out.need = need; hs_out.bad = anybad; hs_out.n = n_pref;
    P.o_status[sc] = anybad ? TG_ST_BAD_ACTION : 0; P.o_total[sc] = 0; P.o_nsel[sc] = 0;
  }
}

template <bool SIDE>
__global__ void __launch_bounds__(256) k_head(const __grid_constant__ Params P, HeadState* hst) {
  const int sc = (int)((blockIdx.x * (unsigned)blockDim.x + threadIdx.x) >> 5);
  if (sc < P.S) head_walk<SIDE>(P, sc, sc, hst[sc], SIDE && P.side_bad[sc], threadIdx.x & 31);
}

// exclusive scan of one int per thread over the CTA; *total = sum.  wsum: 8 ints of scratch.
__device__ __forceinline__ int ks_block_scan(int x, int* wsum, int t, int* total) {
  const int lane = t & 31, warp = t >> 5;
  const int incl = warp_incl_scan32(x, lane);
  if (lane == 31) wsum[warp] = incl;
  __syncthreads();
  int off = 0, tot = 0;
#pragma unroll
  for (int w = 0; w < KS_THREADS / 32; ++w) { const int v = wsum[w]; if (w < warp) off += v; tot += v; }
  __syncthreads();
  *total = tot;
  return off + incl - x;
}

struct StreamShared {
  // usable multiplicities by (pool, unit byte): a record's usable levels are its mask ANDed with the
  // entry, and a record with none is invalid (decode_levels, tabulated once per round description)
  __align__(16) u32 ok[TG_MAX_POOLS * 256];
  int m[TG_MAX_POOLS], first[TG_MAX_POOLS], cur[TG_MAX_POOLS], scan[KS_THREADS / 32];
  int bad;
};
// The waiting lists of a queue that is taken in another order than it stands in: four positions of the order per thread,
// their records gathered from the row, which one block reads whole and so finds in L1.  Bound by the latency of those
// gathers; copying the records into order first, and the results back, took twice the traffic of the round itself.
__device__ __forceinline__ void stream_sorted(const Params& P, int sc, int ws, const HeadState& H, StreamShared& X, int t) {
  const size_t row = (size_t)sc * P.N, prow = (size_t)ws * P.P * P.N;
  const int n_act = min(max(P.n_actions[sc], 0), P.N);
#pragma unroll 1
  for (int tile0 = H.hs; tile0 < n_act; tile0 += KS_THREADS * 4) {
    int src[4], pl[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) { const int i = tile0 + 4 * t + k; src[k] = i < n_act ? P.perm[row + i] : -1; }
#pragma unroll
    for (int k = 0; k < 4; ++k) pl[k] = src[k] >= 0 ? P.a_pool[row + src[k]] : 0xff;
    i64 T[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      T[k] = 0;
      if (pl[k] < P.P && ((H.need >> pl[k]) & 1u)) {
        const u32 eff = P.a_mask[row + src[k]] & X.ok[pl[k] * 256 + P.a_unit[row + src[k]]];
        if (eff) T[k] = duration(clamp_param(P.a_s[row + src[k]]), clamp_param(P.a_p[row + src[k]]), __ffs(eff));   // 0: the scenario is flagged
      }
    }
#pragma unroll 1
    for (u32 nm = H.need; nm; nm &= nm - 1) {
      const int j = __ffs(nm) - 1;
      const int mine = (pl[0] == j) + (pl[1] == j) + (pl[2] == j) + (pl[3] == j), before = X.cur[j];
      int tot;
      int pos = before + ks_block_scan(mine, X.scan, t, &tot);
      if (t == 0) X.cur[j] = before + tot;
      const int m_j = X.m[j];
      i64* dst = P.tmin + prow + (size_t)j * P.N;
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        if (pl[k] != j) continue;
        dst[pos] = T[k];
        if (pos == m_j) X.first[j] = src[k];
        ++pos;
      }
    }
    __syncthreads();
  }
}

// Everything behind the head, by a block of KS_THREADS.  The waiting lists' facts go to the pools' PoolMeta.
// SORTED: the queue is taken in the order P.perm.
template <bool SORTED>
__device__ __forceinline__ void stream_queue(const Params& P, int sc, int ws, const HeadState& H, StreamShared& X, int t) {
  const size_t row = (size_t)sc * P.N;
  const size_t prow = (size_t)ws * P.P * P.N;
  const int n_act = min(max(P.n_actions[sc], 0), P.N);
  const u32 need = SORTED ? 0 : H.need;             // taken in another order: this pass only looks for invalid records
  // 128-bit loads need groups that start at multiples of 16 of the whole array, wherever the row begins: the first tile
  // starts up to 15 records early and skips them
  const bool vec = (((size_t)P.a_pool | (size_t)P.a_unit | (size_t)P.a_mask) & 15) == 0;
  const int hs = SORTED && H.hs < n_act ? 0 : H.hs, skew = vec ? (int)((row + hs) & 15) : 0;
  if (t < TG_MAX_POOLS) {
    X.m[t] = t < P.P ? P.meta[(size_t)ws * P.P + t].m : 0;
    X.first[t] = INT_MAX;
  }
  if (hs >= n_act) {                                 // the head walk has seen every record: 8 KB of table for nothing
  } else if (P.ok_table) {
    for (int x = t; x < TG_MAX_POOLS * 256 / 4; x += KS_THREADS) ((uint4*)X.ok)[x] = ((const uint4*)P.ok_table)[x];
  } else {
#pragma unroll 1
    for (int x = t; x < TG_MAX_POOLS * 256; x += KS_THREADS) {
      int g, gang; u32 eff = 0;
      if (x < P.P * 256) decode_levels(P.pool[x >> 8], (u8)(x & 255), 0xffffffffu, g, gang, eff);
      X.ok[x] = eff;
    }
  }
  if (t == 0) X.bad = H.bad;
  __syncthreads();

  if (t < TG_MAX_POOLS) X.cur[t] = H.cur[t];          // actions of every pool seen so far
  __syncthreads();
  for (int tile0 = hs - skew; tile0 < n_act; tile0 += KS_TILE) {   // a bad scenario is streamed on: its rows are rewritten below
    const int i_first = tile0 + t * KS_ITEMS;
    const bool full = vec && i_first >= hs && i_first + KS_ITEMS <= n_act;
    __align__(16) u8 rp[KS_ITEMS], ru[KS_ITEMS];
    // validate; keep the least multiplicity of the records whose pool may need its list
    bool bad = false;
    u32 rmin4[KS_ITEMS / 4];                          // one byte per record, 0 = not listed
    {
      __align__(16) u32 rm[KS_ITEMS];
      if (full) {
        *(uint4*)rp = *(const uint4*)(P.a_pool + row + i_first);
        *(uint4*)ru = *(const uint4*)(P.a_unit + row + i_first);
#pragma unroll
        for (int k = 0; k < KS_ITEMS; k += 4) *(uint4*)(rm + k) = *(const uint4*)(P.a_mask + row + i_first + k);
      } else {
#pragma unroll
        for (int k = 0; k < KS_ITEMS; ++k) {
          const int i = i_first + k;
          const bool on = i >= hs && i < n_act;
          rp[k] = on ? P.a_pool[row + i] : 0xff;
          ru[k] = on ? P.a_unit[row + i] : 1;
          rm[k] = on ? P.a_mask[row + i] : 1;
        }
      }
#pragma unroll
      for (int k = 0; k < KS_ITEMS / 4; ++k) rmin4[k] = 0;
#pragma unroll
      for (int k = 0; k < KS_ITEMS; ++k) {
        if (!full && (i_first + k < hs || i_first + k >= n_act)) continue;
        const int j = rp[k];
        const u32 eff = j < TG_MAX_POOLS ? rm[k] & X.ok[j * 256 + ru[k]] : 0u;   // pools beyond the description hold zeros
        bad |= eff == 0;
        if ((need >> j) & 1u) rmin4[k >> 2] |= (u32)__ffs(eff) << (8 * (k & 3));
      }
    }
    if (bad) X.bad = 1;
    // waiting lists of the pools that may need them; a position follows from the pool bytes alone
    for (u32 nm = need; nm; nm &= nm - 1) {
      const int j = __ffs(nm) - 1;
      u32 mine = 0;
#pragma unroll
      for (int k = 0; k < KS_ITEMS; ++k) if (rp[k] == j) mine |= 1u << k;
      const int before = X.cur[j];
      int tot;
      int pos = before + ks_block_scan(__popc(mine), X.scan, t, &tot);
      if (t == 0) X.cur[j] = before + tot;               // read again only after the barrier that ends the tile
      if (!mine) continue;
      const int m_j = X.m[j];
      i64* dst = P.tmin + prow + (size_t)j * P.N;
      // the thread's listed records, four at a time: their s / p loads are in flight together
      const u64 rlo = (u64)rmin4[0] | ((u64)rmin4[1] << 32), rhi = (u64)rmin4[2] | ((u64)rmin4[3] << 32);
      for (u32 rest = mine; rest;) {
        i64 sv[4], pv[4]; int kk[4];
#pragma unroll
        for (int x = 0; x < 4; ++x) {
          kk[x] = rest ? __ffs(rest) - 1 : -1;
          rest &= rest - 1;
          sv[x] = kk[x] >= 0 ? P.a_s[row + i_first + kk[x]] : 0;
          pv[x] = kk[x] >= 0 ? P.a_p[row + i_first + kk[x]] : 0;
        }
#pragma unroll
        for (int x = 0; x < 4; ++x) {
          if (kk[x] < 0) continue;
          const int rmin = (int)(((kk[x] < 8 ? rlo : rhi) >> (8 * (kk[x] & 7))) & 0xffu);
          if (rmin) dst[pos] = duration(clamp_param(sv[x]), clamp_param(pv[x]), rmin);   // 0: invalid record, the scenario is flagged
          if (pos == m_j) X.first[j] = i_first + kk[x];   // the pool's first waiting action
          ++pos;
        }
      }
    }
    __syncthreads();
  }
  if (SORTED && H.need) stream_sorted(P, sc, ws, H, X, t);
  __syncthreads();
  const bool bad = X.bad != 0;
  // nobody will write the candidates of a bad scenario: their rows are "not scheduled" too
  if (bad) for (int i = t; i < min(H.n, P.N); i += KS_THREADS) {
    P.o_alloc[row + i] = 0; P.o_node[row + i] = -1; P.o_off[row + i] = -1; P.o_act[row + i] = -1;
  }
  if (t < P.P) {
    PoolMeta* mt = P.meta + (size_t)ws * P.P + t;
    if (bad) { mt->count = 0; mt->m = 0; mt->first_wait = -1; }
    else if ((H.need >> t) & 1u) {
      mt->count = X.cur[t];
      if (X.first[t] != INT_MAX) mt->first_wait = X.first[t];
    } else mt->count = mt->m;                          // a list nobody reads counts as empty
  }
  // (status, total and count were initialised by the head walk)
  if (t == 0 && bad) atomicOr(&P.o_status[sc], TG_ST_BAD_ACTION);
}

template <bool SORTED>
__global__ void __launch_bounds__(KS_THREADS, 5) k_stream(const __grid_constant__ Params P, const HeadState* hst) {
  __shared__ StreamShared X;
  stream_queue<SORTED>(P, blockIdx.x, blockIdx.x, hst[blockIdx.x], X, threadIdx.x);
}

// "not scheduled" (Eq. 2 has no value for an action that stays queued): units 0, node -1, offset -1,
// ACT -1 for every action behind its scenario's candidate prefix (the candidates' rows are written
// by the kernels that decide them, which may run at the same time).  Consecutive threads take
// consecutive groups of four actions, so a warp's store covers whole contiguous sectors.
__device__ __forceinline__ void write_unscheduled(const Params& P, size_t o) {
  P.o_alloc[o] = 0; P.o_node[o] = -1; P.o_off[o] = -1; P.o_act[o] = -1;
}
__device__ __forceinline__ void write_unscheduled4(const Params& P, size_t o) {
  const int4 z = make_int4(0, 0, 0, 0), m1 = make_int4(-1, -1, -1, -1);
  const longlong2 a1 = make_longlong2(-1, -1);
  *(int4*)(P.o_alloc + o) = z; *(int4*)(P.o_node + o) = m1; *(int4*)(P.o_off + o) = m1;
  *(longlong2*)(P.o_act + o) = a1; *(longlong2*)(P.o_act + o + 2) = a1;
}
__device__ __forceinline__ bool outputs_aligned(const Params& P) {
  return (((size_t)P.o_alloc | (size_t)P.o_node | (size_t)P.o_off | (size_t)P.o_act) & 15) == 0;
}
__global__ void __launch_bounds__(256) k_fill(const __grid_constant__ Params P) {
  const u32 stride = gridDim.x * blockDim.x, tid = blockIdx.x * blockDim.x + threadIdx.x, total = (u32)P.S * (u32)P.N;   // S * N <= 2^31
  if (outputs_aligned(P)) {
    for (u32 q = tid; q < total / 4; q += stride) write_unscheduled4(P, (size_t)q * 4);
    if (tid < total % 4) write_unscheduled(P, (size_t)(total - 1 - tid));
  } else
    for (u32 o = tid; o < total; o += stride) write_unscheduled(P, o);
}

// The rows of scenario sc from action n on, by one warp.  Written by a kernel beside k_stream they took the memory that
// that one needs: k_stream 549 us with that kernel beside it, 339 alone, at 16384 x 4096, and the
// call 1675 against 1556.
__device__ __forceinline__ void fill_rows(const Params& P, int sc, int n, int lane) {
  const size_t row = (size_t)sc * P.N, o0 = row + (size_t)min(n, P.N), o1 = row + P.N;
  const size_t a0 = (o0 + 3) & ~(size_t)3, a1 = o1 & ~(size_t)3;           // groups of four of the whole array
  if (a0 >= a1 || !outputs_aligned(P)) {
    for (size_t o = o0 + lane; o < o1; o += 32) write_unscheduled(P, o);
    return;
  }
  if (o0 + lane < a0) write_unscheduled(P, o0 + lane);
  if (a1 + lane < o1) write_unscheduled(P, a1 + lane);
  const u32 groups = (u32)((a1 - a0) / 4);
  const int4 z = make_int4(0, 0, 0, 0), m1 = make_int4(-1, -1, -1, -1);
  int4* const al = (int4*)P.o_alloc + a0 / 4; int4* const nd = (int4*)P.o_node + a0 / 4; int4* const of = (int4*)P.o_off + a0 / 4;
  int4* const ac = (int4*)P.o_act + a0 / 2;
#pragma unroll 2
  for (u32 g = lane; g < groups; g += 32) { al[g] = z; nd[g] = m1; of[g] = m1; }
#pragma unroll 4
  for (u32 g = lane; g < 2 * groups; g += 32) ac[g] = m1;
}
