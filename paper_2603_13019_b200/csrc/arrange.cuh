// Per-pool selection of a round, first half: DPArrange (Algorithms 3 and 4), executed by one warp
// per (scenario, pool).
//
// The problem: every candidate of a prefix gets one of its levels; the duration sum is minimal
// subject to the pool's capacity, for a GPU pool four nested ones (GPUs asked for in chunks of at
// least 1, 2, 4, 8 GPUs against the GPUs held in free aligned blocks of at least that size).  Ties
// follow the canonical order: lowest duration sum, then fewest units, then (k_m, ..., k_1)
// lexicographically smallest.
//
// Two certificates need no search: every candidate's best level fits (each takes the smallest level
// that reaches its lowest duration), or no unit is spare (everybody keeps the least level).
// Otherwise the capacities get PRICES (Lagrange multipliers, whole microseconds per unit, found by
// bisection on the demand that the priced choices add up to).  Under fixed prices every candidate
// has a cheapest level, and any other level costs an EXCESS >= 0 on top; an allocation's duration
// sum is a constant plus its excesses plus price times unused capacity, all three >= 0.  So with U
// known such that the optimum's excess-plus-slack is <= U, no optimal allocation uses a level
// whose excess is above U: most candidates are fixed to their cheapest level and the recurrence of
// Algorithm 3 / 4 only runs over the few that are not, on the few states (demand shifts against the
// priced choices) whose accumulated excess stays <= U.  U starts small and is raised until a solution
// within it is found, which then is the optimum: nothing outside could be better or tie.  The
// result does not depend on the prices, only the work does.  Where nobody is a gang request, a method whose work
// the extents bound takes over from passes that would cost more (dp_classes).
//
// Measured on B200 (fragmented 8-node pools with elastic gang requests, 500 scenarios x 200 actions):
// the table over the product of the four extents has 1e3 .. 1e6 cells per row; the bounded states
// are 5 .. 35 per row (maximum over 1000 pools: 340).
#pragma once
#include "common.cuh"

// Scratch of one worker warp: a window of shared memory first (what is read over and over in
// sequential loops belongs there), its slab in global memory once the window is full.
struct Slab {
  char* base; u64 cap; u64 used;          // global slab
  char* fbase; u32 fcap; u32 fused;       // shared-memory window (generic address), may be empty
  __device__ __forceinline__ void* take(u64 bytes) {
    bytes = (bytes + 15) & ~(u64)15;
    if (used + bytes > cap) return nullptr;
    void* p = base + used; used += bytes; return p;
  }
  // small arrays that sequential loops read again and again: the window if there is room
  __device__ __forceinline__ void* take_fast(u64 bytes) {
    bytes = (bytes + 15) & ~(u64)15;
    if (fused + bytes <= fcap) { void* p = fbase + fused; fused += (u32)bytes; return p; }
    return take(bytes);
  }
};

// warp-uniform bump allocation from the bump part of the arena
__device__ __forceinline__ void* arena_take(const Params& P, u64 bytes, int lane) {
  bytes = (bytes + 255) & ~(u64)255;
  const u64 half = arena_bump_base(P);
  u64 off = 0;
  if (lane == 0) off = atomicAdd(P.arena_top, bytes);
  off = __shfl_sync(TG_FULL, off, 0);
  if (half + off + bytes > P.arena_bytes) return nullptr;
  return P.arena + half + off;
}
// Borrow a slot (warp-uniform).  Waits, with a limit, for another warp to give one back; the
// holders never wait for anything, so the wait ends.  Returns -1 if the table does not fit a
// slot or the limit ran out.
__device__ __forceinline__ int slot_acquire(const Params& P, u64 bytes, int lane) {
  const u64 slot_bytes = arena_slot_bytes(P);
  int got = -1;
  if (lane == 0 && bytes <= slot_bytes) {
    int* flags = (int*)(P.arena_top + 8);
    const int ns = arena_n_slots(P);
    const int start = (int)((blockIdx.x * blockDim.x + threadIdx.x) >> 5) % ns;
#pragma unroll 1
    for (int tries = 0; tries < P.slot_tries && got < 0; ++tries) {   // gives up after the round's slot_wait_us
#pragma unroll 1
      for (int k = 0; k < ns && got < 0; ++k) {
        const int s = (start + k) % ns;
        if (atomicCAS(&flags[s], 0, 1) == 0) got = s;
      }
      if (got < 0) __nanosleep(2000);
    }
  }
  return __shfl_sync(TG_FULL, got, 0);
}
__device__ __forceinline__ char* slot_ptr(const Params& P, int s) {
  return P.arena + (u64)s * arena_slot_bytes(P);
}
__device__ __forceinline__ void slot_release(const Params& P, int s, int lane) {
  __syncwarp();
  if (lane == 0 && s >= 0) { __threadfence(); atomicExch((int*)(P.arena_top + 8) + s, 0); }
}

// One (scenario, pool) at hand.  It lives in the warp's shared memory: the same for all lanes, and the routines
// below take what they need of it into locals.  They are inlined, one place each in every kernel: a warp that calls
// waits for the instructions at the other end (a third of all warp cycles at 8192 x 1024 was waiting for instructions; k_pool at 16384 x
// 4096 1555 us with the routines out of line, 1316 us inlined).
struct PoolTask {
  // the pool
  int type, group;
  int cap[4];             // free capacity per chunk level (core / quota pools: cap[0] only)
  // candidates of the pool in queue order
  int m;
  const i64* cs; const i64* cp; const u32* cmask; const u8* cg;
  // what waits behind them on this pool: durations at the least level, and the first record
  const i64* ac_tmin; int n_ac;
  Act ac_first;
  // completion times (relative to now) of what is running on the pool
  const i64* seeds; int n_seeds;
  int depth;
  // results: multiplicity per candidate of the prefix under evaluation / of the accepted one
  u8* rsel; u8* rkeep;
  int* rowcand;           // scratch, m ints
  // work area of this warp in shared memory (generic address, 16-byte aligned)
  char* wk; u32 wk_bytes;
  float lam[4];           // prices of the prefix solved last (0: none known)
  i64 opt;                // duration sum of the prefix solved last
  // sums over the candidates of prefix sq (0: none yet): demand per chunk level at the least and at the best levels,
  // largest extra demand, duration sums; elastic candidates and their levels
  int sq, dmin[4], dbest[4], maxex[4], nrows, n_levels;
  i64 tmin_sum, tbest_sum;
  // table of at most 32 cells over the elastic rows (small_table): values and choices, [row][32]; rows in it (0: not
  // built, -1: not possible)
  i64* cell_val; unsigned short* cell_ch; int cell_rows;
  // nested capacities bind and nobody is an elastic gang request (dp_classes applies): upgrade steps and candidates
  // with gaps in their levels; upgrades -1: another pool
  int upgrades, gaps;
  int limit;              // what a pass of bounded_dp may cost, in rows times 32 states
};

// a level as one number pair: units of multiplicity r and the chunk class they are asked for at
__device__ __forceinline__ int class_of(int type, int g, int gang, int r) {
  return type == TG_POOL_GPU ? level_of(g, gang, r) : 0;
}

// extra demand, per chunk level, of multiplicity r over the least multiplicity r0
__device__ __forceinline__ void extra_demand(int type, int g, int gang, int r0, int r, int d[4]) {
  d[0] = d[1] = d[2] = d[3] = 0;
  if (type != TG_POOL_GPU) { d[0] = g * (r - r0); return; }
  if (gang) {
    int z = g * r, z0 = g * r0, lz = ilog2(z), lz0 = ilog2(z0);
#pragma unroll
    for (int l = 0; l < 4; ++l) if (l <= lz) d[l] = z - (l <= lz0 ? z0 : 0);
  } else {
    int lz = ilog2(g);
#pragma unroll
    for (int l = 0; l < 4; ++l) if (l <= lz) d[l] = g * (r - r0);
  }
}

// smallest multiplicity that already reaches the duration of the largest one (durations do not grow
// with the level, so the levels that reach it are the topmost ones)
__device__ __forceinline__ int best_level(i64 p, u32 mask) {
  int r = 32 - __clz(mask);
  const i64 tb = div_small(p, r);
#pragma unroll 1
  for (u32 mm = mask & ~(1u << (r - 1)); mm;) {
    const int x = 32 - __clz(mm);
    if (div_small(p, x) != tb) break;
    r = x; mm &= ~(1u << (x - 1));
  }
  return r;
}

// ---- prices ---------------------------------------------------------------------------------
// Level table of the elastic rows T.rowcand[0 .. nrows): row t's levels are entries off[t] .. off[t+1].
// x: gain over the least level (float bits); y: units (float bits, whole) with the chunk class in
// the two lowest mantissa bits (units stay below 2^20, so those bits are free).
struct Levels { const uint2* lv; const u32* off; int nrows; };
#define LV_UNITS(y) ((int)__uint_as_float((y) & ~3u))
#define LV_CLASS(y) ((int)((y) & 3u))

// four values by a run-time index without an array in memory
template <class V>
__device__ __forceinline__ V pick4(const V v[4], int l) { return l == 0 ? v[0] : (l == 1 ? v[1] : (l == 2 ? v[2] : v[3])); }

// Demand at level `l` of the rows' cheapest levels under the prices lam (per unit, added up from class 0 to
// the level's class).
__device__ __forceinline__ int priced_demand(const Levels& V, const float lam[4], int l, int lane) {
  const float p0 = lam[0], p1 = p0 + lam[1], p2 = p1 + lam[2], p3 = p2 + lam[3];
  int x = 0;
#pragma unroll 1
  for (int t = lane; t < V.nrows; t += 32) {
    u32 by = 0; float best = 3.0e38f;
#pragma unroll 1
    for (u32 k = V.off[t], e = V.off[t + 1]; k < e; ++k) {
      const uint2 v = V.lv[k];
      const float p = (v.y & 2u) ? ((v.y & 1u) ? p3 : p2) : ((v.y & 1u) ? p1 : p0);
      const float cost = fmaf(__uint_as_float(v.y), p, -__uint_as_float(v.x));
      if (cost < best) { best = cost; by = v.y; }
    }
    if (LV_CLASS(by) >= l) x += LV_UNITS(by);
  }
  return warp_sum32(x);
}

// Prices under which the rows' cheapest levels (about) fill the capacities.  Level 0 first; then, where the
// pool has nested capacities that bind, the others and level 0 again, at most four times.  A level's price moves to (about) the
// smallest one at which the demand is within the capacity: a bracket grown from the current price by factors that
// square from step to step, then bisection to one part in 1000; it stops early where the demand meets the
// capacity exactly.  first: average gain per unit, where no price is known.
__device__ __forceinline__ void search_prices(const Levels& V, float lam[4], u32 kept, const int cap[4], float first, int lane) {
  const int n_turns = kept == 1u ? 1 : 17;               // levels 0 | 1 2 3 0 | 1 2 3 0 | ...
  bool moved = false;
#pragma unroll 1
  for (int turn = 0; turn < n_turns; ++turn) {
    const int l = turn & 3;
    if (!((kept >> l) & 1u)) continue;
    if (l == 0 && turn > 0) { if (!moved) break; moved = false; }
    const float was = pick4(lam, l);
    const int c = pick4(cap, l);
    float lo = 0.f, hi = -1.f, grow = was > 0.f ? 1.125f : 2.f;
    float x = l > 0 ? 0.f : (was > 0.f ? was : first);   // an inner level may not bind at all
#pragma unroll 1
    for (int it = 0; it < 64; ++it) {
#pragma unroll
      for (int k = 0; k < 4; ++k) if (k == l) lam[k] = x;
      const int d = priced_demand(V, lam, l, lane);
      if (d == c || (d < c && x == 0.f)) { hi = x; break; }
      if (x == 0.f) { x = was > 0.f ? was : fmaxf(0.25f * lam[0], 1.f); continue; }
      if (d > c) lo = x; else hi = x;
      if (hi < 0.f) { x = lo * grow; grow *= grow; }
      else if (lo == 0.f) {
        if (hi < 1.f) break;                             // prices are whole microseconds
        x = fmaxf(hi / grow, 0.5f); grow *= grow;
      } else {
        if (hi - lo <= hi * (1.f / 1024.f)) break;
        x = 0.5f * (lo + hi);
      }
      if (x > 4.0e12f) break;                            // beyond any gain per unit: durations are below 2^41
    }
    x = hi >= 0.f ? hi : lo;
#pragma unroll
    for (int k = 0; k < 4; ++k) if (k == l) lam[k] = x;
    moved |= l > 0 && x != was;
  }
}

// ---- the bounded recurrence -----------------------------------------------------------------
// A state's key is the demand shift against the priced choices: level 0 in the upper bits, levels 1 .. 3
// (multiples of 2, 4, 8 GPUs, counted in those) in 13 bits each, biased.
#define BD_SHIFT0 39
#define BD_EMPTY 0xffffffffffffffffull
#define BD_ZERO (((u64)1 << 63) | ((u64)4096 << 26) | ((u64)4096 << 13) | (u64)4096)
__device__ __forceinline__ u64 bd_pack(const int d[4], u32 kept) {
  u64 k = (u64)(i64)d[0] << BD_SHIFT0;
#pragma unroll
  for (int l = 1; l < 4; ++l) if ((kept >> l) & 1u) k += (u64)(i64)(d[l] >> l) << (13 * (3 - l));
  return k;
}
__device__ __forceinline__ int bd_field(u64 key, int l) {
  return l == 0 ? (int)((i64)(key ^ ((u64)1 << 63)) >> BD_SHIFT0) : ((int)((key >> (13 * (3 - l))) & 8191u) - 4096) << l;
}
__device__ __forceinline__ u32 bd_hash(u64 k) { k ^= k >> 32; k *= 0x9e3779b97f4a7c15ull; return (u32)(k >> 40); }

// States, numbered as they come up, in [mem, mem + bytes): key; excess after the row before; (excess << 6 |
// multiplicity) of the row at hand.  tab finds a state's number by its key (open addressing, at most half full).
struct BdTable {
  u64* key; u64* exc; u64* val; u64* fresh;   // fresh: 32 keys on their way in, one per lane
  unsigned short* tab;
  u32 mask; int cap;
};
#define BD_NONE 0xffffu
#define BD_ON_ITS_WAY 0x8000u       // | lane
__device__ __forceinline__ bool bd_table(BdTable& B, char* mem, u64 bytes) {
  u32 cap = 32;
  if (cap * 28 + 256 > bytes) return false;
#pragma unroll 1
  while (cap < 4096 && (u64)cap * 56 + 256 <= bytes) cap *= 2;
  B.key = (u64*)mem; B.exc = B.key + cap; B.val = B.exc + cap; B.fresh = B.val + cap;
  B.tab = (unsigned short*)(B.fresh + 32);
  B.mask = 2 * cap - 1; B.cap = (int)cap;
  return true;
}
__device__ __forceinline__ int bd_find(const BdTable& B, u64 key) {      // the key is there
  u32 h = bd_hash(key) & B.mask;
#pragma unroll 1
  for (u32 k = 0; k < B.mask; ++k) {
    const u32 x = B.tab[h];
    if (x == BD_NONE || B.key[x] == key) return (int)x;
    h = (h + 1) & B.mask;
  }
  return 0;
}

// One level of row i under the prices: excess over the row's cheapest level (lane r - 1 holds multiplicity r;
// -1 where the row has no such level), the cheapest level itself (smallest multiplicity among equals) and the
// demand shift of every level against it.
struct RowCost { i64 x; int rstar; u64 shift; };
__device__ __forceinline__ RowCost bd_row(const PoolTask& T, int i, const i64 price[4], u32 kept, int lane) {
  RowCost R;
  const u32 mk = T.cmask[i];
  const int g = T.cg[i] & 0x7f, gang = T.cg[i] >> 7, r = lane + 1;
  const bool on = (mk >> lane) & 1u;
  const int u = g * r, c = on ? class_of(T.type, g, gang, r) : 0;
  const i64 pc = pick4(price, c);
  const i64 cost = on ? duration(T.cs[i], T.cp[i], r) + (i64)u * pc : TG_INF;
  const i64 b = warp_min64(cost);
  const int rs = __ffs(__ballot_sync(TG_FULL, cost == b));
  const int us = g * rs, csr = class_of(T.type, g, gang, rs);
  int d[4];
#pragma unroll
  for (int l = 0; l < 4; ++l) d[l] = (l <= c ? u : 0) - (l <= csr ? us : 0);
  R.x = on ? cost - b : -1; R.rstar = rs; R.shift = on ? bd_pack(d, kept) : 0;
  return R;
}

// The recurrence over the rows of frow[0 .. nfree), levels and states with excess <= delta.  slack[l] = capacity
// the priced choices leave (may be negative).  choice: the states' multiplicities row by row, crow[f] = where row f's
// start; lim[f]: smallest and largest demand shift of row f's usable levels, per level (eight 16-bit numbers), by which
// a state is dropped that the rows behind cannot bring within the capacities, or cannot fill enough.  On success
// the rows' multiplicities are in T.rsel.  Returns 1 solved, 0 nothing within delta, -1 out of room (or more than 32 end states tie).
__device__ __forceinline__ int bounded_dp(const PoolTask& T, const int* frow, u32* crow, const uint4* lim, int nfree, const i64 price[4], const i64 lam[4],
                                       u32 kept, const int slack[4], i64 delta, BdTable B, u8* choice, u64 choice_bytes,
                                       int lane) {
  u64 used = 0;
  // smallest and largest shift of all the rows behind the current one
  int lo[4] = {0, 0, 0, 0}, hi[4] = {0, 0, 0, 0};
#pragma unroll 1
  for (int f = lane; f < nfree; f += 32) {
    const uint4 v = lim[f];
    lo[0] += (short)v.x; hi[0] += (short)(v.x >> 16); lo[1] += (short)v.y; hi[1] += (short)(v.y >> 16);
    lo[2] += (short)v.z; hi[2] += (short)(v.z >> 16); lo[3] += (short)v.w; hi[3] += (short)(v.w >> 16);
  }
#pragma unroll
  for (int l = 0; l < 4; ++l) { lo[l] = warp_sum32(lo[l]); hi[l] = warp_sum32(hi[l]); }
#pragma unroll 1
  for (u32 h = lane; h <= B.mask; h += 32) B.tab[h] = BD_NONE;
  __syncwarp();
  int n = 1;
  if (lane == 0) { B.tab[bd_hash(BD_ZERO) & B.mask] = 0; B.key[0] = BD_ZERO; B.exc[0] = 0; }
  __syncwarp();
#pragma unroll 1
  for (int f = 0; f < nfree; ++f) {
    const RowCost R = bd_row(T, frow[f], price, kept, lane);
    const u32 alts = __ballot_sync(TG_FULL, R.x >= 0 && R.x <= delta && lane + 1 != R.rstar);
    {
      const uint4 v = lim[f];
      lo[0] -= (short)v.x; hi[0] -= (short)(v.x >> 16); lo[1] -= (short)v.y; hi[1] -= (short)(v.y >> 16);
      lo[2] -= (short)v.z; hi[2] -= (short)(v.z >> 16); lo[3] -= (short)v.w; hi[3] -= (short)(v.w >> 16);
    }
    const int n0 = n;
#pragma unroll 1
    for (int x = lane; x < n0; x += 32) B.val[x] = (B.exc[x] << 6) | (u64)R.rstar;
    __syncwarp();
#pragma unroll 1
    for (u32 am = alts; am; am &= am - 1) {
      const int a = __ffs(am) - 1;
      const i64 xa = __shfl_sync(TG_FULL, R.x, a);
      const u64 sh = __shfl_sync(TG_FULL, R.shift, a);
#pragma unroll 1
      for (int x0 = 0; x0 < n0; x0 += 32) {
        bool ok = x0 + lane < n0, fresh = false;
        u64 k = 0; i64 e = 0; u32 h = 0;
        if (ok) {
          e = (i64)B.exc[x0 + lane] + xa; k = B.key[x0 + lane] + sh;
          i64 least = e;                                 // with the price of what must stay unused
#pragma unroll
          for (int l = 0; l < 4; ++l)
            if ((kept >> l) & 1u) {
              const int left = slack[l] - bd_field(k, l);
              ok &= left >= lo[l];
              least += lam[l] * (i64)max(0, left - hi[l]);
            }
          ok &= least <= delta;
          B.fresh[lane] = k;
        }
        __syncwarp();
        if (ok) {
          h = bd_hash(k) & B.mask;
#pragma unroll 1
          for (u32 probe = 0; probe <= B.mask; ++probe) {
            u32 x = B.tab[h];
            if (x == BD_NONE) x = atomicCAS(&B.tab[h], (unsigned short)BD_NONE, (unsigned short)(BD_ON_ITS_WAY | lane));
            if (x == BD_NONE) { fresh = true; break; }
            if ((x & BD_ON_ITS_WAY ? B.fresh[x & 31u] : B.key[x]) == k) break;
            h = (h + 1) & B.mask;
          }
        }
        const u32 fb = __ballot_sync(TG_FULL, fresh);
        if (n + __popc(fb) > B.cap) return -1;
        if (fresh) {
          const int y = n + __popc(fb & ((1u << lane) - 1u));
          B.key[y] = k; B.val[y] = ~0ull; B.tab[h] = (unsigned short)y;
        }
        n += __popc(fb);
        __syncwarp();
        if (ok) atomicMin((unsigned long long*)&B.val[B.tab[h]], ((u64)e << 6) | (u64)(a + 1));
      }
    }
    __syncwarp();
    if (used + n > choice_bytes) return -1;
    u8* ch = choice + used;
    if (lane == 0) crow[f] = (u32)used;
    used += n;
#pragma unroll 1
    for (int x = lane; x < n; x += 32) {
      const u64 v = B.val[x];
      B.exc[x] = v >> 6; ch[x] = (u8)(v & 63u);
    }
    __syncwarp();
  }
  // best end state within the capacities: lowest value (excess plus price of what stays unused), then fewest units
  i64 bv = TG_INF;
#pragma unroll 1
  for (int x = lane; x < n; x += 32) {
    const u64 k = B.key[x];
    i64 v = (i64)B.exc[x];
    bool in = true;
#pragma unroll
    for (int l = 0; l < 4; ++l)
      if ((kept >> l) & 1u) { const int left = slack[l] - bd_field(k, l); in &= left >= 0; v += lam[l] * (i64)left; }
    if (!in) v = TG_INF;
    B.val[x] = (u64)v;
    bv = min(bv, v);
  }
  bv = warp_min64(bv);
  if (bv > delta) return 0;
  int bu = INT_MAX;
#pragma unroll 1
  for (int x = lane; x < n; x += 32) if ((i64)B.val[x] == bv) bu = min(bu, bd_field(B.key[x], 0));
  bu = warp_min32(bu);
  // the tied end states walk back together, one per lane; at each row (last first) those with the smallest
  // multiplicity stay
  u64 mine = BD_EMPTY;
  int nt = 0;
#pragma unroll 1
  for (int x0 = 0; x0 < n; x0 += 32) {
    const int x = x0 + lane;
    const u64 k = B.key[x < n ? x : 0];
    u32 b = __ballot_sync(TG_FULL, x < n && (i64)B.val[x < n ? x : 0] == bv && bd_field(k, 0) == bu);
    if (nt + __popc(b) > 32) return -1;
#pragma unroll 1
    for (; b; b &= b - 1) {
      const u64 kk = __shfl_sync(TG_FULL, k, __ffs(b) - 1);
      if (lane == nt) mine = kk;
      ++nt;
    }
  }
#pragma unroll 1
  for (int f = nfree - 1; f >= 0; --f) {
    const int i = frow[f];
    const RowCost R = bd_row(T, i, price, kept, lane);
    int r = 255;
    if (mine != BD_EMPTY) r = choice[crow[f] + bd_find(B, mine)];
    const int rm = warp_min32(r);
    if (lane == 0) T.rsel[i] = (u8)rm;
    const u64 sh = __shfl_sync(TG_FULL, R.shift, rm - 1);
    mine = (mine != BD_EMPTY && r == rm) ? mine - sh : BD_EMPTY;
  }
  __syncwarp();
  return 1;
}

// ---- replica requests only: one dimension per chunk size --------------------------------------
// Without gang requests a row of chunk size 2^c only ever adds requests of that size, so the rows fall into four
// classes that meet in nothing but the nested capacities (extra GPUs at sizes >= 2^l at most cap[l] - dmin[l]).  Per
// class, f_c(x) = least duration sum with exactly x extra chunks; the classes are merged from the largest size down,
//   G_c(e) = min over x of G_{c+1}((e - x) / 2) + f_c(x),   e in chunks of 2^c,
// tables over each extent instead of one over their product.  The work depends on the extents and hardly on the
// durations.  f_c: where every row's multiplicities are contiguous and its gains T(r) - T(r+1) do not grow (the
// floor in Eq. 1 can break that), f_c(x) is the sum at the least levels minus the x largest gains (separable
// convex resource allocation), and equal gains go to the earliest rows first (a later queue position gets less), so
// one sort of the steps by (gain descending, row, step) serves every x; other classes go through Algorithm 3's
// recurrence.  Two splits between classes that tie on a cell of the chosen path are not decided here.
#define MG_GAIN_BITS 41
#define MG_ROW_BITS 18
#define MG_GAIN_MAX ((1ull << MG_GAIN_BITS) - 1ull)
__device__ __forceinline__ u64 mg_key(i64 gain, int row, int step) {     // step 1-based, at most 31
  return ((MG_GAIN_MAX - (u64)gain) << (MG_ROW_BITS + 5)) | ((u64)row << 5) | (u64)(step - 1);
}
__device__ __forceinline__ i64 mg_gain(u64 key) { return (i64)(MG_GAIN_MAX - (key >> (MG_ROW_BITS + 5))); }
// contiguous multiplicities and gains that do not grow
__device__ __forceinline__ bool mg_row_ok(i64 p, u32 mk) {
  const int r0 = __ffs(mk), rx = 32 - __clz(mk);
  if (__popc(mk) != rx - r0 + 1) return false;
  i64 before = div_small(p, r0), last = TG_INF;
#pragma unroll 1
  for (int r = r0 + 1; r <= rx; ++r) {
    const i64 now = div_small(p, r), gain = before - now;
    if (gain > last) return false;
    last = gain; before = now;
  }
  return true;
}
// ascending bitonic sort of n (a power of two) keys by the calling warp
__device__ __forceinline__ void warp_sort_u64(u64* a, int n, int lane) {
#pragma unroll 1
  for (int k = 2; k <= n; k <<= 1)
#pragma unroll 1
    for (int j = k >> 1; j > 0; j >>= 1) {
#pragma unroll 1
      for (int i = lane; i < n; i += 32) {
        const int l = i ^ j;
        if (l > i) {
          const u64 x = a[i], y = a[l];
          if ((x > y) == ((i & k) == 0)) { a[i] = y; a[l] = x; }
        }
      }
      __syncwarp();
    }
}

// What dp_classes knows of one class; on the warp's slab, so that loops over the classes need no registers per class.
struct ChunkClass {
  int rows, most;          // rows; extra chunks they could use
  int by_gain;             // the steps sorted by gain serve every count
  int U;                   // extra chunks that may be given: min(most, units left >> class)
  int E;                   // merged table: cells 0 .. E, in chunks of this size
  int npad;                // sorted steps, padded to a power of two
  i64 base;                // duration sum at the least levels
  i64* f; u64* keys; u8* ch;
  i64* G; int* sel; u8* tie;
};
#define DPC_MAX_CELLS 4096
// Rows T.rowcand[0 .. T.nrows), none of them a gang request.  Returns 1 with the rows' multiplicities in T.rsel, 0 (T.rsel
// untouched) where splits tie or the slab does not suffice.  This and solve_box are out of line, so that the usual path keeps its
// registers (16384 x 4096, where nothing calls them: 0.3 % slower than without this routine, both inlined 1.5 %,
// only this one out of line 0.7 %).
__device__ __noinline__ int dp_classes(const PoolTask& T, Slab slab, int lane) {
  const int nrows = T.nrows;
  if (nrows >= (1 << MG_ROW_BITS)) return 0;
  ChunkClass* C = (ChunkClass*)slab.take(4 * sizeof(ChunkClass));
  if (!C) return 0;
  int Umax = 0;
#pragma unroll 1
  for (int c = 0; c < 4; ++c) {
    int rows = 0, most = 0; i64 base = 0; bool convex = true;
#pragma unroll 1
    for (int t = lane; t < nrows; t += 32) {
      const int i = T.rowcand[t];
      if (ilog2(T.cg[i]) != c) continue;
      const u32 mk = T.cmask[i];
      ++rows; most += (32 - __clz(mk)) - __ffs(mk);
      base += duration(T.cs[i], T.cp[i], __ffs(mk));
      convex &= mg_row_ok(T.cp[i], mk);
    }
    rows = warp_sum32(rows); most = warp_sum32(most); base = warp_sum64(base);
    const bool by_gain = __all_sync(TG_FULL, convex) && most >= 1;
    const int E = max(T.cap[c] - T.dmin[c], 0) >> c, U = min(E, most);
    if (U + 1 > DPC_MAX_CELLS || E + 1 > 2 * DPC_MAX_CELLS) return 0;
    Umax = max(Umax, U);
    int npad = 1;
    while (npad < most) npad <<= 1;
    i64* f = (i64*)slab.take((u64)(U + 1) * 8);
    u64* keys = by_gain ? (u64*)slab.take((u64)npad * 8) : nullptr;
    u8* ch = by_gain ? nullptr : (u8*)slab.take((u64)max(rows, 1) * (U + 1));
    i64* G = (i64*)slab.take((u64)(E + 1) * 8);
    int* sel = (int*)slab.take((u64)(E + 1) * 4);
    u8* tie = (u8*)slab.take((u64)(E + 1));
    if (!f || (by_gain ? !keys : !ch) || !G || !sel || !tie) return 0;
    if (lane == 0) {
      ChunkClass& k = C[c];
      k.rows = rows; k.most = most; k.by_gain = by_gain; k.U = U; k.E = E; k.npad = npad; k.base = base;
      k.f = f; k.keys = keys; k.ch = ch; k.G = G; k.sel = sel; k.tie = tie;
    }
  }
  i64* work = (i64*)slab.take(2 * (u64)(Umax + 1) * 8);
  if (!work) return 0;
  __syncwarp();
  // ---- per class: f_c(x), least duration sum with exactly x extra chunks
#pragma unroll 1
  for (int c = 0; c < 4; ++c) {
    const ChunkClass& k = C[c];
    const int U = uniform(k.U);
    i64* f = k.f;
    if (k.by_gain) {
      const int n = uniform(k.npad), most = uniform(k.most);
      u64* srt = (u64)n * 8 <= T.wk_bytes ? (u64*)T.wk : k.keys;
      int fill = 0;                                      // every row writes its steps behind those of the rows before it
#pragma unroll 1
      for (int t0 = 0; t0 < nrows; t0 += 32) {
        const int t = t0 + lane;
        int ex = 0, r0 = 1; i64 p = 0;
        if (t < nrows) {
          const int i = T.rowcand[t];
          const u32 mk = T.cmask[i];
          if (ilog2(T.cg[i]) == c) { r0 = __ffs(mk); ex = (32 - __clz(mk)) - r0; p = T.cp[i]; }
        }
        int incl = ex;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) { const int y = __shfl_up_sync(TG_FULL, incl, o); if (lane >= o) incl += y; }
        u64* dst = srt + fill + incl - ex;
        i64 before = div_small(p, r0);
#pragma unroll 1
        for (int x = 1; x <= ex; ++x) {
          const i64 now = div_small(p, r0 + x);
          dst[x - 1] = mg_key(before - now, t, x);
          before = now;
        }
        fill += __shfl_sync(TG_FULL, incl, 31);
      }
#pragma unroll 1
      for (int x = most + lane; x < n; x += 32) srt[x] = ~0ull;
      __syncwarp();
      warp_sort_u64(srt, n, lane);
      i64 run = k.base;                                  // f_c at the start of the block of 32
#pragma unroll 1
      for (int x0 = 0; x0 <= U; x0 += 32) {
        // f_c(x0 + lane) = run - gains of the steps x0 .. x0 + lane - 1
        const int x = x0 + lane;
        const i64 g = x < U ? mg_gain(srt[x]) : 0;
        i64 incl = g;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) { const i64 y = __shfl_up_sync(TG_FULL, incl, o); if (lane >= o) incl += y; }
        if (x <= U) f[x] = run - (incl - g);
        run -= __shfl_sync(TG_FULL, incl, 31);
      }
      if (srt != k.keys) {
#pragma unroll 1
        for (int x = lane; x < U; x += 32) k.keys[x] = srt[x];
      }
      __syncwarp();
      continue;
    }
    i64* prev = work; i64* cur = work + (Umax + 1);
#pragma unroll 1
    for (int u = lane; u <= U; u += 32) prev[u] = u == 0 ? 0 : TG_INF;
    __syncwarp();
    u8* ch = k.ch;
#pragma unroll 1
    for (int t = 0; t < nrows; ++t) {
      const int i = T.rowcand[t];
      if (ilog2(T.cg[i]) != c) continue;
      const u32 mk = T.cmask[i];
      const int r0 = __ffs(mk);
      const i64 s = T.cs[i], p = T.cp[i];
#pragma unroll 1
      for (int u = lane; u <= U; u += 32) {
        i64 best = TG_INF; int bestr = 0;
#pragma unroll 1
        for (u32 mm = mk; mm; mm &= mm - 1) {
          const int r = __ffs(mm), du = r - r0;
          if (du > u) break;                             // levels ascend
          const i64 pv = prev[u - du];
          if (pv == TG_INF) continue;
          const i64 cand = pv + duration(s, p, r);
          if (cand < best) { best = cand; bestr = r; }
        }
        cur[u] = best; ch[u] = (u8)bestr;
      }
      __syncwarp();
      i64* tmp = prev; prev = cur; cur = tmp;
      ch += U + 1;
    }
#pragma unroll 1
    for (int u = lane; u <= U; u += 32) f[u] = prev[u];
    __syncwarp();
  }
  // ---- merge, largest chunks first
#pragma unroll 1
  for (int c = 3; c >= 0; --c) {
    const ChunkClass& k = C[c];
    const int E = uniform(k.E), U = uniform(k.U), Eup = c < 3 ? uniform(C[c + 1].E) : 0;
    const i64* f = k.f;
    const i64* up_G = c < 3 ? C[c + 1].G : nullptr;
    const u8* up_tie = c < 3 ? C[c + 1].tie : nullptr;
    i64* G = k.G; int* sel = k.sel; u8* tie = k.tie;
#pragma unroll 1
    for (int e = lane; e <= E; e += 32) {
      i64 best = TG_INF; int bu = 0; bool tied = false;
      if (c == 3) { if (e <= U) best = f[e]; }
      else {
        const int hi = min(Eup, e >> 1);
#pragma unroll 1
        for (int up = max(e - U + 1, 0) >> 1; up <= hi; ++up) {       // e - 2 up <= U
          const i64 a = up_G[up], b = f[e - 2 * up];
          if (a == TG_INF || b == TG_INF) continue;
          const i64 cand = a + b;
          if (cand < best) { best = cand; bu = up; tied = up_tie[up] != 0; }
          else if (cand == best) tied = true;
        }
      }
      G[e] = best; sel[e] = bu; tie[e] = tied ? 1 : 0;
    }
    __syncwarp();
  }
  // ---- best end cell: lowest value, then fewest extra GPUs
  const i64* G0 = C[0].G;
  const int E0 = uniform(C[0].E);
  i64 bv = TG_INF;
#pragma unroll 1
  for (int e = lane; e <= E0; e += 32) bv = min(bv, G0[e]);
  bv = warp_min64(bv);
  if (bv == TG_INF) return 0;
  int at = INT_MAX;
#pragma unroll 1
  for (int e = lane; e <= E0; e += 32) if (G0[e] == bv) at = min(at, e);
  at = warp_min32(at);
  if (C[0].tie[at]) return 0;
  // ---- walk back: cells of the merged tables, then the rows of every class
#pragma unroll 1
  for (int c = 0; c < 4; ++c) {
    const ChunkClass& k = C[c];
    const int up = c < 3 ? k.sel[at] : 0;
    int u = at - 2 * up;                                 // extra chunks of this class
    at = up;
    if (k.by_gain) {
      // the steps in front of the cut are taken: a row gets its steps up to the threshold key
      const u64 thr = u >= 1 ? k.keys[u - 1] : 0ull;
#pragma unroll 1
      for (int t = lane; t < nrows; t += 32) {
        const int i = T.rowcand[t];
        if (ilog2(T.cg[i]) != c) continue;
        const u32 mk = T.cmask[i];
        const int r0 = __ffs(mk), ex = u >= 1 ? (32 - __clz(mk)) - r0 : 0;
        const i64 p = T.cp[i];
        i64 before = div_small(p, r0);
        int take = 0;
#pragma unroll 1
        for (int x = 1; x <= ex; ++x) {
          const i64 now = div_small(p, r0 + x);
          if (mg_key(before - now, t, x) > thr) break;   // a row's keys ascend with the step
          take = x; before = now;
        }
        T.rsel[i] = (u8)(r0 + take);
      }
    } else if (lane == 0) {
      const u8* ch = k.ch + (u64)k.rows * (k.U + 1);
#pragma unroll 1
      for (int t = nrows - 1; t >= 0; --t) {
        const int i = T.rowcand[t];
        if (ilog2(T.cg[i]) != c) continue;
        ch -= k.U + 1;
        const int r = ch[u];
        T.rsel[i] = (u8)r;
        u -= r - __ffs(T.cmask[i]);
      }
    }
  }
  __syncwarp();
  return 1;
}

// Once per task whose nested capacities bind: does dp_classes apply?  -> T.upgrades, T.gaps
__device__ __forceinline__ void find_replicas(PoolTask& T, int lane) {
  bool gang = false;
  int gaps = 0, up = 0;
#pragma unroll 1
  for (int i = lane; i < T.m; i += 32) {
    const u32 mk = T.cmask[i];
    const int span = 32 - __clz(mk) - __ffs(mk);
    gang |= (T.cg[i] >> 7) != 0 && span > 0;
    gaps += __popc(mk) != span + 1 ? 1 : 0;
    up += span;
  }
  gang = __any_sync(TG_FULL, gang);
  gaps = warp_sum32(gaps); up = warp_sum32(up);
  if (lane == 0) { T.upgrades = gang ? -1 : up; T.gaps = gaps; }
  __syncwarp();
}
// Prices settle most boxes with few rows, but what a pass of bounded_dp costs is up to the durations; dp_classes costs what
// the extents make of it.  In units of a row times 32 states (1500 to 3300 cycles) that is 40, one per 5 upgrade steps (sorts),
// one per 9 rounds of the largest merge, 1.5 per 32 cells and row with gaps in its levels (recurrence).  A pass may cost
// a quarter of it (at least 24: the first passes, of four rows): the state table is that much smaller.
// Measured, us a call, lowest .. highest of 9 to 16 inputs (64 nodes, 30 % of the GPUs busy, levels 1..4):
//                                       without dp_classes  at once         after one pass  with this limit
//   1024 scenarios x 2048               790 .. 4140         800 .. 1014     757 .. 872      746 .. 895
//   400 x 200                           1075 .. 4770        1600 .. 1900    1120 .. 1646    1083 .. 1792
//   12 x 256, alike durations           495000              1140            1200            1270
//   12 x 256, 128 nodes, levels 1 2 4 8 1090                6550            3110            1080
//   12 x 256, levels 1 2 4 8            350                 680             650             630
// (alike durations: the states outgrow every table but the arena's).  A pass that may cost half or all of dp_classes: 1540
// and 1600 for the alike durations, 1118 .. 1750 and 1099 .. 2040 for 400 x 200.
__device__ __forceinline__ void set_limit(PoolTask& T, int lane) {
  const int Y0 = T.cap[0] - T.dmin[0], Y1 = T.cap[1] - T.dmin[1];
  const int blocks = (min(Y0, 1 << 14) >> 5) + 1, span = min(min(Y1, T.upgrades), 1 << 14) >> 1;
  const int cost = 40 + T.upgrades / 5 + blocks * span / 9 + min(T.gaps, 1 << 14) * blocks * 3 / 2;
  if (lane == 0) T.limit = max(cost / 4, 24);
  __syncwarp();
}

// The optimum under prices, over the elastic rows T.rowcand[0 .. nrows) with Y[l] units to give beyond everybody's
// least level (Y[0] > 0).  lam: prices to start from and the prices found (all 0: none known).  T.rsel holds the
// only level of every inelastic candidate on entry and the optimum on success.  T0.limit: what a pass may cost (INT_MAX:
// anything); where it would cost more, dp_classes decides.  Returns 0 if the state tables do not suffice (the caller
// then goes through the general tables).
__device__ __forceinline__ int solve_priced(const PoolTask& T0, const PoolTask& T, int nrows, int n_levels, const int Y[4], u32 kept,
                                            Slab slab, int lane) {
  float lam[4] = {T0.lam[0], T0.lam[1], T0.lam[2], T0.lam[3]};
  // ---- level table, in the work area if it fits
  const u64 off_bytes = ((u64)(nrows + 1) * 4 + 15) & ~(u64)15, lv_bytes = off_bytes + (u64)n_levels * 8;
  char* lmem = lv_bytes <= T.wk_bytes ? T.wk : (char*)slab.take(lv_bytes);
  if (!lmem) return 0;
  u32* off = (u32*)lmem;
  uint2* lv = (uint2*)(lmem + off_bytes);
  int base[4] = {0, 0, 0, 0}, at = 0;
  float gsum = 0.f;                                      // average gain per unit: a first price
  int usum = 0;
#pragma unroll 1
  for (int t0 = 0; t0 < nrows; t0 += 32) {
    const int t = t0 + lane;
    u32 mk = 0; int i = 0;
    if (t < nrows) { i = T.rowcand[t]; mk = T.cmask[i]; }
    int incl = __popc(mk);
    const int cnt = incl;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) { const int y = __shfl_up_sync(TG_FULL, incl, o); if (lane >= o) incl += y; }
    if (t < nrows) {
      u32 k = (u32)(at + incl - cnt);
      off[t] = k;
      const int g = T.cg[i] & 0x7f, gang = T.cg[i] >> 7, r0 = __ffs(mk), c0 = class_of(T.type, g, gang, r0);
      const i64 p = T.cp[i], q0 = div_small(p, r0);
      float gain = 0.f; int r = r0;
#pragma unroll 1
      for (u32 mm = mk; mm; mm &= mm - 1) {
        r = __ffs(mm);
        gain = (float)(q0 - div_small(p, r));
        lv[k++] = make_uint2(__float_as_uint(gain), __float_as_uint((float)(g * r)) | (u32)class_of(T.type, g, gang, r));
      }
      gsum += gain; usum += g * (r - r0);
#pragma unroll
      for (int l = 0; l < 4; ++l) if (l <= c0) base[l] += g * r0;
    }
    at += __shfl_sync(TG_FULL, incl, 31);
  }
  if (lane == 0) off[nrows] = (u32)at;
  int cap[4];
#pragma unroll
  for (int l = 0; l < 4; ++l) cap[l] = Y[l] + warp_sum32(base[l]);
#pragma unroll 1
  for (int o = 16; o; o >>= 1) gsum += __shfl_xor_sync(TG_FULL, gsum, o);
  usum = warp_sum32(usum);
  __syncwarp();
  const Levels V = {lv, off, nrows};
  const float first = fmaxf(gsum / fmaxf((float)usum, 1.f), 1.f);
  search_prices(V, lam, kept, cap, first, lane);
  if (lane == 0) {
#pragma unroll
    for (int l = 0; l < 4; ++l) ((PoolTask&)T0).lam[l] = lam[l];
  }
  __syncwarp();
  // ---- exact: cheapest levels, excess of the second cheapest, what the priced choices leave of the capacities
  i64 li[4], price[4];
#pragma unroll
  for (int l = 0; l < 4; ++l) { li[l] = (i64)rintf(lam[l]); price[l] = li[l] + (l ? price[l - 1] : 0); }
  i64* x2 = (i64*)slab.take((u64)nrows * 8);
  int* frow = (int*)slab.take((u64)nrows * 4);
  u32* crow = (u32*)slab.take((u64)nrows * 4);
  uint4* lim = (uint4*)slab.take((u64)nrows * 16);
  if (!x2 || !frow || !crow || !lim) return 0;
  int slack[4] = {0, 0, 0, 0};
  i64 xmin = TG_INF;
#pragma unroll 1
  for (int t = lane; t < nrows; t += 32) {
    const int i = T.rowcand[t];
    const u32 mk = T.cmask[i];
    const int g = T.cg[i] & 0x7f, gang = T.cg[i] >> 7;
    const i64 p = T.cp[i];
    i64 b = TG_INF, b2 = TG_INF; int rs = 0, cs = 0;
#pragma unroll 1
    for (u32 mm = mk; mm; mm &= mm - 1) {
      const int r = __ffs(mm), c = class_of(T.type, g, gang, r);
      const i64 pc = pick4(price, c);
      const i64 cost = div_small(p, r) + (i64)(g * r) * pc;
      if (cost < b) { b2 = b; b = cost; rs = r; cs = c; } else b2 = min(b2, cost);
    }
    x2[t] = b2 - b;
    xmin = min(xmin, b2 - b);
    T.rsel[i] = (u8)rs;
#pragma unroll
    for (int l = 0; l < 4; ++l) if (l <= cs) slack[l] += g * rs;
  }
  xmin = warp_min64(xmin);
  bool feasible = true;
  i64 s0 = 0;                                            // price of the capacity that the priced choices leave unused
#pragma unroll
  for (int l = 0; l < 4; ++l) {
    slack[l] = cap[l] - warp_sum32(slack[l]);
    if ((kept >> l) & 1u) { feasible &= slack[l] >= 0; s0 += li[l] * (i64)slack[l]; }
  }
  __syncwarp();
  if (feasible && s0 < xmin) return 1;                   // any other choice costs more than it could save
  // ---- how far to look: the priced choices themselves are within s0; else a few rows' worth of excess
  i64 delta = s0;
  if (!feasible || s0 > xmin) {
    i64 last = xmin;                                     // fourth smallest second excess
#pragma unroll 1
    for (int k = 0; k < 3; ++k) {
      i64 nx = TG_INF;
#pragma unroll 1
      for (int t = lane; t < nrows; t += 32) if (x2[t] > last) nx = min(nx, x2[t]);
      nx = warp_min64(nx);
      if (nx == TG_INF) break;
      last = nx;
    }
    delta = feasible ? min(s0, last) : last;
  }
  const u64 room = slab.cap - slab.used;
#pragma unroll 1
  for (int pass = 0; pass < 40; ++pass) {
    if (delta >= (1ll << 56)) return 0;
    int nfree = 0, reach = 0;
#pragma unroll 1
    for (int t0 = 0; t0 < nrows; t0 += 32) {
      const int t = t0 + lane;
      const bool fr = t < nrows && x2[t] <= delta;
      const u32 b = __ballot_sync(TG_FULL, fr);
      if (fr) {
        const int i = T.rowcand[t];
        // its usable levels' smallest and largest demand shifts
        const u32 mk = T.cmask[i];
        const int g = T.cg[i] & 0x7f, gang = T.cg[i] >> 7, rs = T.rsel[i], cs = class_of(T.type, g, gang, rs);
        const i64 p = T.cp[i], most = div_small(p, rs) + (i64)(g * rs) * pick4(price, cs) + delta;
        int dl[4] = {0, 0, 0, 0}, dh[4] = {0, 0, 0, 0};
#pragma unroll 1
        for (u32 mm = mk; mm; mm &= mm - 1) {
          const int r = __ffs(mm), c = class_of(T.type, g, gang, r);
          if (div_small(p, r) + (i64)(g * r) * pick4(price, c) > most) continue;
#pragma unroll
          for (int l = 0; l < 4; ++l) {
            const int d = (l <= c ? g * r : 0) - (l <= cs ? g * rs : 0);
            dl[l] = min(dl[l], d); dh[l] = max(dh[l], d);
          }
        }
        const int f = nfree + __popc(b & ((1u << lane) - 1u));
        frow[f] = i;
        lim[f] = make_uint4((u32)(dl[0] & 0xffff) | ((u32)dh[0] << 16), (u32)(dl[1] & 0xffff) | ((u32)dh[1] << 16),
                            (u32)(dl[2] & 0xffff) | ((u32)dh[2] << 16), (u32)(dl[3] & 0xffff) | ((u32)dh[3] << 16));
        reach += (dh[1] - dl[1]) >> 1;
      }
      nfree += __popc(b);
    }
    if (kept != 1u && warp_sum32(reach) > 4000) return 0;   // (levels 2 and 3 move no further)
    __syncwarp();
    const int per_row = T0.limit / max(nfree, 1);        // blocks of 32 states
    int got = -1;
#pragma unroll 1
    for (int where = 0; where < 2 && got < 0 && per_row > 0; ++where) { // the work area, then the slab
      const u64 half = where == 0 ? 0 : (room / 2) & ~(u64)15;
      BdTable B;
      if (!bd_table(B, where == 0 ? T.wk : slab.base + slab.used, where == 0 ? (u64)T.wk_bytes : half)) break;
      B.cap = min(B.cap, 32 * min(per_row, 128));
      got = bounded_dp(T, frow, crow, lim, nfree, price, li, kept, slack, delta, B, (u8*)slab.base + slab.used + half, room - half, lane);
    }
    if (got > 0) return 1;
    if (got < 0) {
      if (T0.limit == INT_MAX) return 0;
      if (dp_classes(T0, slab, lane)) return 1;
      if (lane == 0) ((PoolTask&)T0).limit = INT_MAX;    // (splits tie: this pass once more, without a limit)
      --pass;
      continue;
    }
    delta = max(nfree <= 16 ? 8 * delta : 2 * delta, (i64)16);
    if (feasible) delta = min(delta, s0);
  }
  return 0;
}

// The box DP on the REACHABLE cells only, for boxes whose dense table would not fit: Algorithm 4's
// state space is the product of the four chunk-count ranges, but a row only moves a state by one of
// a handful of demand vectors, so few cells are ever reached.  A state is the extra-demand vector
// packed into one key (one bit field per kept dimension); the states of a row are built from those
// of the row before through a hash table (open addressing; a cell keeps the least
// duration sum << 6 | multiplicity, i.e. the lowest value and among equals the smallest level,
// which is what the dense loop's ascending levels with strict '<' keep), compacted into the next
// list, and their (key, multiplicity) pairs are kept per row for the walk back.  Same end-cell rule
// as the dense loop: lowest value, then fewest extra units, then the allocations compared from the
// last row down.  Everything lives in [mem, mem + bytes).  Returns 1 (T.rsel written), 0 if the
// memory does not suffice or a value outgrows its field.
#define SP_EMPTY 0xffffffffffffffffull
__device__ __forceinline__ u64 sp_hash(u64 k) { k ^= k >> 29; k *= 0xbf58476d1ce4e5b9ull; k ^= k >> 32; return k; }
__device__ __forceinline__ int dp_sparse(const PoolTask& T, int nrows, const int ext[4], u32 kept,
                                      char* mem, u64 bytes, int lane) {
  // bit fields of a key
  int shift[4], width[4], total_bits = 0;
#pragma unroll
  for (int l = 0; l < 4; ++l) {
    width[l] = ((kept >> l) & 1u) ? 32 - __clz(max(ext[l] - 1, 1)) : 0;
    shift[l] = total_bits; total_bits += width[l];
  }
  if (total_bits > 60) return 0;
  // memory: two state lists and the hash table at the end, the rows' (key, multiplicity) pairs from the front
  const u64 cap_states = bytes / 2 / (2 * 16 + 4 * 16);          // each list 16 B per state, table 4 slots of 16 B per state
  if (cap_states < 64) return 0;
  u64* lk[2]; i64* lv[2];
  char* top = mem + bytes;
  u64 tab_slots = 1; while (tab_slots < 4 * cap_states) tab_slots <<= 1; tab_slots >>= 1;   // largest power of two <= 4 cap
  top -= tab_slots * 16; u64* tk = (u64*)top; u64* tv = tk + tab_slots;
#pragma unroll 1
  for (int x = 0; x < 2; ++x) { top -= cap_states * 16; lk[x] = (u64*)top; lv[x] = (i64*)(lk[x] + cap_states); }
  char* store = mem;                                             // grows towards `top`
  // per row: where its pairs start and how many (kept in the store itself, in front of the pairs)
  u64* row_dir = (u64*)store; store += (u64)nrows * 16;
  if (store > top) return 0;
  u64 n = 1;
  if (lane == 0) { lk[0][0] = 0; lv[0][0] = 0; }
  __syncwarp();
  int cur = 0;
#pragma unroll 1
  for (int t = 0; t < nrows; ++t) {
    const int i = T.rowcand[t];
    const int g = T.cg[i] & 0x7f, gang = T.cg[i] >> 7;
    const u32 mk = T.cmask[i];
    const int r0 = __ffs(mk), nlev = __popc(mk);
    const i64 s = T.cs[i], p = T.cp[i];
    // table of this row: a power of two of at least four slots per candidate state
    u64 want = n * (u64)nlev * 2, slots = 64;
#pragma unroll 1
    while (slots < want && slots < tab_slots) slots <<= 1;
#pragma unroll 1
    for (u64 x = lane; x < slots; x += 32) { tk[x] = SP_EMPTY; tv[x] = ~0ull; }
    __syncwarp();
    u64 distinct = 0;
    bool fail = false;
#pragma unroll 1
    for (u64 x0 = 0; x0 < n; x0 += 32) {
      const u64 x = x0 + lane;
      const bool on = x < n;
      const u64 key = on ? lk[cur][x] : 0;
      const i64 val = on ? lv[cur][x] : 0;
      u32 mm = mk;
#pragma unroll 1
      while (mm) {
        const int r = __ffs(mm); mm &= mm - 1;
        int d[4];
        extra_demand(T.type, g, gang, r0, r, d);
        u64 nk = key; bool inside = on;
#pragma unroll
        for (int l = 0; l < 4; ++l)
          if ((kept >> l) & 1u) {
            const int dl = d[l] >> l;
            const int e = (int)((key >> shift[l]) & ((1ull << width[l]) - 1ull));
            inside &= e + dl < ext[l];
            nk += (u64)dl << shift[l];
          }
        const i64 cand = val + duration(s, p, r);
        if (inside && cand >= (1ll << 56)) { fail = true; inside = false; }
        if (inside) {
          const u64 packed = ((u64)cand << 6) | (u64)r;
          u64 h = sp_hash(nk) & (slots - 1);
#pragma unroll 1
          for (u64 probe = 0; probe < slots; ++probe) {
            const u64 seen = atomicCAS((unsigned long long*)&tk[h], SP_EMPTY, nk);
            if (seen == SP_EMPTY || seen == nk) { atomicMin((unsigned long long*)&tv[h], packed); if (seen == SP_EMPTY) ++distinct; break; }
            h = (h + 1) & (slots - 1);
            if (probe + 1 == slots) fail = true;
          }
        }
      }
    }
    __syncwarp();
    distinct = (u64)warp_sum64((i64)distinct);
    if (__any_sync(TG_FULL, fail) || distinct > cap_states || distinct > slots / 2 + 32) return 0;
    // compact the table into the next list and into the row's store
    if (store + distinct * 16 > top) return 0;
    u64* sk = (u64*)store; u64* sr = sk + distinct;
    if (lane == 0) { row_dir[2 * t] = (u64)(store - mem); row_dir[2 * t + 1] = distinct; }
    store += distinct * 16;
    u64 filled = 0;
#pragma unroll 1
    for (u64 x0 = 0; x0 < slots; x0 += 32) {
      const u64 x = x0 + lane;
      const u64 k = tk[x];
      const bool has = k != SP_EMPTY;
      const u32 b = __ballot_sync(TG_FULL, has);
      if (has) {
        const u64 at = filled + __popc(b & ((1u << lane) - 1u));
        const u64 pv = tv[x];
        lk[cur ^ 1][at] = k; lv[cur ^ 1][at] = (i64)(pv >> 6);
        sk[at] = k; sr[at] = pv & 63ull;
      }
      filled += __popc(b);
    }
    __syncwarp();
    n = distinct; cur ^= 1;
  }
  // best end state: lowest value, then fewest extra units (dimension 0)
  const u64 m0 = (1ull << width[0]) - 1ull;
  i64 bv = TG_INF;
#pragma unroll 1
  for (u64 x = lane; x < n; x += 32) bv = min(bv, lv[cur][x]);
  bv = warp_min64(bv);
  if (bv == TG_INF) return 0;
  int be = INT_MAX;
#pragma unroll 1
  for (u64 x = lane; x < n; x += 32) if (lv[cur][x] == bv) be = min(be, (int)((lk[cur][x] >> shift[0]) & m0));
  be = warp_min32(be);
  // the tied end states walk back together; at each row (last first) those with the smallest multiplicity stay
  const int TIE_CAP = 32;
  u64 tied = SP_EMPTY;                                     // lane x holds the x-th tied key
  int nt = 0;
#pragma unroll 1
  for (u64 x0 = 0; x0 < n; x0 += 32) {
    const u64 x = x0 + lane;
    const bool hit = x < n && lv[cur][x] == bv && (int)((lk[cur][x] >> shift[0]) & m0) == be;
    const u32 b = __ballot_sync(TG_FULL, hit);
    if (nt + __popc(b) > TIE_CAP) return 0;
    // hand the hits to lanes nt, nt+1, ...
#pragma unroll 1
    for (u32 bb = b; bb; bb &= bb - 1) {
      const int src = __ffs(bb) - 1;
      const u64 k = __shfl_sync(TG_FULL, hit ? lk[cur][x] : 0ull, src);
      if (lane == nt) tied = k;
      ++nt;
    }
  }
#pragma unroll 1
  for (int t = nrows - 1; t >= 0; --t) {
    const int i = T.rowcand[t];
    const u64* sk = (const u64*)(mem + row_dir[2 * t]);
    const u64 cnt = row_dir[2 * t + 1];
    const u64* sr = sk + cnt;
    // every tied key looks up its multiplicity in this row (all lanes scan for one key at a time)
    int myr = 255;
#pragma unroll 1
    for (int y = 0; y < nt; ++y) {
      const u64 k = __shfl_sync(TG_FULL, tied, y);
      int found = 255;
#pragma unroll 1
      for (u64 x = lane; x < cnt; x += 32) if (sk[x] == k) found = (int)sr[x];
      found = warp_min32(found);
      if (lane == y) myr = found;
    }
    const int rm = warp_min32(lane < nt ? myr : 255);
    if (rm == 255) return 0;                               // cannot happen: every kept key was written by this row
    if (lane == 0) T.rsel[i] = (u8)rm;
    int d[4];
    extra_demand(T.type, T.cg[i] & 0x7f, T.cg[i] >> 7, __ffs(T.cmask[i]), rm, d);
    u64 delta = 0;
#pragma unroll
    for (int l = 0; l < 4; ++l) if ((kept >> l) & 1u) delta += (u64)(d[l] >> l) << shift[l];
    // keep the keys whose multiplicity is the smallest, move them to the row before, drop duplicates
    const bool stay = lane < nt && myr == rm;
    const u64 prevk = tied - delta;
    const u32 sb = __ballot_sync(TG_FULL, stay);
    u64 next = SP_EMPTY;
    int nn = 0;
#pragma unroll 1
    for (u32 bb = sb; bb; bb &= bb - 1) {
      const int src = __ffs(bb) - 1;
      const u64 k = __shfl_sync(TG_FULL, prevk, src);
      const bool dup = __any_sync(TG_FULL, lane < nn && next == k);
      if (!dup) { if (lane == nn) next = k; ++nn; }
    }
    tied = next; nt = nn;
  }
  __syncwarp();
  return 1;
}

// The whole box of feasible extra-demand vectors (T.rowcand; T.maxex[l] = largest extra demand at level l), where the states
// within a bound do not fit their table, or very many end states tie.  -> T.rsel, T.opt
__device__ __noinline__ bool solve_box(const Params& P, PoolTask& T, int q, Slab slab, int lane) {
  const int nrows = T.nrows;
  int maxex[4] = {0, 0, 0, 0};
  u32 kept = 1u;
#pragma unroll
  for (int l = 0; l < 4; ++l) {
    if (l > 0 && T.type != TG_POOL_GPU) continue;
    maxex[l] = min(T.cap[l] - T.dmin[l], T.maxex[l]);
    if (l > 0 && T.cap[l] < T.cap[l - 1]) kept |= 1u << l;
  }
#pragma unroll 1
  for (int t = lane; t < nrows; t += 32) { const int i = T.rowcand[t]; T.rsel[i] = (u8)__ffs(T.cmask[i]); }
  __syncwarp();
  int ext[4], stride[4];
  u64 cells = 1;
#pragma unroll
  for (int l = 0; l < 4; ++l) {
    ext[l] = ((kept >> l) & 1u) ? (max(maxex[l], 0) >> l) + 1 : 1;
    stride[l] = (int)cells;
    if (cells <= (1ull << 30)) cells *= (u64)ext[l];
  }
  if (cells > (1ull << 30)) cells = (1ull << 30) + 1;       // (never dense: the reachable cells only, below)
  const int ncell = (int)cells;
  i64* val = (i64*)slab.take(2 * cells * sizeof(i64));
  u8* choice = val ? (u8*)slab.take((u64)nrows * cells) : nullptr;
  if (!choice) {
    // the dense table does not fit the warp's slab: only the reachable cells, in a borrowed slot of the arena
    const int sl = slot_acquire(P, 1, lane);
    if (sl < 0) return false;
    const int done = dp_sparse(T, nrows, ext, kept, slot_ptr(P, sl), arena_slot_bytes(P), lane);
    slot_release(P, sl, lane);
    if (!done) return false;
    i64 sum = 0;
#pragma unroll 1
    for (int i = lane; i < q; i += 32) sum += duration(T.cs[i], T.cp[i], T.rsel[i]);
    sum = warp_sum64(sum);
    if (lane == 0) T.opt = sum;
    __syncwarp();
    return true;
  }
  i64* prev = val; i64* cur = val + cells;
#pragma unroll 1
  for (int c = lane; c < ncell; c += 32) prev[c] = c == 0 ? 0 : TG_INF;
  __syncwarp();
#pragma unroll 1
  for (int t = 0; t < nrows; ++t) {
    const int i = T.rowcand[t];
    const int g = T.cg[i] & 0x7f, gang = T.cg[i] >> 7;
    const u32 mk = T.cmask[i];
    const int r0 = __ffs(mk);
    const i64 s = T.cs[i], p = T.cp[i];
    u8* ch = choice + (u64)t * cells;
#pragma unroll 1
    for (int c = lane; c < ncell; c += 32) {
      int e[4];
#pragma unroll
      for (int l = 0; l < 4; ++l) e[l] = (c / stride[l]) % ext[l];
      i64 best = TG_INF; int bestr = 0;
      u32 mm = mk;
#pragma unroll 1
      while (mm) {
        int r = __ffs(mm); mm &= mm - 1;
        int d[4];
        extra_demand(T.type, g, gang, r0, r, d);
        int off = 0; bool ok = true;
#pragma unroll
        for (int l = 0; l < 4; ++l)
          if ((kept >> l) & 1u) { int dl = d[l] >> l; ok &= dl <= e[l]; off += dl * stride[l]; }
        if (!ok) continue;
        i64 pv = prev[c - off];
        if (pv == TG_INF) continue;
        i64 cand = pv + duration(s, p, r);
        if (cand < best) { best = cand; bestr = r; }
      }
      cur[c] = best; ch[c] = (u8)bestr;
    }
    __syncwarp();
    i64* tmp = prev; prev = cur; cur = tmp;
  }
  // best cell of the last row: lowest value, then fewest extra units (e_1 = index along dim 0)
  i64 bv = TG_INF;
#pragma unroll 1
  for (int c = lane; c < ncell; c += 32) bv = min(bv, prev[c]);
  bv = warp_min64(bv);
  if (bv == TG_INF) { return false; }   // cannot happen for an accommodated prefix
  int be = INT_MAX;
#pragma unroll 1
  for (int c = lane; c < ncell; c += 32) if (prev[c] == bv) be = min(be, c % ext[0]);
  be = warp_min32(be);
  int cnt = 0, bc = -1;
#pragma unroll 1
  for (int c = lane; c < ncell; c += 32) if (prev[c] == bv && c % ext[0] == be) { ++cnt; bc = max(bc, c); }
  cnt = warp_sum32(cnt); bc = warp_max32(bc);
  int fail = 0;
  if (lane == 0) {
    if (cnt == 1) {
      int c = bc;
#pragma unroll 1
      for (int t = nrows - 1; t >= 0; --t) {
        int i = T.rowcand[t];
        int r = choice[(u64)t * cells + c];
        T.rsel[i] = (u8)r;
        int d[4];
        extra_demand(T.type, T.cg[i] & 0x7f, T.cg[i] >> 7, __ffs(T.cmask[i]), r, d);
#pragma unroll
        for (int l = 0; l < 4; ++l) if ((kept >> l) & 1u) c -= (d[l] >> l) * stride[l];
      }
    } else {
      // several end cells tie on value and units: walk back all of them at once, keeping at
      // each task (latest first) the cells whose choice is the smallest
      const int TIE_CAP = 64;
      int lst[TIE_CAP], nl = 0;
#pragma unroll 1
      for (int c = 0; c < ncell; ++c)
        if (prev[c] == bv && c % ext[0] == be) { if (nl < TIE_CAP) lst[nl++] = c; else fail = 1; }
#pragma unroll 1
      for (int t = nrows - 1; t >= 0; --t) {
        int i = T.rowcand[t];
        const u8* ch = choice + (u64)t * cells;
        int rm = 255;
#pragma unroll 1
        for (int x = 0; x < nl; ++x) rm = min(rm, (int)ch[lst[x]]);
        T.rsel[i] = (u8)rm;
        int d[4];
        extra_demand(T.type, T.cg[i] & 0x7f, T.cg[i] >> 7, __ffs(T.cmask[i]), rm, d);
        int off = 0;
#pragma unroll
        for (int l = 0; l < 4; ++l) if ((kept >> l) & 1u) off += (d[l] >> l) * stride[l];
        int nn = 0;
#pragma unroll 1
        for (int x = 0; x < nl; ++x) {
          if (ch[lst[x]] != rm) continue;
          int c = lst[x] - off;
          bool dup = false;
#pragma unroll 1
          for (int y = 0; y < nn; ++y) dup |= lst[y] == c;
          if (!dup) lst[nn++] = c;
        }
        nl = nn;
      }
    }
  }
  fail = __shfl_sync(TG_FULL, fail, 0);
  if (fail) return false;
  __syncwarp();
  i64 sum = 0;
#pragma unroll 1
  for (int i = lane; i < q; i += 32) sum += duration(T.cs[i], T.cp[i], T.rsel[i]);
  sum = warp_sum64(sum);
  if (lane == 0) T.opt = sum;
  __syncwarp();
  return true;
}

// ---- one capacity and little to give: a table of 32 cells ------------------------------------
// Where a pool has one capacity (core and quota pools, GPU pools without binding nested ones) and at most 31 units
// beyond everybody's least level, the recurrence of Algorithm 3 runs over at most 32 cells ("extra units"): lane c owns
// cell c, a predecessor is one shuffle away.  The rows (elastic candidates) do not depend on how long the prefix is,
// and a shorter prefix only reads an earlier row inside a larger box, so ONE pass serves every prefix of an eviction
// chain: the values of every row are kept (256 B each), and the choices for the walk back (64 B).
// About 100 cycles per row: bound by the chain of shuffle, add and compare from row to row.
#define CELL_LEVELS 6
#define CELL_FAR (1ll << 61)        // an unreachable cell
#define CELL_SHARED_ROWS 68         // rows whose choices fit the work area (7424 bytes)
__device__ __forceinline__ bool small_table(const PoolTask& T, int nrows, i64* val, unsigned short* ch, int lane) {
  i64 prev = lane == 0 ? 0 : CELL_FAR;
#pragma unroll 1
  for (int t0 = 0; t0 < nrows; t0 += 32) {
    // every lane lists the levels of its own row: multiplicity | extra units << 8, change of the duration
    int nl = 0;
    uint4* mine = (uint4*)T.wk + lane * CELL_LEVELS;
    __syncwarp();
    if (t0 + lane < nrows) {
      const int i = T.rowcand[t0 + lane];
      const i64 p = T.cp[i];
      const int g = T.cg[i] & 0x7f, r0 = __ffs(T.cmask[i]);
      const i64 q0 = div_small(p, r0);
#pragma unroll 1
      for (u32 mm = T.cmask[i]; mm; mm &= mm - 1) {
        const int r = __ffs(mm), off = g * (r - r0);
        if (off > 31) break;                             // (levels ascend)
        if (nl < CELL_LEVELS) {
          const u64 d = (u64)(div_small(p, r) - q0);
          mine[nl] = make_uint4((u32)r | ((u32)off << 8), (u32)d, (u32)(d >> 32), 0u);
        }
        ++nl;
      }
#pragma unroll 1
      for (int k = nl; k < CELL_LEVELS; ++k) mine[k] = make_uint4(0u, 0u, 0u, 0u);
    }
    if (__any_sync(TG_FULL, nl > CELL_LEVELS)) return false;
    const int widest = warp_max32(nl), nb = min(32, nrows - t0);
    __syncwarp();
    const uint4* row = (const uint4*)T.wk;
#pragma unroll 1
    for (int b = 0; b < nb; ++b, row += CELL_LEVELS) {
      // (levels ascend, so the first of equal values is the smallest multiplicity; the first level always applies)
      i64 best = prev; u32 bestv = row[0].x;
#pragma unroll
      for (int k = 1; k < CELL_LEVELS; ++k) {
        if (k >= 4 && k >= widest) break;
        const uint4 v = row[k];
        const int off = (int)(v.x >> 8);
        const i64 c = __shfl_up_sync(TG_FULL, prev, off) + (i64)(((u64)v.z << 32) | v.y);
        if (v.x != 0u && lane >= off && c < best) { best = c; bestv = v.x; }
      }
      prev = best;
      val[(t0 + b) * 32 + lane] = best;
      ch[(t0 + b) * 32 + lane] = (unsigned short)bestv;
    }
  }
  __syncwarp();
  return true;
}
// the best allocation of the first nrows rows with at most y <= 31 extra units -> T.rsel; returns the change of the
// duration sum against the least levels
__device__ __forceinline__ i64 small_answer(const PoolTask& T, int nrows, int y, const i64* val, const unsigned short* ch, int lane) {
  const i64 v = lane <= y ? val[(nrows - 1) * 32 + lane] : TG_INF;
  const i64 bv = warp_min64(v);
  int c = __ffs(__ballot_sync(TG_FULL, v == bv)) - 1;    // lowest value, then fewest units
#pragma unroll 1
  for (int t0 = (nrows - 1) & ~7; t0 >= 0; t0 -= 8) {    // eight rows' choices at a time, then the walk through them
    u32 x[8];
#pragma unroll
    for (int k = 0; k < 8; ++k) x[k] = t0 + k < nrows ? ch[(t0 + k) * 32 + lane] : 0u;
#pragma unroll
    for (int k = 7; k >= 0; --k) {
      if (t0 + k >= nrows) continue;
      const u32 w = __shfl_sync(TG_FULL, x[k], c);
      if (lane == k) T.rsel[T.rowcand[t0 + k]] = (u8)(w & 0xffu);
      c -= (int)(w >> 8);
    }
  }
  __syncwarp();
  return bv;
}

// Two or three candidates: all combinations of their levels, one per lane (a replay's rounds seldom have more).
#define FEW_MAX 3
__device__ __forceinline__ bool solve_few(PoolTask& T0, int q, int lane) {
  const int type = T0.type;
  u32 mk[FEW_MAX]; i64 s[FEW_MAX], p[FEW_MAX]; int cg[FEW_MAX], nl[FEW_MAX], total = 1;
#pragma unroll
  for (int i = 0; i < FEW_MAX; ++i) {
    mk[i] = i < q ? T0.cmask[i] : 1u; s[i] = i < q ? T0.cs[i] : 0; p[i] = i < q ? T0.cp[i] : 0; cg[i] = i < q ? (int)T0.cg[i] : 0;
    nl[i] = __popc(mk[i]); total *= nl[i];
  }
  if (total > 256) return false;
  i64 bv = TG_INF; int bu = INT_MAX; u32 bs = 0;
#pragma unroll 1
  for (int c = lane; c < total; c += 32) {
    int rest = c, dem[4] = {0, 0, 0, 0};
    i64 v = 0; u32 seq = 0;
#pragma unroll
    for (int i = 0; i < FEW_MAX; ++i) {
      const int d = rest % nl[i];
      rest /= nl[i];
      u32 mm = mk[i];
#pragma unroll 1
      for (int k = 0; k < d; ++k) mm &= mm - 1;
      const int r = __ffs(mm), g = cg[i] & 0x7f, cl = class_of(type, max(g, 1), cg[i] >> 7, r);
#pragma unroll
      for (int l = 0; l < 4; ++l) if (l <= cl) dem[l] += g * r;
      v += duration(s[i], p[i], r);
      seq |= (u32)r << (6 * i);                          // (a later candidate counts more)
    }
    bool fit = dem[0] <= T0.cap[0];
    if (type == TG_POOL_GPU) {
#pragma unroll
      for (int l = 1; l < 4; ++l) fit &= dem[l] <= T0.cap[l];
    }
    if (fit && (v < bv || (v == bv && (dem[0] < bu || (dem[0] == bu && seq < bs))))) { bv = v; bu = dem[0]; bs = seq; }
  }
  const i64 v = warp_min64(bv);
  const int u = warp_min32(bv == v ? bu : INT_MAX);
  const u32 w = __reduce_min_sync(TG_FULL, bv == v && bu == u ? bs : 0xffffffffu);
  if (lane < q) T0.rsel[lane] = (u8)((w >> (6 * lane)) & 63u);
  if (lane == 0) T0.opt = v;
  __syncwarp();
  return v != TG_INF;
}

// Optimal allocation of candidates [0, q) -> T.rsel[0..q), duration sum -> T.opt.  Prefixes are asked for in descending
// order.
#define SOLVED_ALL_BEST 2   // every candidate got its best level (then so does every shorter prefix)
#define SOLVED 1
#define UNSOLVED 0          // the workspace is too small
__device__ __forceinline__ int solve_prefix(const Params& P, PoolTask& T0, int q, Slab slab, int lane) {
  if (q <= FEW_MAX && solve_few(T0, q, lane)) return SOLVED;
  PoolTask T;                                            // (what is used of it, in registers)
  T.type = T0.type; T.cs = T0.cs; T.cp = T0.cp; T.cmask = T0.cmask; T.cg = T0.cg; T.rsel = T0.rsel; T.rowcand = T0.rowcand;
  T.wk = T0.wk; T.wk_bytes = T0.wk_bytes;
  const bool gpu = T.type == TG_POOL_GPU;
  // ---- sums over the candidates: from scratch, or from the prefix before by taking the last candidate out
  int dmin[4] = {0, 0, 0, 0}, dbest[4] = {0, 0, 0, 0}, maxex[4] = {0, 0, 0, 0};
  i64 tmin_sum = 0, tbest_sum = 0;
  int nrows = 0, n_levels = 0;
  const bool shorter = T0.sq == q + 1;
#pragma unroll 1
  for (int i0 = shorter ? q : 0; i0 < (shorter ? q + 1 : q); i0 += 32) {
    const int i = i0 + lane;
    bool el = false;
    if (shorter ? lane == 0 : i < q) {
      const int g = T.cg[i] & 0x7f, gang = T.cg[i] >> 7;
      const u32 mk = T.cmask[i];
      const i64 s = T.cs[i], p = T.cp[i];
      const int r0 = __ffs(mk), rx = 32 - __clz(mk);
      el = rx != r0;
      const int rb = el ? best_level(p, mk) : r0;
      const int c0 = class_of(T.type, g, gang, r0), cb = class_of(T.type, g, gang, rb);
#pragma unroll
      for (int l = 0; l < 4; ++l) {
        if (l <= c0) dmin[l] += g * r0;
        if (l <= cb) dbest[l] += g * rb;
      }
      tmin_sum += duration(s, p, r0);
      tbest_sum += duration(s, p, rb);
      if (!shorter) T.rsel[i] = (u8)rb;
      if (el) {
        n_levels += __popc(mk);
        const int cx = class_of(T.type, g, gang, rx);
#pragma unroll
        for (int l = 0; l < 4; ++l) if (l <= cx) maxex[l] += g * rx - (l <= c0 ? g * r0 : 0);
      }
    }
    const u32 b = __ballot_sync(TG_FULL, el);
    if (el && !shorter) T.rowcand[nrows + __popc(b & ((1u << lane) - 1u))] = i;
    nrows += __popc(b);
  }
  if (shorter) {
    // (lane 0 has the candidate's share; the sums are kept by lane 0 too)
    if (lane == 0) {
#pragma unroll
      for (int l = 0; l < 4; ++l) { T0.dmin[l] -= dmin[l]; T0.dbest[l] -= dbest[l]; T0.maxex[l] -= maxex[l]; }
      T0.nrows -= nrows; T0.n_levels -= n_levels; T0.tmin_sum -= tmin_sum; T0.tbest_sum -= tbest_sum;
      T0.sq = q;
    }
  } else {
#pragma unroll
    for (int l = 0; l < 4; ++l) {
      dmin[l] = warp_sum32(dmin[l]); dbest[l] = warp_sum32(dbest[l]); maxex[l] = warp_sum32(maxex[l]);
      if (lane == 0) { T0.dmin[l] = dmin[l]; T0.dbest[l] = dbest[l]; T0.maxex[l] = maxex[l]; }
    }
    n_levels = warp_sum32(n_levels); tmin_sum = warp_sum64(tmin_sum); tbest_sum = warp_sum64(tbest_sum);
    if (lane == 0) { T0.nrows = nrows; T0.n_levels = n_levels; T0.tmin_sum = tmin_sum; T0.tbest_sum = tbest_sum; T0.sq = q; }
  }
  __syncwarp();
  nrows = uniform(T0.nrows);
  bool fits_best = true;
  int Y[4];
  u32 kept = 1u;
#pragma unroll
  for (int l = 0; l < 4; ++l) {
    T.cap[l] = T0.cap[l];
    Y[l] = 0;
    if (l > 0 && !gpu) continue;
    Y[l] = T.cap[l] - T0.dmin[l];
    fits_best &= T0.dbest[l] <= T.cap[l];
    if (l > 0 && T.cap[l] < T.cap[l - 1]) kept |= 1u << l;
  }
  if (fits_best) {
#pragma unroll 1
    for (int i = lane; i < q && shorter; i += 32) T.rsel[i] = (u8)best_level(T.cp[i], T.cmask[i]);
    if (lane == 0) T0.opt = T0.tbest_sum;
    __syncwarp();
    return SOLVED_ALL_BEST;
  }
  if (Y[0] <= 0) {
#pragma unroll 1
    for (int i = lane; i < q; i += 32) T.rsel[i] = (u8)__ffs(T.cmask[i]);
    if (lane == 0) T0.opt = T0.tmin_sum;
    __syncwarp();
    return SOLVED;
  }
  if (kept == 1u && Y[0] <= 31 && T0.cell_rows >= 0) {
    i64* val = T0.cell_val; unsigned short* ch = T0.cell_ch;
    int built = uniform(T0.cell_rows);
    if (built < nrows) {
      // the choices behind the staged levels in the work area, which the simulations of up to 256 times leave alone: read
      // back from the slab, every eight rows of the walk wait for the L2 (15000 cycles for 43 rows; cost vectors 2048 x 4096
      // 403 us a call against 388, 16384 x 4096 1692 against 1685)
      if (nrows <= CELL_SHARED_ROWS && T0.n_seeds + T0.m <= 256) ch = (unsigned short*)(T.wk + 32 * CELL_LEVELS * 16);
      built = small_table(T, nrows, val, ch, lane) ? nrows : -1;
      if (lane == 0) { T0.cell_rows = built; T0.cell_ch = ch; }
    }
    if (built > 0) {
      const i64 change = small_answer(T, nrows, Y[0], val, ch, lane);
      if (lane == 0) T0.opt = T0.tmin_sum + change;
      __syncwarp();
      return SOLVED;
    }
  }
#pragma unroll
  for (int l = 0; l < 4; ++l) maxex[l] = min(Y[l], T0.maxex[l]);
  u64 cells = 1;                                         // of the box of feasible extra-demand vectors
#pragma unroll
  for (int l = 0; l < 4; ++l) if (cells <= (1ull << 30)) cells *= ((kept >> l) & 1u) ? (u64)(max(maxex[l], 0) >> l) + 1 : 1;
  // Gang requests couple the chunk sizes; the header asks that the table of such a pool's reachable states fits a slot
  // of the workspace.  With slots below TG_MIN_SLOT_BYTES (workspace_bytes under 2.3 MB) that rule decides alone: a box
  // whose table fits neither the slab nor the slot gets its status word whatever its durations.  All other pools need
  // nothing but the slab, on any workspace.
  const bool dense_fits = slab.used + 2 * cells * sizeof(i64) + (u64)nrows * cells + 64 <= slab.cap;
  bool by_table = false;
  if (!dense_fits && arena_slot_bytes(P) < TG_MIN_SLOT_BYTES) {
#pragma unroll 1
    for (int t = lane; t < nrows; t += 32) by_table |= (T.cg[T.rowcand[t]] >> 7) != 0;
    by_table = __any_sync(TG_FULL, by_table);
  }
  if (T0.upgrades >= 0) set_limit(T0, lane);
  if (!by_table && solve_priced(T0, T, nrows, uniform(T0.n_levels), Y, kept, slab, lane)) {
    i64 sum = 0;
#pragma unroll 1
    for (int i = lane; i < q; i += 32) sum += duration(T.cs[i], T.cp[i], T.rsel[i]);
    sum = warp_sum64(sum);
    if (lane == 0) T0.opt = sum;
    __syncwarp();
    return SOLVED;
  }
  return solve_box(P, T0, q, slab, lane) ? SOLVED : UNSOLVED;
}
