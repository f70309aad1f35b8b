// Per-pool selection of a round, second half: the greedy eviction loop (Algorithm 1, lines 8-14)
// and the completion-heap simulations it compares (Algorithm 2), one warp per (scenario, pool).
//
// An eviction step compares the objective of q+1 kept candidates with that of q: the optimal
// duration sum of the kept ones plus the sum of completions of everything that keeps waiting, put
// one after the other on the slot that frees earliest ("pop the earliest completion ts, push
// ts + T").  Only the SIGN of the difference matters, so the two simulations run side by side, in
// blocks of EV_BLOCK steps, and stop as soon as the sign cannot change any more: if every completion
// of the shorter prefix's heap is at or behind its counterpart in the longer one's (both sorted; the
// slot the shorter one lacks counts as never free), it stays so after every further step with the
// same T, so every later completion is at or behind as well and the difference only grows.  Once it
// is >= 0 and the heaps are ordered that way, the step does not pay and Algorithm 1 stops.  The
// durations cancel in the difference, only popped times are summed.
//
// One level of the first waiting action is enough although Algorithm 2 tries `depth` of them: by
// the same ordering the sum is non-decreasing in that action's duration, durations do not grow with
// the level, hence the best depth is always the largest level tried.
//
// A heap of up to 256 times sits in lane registers, unsorted (ev_compare_regs); a larger one is a window of up to
// 32 earliest times, sorted over the lanes, and an unsorted rest, all of it at or behind the window's last time
// (ev_compare).  With w the window and d the next durations, w + d are the completions of the next actions as
// long as none of them comes before a later window entry: up to the smallest of them, all pops are known at once.
// The new times go to the rest, or one by one into the window where they belong in it; an empty window is
// refilled with the rest's earliest.  Measured on B200, 66 waiting slots, both heaps, cycles per step: one pop
// after the other on sorted arrays about 600, windows 320, registers 113.
//
// Times are 32-bit microseconds that saturate (71 minutes); sums are exact as long as no saturated
// time is popped, and if one is, both objectives are computed on an exact 64-bit heap.
#pragma once
#include "common.cuh"
#include "arrange.cuh"

#define EV_BLOCK 64
#define EV_SAT 0xfffffffeu
#define EV_NONE 0xffffffffu

__device__ __forceinline__ u32 ev_key(i64 v) { return v >= (i64)EV_SAT ? EV_SAT : (u32)v; }

// d-th smallest set bit (d = 0 is the lowest) as a multiplicity
__device__ __forceinline__ int nth_level(u32 mask, int d) {
#pragma unroll 1
  for (int k = 0; k < d; ++k) mask &= mask - 1;
  return __ffs(mask);
}

// The unsorted rest of a heap (and the staged durations): shared memory, or the slab where it does not fit.
struct EvShared {
  u32 base;
  __device__ __forceinline__ u32 get(int i) const { u32 v; asm volatile("ld.shared.u32 %0, [%1];" : "=r"(v) : "r"(base + (u32)i * 4u) : "memory"); return v; }
  __device__ __forceinline__ void put(int i, u32 v) const { asm volatile("st.shared.u32 [%0], %1;" :: "r"(base + (u32)i * 4u), "r"(v) : "memory"); }
  __device__ __forceinline__ EvShared at(int i) const { return EvShared{base + (u32)i * 4u}; }
};
struct EvGlobal {
  u32* p;
  __device__ __forceinline__ u32 get(int i) const { return p[i]; }
  __device__ __forceinline__ void put(int i, u32 v) const { p[i] = v; }
  __device__ __forceinline__ EvGlobal at(int i) const { return EvGlobal{p + i}; }
};

struct EvHeap {
  u32 w;          // window: lane k < n holds the k-th earliest time, the others EV_NONE
  int n;          // times in the window
  u32 edge;       // every time of the rest is >= edge
  int n_rest;
  u32 width;      // width of the last refill (a first guess for the next)
  u64 pops;       // this lane's share of the popped times
  bool sat;       // a saturated time was popped
};

__device__ __forceinline__ u32 ev_sort(u32 v, int lane) {      // ascending over the lanes
#pragma unroll
  for (int k = 2; k <= 32; k <<= 1)
#pragma unroll
    for (int j = k >> 1; j > 0; j >>= 1) {
      const u32 o = __shfl_xor_sync(TG_FULL, v, j);
      const bool lower = ((lane & j) == 0) == ((lane & k) == 0);
      v = lower ? min(v, o) : max(v, o);
    }
  return v;
}

// Empty window: the earliest of the rest, at most 32 of them, sorted.  tmp: 32 words.
template <class Buf>
__device__ __forceinline__ void ev_refill(EvHeap& H, const Buf& rest, const Buf& tmp, int lane) {
  const int n = H.n_rest;
  if (n <= 32) {                                         // everything fits: nothing is left outside
    H.w = ev_sort(lane < n ? rest.get(lane) : EV_NONE, lane);
    H.n = n; H.n_rest = 0; H.edge = EV_NONE;
    return;
  }
  // A threshold with 12 to 32 times at or below it (fewer, at least one, if none is found soon); the last window's
  // width is the first guess.  Up to 128 times are looked at in registers.
  u32 v[4];
#pragma unroll
  for (int r = 0; r < 4; ++r) v[r] = 32 * r + lane < n ? rest.get(32 * r + lane) : EV_NONE;
  auto count = [&](u32 y) {
    int k = 0;
#pragma unroll
    for (int r = 0; r < 4; ++r) k += v[r] <= y ? 1 : 0;
#pragma unroll 1
    for (int i = 128 + lane; i < n; i += 32) k += rest.get(i) <= y ? 1 : 0;
    return __reduce_add_sync(TG_FULL, k);
  };
  u32 lo = H.edge, hi = EV_NONE, x = lo + min(H.width, EV_SAT - lo);
  int c = 0, c_lo = 0;                                   // times at or below x / lo (0: not known for the edge itself)
#pragma unroll 1
  for (int it = 0; it < 64; ++it) {
    c = count(x);
    if (c >= 12 && c <= 32) break;
    if (c > 32) hi = x; else { lo = x; c_lo = c; if (it >= 4 && c > 0) break; }
    if (hi == EV_NONE) { const u32 g = max(x - H.edge, 1u); x = H.edge + min(g >= 0x40000000u ? EV_SAT : g * 4u, EV_SAT - H.edge); }
    else {
      if (hi - lo <= 1u) {                               // those at hi, or at lo, are equal: any 32 of them will do
        if (c_lo == 0) c_lo = count(lo);
        x = c_lo > 0 ? lo : hi;
        break;
      }
      x = lo + ((hi - lo) >> 1);
    }
  }
  // (aim at about 24 times next)
  const u32 width = max(x - H.edge, 16u);
  H.width = c < 18 ? width + (width >> 1) : (c > 28 ? width - (width >> 3) : width);
  if (H.width < width && c < 18) H.width = EV_SAT;
  H.edge = x;
  int at = 0, left = 0;
#pragma unroll 1
  for (int i0 = 0; i0 < n; i0 += 32) {
    const int i = i0 + lane;
    const u32 y = i0 == 0 ? v[0] : (i0 == 32 ? v[1] : (i0 == 64 ? v[2] : (i0 == 96 ? v[3] : (i < n ? rest.get(i) : EV_NONE))));
    const u32 b = __ballot_sync(TG_FULL, i < n && y <= x), below = (1u << lane) - 1u;
    const bool take = ((b >> lane) & 1u) && at + __popc(b & below) < 32;
    const u32 tb = __ballot_sync(TG_FULL, take), kb = __ballot_sync(TG_FULL, i < n && !take);
    if (take) tmp.put(at + __popc(tb & below), y);
    else if (i < n) rest.put(left + __popc(kb & below), y);
    at += __popc(tb); left += __popc(kb);
  }
  __syncwarp();
  H.w = ev_sort(lane < at ? tmp.get(lane) : EV_NONE, lane);
  H.n = at; H.n_rest = left;
  __syncwarp();
}

// The next pops ("pop the earliest, push earliest + T"), at most `steps` of them and at least one, with the durations
// dur.get(0 ..).  Returns their number.
template <class Buf>
__device__ __forceinline__ int ev_round(EvHeap& H, const Buf& rest, const Buf& tmp, const EvShared& dur, int steps, int lane) {
  if (H.n == 0) ev_refill(H, rest, tmp, lane);
  const int len = min(H.n, steps);
  const bool on = lane < len;
  u32 c = EV_NONE;
  if (on) { const u32 d = dur.get(lane); c = H.w >= EV_SAT - d ? EV_SAT : H.w + d; }
  const u32 first = __reduce_min_sync(TG_FULL, c);       // the first completion: window entries up to it are the next pops
  const u32 pb = __ballot_sync(TG_FULL, on && H.w <= first);
  const int np = __popc(pb);
  const bool popped = lane < np;
  if (popped) { H.pops += H.w; H.sat |= H.w >= EV_SAT; }
  u32 nw = __shfl_down_sync(TG_FULL, H.w, np & 31);
  if (np == 32 || lane >= H.n - np) nw = EV_NONE;
  u32 ins = __ballot_sync(TG_FULL, popped && c < H.edge);
  const u32 out = pb & ~ins;
  if (popped && c >= H.edge) rest.put(H.n_rest + __popc(out & ((1u << lane) - 1u)), c);
  H.n_rest += __popc(out);
  H.n += __popc(ins) - np;
#pragma unroll 1
  for (; ins; ins &= ins - 1) {                          // into the window, one after the other
    const u32 v = __shfl_sync(TG_FULL, c, __ffs(ins) - 1);
    const int pos = __popc(__ballot_sync(TG_FULL, nw < v));
    const u32 up = __shfl_up_sync(TG_FULL, nw, 1);
    nw = lane < pos ? nw : (lane == pos ? v : up);
  }
  H.w = nw;
  __syncwarp();
  return np;
}

// Are B's times (n - 1 of them) at or behind A's (n) position by position, both sorted?  Counted: for every time of B,
// no more times of B than of A are at or before it.  A saturated time may stand for any later one, so A may
// hold at most one (its last, which has no counterpart).
template <class Buf>
__device__ __forceinline__ bool ev_behind(const EvHeap& A, const Buf& ra, const EvHeap& B, const Buf& rb, int lane) {
  // the windows behind the rests, so that both heaps are plain lists
  if (lane < A.n) ra.put(A.n_rest + lane, A.w);
  if (lane < B.n) rb.put(B.n_rest + lane, B.w);
  __syncwarp();
  const int na = A.n_rest + A.n, nb = B.n_rest + B.n;
  int sat = 0;
#pragma unroll 1
  for (int i = lane; i < na; i += 32) sat += ra.get(i) >= EV_SAT ? 1 : 0;
  bool ok = __reduce_add_sync(TG_FULL, sat) <= 1;
#pragma unroll 1
  for (int i0 = 0; i0 < nb && ok; i0 += 32) {
    const u32 v = i0 + lane < nb ? rb.get(i0 + lane) : EV_NONE;
    int ca = 0, cb = 0;
#pragma unroll 1
    for (int j = 0; j < na; ++j) ca += ra.get(j) <= v ? 1 : 0;
#pragma unroll 1
    for (int j = 0; j < nb; ++j) cb += rb.get(j) <= v ? 1 : 0;
    ok = __all_sync(TG_FULL, i0 + lane >= nb || v >= EV_SAT || cb <= ca);
  }
  __syncwarp();
  return ok;
}

// What keeps waiting when the first q candidates are kept: the evicted candidates in queue order, then the pool's
// waiting actions, all at their least level; the first of all takes the largest of its first `depth` levels.
__device__ __forceinline__ i64 rest_least(const PoolTask& T, int keep, int j) {      // j-th behind the first `keep` candidates
  const int i = keep + j;
  return i < T.m ? duration(T.cs[i], T.cp[i], __ffs(T.cmask[i])) : T.ac_tmin[i - T.m];
}
__device__ __forceinline__ i64 rest_first(const PoolTask& T, int q) {
  const i64 s = q < T.m ? T.cs[q] : T.ac_first.s, p = q < T.m ? T.cp[q] : T.ac_first.p;
  const u32 mk = q < T.m ? T.cmask[q] : T.ac_first.mask;
  return duration(s, p, nth_level(mk, min(T.depth, __popc(mk)) - 1));
}

// Completion-heap estimate (Algorithm 2) on an exact 64-bit heap, one lane; for what leaves 32-bit times.
__device__ __noinline__ bool estimate_exact(const Params& P, const PoolTask& T, int q, const u8* alloc, Slab slab, int lane, i64* est) {
  const int n_rest = T.m - q + T.n_ac, H = T.n_seeds + q;
  if (n_rest == 0) { *est = 0; return true; }
  i64* h = (i64*)slab.take((u64)H * sizeof(i64));
  if (!h) h = (i64*)arena_take(P, (u64)H * sizeof(i64), lane);
  if (!h) return false;
#pragma unroll 1
  for (int i = lane; i < H; i += 32)
    h[i] = i < T.n_seeds ? T.seeds[i] : duration(T.cs[i - T.n_seeds], T.cp[i - T.n_seeds], alloc[i - T.n_seeds]);
  __syncwarp();
  i64 tmp = 0;
  if (lane == 0) {
#pragma unroll 1
    for (int st = H / 2 - 1; st >= 0; --st) {             // heapify
      const i64 v = h[st]; int pos = st;
#pragma unroll 1
      for (;;) {
        int c = 2 * pos + 1;
        if (c >= H) break;
        if (c + 1 < H && h[c + 1] < h[c]) ++c;
        if (h[c] < v) { h[pos] = h[c]; pos = c; } else break;
      }
      h[pos] = v;
    }
#pragma unroll 1
    for (int e = 0; e < n_rest; ++e) {
      const i64 v = h[0] + (e == 0 ? rest_first(T, q) : rest_least(T, q, e));   // pop the earliest completion, push ts + T
      tmp = sat_add(tmp, v);
      int pos = 0;
#pragma unroll 1
      for (;;) {
        int c = 2 * pos + 1;
        if (c >= H) break;
        i64 hc = h[c];
        if (c + 1 < H) { const i64 h2 = h[c + 1]; if (h2 < hc) { hc = h2; ++c; } }
        if (hc < v) { h[pos] = hc; pos = c; } else break;
      }
      h[pos] = v;
    }
  }
  *est = __shfl_sync(TG_FULL, tmp, 0);
  __syncwarp();
  return true;
}

// An eviction step that cannot pay.  Let the first q+1 candidates be kept with multiplicities
// `kept`, and let `fewer` be the optimal multiplicities of the first q alone.  If the two agree on
// the first q candidates and candidate q's kept duration is no longer than at the largest level
// the estimate would try for it, then objective(q) >= objective(q+1):
//   * both objectives share the duration sum of the first q candidates;
//   * with q+1 kept, candidate q adds T_q(kept) and occupies one completion slot from T_q(kept) on;
//     with q kept, it is the first waiting action: it adds ts + T_q(level d) >= T_q(kept), where
//     ts >= 0 is the earliest completion, and that slot is busy until then;
//   * so the completion multiset after the step dominates the other one slot by slot (the slot
//     the smaller list lacks counts as never free), dominance survives every further
//     "pop the earliest, push earliest + T" step, every popped time is >=, and every later
//     waiting action runs at its least level in the first sum and at that or a larger level in
//     the second.
// Algorithm 1 stops at the first step whose objective does not decrease, so no simulation is needed.
// Warp-uniform result.
__device__ __forceinline__ bool eviction_cannot_pay(const PoolTask& T, int q, const u8* kept, const u8* fewer,
                                                    int lane) {
  bool same = true;
#pragma unroll 1
  for (int i = lane; i < q; i += 32) same &= kept[i] == fewer[i];
  if (!__all_sync(TG_FULL, same)) return false;
  return duration(T.cs[q], T.cp[q], kept[q]) <= rest_first(T, q);
}

// ---- heaps of up to 256 times: 32 NS of them in lane registers -----------------------------------
// Every lane keeps its own times in ascending order, the lanes among each other are in none.  One pop: a warp minimum over
// the lanes' first times, and the (highest) lane that holds it sorts the new time in among its own; the chain is warp
// minimum, vote, insertion.  (Not waiting for the vote and mending ties one step later was slower: the branch costs
// more than the vote.  Without an order every step looks for a lane's minimum and its place: 16384 x 4096 1936 us a call
// against 1780, 64 nodes of 8 GPUs, 1024 x 2048, 762 against 589; the insertion in a branch 866.)
template <int NS>
__device__ __forceinline__ void ev_order(u32 (&key)[NS]) {
#pragma unroll
  for (int i = 1; i < NS; ++i)
#pragma unroll
    for (int j = NS - 1; j >= i; --j) { const u32 x = key[j - 1], y = key[j]; key[j - 1] = min(x, y); key[j] = max(x, y); }
}
// above: the lanes above this one
template <int NS>
__device__ __forceinline__ void ev_replace(u32 (&key)[NS], u32 mn, u32 holders, u32 d, u32 above) {
  // (a lane whose time stays sorts that one in again: no branch; every place on its own: no chain through the registers)
  const u32 c = key[0] == mn && (holders & above) == 0u ? min(mn, EV_SAT - d) + d : key[0];      // d <= EV_SAT
#pragma unroll
  for (int j = 0; j < NS; ++j) {
    const u32 x = j == 0 ? c : max(c, key[j]);
    key[j] = j + 1 < NS ? min(x, key[j + 1]) : x;
  }
}

__device__ __forceinline__ void ev_load(u32 (&d)[2], u32 at) {
  asm volatile("ld.shared.v2.u32 {%0, %1}, [%2];" : "=r"(d[0]), "=r"(d[1]) : "r"(at) : "memory");
}
__device__ __forceinline__ void ev_load(u32 (&d)[4], u32 at) {
  asm volatile("ld.shared.v4.u32 {%0, %1, %2, %3}, [%4];" : "=r"(d[0]), "=r"(d[1]), "=r"(d[2]), "=r"(d[3]) : "r"(at) : "memory");
}

template <int NS>
__device__ __forceinline__ void ev_step(u32 (&a)[NS], u32 (&b)[NS], u32 da, u32 db, u32 above, u32& ma, u32& mb) {
  mb = __reduce_min_sync(TG_FULL, b[0]);
  ma = __reduce_min_sync(TG_FULL, a[0]);
  const u32 hb = __ballot_sync(TG_FULL, b[0] == mb), ha = __ballot_sync(TG_FULL, a[0] == ma);
  ev_replace(b, mb, hb, db, above);
  ev_replace(a, ma, ha, da, above);
}

// ev_behind for register heaps (a: n + 1 times, b: n); list: 64 NS words of shared memory
template <int NS>
__device__ __forceinline__ bool ev_behind_regs(const u32 (&a)[NS], const u32 (&b)[NS], int ha, u32 list, int lane) {
  int sat = 0;
  const u32 la = list, lb = list + NS * 128u;
#pragma unroll
  for (int j = 0; j < NS; ++j) {
    sat += a[j] == EV_SAT ? 1 : 0;
    asm volatile("st.shared.u32 [%0], %1;" :: "r"(la + (u32)(j * 32 + lane) * 4u), "r"(a[j]) : "memory");
    asm volatile("st.shared.u32 [%0], %1;" :: "r"(lb + (u32)(j * 32 + lane) * 4u), "r"(b[j]) : "memory");
  }
  if (__reduce_add_sync(TG_FULL, sat) > 1) return false;
  __syncwarp();
  int excess[NS];                                        // per time of b: times of a less times of b at or before it
#pragma unroll
  for (int j = 0; j < NS; ++j) excess[j] = 0;
#pragma unroll 1
  for (int k = 0; k < ha; k += 4) {                      // (unused entries are EV_NONE: behind everything)
    u32 x[4], y[4];
    asm volatile("ld.shared.v4.u32 {%0, %1, %2, %3}, [%4];" : "=r"(x[0]), "=r"(x[1]), "=r"(x[2]), "=r"(x[3]) : "r"(la + (u32)k * 4u) : "memory");
    asm volatile("ld.shared.v4.u32 {%0, %1, %2, %3}, [%4];" : "=r"(y[0]), "=r"(y[1]), "=r"(y[2]), "=r"(y[3]) : "r"(lb + (u32)k * 4u) : "memory");
#pragma unroll
    for (int z = 0; z < 4; ++z)
#pragma unroll
      for (int j = 0; j < NS; ++j) excess[j] += (x[z] <= b[j] ? 1 : 0) - (y[z] <= b[j] ? 1 : 0);
  }
  bool ok = true;
#pragma unroll
  for (int j = 0; j < NS; ++j) ok &= b[j] >= EV_SAT || excess[j] >= 0;
  __syncwarp();
  return __all_sync(TG_FULL, ok);
}

// The two heaps side by side (see ev_compare for the conventions).  a: heap of the longer prefix, in the first ha places; b:
// of the shorter one, before the evicted candidate of duration `evicted`.  dur_of(k): duration of the k-th of n that wait behind
// both, first_a: of the first one as `a` takes it; diff: the part of the difference that is no popped time.
// wk: 64 NS + 2 EV_BLOCK + 4 words of shared memory.
template <int NS, int U, class Dur>
__device__ __forceinline__ int ev_run_regs(u32 (&a)[NS], u32 (&b)[NS], int ha, int n, u32 evicted, u32 first_a, i64 diff, const Dur& dur_of, u32 wk,
                                           int lane) {
  const EvShared dur = {wk + NS * 256u};
  const u32 above = lane == 31 ? 0u : TG_FULL << (lane + 1);
  u32 last_a = 0, last_b;
  ev_order(a); ev_order(b);
  last_b = __reduce_min_sync(TG_FULL, b[0]);             // the evicted candidate
  ev_replace(b, last_b, __ballot_sync(TG_FULL, b[0] == last_b), evicted, above);
  diff += (i64)last_b;
  int wait = 0;                                          // blocks until the heaps are compared again
#pragma unroll 1
  for (int k0 = 0; k0 < n; k0 += EV_BLOCK) {
    const int steps = min(EV_BLOCK, n - k0);
#pragma unroll 1
    for (int x = lane; x < steps; x += 32) dur.put(x, dur_of(k0 + x));
    __syncwarp();
    // The two chains, step by step side by side (warp-wide operations keep their order, so it is written this way).
    // A's first action takes its own level.
    // The next durations are loaded while these are worked on.  U steps per turn of the loop: two in k_pool, where all warps are
    // busy and wait for instructions, so that the text of this loop counts (16384 x 4096, 66 slots: four steps 1585 us a call,
    // two 1510, one 1600), for 0.5 to 2 % where a few pools set the time (4096 x 1024: four 251, two 256; 64 nodes,
    // 1024 x 2048: 527 and 550); four in k_round and k_replay, where few warps wait for this chain.
    u32 d[U];
    ev_load(d, dur.base);
    u32 da = k0 == 0 ? first_a : d[0];
    int k = 0;
#pragma unroll 1
    for (; k + U <= steps; k += U) {
      u32 next[U];
      ev_load(next, dur.base + (u32)(k + U) * 4u);          // (behind the last ones lies room for a block more)
#pragma unroll
      for (int z = 0; z < U; ++z) {
        ev_step(a, b, z == 0 ? da : d[z], d[z], above, last_a, last_b);
        diff += (i64)last_b - (i64)last_a;
      }
      da = next[0];
#pragma unroll
      for (int z = 0; z < U; ++z) d[z] = next[z];
    }
#pragma unroll 1
    for (; k < steps; ++k) {
      const u32 e = dur.get(k);
      ev_step(a, b, k > 0 ? e : da, e, above, last_a, last_b);
      diff += (i64)last_b - (i64)last_a;
    }
    __syncwarp();
    if (last_a >= EV_SAT || last_b >= EV_SAT) return -1; // (pops do not decrease)
    if (k0 + EV_BLOCK >= n) break;
    if (diff >= 0) {
      if (wait == 0) { if (ev_behind_regs(a, b, ha, wk, lane)) return 0; wait = 1; }
      else --wait;
    }
  }
  if (last_b >= EV_SAT) return -1;
  return diff < 0 ? 1 : 0;
}
template <int NS, int U>
__device__ __forceinline__ int ev_compare_regs(const PoolTask& T, int q, const u8* kept, const u8* fewer, i64 fixed, u32 wk, int lane) {
  const int ha = T.n_seeds + q + 1, n = T.m - q - 1 + T.n_ac;
  u32 a[NS], b[NS];
#pragma unroll
  for (int j = 0; j < NS; ++j) {
    const int i = j * 32 + lane, c = i - T.n_seeds;
    a[j] = b[j] = EV_NONE;
    if (i >= ha) continue;
    if (c < 0) a[j] = b[j] = ev_key(T.seeds[i]);
    else {
      const i64 s = T.cs[c], p = T.cp[c];
      a[j] = ev_key(duration(s, p, kept[c]));
      if (c < q) b[j] = ev_key(duration(s, p, fewer[c]));
    }
  }
  return ev_run_regs<NS, U>(a, b, ha, n, ev_key(rest_first(T, q)), n > 0 ? ev_key(rest_first(T, q + 1)) : 0u, fixed,
                         [&](int k) { return ev_key(rest_least(T, q + 1, k)); }, wk, lane);
}

// The two heaps side by side.  fixed: the part of objective(q) - objective(q+1) that is no popped time.
// Returns 1 if the difference is negative (the step pays), 0 if not, -1 if a saturated time was popped.
template <class Buf>
__device__ __forceinline__ int ev_compare(const PoolTask& T, int q, const u8* kept, const u8* fewer, i64 fixed, const Buf& mem,
                                          const EvShared& dur, int lane) {
  const int ha = T.n_seeds + q + 1, hb = ha - 1, n = T.m - q - 1 + T.n_ac;
  const Buf ra = mem, rb = mem.at(ha), tmp = mem.at(2 * ha);
#pragma unroll 1
  for (int i = lane; i < ha; i += 32) {
    i64 a, b = 0;
    if (i < T.n_seeds) a = b = T.seeds[i];
    else {
      const int c = i - T.n_seeds;
      const i64 s = T.cs[c], p = T.cp[c];
      a = duration(s, p, kept[c]);
      if (c < q) b = duration(s, p, fewer[c]);
    }
    ra.put(i, ev_key(a));
    if (i < hb) rb.put(i, ev_key(b));
  }
  EvHeap A, B;
  A.w = B.w = EV_NONE; A.n = B.n = 0; A.edge = B.edge = 0; A.n_rest = ha; B.n_rest = hb;
  A.width = B.width = 1u << 16; A.pops = B.pops = 0; A.sat = B.sat = false;
  // Block by block, a round of either heap in turn (their chains are independent).  B is one step ahead: its first
  // is the evicted candidate.  dur: [0] that one, [1 ..] the block's durations as B takes them, dur_a[0] the first as A
  // takes it.
  i64 diff = fixed;
  int wait = 0;                                          // blocks until the heaps are compared again
#pragma unroll 1
  for (int k0 = 0; k0 < n || k0 == 0; k0 += EV_BLOCK) {
    const int steps = min(EV_BLOCK, n - k0);
#pragma unroll 1
    for (int x = lane; x < steps; x += 32) {
      const u32 d = ev_key(rest_least(T, q + 1, k0 + x));
      dur.put(1 + x, d);
      if (k0 == 0) dur.put(EV_BLOCK + 1 + x, x == 0 ? ev_key(rest_first(T, q + 1)) : d);
    }
    if (k0 == 0 && lane == 0) dur.put(0, ev_key(rest_first(T, q)));
    __syncwarp();
    int kb = k0 == 0 ? 0 : 1, ka = k0 == 0 ? EV_BLOCK + 1 : 1;
    const int eb = steps + 1, ea = ka + steps;
#pragma unroll 1
    while (kb < eb || ka < ea) {
      if (kb < eb) kb += ev_round(B, rb, tmp, dur.at(kb), eb - kb, lane);
      if (ka < ea) ka += ev_round(A, ra, tmp, dur.at(ka), ea - ka, lane);
    }
    if (__any_sync(TG_FULL, A.sat || B.sat)) return -1;
    diff = fixed + warp_sum64((i64)B.pops) - warp_sum64((i64)A.pops);
    if (k0 + EV_BLOCK >= n) break;
    if (diff >= 0) {
      if (wait == 0) { if (ev_behind(A, ra, B, rb, lane)) return 0; wait = 1; }
      else --wait;
    }
  }
  return diff < 0 ? 1 : 0;
}

// heaps beyond 256 times: windows with the rests in shared memory, or in the slab where they do not fit
__device__ __forceinline__ int ev_compare_windows(const PoolTask& T, int q, const u8* kept, const u8* fewer, i64 fixed, Slab slab, u32 wk, int lane) {
  const u32 words = 2u * (u32)(T.n_seeds + q + 1) + 32u, stage = 2 * EV_BLOCK + 4;   // rests; staged durations
  if ((stage + words) * 4u <= T.wk_bytes) return ev_compare(T, q, kept, fewer, fixed, EvShared{wk + stage * 4u}, EvShared{wk}, lane);
  u32* g = (u32*)slab.take((u64)words * 4);
  return g ? ev_compare(T, q, kept, fewer, fixed, EvGlobal{g}, EvShared{wk}, lane) : -1;
}

// Does evicting candidate q (the last of the q+1 kept, multiplicities rkeep) lower the objective (rsel, T0.opt: the
// optimum without it)?  opt_kept: duration sum with it.  1 yes, 0 no, -1 workspace too small.
template <int U>
__device__ __forceinline__ int eviction_pays(const Params& P, const PoolTask& T0, int q, i64 opt_kept, Slab slab, int lane) {
  PoolTask T;                                            // (what is used of it, in registers)
  T.m = uniform(T0.m); T.n_ac = uniform(T0.n_ac); T.n_seeds = uniform(T0.n_seeds); T.depth = T0.depth;
  T.cs = T0.cs; T.cp = T0.cp; T.cmask = T0.cmask; T.ac_tmin = T0.ac_tmin; T.seeds = T0.seeds;
  T.ac_first = T0.ac_first; T.wk = T0.wk; T.wk_bytes = T0.wk_bytes;
  const u8* kept = T0.rkeep; const u8* fewer = T0.rsel;
  const i64 opt_fewer = T0.opt;
  const int n = T.m - q - 1 + T.n_ac;                    // what waits behind candidate q
  const int ha = T.n_seeds + q + 1;
  if (n < (1 << 20)) {                                   // (sums then stay below 2^63 whatever the durations)
    i64 fixed = opt_fewer - opt_kept + rest_first(T, q);
    if (n > 0) fixed += rest_least(T, q + 1, 0) - rest_first(T, q + 1);
    const u32 wk = (u32)__cvta_generic_to_shared(T.wk);
    int got = -1;
    if (ha <= 32) got = ev_compare_regs<1, U>(T, q, kept, fewer, fixed, wk, lane);
    else if (ha <= 64) got = ev_compare_regs<2, U>(T, q, kept, fewer, fixed, wk, lane);
    else if (ha <= 96) got = ev_compare_regs<3, U>(T, q, kept, fewer, fixed, wk, lane);
    else if (ha <= 128) got = ev_compare_regs<4, U>(T, q, kept, fewer, fixed, wk, lane);
    else if (ha <= 192) got = ev_compare_regs<6, U>(T, q, kept, fewer, fixed, wk, lane);
    else if (ha <= 256) got = ev_compare_regs<8, U>(T, q, kept, fewer, fixed, wk, lane);
    else got = ev_compare_windows(T0, q, kept, fewer, fixed, slab, wk, lane);
    if (got >= 0) return got;
  }
  i64 ek, ef;
  if (!estimate_exact(P, T0, q + 1, kept, slab, lane, &ek) || !estimate_exact(P, T0, q, fewer, slab, lane, &ef)) return -1;
  return sat_add(opt_fewer, ef) < sat_add(opt_kept, ek) ? 1 : 0;
}

// A single candidate: nothing can be evicted (the head stays), and DPArrange for one task is the feasible
// level of least duration, the smallest one among equals (value, then units).  Lane r-1 tries multiplicity r.
__device__ __forceinline__ void solve_single(const PoolTask& T, int lane) {
  const int g = T.cg[0] & 0x7f, gang = T.cg[0] >> 7, r = lane + 1;
  const u32 mk = T.cmask[0];
  bool ok = (mk >> lane) & 1u;
  if (ok) {
    const int lz = class_of(T.type, g, gang, r);
    int cap = T.cap[0];
#pragma unroll
    for (int l = 1; l < 4; ++l) if (l == lz) cap = T.cap[l];
    ok = g * r <= cap;
  }
  const i64 key = ok ? ((duration(T.cs[0], T.cp[0], r) << 6) | (i64)r) : TG_INF;
  const i64 best = warp_min64(key);
  // (the least level fits: the prefix admitted the action)
  if (lane == 0) { const u8 rr = best == TG_INF ? (u8)__ffs(mk) : (u8)(best & 63); T.rsel[0] = rr; T.rkeep[0] = rr; }
  __syncwarp();
}

// Greedy eviction (Algorithm 1, lines 8-14) from the full candidate list.  The accepted multiplicities are in
// T.rkeep; returns the number of candidates kept, or -1 if the workspace is too small.
template <int U>
__device__ __forceinline__ int evict_loop(const Params& P, PoolTask& T, Slab slab, int lane) {
  const int m = uniform(T.m);
  if (m == 1) { solve_single(T, lane); return 1; }
  u8* rkeep = T.rkeep; const u8* rsel = T.rsel;
  // room for the small table of a pool with one capacity and up to 256 elastic candidates (the routines below get the
  // rest of the slab; a pool whose nested capacities bind never builds that table and keeps all of it)
  const bool one_capacity = T.type != TG_POOL_GPU || T.cap[3] >= T.cap[0];
  i64* cells = m <= 256 && one_capacity ? (i64*)slab.take((u64)m * (256 + 64)) : nullptr;
  if (lane < 4) T.lam[lane] = 0.f;
  if (lane == 0) { T.upgrades = -1; T.limit = INT_MAX; T.sq = 0; T.cell_rows = cells ? 0 : -1; T.cell_val = cells; T.cell_ch = (unsigned short*)(cells + (size_t)m * 32); }
  __syncwarp();
  if (!one_capacity) find_replicas(T, lane);
  i64 opt = 0;
  int keep = m;
#pragma unroll 1
  for (int q = m; q >= 1; --q) {                         // q = m: the full list itself
    const int got = solve_prefix(P, T, q, slab, lane);
    if (got == UNSOLVED) return -1;
    if (q < m) {
      if (eviction_cannot_pay(T, q, rkeep, rsel, lane)) break;
      const int pays = eviction_pays<U>(P, T, q, opt, slab, lane);
      if (pays < 0) return -1;
      if (!pays) break;
    }
    keep = q; opt = T.opt;
#pragma unroll 1
    for (int i = lane; i < q; i += 32) rkeep[i] = rsel[i];
    __syncwarp();
    if (got == SOLVED_ALL_BEST && q == m) break;         // then so does every prefix: no eviction can pay
  }
  return keep;
}
