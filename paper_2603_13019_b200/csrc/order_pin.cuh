// Front ends of a round that change what the scheduler sees as its queue.
//
// k_order (Section 4.2: Algorithm 1 takes the queue in any order): one block per scenario sorts the
// queue by a policy key -- least-level duration (Eq. 1) ascending or descending, or arrival time --
// with the queue position as second key, so equal keys keep their order.  The round then walks the queue through
// the sorted positions (P.perm) and leaves records and results where the caller has them.
//
// k_pin (Section 5.2: per-node CPU scheduling): one warp per scenario walks the queue; the first
// action of a trajectory pins it to the CPU node (= CPU pool) with the most free memory among those
// with enough cores for the action's least level and enough free memory for the whole trajectory;
// every action of a pinned trajectory gets its node as pool.
#pragma once
#include "common.cuh"

#define KO_MAX_N 16384
#define KO_MAX_THREADS 512

struct OrderIo {
  int policy;            // 1: shortest least-level duration first, 2: longest first, 3: earliest arrival first
  int* perm;             // [S][N] action index at each sorted position
};

// maximum over the warp of values >= -1
__device__ __forceinline__ i64 warp_max64_from_m1(i64 v) {
  const u64 u = (u64)(v + 1);
  const u32 hi = (u32)(u >> 32);
  const u32 mhi = __reduce_max_sync(TG_FULL, hi);
  const u32 mlo = __reduce_max_sync(TG_FULL, hi == mhi ? (u32)u : 0u);
  return (i64)(((u64)mhi << 32) | mlo) - 1;
}

// The key an action is sorted by, smallest first.
__device__ __forceinline__ u64 order_key(const Params& P, int policy, size_t o) {
  if (policy == 3) return (u64)(P.a_arrival ? P.a_arrival[o] : 0) ^ 0x8000000000000000ull;
  const int j = P.a_pool[o];
  int g, gang; u32 eff;
  i64 T = 0;                                           // a record no pool can serve has key 0
  if (j < P.P && decode_levels(P.pool[j], P.a_unit[o], P.a_mask[o], g, gang, eff))
    T = duration(clamp_param(P.a_s[o]), clamp_param(P.a_p[o]), __ffs(eff));
  return policy == 2 ? (u64)((1ll << 42) - T) : (u64)T;
}

// A duration key in 16 bits that keep its order: exact below 2048 us, then eleven bits behind the leading one.
__device__ __forceinline__ u32 short_key(u64 key, int policy) {
  const u64 T = policy == 2 ? (1ull << 42) - key : key;
  const int e = 63 - __clzll((i64)(T | 1));
  const u32 c = e < 11 ? (u32)T : ((u32)(e - 10) << 11) | ((u32)(T >> (e - 11)) & 2047u);
  return policy == 2 ? 65535u - c : c;
}

// One block per scenario, EPT actions per thread in registers: element e of a lane is position warp * 32 * EPT + 32 * e + lane
// of the queue.  A queue in order is left alone.  Durations go into buckets of equal width on the logarithmic scale of
// short_key, twice as many as the queue has places, and every action counts the smaller ones among the few in its
// bucket: three trips through shared memory.  A queue that fills a bucket with more than KO_BUCKET_MAX (equal or nearly equal
// durations), and arrival times out of order, take a radix sort from the low end, eight bits at a time where the keys
// differ: a warp ranks its elements by eight ballots and its own counters, one scan over (digit, warp) gives every
// warp its place for every digit, and one trip through shared memory puts the elements there; each step keeps the
// order of equal digits.  Bound by instructions issued (ranking costs some hundred per element and pass).
// 3000 x 2001 durations: bitonic network 250 us, radix sort 217 us, buckets 111 us.
// Key and position share a 64-bit word (50 + 14 bits); where arrival times differ in higher bits than that, the
// word holds the position alone and the key is read again in every pass.
#define KO_BUCKET_MAX 32
__host__ __device__ constexpr int ko_buckets(int ept, int threads) { return (ept <= 16 ? 2 : 1) * ept * threads; }
// bytes behind the elements: the radix sort's counters, or the buckets' (one in 33 idle: no bank conflicts in the scan)
__host__ __device__ constexpr int ko_counter_bytes(int ept, int threads) {
  const int b = ko_buckets(ept, threads), x = (b + b / 32 + 1) * 4, y = threads / 32 * 1024;
  return x > y ? x : y;
}
// exclusive scan of one count per thread over the block
__device__ __forceinline__ u32 ko_block_scan(u32 sum, u32* wsum, int lane, int warp) {
  u32 incl = sum;
#pragma unroll
  for (int s = 1; s < 32; s <<= 1) { const u32 y = __shfl_up_sync(TG_FULL, incl, s); if (lane >= s) incl += y; }
  if (lane == 31) wsum[warp] = incl;
  __syncthreads();
  u32 off = incl - sum;
  for (int w = 0; w < warp; ++w) off += wsum[w];
  return off;
}
template <int EPT>
__global__ void __launch_bounds__(KO_MAX_THREADS) k_order(const __grid_constant__ Params P, const OrderIo O) {
  extern __shared__ __align__(16) unsigned char ko_smem[];
  __shared__ u64 s_diff;
  __shared__ int s_unsorted;
  __shared__ u32 s_cmin, s_cmax;
  __shared__ int s_full;
  __shared__ u32 wsum[KO_MAX_THREADS / 32];
  u64* buf = (u64*)ko_smem;                            // [EPT * blockDim.x]
  const int t = threadIdx.x, lane = t & 31, warp = t >> 5, nw = blockDim.x >> 5;
  u32* hist = (u32*)(buf + EPT * blockDim.x);          // [nw][256]
  u32* mine = hist + warp * 256;
  const int sc = blockIdx.x, wb = warp * 32 * EPT + lane;
  const size_t row = (size_t)sc * P.N;
  const int n = min(max(P.n_actions[sc], 0), P.N);
  const u32 lt = (1u << lane) - 1u;
  if (t == 0) { s_diff = 0; s_cmin = ~0u; s_cmax = 0; s_full = 0; s_unsorted = 0; }
  u64 v[EPT];
#pragma unroll
  for (int e = 0; e < EPT; ++e) {
    const int i = wb + 32 * e;
    if (i < n) { v[e] = order_key(P, O.policy, row + i); buf[i] = v[e]; }
  }
  __syncthreads();
  u64 diff = 0;
  u32 cmin = ~0u, cmax = 0;
  bool unsorted = false;
  const bool timed = O.policy != 3;                    // keys are durations
#pragma unroll
  for (int e = 0; e < EPT; ++e) {
    const int i = wb + 32 * e;
    if (i < n) {
      diff |= v[e] ^ buf[0]; unsorted |= i + 1 < n && buf[i + 1] < v[e];
      if (timed) { const u32 c = short_key(v[e], O.policy); cmin = min(cmin, c); cmax = max(cmax, c); }
    }
  }
  if (unsorted) s_unsorted = 1;
  const u32 dlo = __reduce_or_sync(TG_FULL, (u32)diff), dhi = __reduce_or_sync(TG_FULL, (u32)(diff >> 32));
  cmin = __reduce_min_sync(TG_FULL, cmin); cmax = __reduce_max_sync(TG_FULL, cmax);
  if (lane == 0) {
    atomicOr((unsigned long long*)&s_diff, ((u64)dhi << 32) | dlo);
    if (timed) { atomicMin(&s_cmin, cmin); atomicMax(&s_cmax, cmax); }
  }
  __syncthreads();
  diff = s_unsorted ? s_diff : 0;
  const bool wide = (diff >> 50) != 0;
#pragma unroll
  for (int e = 0; e < EPT; ++e) v[e] = (wide ? 0 : v[e] << 14) | (u64)(u32)(wb + 32 * e);

  if (timed && diff) {
    const int B = ko_buckets(EPT, blockDim.x);
    const float scale = (float)B / (float)(s_cmax - s_cmin + 1);
    auto place = [](int b) { return b + (b >> 5); };
    u32 at[EPT];                                       // bucket and number in it
    for (int x = t; x <= place(B); x += blockDim.x) hist[x] = 0;
    __syncthreads();
    bool full = false;
#pragma unroll
    for (int e = 0; e < EPT; ++e) {
      if (wb + 32 * e >= n) continue;
      const int b = min(B - 1, (int)((float)(short_key(v[e] >> 14, O.policy) - s_cmin) * scale));
      const u32 r = atomicAdd(&hist[place(b)], 1u);
      at[e] = (u32)b | r << 16;
      full |= r >= KO_BUCKET_MAX;
    }
    if (full) s_full = 1;
    __syncthreads();
    if (!s_full) {
      constexpr int per = EPT <= 16 ? 2 * EPT : EPT;   // buckets per thread
      u32 sum = 0;
#pragma unroll 4
      for (int x = 0; x < per; ++x) sum += hist[place(t * per + x)];
      u32 off = ko_block_scan(sum, wsum, lane, warp);
#pragma unroll 4
      for (int x = 0; x < per; ++x) { u32& h = hist[place(t * per + x)]; const u32 c = h; h = off; off += c; }
      if (t == 0) hist[place(B)] = n;
      __syncthreads();
#pragma unroll
      for (int e = 0; e < EPT; ++e)
        if (wb + 32 * e < n) buf[hist[place(at[e] & 0xffff)] + (at[e] >> 16)] = v[e];
      __syncthreads();
#pragma unroll
      for (int e = 0; e < EPT; ++e) {
        if (wb + 32 * e >= n) continue;
        const int b = at[e] & 0xffff, lo = hist[place(b)], hi = hist[place(b + 1)];
        u32 pos = lo;
#pragma unroll 1
        for (int k = lo; k < hi; ++k) pos += buf[k] < v[e];
        at[e] = pos;
      }
      __syncthreads();
#pragma unroll
      for (int e = 0; e < EPT; ++e) if (wb + 32 * e < n) ((u32*)buf)[at[e]] = (u32)v[e] & 0x3fff;
      __syncthreads();
#pragma unroll
      for (int e = 0; e < EPT; ++e) if (wb + 32 * e < n) v[e] = ((u32*)buf)[wb + 32 * e];
      diff = 0;
    }
  }
#pragma unroll 1
  for (int sh = 0; sh < 64; sh += 8) {
    if (((diff >> sh) & 255) == 0) continue;
    auto digit = [&](u64 x) -> u32 {
      return (u32)((wide ? order_key(P, O.policy, row + (size_t)(x & 0x3fff)) : x >> 14) >> sh) & 255u;
    };
    u32 rank[EPT];
#pragma unroll
    for (int x = 0; x < 8; ++x) mine[32 * x + lane] = 0;
    __syncwarp();
#pragma unroll
    for (int e = 0; e < EPT; ++e) {
      if (wb - lane + 32 * e >= n) continue;           // nothing there for the whole warp
      const bool on = wb + 32 * e < n;
      const u32 d = on ? digit(v[e]) : 0;
      u32 peers = __ballot_sync(TG_FULL, on);
#pragma unroll
      for (int b = 0; b < 8; ++b) {
        const u32 q = __ballot_sync(TG_FULL, (d >> b) & 1u);
        peers &= (d >> b) & 1u ? q : ~q;
      }
      const u32 before = on ? mine[d] : 0;
      rank[e] = before + __popc(peers & lt);
      __syncwarp();
      if (on && !(peers & lt)) mine[d] = before + __popc(peers);
      __syncwarp();
    }
    __syncthreads();
    // the digits in order, and for every digit the warps in order: where each warp's elements begin
    const int dp = blockDim.x < 256 ? 256 / blockDim.x : 1;
    u32 sum = 0;
    if (t * dp < 256)
#pragma unroll 1
      for (int x = 0; x < dp; ++x)
        for (int w = 0; w < nw; ++w) sum += hist[w * 256 + t * dp + x];
    u32 off = ko_block_scan(sum, wsum, lane, warp);
    if (t * dp < 256)
#pragma unroll 1
      for (int x = 0; x < dp; ++x)
        for (int w = 0; w < nw; ++w) { u32& h = hist[w * 256 + t * dp + x]; const u32 c = h; h = off; off += c; }
    __syncthreads();
#pragma unroll
    for (int e = 0; e < EPT; ++e)
      if (wb + 32 * e < n) buf[mine[digit(v[e])] + rank[e]] = v[e];
    __syncthreads();
#pragma unroll
    for (int e = 0; e < EPT; ++e)
      if (wb + 32 * e < n) v[e] = buf[wb + 32 * e];
  }
#pragma unroll
  for (int e = 0; e < EPT; ++e)                        // the positions behind the queue stay where they are
    if (wb + 32 * e < P.N) O.perm[row + wb + 32 * e] = (int)(v[e] & 0x3fff);
}

struct PinIo {
  const int* trajectory; const u32* traj_mem; int max_traj;
  int* traj_node; i64* mem_free; u8* pool_out; int* n_admitted;
};

// One chunk of up to 32 consecutive queue actions, one per lane (`have`: the lane holds one, of pool pj; `mine`: an action of
// the CPU manager, of trajectory t that needs `mem` and least-level cores `need`).  Lane j < P keeps node j's free memory (mf) and cores (-1: not a CPU node).  The actions whose
// trajectory has no node yet are taken one after the other, lowest lane first.  Returns the lane of the first
// action whose trajectory finds no node (32 if none); pool_of = the lane's pool afterwards (its trajectory's
// node, or its own pool; untouched for a lane without an action); the actions from the returned lane on keep
// their pools.
__device__ __forceinline__ int pin_chunk(bool mine, int t, u32 mem, int need, int pj, bool have, int* tn, i64& mf, int cores, int lane,
                                         int& pool_of) {
  int node = mine ? tn[t] : -1;
  __syncwarp();                                         // (lane 0 writes tn below)
  int first_out = 32;
  u32 open = __ballot_sync(TG_FULL, mine && node < 0);
  while (open) {
    const int b = __ffs(open) - 1;
    const int bt = __shfl_sync(TG_FULL, t, b), bneed = __shfl_sync(TG_FULL, need, b);
    const u32 bmem = __shfl_sync(TG_FULL, mem, b);
    // the eligible node with the most free memory, lowest index on ties
    const bool ok = cores >= 0 && cores >= bneed && mf >= (i64)bmem;
    const i64 best = warp_max64_from_m1(ok ? mf : -1);
    const u32 who = __ballot_sync(TG_FULL, ok && mf == best);
    if (!who) {                                         // no node: the admitted queue ends before this action
      first_out = b;
      if (lane >= b) mine = false;                      // nothing from it on is touched
      break;
    }
    const int bn = __ffs(who) - 1;
    if (lane == bn) mf -= (i64)bmem;
    if (lane == 0) tn[bt] = bn;
    if (mine && t == bt) node = bn;                     // later actions of the trajectory in this chunk follow
    open = __ballot_sync(TG_FULL, mine && node < 0) & ~((2u << b) - 1u);
  }
  if (have) pool_of = (mine && node >= 0) ? node : pj;
  __syncwarp();
  return first_out;
}

__global__ void __launch_bounds__(256) k_pin(const __grid_constant__ Params P, const PinIo X) {
  const int lane = threadIdx.x & 31;
  const int sc = (int)((blockIdx.x * (unsigned)blockDim.x + threadIdx.x) >> 5);
  if (sc >= P.S) return;
  const size_t row = (size_t)sc * P.N;
  const int n = min(max(P.n_actions[sc], 0), P.N);
  int* tn = X.traj_node + (size_t)sc * X.max_traj;
  // lane j < P: node j's free memory and cores (-1 cores: not a CPU node)
  i64 mf = 0; int cores = -1;
  if (lane < P.P && P.pool[lane].type == TG_POOL_CPU) { mf = X.mem_free[(size_t)sc * P.P + lane]; cores = P.pool[lane].capacity; }
  int admitted = n;
  for (int c0 = 0; c0 < P.N; c0 += 32) {
    const int i = c0 + lane;
    int pool_of = i < P.N ? P.a_pool[row + i] : 0xff;
    if (admitted == n && c0 < n) {                      // (behind the admitted queue the pool column is copied)
      int pj = 0xff, t = -1, need = 0; u32 mem = 0;
      bool mine = false;                                // an action of the CPU manager with a trajectory
      if (i < n) {
        pj = P.a_pool[row + i];
        t = X.trajectory[row + i];
        mine = t >= 0 && t < X.max_traj && pj < P.P && P.pool[pj].type == TG_POOL_CPU;
        if (mine) {
          mem = X.traj_mem[row + i];
          const u32 mk = P.a_mask[row + i];
          need = (int)(P.a_unit[row + i] & 0x7f) * (mk ? __ffs(mk) : 0);
        }
      }
      const int out = pin_chunk(mine, t, mem, need, pj, i < n, tn, mf, cores, lane, pool_of);
      if (out < 32) admitted = c0 + out;
    }
    if (i < P.N) X.pool_out[row + i] = (u8)pool_of;
  }
  if (lane < P.P && cores >= 0) X.mem_free[(size_t)sc * P.P + lane] = mf;
  if (lane == 0) X.n_admitted[sc] = admitted;
}
