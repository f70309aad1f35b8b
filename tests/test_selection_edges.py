"""Edges of the per-pool selection on the CUDA path: heap sizes around every register count, spare units around the 32-cell
table, rows beyond its size and level lists beyond its width, against the oracle."""
import numpy as np
import pytest

from test_gpu_parity import _gpu_round_ws, assert_same, gpu_round
from workloads import POOL_API, POOL_CPU, POOL_GPU, GANG, Pool, contiguous_replica_round

pytestmark = pytest.mark.gpu


def _round(seed, pools, head, mask, spare_pool, behind, tiny=False):
    """`head` core actions, two actions of a quota pool with one token (the second one ends the candidate prefix), then
    `behind` waiting core actions; durations drawn per scenario."""
    rng = np.random.Generator(np.random.PCG64(seed))
    S, N = 6, head + 2 + behind
    pool = np.zeros((S, N), np.uint8)
    pool[:, head:head + 2] = spare_pool
    masks = np.array(mask, np.uint32)[rng.integers(0, len(mask), (S, N))]
    masks[:, head:head + 2] = 1
    hi = (4, 12) if tiny else (50_000, 500_000)
    return dict(pool=pool, unit=np.ones((S, N), np.uint8), level_mask=masks, arrival_us=None, gpu_busy=None,
                s_us=rng.integers(0, hi[0], (S, N)).astype(np.int64), p_us=rng.integers(0, hi[1], (S, N)).astype(np.int64),
                n_actions=np.full(S, N, np.int32))


@pytest.mark.parametrize("m", [2, 31, 32, 33, 64, 65, 96, 97, 128, 129, 192, 193, 256, 257, 300])
def test_heap_sizes_match_oracle(oracle, m):
    # no spare unit with all m candidates, one more with every eviction; 150 actions wait
    pools = (Pool(POOL_CPU, m, m), Pool(POOL_API, 1, 0, 0))
    a = _round(m, pools, m, [0b11, 0b1011, 0b1], 1, 150, tiny=m in (64, 257))
    assert_same(oracle.schedule_batch(pools, a), gpu_round(pools, a))


@pytest.mark.parametrize("m,spare", [(2, 1), (33, 30), (33, 31), (40, 32), (64, 33), (200, 31), (256, 20), (257, 20), (90, 200)])
@pytest.mark.parametrize("mask", [[0b1000_0000_1000_1011, 0x80008_08B, 0b1], [0x1FF, 0b1]])
def test_spare_units_match_oracle(oracle, m, spare, mask):
    # powers of two up to 32 (at most six levels inside the small table), or contiguous levels 1..9 (more than six)
    pools = (Pool(POOL_CPU, m + spare, m + spare), Pool(POOL_API, 1, 0, 0))
    for tiny in (False, True):
        a = _round(1000 + m + spare, pools, m, mask, 1, 40, tiny=tiny)
        assert_same(oracle.schedule_batch(pools, a), gpu_round(pools, a))


@pytest.mark.parametrize("nodes,m,tiny", [(3, 9, False), (8, 20, True), (12, 40, False), (20, 30, False)])
def test_gang_requests_on_fragmented_nodes_match_oracle(oracle, nodes, m, tiny):
    # all four nested capacities bind: priced selection over the states within a bound, tied values with tiny durations
    pools = (Pool(POOL_GPU, 8 * nodes, 8), Pool(POOL_API, 1, 0, 0))
    a = _round(77 + nodes, pools, m, [0x8B, 0xB, 0x3, 0x80, 0x1], 1, 30, tiny=tiny)
    a["unit"] = np.where(a["pool"] == 0, 1 | GANG, 1).astype(np.uint8)
    rng = np.random.Generator(np.random.PCG64(nodes))
    a["gpu_busy"] = np.where(rng.random((6, nodes)) < 0.5, rng.integers(0, 256, (6, nodes)), 0).astype(np.uint8)
    assert_same(oracle.schedule_batch(pools, a), gpu_round(pools, a))


@pytest.mark.parametrize("kind,S,nodes,N,seed", [
    ("alike", 12, 64, 256, 320),     # more states within reach of the prices than a table holds
    ("alike", 2, 256, 512, 768),     # more than 512 upgrade steps in a class: sorted in global memory
    ("gaps", 6, 40, 120, 8168),      # levels 1, 2, 4, 8: the recurrence instead of the sorted gains
    ("equal", 6, 64, 256, 8328),     # splits between chunk sizes tie in some pools
])
def test_alike_replica_requests_match_oracle(oracle, kind, S, nodes, N, seed):
    # durations so close to each other that the prices settle nothing and a pass over the states within their reach costs
    # more than the chunk sizes one by one; that way needs the slab only, so one MiB of workspace does
    w, a = contiguous_replica_round(seed, S, N, nodes, 8)
    rng = np.random.default_rng(seed % 8000)
    a["p_us"] = rng.integers(400_000_000, 400_001_000, a["p_us"].shape)
    if kind == "gaps":
        a["level_mask"] = rng.choice(np.array([0x8B, 0xB, 0x5, 0x1], np.uint32), a["level_mask"].shape)
    if kind == "equal":
        a["p_us"] = 4000 * rng.integers(50, 52, a["p_us"].shape)
    g = _gpu_round_ws(w.pools, a, workspace_bytes=1 << 20)
    assert np.all(g["status"] == 0)
    assert_same(oracle.schedule_batch(w.pools, a), g)


def test_states_that_outgrow_the_priced_table_take_a_slot(oracle):
    # an elastic gang request among replica requests of close durations: neither the prices nor the chunk sizes one by one
    # settle it, the table of all reachable states in a slot of the workspace does.  Twelve copies for four slots:
    # with a wait of a millisecond some give up, with a long one every copy gets its turn
    w, a = contiguous_replica_round(96, 12, 64, 32, 8)
    a["p_us"] = np.random.default_rng(96).integers(400_000_000, 400_001_000, a["p_us"].shape)
    a["unit"][:, 0] = 1 | GANG
    a["level_mask"][:, 0] = 0xB
    a = {k: None if v is None else np.repeat(v[4:5], 12, axis=0) for k, v in a.items()}
    want = oracle.schedule_batch(w.pools, a)
    assert_same(want, _gpu_round_ws(w.pools, a))
    short = _gpu_round_ws(w.pools, a, workspace_bytes=320 << 20, slot_wait_us=1000)
    assert set(np.unique(short["status"])) == {0, 4}
    solved = short["status"] == 0
    assert_same({k: v[solved] for k, v in want.items()}, {k: v[solved] for k, v in short.items()})
    assert_same(want, _gpu_round_ws(w.pools, a, workspace_bytes=320 << 20, slot_wait_us=5_000_000))


def test_many_tied_end_states_take_the_dense_table(oracle):
    # 70 gang requests and 40 requests for chunks of two, all with the same gain per GPU, share 70 GPUs: 36 splits tie on
    # duration and units, more than a warp's lanes; long rows make a slab that holds the box
    S, N, n = 3, 16384, 110
    busy = np.array([0] * 27 + [0x3F] + [0x7F] * 2, np.uint8)
    pools = (Pool(POOL_GPU, 8 * len(busy), 8),)
    rng = np.random.default_rng(5)
    a = dict(pool=np.zeros((S, N), np.uint8), unit=np.ones((S, N), np.uint8), level_mask=np.ones((S, N), np.uint32),
             s_us=np.zeros((S, N), np.int64), p_us=np.zeros((S, N), np.int64), arrival_us=None,
             n_actions=np.full(S, n, np.int32), gpu_busy=np.tile(busy, (S, 1)))
    for sc in range(S):
        gang = rng.permutation(n) < 70
        a["unit"][sc, :n] = np.where(gang, 1 | GANG, 2)
        a["level_mask"][sc, :n] = 3
        a["p_us"][sc, :n] = np.where(gang, 80_000, 160_000)
        a["s_us"][sc, :n] = rng.integers(0, 50_000, n)
    g = gpu_round(pools, a)
    assert np.all(g["status"] == 0)
    assert_same(oracle.schedule_batch(pools, a), g)


@pytest.mark.parametrize("policy", [0, 1, 2])
def test_replay_queues_beyond_shared_memory_match_oracle(oracle, policy):
    # so many scenarios that a block keeps few waiting records in shared memory: with bursts of long actions on
    # four cores the tail of every queue lives in global memory, and comes back as the queue drains
    import torch
    from paper_2603_13019_b200 import binding
    pools = (Pool(POOL_CPU, 2040, 1020), Pool(POOL_GPU, 8, 8))
    S, N = 900, 420
    rng = np.random.Generator(np.random.PCG64(policy))
    gpu = rng.random((S, N)) < 0.4
    a = dict(pool=gpu.astype(np.uint8), unit=np.where(gpu, 1 | GANG, 100).astype(np.uint8),
             level_mask=np.where(gpu, 0x8B, np.where(rng.random((S, N)) < 0.5, 0x80, 0xC0)).astype(np.uint32),
             s_us=rng.integers(5_000, 60_000, (S, N)).astype(np.int64), p_us=rng.integers(0, 60_000, (S, N)).astype(np.int64),
             arrival_us=np.sort(rng.integers(0, 400_000, (S, N)), axis=1).astype(np.int64),
             n_actions=np.full(S, N, np.int32), gpu_busy=None)
    rnd = binding.Round(S, N, pools, round_us=10_000, max_rounds=3000)
    g = rnd.replay_trace(binding.to_device(a), policy=policy)
    torch.cuda.synchronize()
    o = oracle.replay_trace(pools, a, round_us=10_000, max_rounds=3000, policy=policy, lo=0, hi=6)
    for k in ("status", "n_selected", "total_act_us", "alloc_units", "place_node", "place_off", "act_us", "occupancy", "rounds_used"):
        assert np.array_equal(o[k], g[k][:6].cpu().numpy()), k
    assert np.all(o["n_selected"] == N)
    rnd.destroy()


def _copies(a, o, n):
    S = a["n_actions"].shape[0]
    pick = np.arange(n) % S
    return {k: None if v is None else v[pick] for k, v in a.items()}, {k: v[pick] for k, v in o.items()}


@pytest.mark.parametrize("n", [295, 296, 297, 301])
@pytest.mark.parametrize("behind", [0, 29, 150])
def test_batches_around_one_launch_match_oracle(oracle, n, behind):
    # two blocks on each of 148 multiprocessors: the last batch that is one launch, and the first that is not
    pools = (Pool(POOL_CPU, 40, 40), Pool(POOL_API, 1, 0, 0))
    a = _round(n, pools, 33, [0b11, 0b1011, 0b1], 1, behind)
    a["n_actions"] = np.array([0, 1, 33, 34, a["pool"].shape[1], a["pool"].shape[1] // 2], np.int32)
    b, want = _copies(a, oracle.schedule_batch(pools, a), n)
    assert_same(want, gpu_round(pools, b))


@pytest.mark.parametrize("n", [3, 40000])
def test_static_entry_point_with_fewer_warps_than_pools_matches_oracle(oracle, n):
    # eight pools with rows of 40000 actions leave room for seven worker warps
    import torch
    from paper_2603_13019_b200 import binding
    pools = tuple(Pool(POOL_CPU, 40 + j, 40 + j) for j in range(8))
    rng = np.random.Generator(np.random.PCG64(n))
    a = dict(pool=rng.integers(0, 8, (1, n)).astype(np.uint8), unit=np.ones((1, n), np.uint8),
             level_mask=np.full((1, n), 0b1011, np.uint32), arrival_us=None, gpu_busy=None,
             s_us=rng.integers(0, 50_000, (1, n)), p_us=rng.integers(0, 500_000, (1, n)), n_actions=np.full(1, n, np.int32))
    want = oracle.schedule_batch(pools, a)
    got = {k: torch.full(v.shape, -7, dtype=torch.int64 if v.dtype == np.int64 else torch.int32, device="cuda")
           for k, v in want.items()}
    assert binding.schedule_batch_static(pools, binding.to_device(a), got) == 0
    assert_same(want, {k: v.cpu().numpy() for k, v in got.items()})


@pytest.mark.parametrize("n", [1, 31, 128, 129, 512, 513, 2049, 16384])
@pytest.mark.parametrize("lo,hi", [(0, 3), (-40, 40), (-2**62, 2**62), (7, 8)])
def test_sorted_orders_match_oracle(oracle, n, lo, hi):
    # edges of the sort's tiles; few, mixed-sign, 64-bit and equal arrival times; one queue in order already
    from paper_2603_13019_b200 import binding
    pools = (Pool(POOL_CPU, 64, 64), Pool(POOL_API, 1, 0, 0))
    rng = np.random.Generator(np.random.PCG64(n))
    a = dict(pool=np.zeros((4, n), np.uint8), unit=np.ones((4, n), np.uint8), level_mask=np.full((4, n), 0b1011, np.uint32),
             gpu_busy=None, s_us=rng.integers(0, 50, (4, n)), p_us=rng.integers(0, 1 << 40, (4, n)),
             arrival_us=rng.integers(lo, hi, (4, n)), n_actions=np.array([n, n // 2, n, 0], np.int32))
    a["arrival_us"][2].sort()
    rnd, dev = binding.Round(4, n, pools), binding.to_device(a)
    for policy in (1, 2, 3):
        assert np.array_equal(oracle.order_queue(pools, a, policy), rnd.order_queue(dev, policy).cpu().numpy())


@pytest.mark.parametrize("m", [68, 69])
def test_rows_around_the_shared_table_match_oracle(oracle, m):
    # m elastic candidates, ten spare cores; the last ones pay to be evicted in one scenario, everything ties in another
    pools = (Pool(POOL_CPU, m + 10, m + 10), Pool(POOL_API, 1, 0, 0))
    a = _round(m, pools, m, [0b1011], 1, 150)
    a["p_us"][1, :m] = 50_000
    a["s_us"][1] = 1000
    a["p_us"][2, m - 4:m] = 4_000_000
    assert_same(oracle.schedule_batch(pools, a), gpu_round(pools, a))


@pytest.mark.parametrize("gpus,group,busy", [(8, 8, 0.0), (256, 8, 0.3), (264, 8, 0.3), (1032, 8, 0.1), (4800, 8, 0.2), (140, 4, 0.3),
                                             (70, 2, 0.2), (33, 1, 0.3)])
def test_gpu_placement_at_the_edges_match_oracle(oracle, gpus, group, busy):
    # one node, 32 and 33 nodes, more than 128; more requests than the warp's work area lists (4800 GPUs, mostly single requests)
    S, N = 4, gpus + 40
    pools = (Pool(POOL_GPU, gpus, group),)
    rng = np.random.default_rng(gpus)
    top = int(np.log2(group))
    unit = (1 << np.minimum(rng.geometric(0.7, (S, N)) - 1, top)).astype(np.uint8)
    gang = rng.random((S, N)) < 0.5
    mask = np.where(gang, 1, np.where(rng.random((S, N)) < 0.2, 4, 1))
    a = dict(pool=np.zeros((S, N), np.uint8), unit=np.where(gang, unit | GANG, unit).astype(np.uint8), level_mask=mask.astype(np.uint32),
             s_us=rng.integers(0, 20_000, (S, N)).astype(np.int64), p_us=rng.integers(0, 200_000, (S, N)).astype(np.int64),
             arrival_us=None, n_actions=np.full(S, N, np.int32), gpu_busy=(rng.random((S, gpus // group, group)) < busy))
    a["gpu_busy"] = (a["gpu_busy"] << np.arange(group)).sum(2).astype(np.uint8)
    a["gpu_busy"][rng.random(a["gpu_busy"].shape) < 0.6] = 0
    a["gpu_busy"][0] = 0
    a["level_mask"][1] = np.where(gang[1] & (unit[1] * 2 <= group), 3, a["level_mask"][1])     # elastic gangs
    o = oracle.schedule_batch(pools, a)
    assert_same(o, gpu_round(pools, a))
    assert o["n_selected"].sum() > gpus // 4


@pytest.mark.parametrize("n", [2950, 3200])
def test_requests_by_the_ten_thousands_are_placed(n):
    # n actions of 32 replicas of one GPU each on free nodes of eight: every action gets the next four nodes.  2950: a list of
    # all requests fits the scratch of one pool, but not beside the masks of its 11840 nodes; 3200: the list alone does not fit.
    # Both are placed one request after the other.
    pools = (Pool(POOL_GPU, 32 * n + 320, 8),)
    a = dict(pool=np.zeros((2, n), np.uint8), unit=np.ones((2, n), np.uint8), level_mask=np.full((2, n), 1 << 31, np.uint32),
             s_us=np.full((2, n), 1000, np.int64), p_us=np.full((2, n), 32_000, np.int64), arrival_us=None,
             n_actions=np.full(2, n, np.int32), gpu_busy=None)
    g = gpu_round(pools, a, depth=1)
    assert np.all(g["status"] == 0) and np.all(g["n_selected"] == n) and np.all(g["alloc_units"] == 32)
    assert np.array_equal(g["place_node"], np.tile(4 * np.arange(n), (2, 1))) and np.all(g["place_off"] == 0) and np.all(g["act_us"] == 2000)


@pytest.mark.parametrize("m", [255, 256, 257])
def test_shared_table_beside_the_largest_register_heaps_matches_oracle(oracle, m):
    # 60 elastic candidates among m, ten spare units: their choices share the work area with heaps of up to 256 times (with
    # more, both go elsewhere); some of the last ones pay to be evicted
    pools = (Pool(POOL_CPU, m + 10, m + 10), Pool(POOL_API, 1, 0, 0))
    a = _round(500 + m, pools, m, [1], 1, 150)
    rows = np.random.Generator(np.random.PCG64(m)).permutation(m)[:60]
    a["level_mask"][:, rows] = 0b1011
    a["level_mask"][:, m - 6:m] = 0b1011
    a["p_us"][1, m - 8:m] = 4_000_000
    a["s_us"][2] = 0
    a["p_us"][3, rows] = 60_000
    o = oracle.schedule_batch(pools, a)
    assert_same(o, gpu_round(pools, a))
    assert (o["n_selected"] < m + 1).sum() >= 2          # (one token beside the m)
