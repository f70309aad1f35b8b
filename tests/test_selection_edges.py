"""Edges of the per-pool selection on the CUDA path: heap sizes around every register count, spare units around the 32-cell
table, rows beyond its size and level lists beyond its width, against the oracle."""
import numpy as np
import pytest

from test_gpu_parity import assert_same, gpu_round
from workloads import POOL_API, POOL_CPU, POOL_GPU, GANG, Pool

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
