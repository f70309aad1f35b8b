"""Parity of the device-resident trace replay with the CPU oracle, through the C ABI."""
import numpy as np
import pytest

from workloads import POOL_API, POOL_CPU, POOL_GPU, Pool, generate, make_workload, random_round

pytestmark = pytest.mark.gpu

KEYS = ("status", "n_selected", "total_act_us", "alloc_units", "place_node", "place_off", "act_us",
        "rounds_used", "occupancy")


def gpu_replay(pools, a, depth, round_us, max_rounds, host_buffers=False):
    import torch
    from paper_2603_13019_b200 import binding
    S, N = a["pool"].shape
    rnd = binding.Round(S, N, pools, depth=depth, round_us=round_us, max_rounds=max_rounds,
                        host_buffers=host_buffers)
    out = rnd.replay_trace(binding.to_device(a, pin=host_buffers))
    torch.cuda.synchronize()
    res = {k: v.cpu().numpy() for k, v in out.items()}
    rnd.destroy()
    return res


def assert_same(o, g):
    for k in KEYS:
        if not np.array_equal(o[k], g[k]):
            bad = np.argwhere(o[k] != g[k])
            first = tuple(bad[0])
            raise AssertionError(
                f"{k} differs at {first}: oracle {o[k][first]} cuda {g[k][first]} ({len(bad)} mismatches)")


def test_cfg2_shape_matches_oracle(oracle):
    w = make_workload("cfg2", n_scenarios=12, max_actions=900)
    a = generate(w)
    max_rounds = 3000
    o = oracle.replay_trace(w.pools, a, depth=w.depth, round_us=w.round_us, max_rounds=max_rounds)
    g = gpu_replay(w.pools, a, w.depth, w.round_us, max_rounds)
    assert_same(o, g)
    assert np.all(g["status"] == 0) and np.all(g["n_selected"] == 900)
    assert_same(o, gpu_replay(w.pools, a, w.depth, w.round_us, max_rounds, host_buffers=True))


POOLSETS = [
    (Pool(POOL_CPU, 16, 4), Pool(POOL_GPU, 16, 8), Pool(POOL_API, 5, 0, 200_000)),
    (Pool(POOL_GPU, 24, 8),),
    (Pool(POOL_CPU, 40, 8), Pool(POOL_GPU, 8, 4), Pool(POOL_API, 3, 0, 0)),
]


@pytest.mark.parametrize("seed", range(6))
def test_random_traces_match_oracle(oracle, seed):
    pools = POOLSETS[seed % len(POOLSETS)]
    N = 120
    w, a = random_round(700 + seed, 16, N, pools, small_durations=0.2, busy_fraction=0.25 if seed % 2 else 0.0,
                        max_mult=4)
    rng = np.random.default_rng(seed)
    # bursts: arrivals every ~2 ms on average while actions last up to 0.5 s
    a["arrival_us"] = np.cumsum(rng.integers(0, 4000, a["pool"].shape), axis=1).astype(np.int64)
    for depth, max_rounds in ((2, 4000), (1, 40)):
        o = oracle.replay_trace(pools, a, depth=depth, round_us=10_000, max_rounds=max_rounds)
        g = gpu_replay(pools, a, depth, 10_000, max_rounds)
        assert_same(o, g)
    assert o["n_selected"].sum() > 0


def test_replay_flags_bad_input(oracle):
    pools = (Pool(POOL_CPU, 8, 4),)
    w, a = random_round(5, 4, 10, pools, ragged=False)
    a["arrival_us"] = np.cumsum(np.full(a["pool"].shape, 1000), axis=1).astype(np.int64)
    a["arrival_us"][1, 3] = 0                       # not sorted
    a["level_mask"][2, 0] = 0                       # no usable level
    o = oracle.replay_trace(pools, a, depth=2, round_us=10_000, max_rounds=200)
    g = gpu_replay(pools, a, 2, 10_000, 200)
    assert_same(o, g)
    assert list(g["status"]) == [0, 2, 1, 0]


def test_cfg2_full_size_sampled_scenarios_match_oracle(oracle):
    # the whole 256 x 20000 trace on the GPU; eight scenarios recomputed by the oracle, everything compared
    w = make_workload("cfg2")
    a = generate(w)
    g = gpu_replay(w.pools, a, w.depth, w.round_us, w.max_rounds)
    assert np.all(g["status"] == 0) and np.all(g["n_selected"] == w.max_actions)
    rng = np.random.default_rng(3)
    for sc in np.unique(np.concatenate([[0, w.n_scenarios - 1], rng.integers(0, w.n_scenarios, 6)])):
        o = oracle.replay_trace(w.pools, a, depth=w.depth, round_us=w.round_us, max_rounds=w.max_rounds,
                                lo=int(sc), hi=int(sc) + 1)
        for k in KEYS:
            assert np.array_equal(o[k][0], g[k][sc]), f"scenario {sc}: {k} differs"
    # conservation on every scenario: each action ran once, with a legal allocation
    assert np.all(g["alloc_units"] > 0) and np.all(g["act_us"] >= 0)
    assert np.array_equal(g["act_us"].sum(1), g["total_act_us"])


def test_long_running_sets_match_oracle(oracle):
    # a burst of long single-core actions on a pool of 600 cores: more than 448 actions run at once,
    # so the completion heap of the estimates outgrows the warp's shared-memory tree
    pools = (Pool(POOL_CPU, 600, 60),)
    S, N = 4, 1400
    rng = np.random.default_rng(17)
    elastic = rng.random((S, N)) < 0.3
    a = dict(pool=np.zeros((S, N), np.uint8), unit=np.ones((S, N), np.uint8),
             level_mask=np.where(elastic, 0xB, 1).astype(np.uint32),
             s_us=rng.integers(200_000, 900_000, (S, N)).astype(np.int64),
             p_us=np.where(elastic, rng.integers(0, 2_000_000, (S, N)), 0).astype(np.int64),
             arrival_us=np.cumsum(rng.integers(0, 600, (S, N)), axis=1).astype(np.int64),
             n_actions=np.full(S, N, np.int32), gpu_busy=None)
    o = oracle.replay_trace(pools, a, depth=2, round_us=10_000, max_rounds=600)
    g = gpu_replay(pools, a, 2, 10_000, 600)
    assert_same(o, g)
    assert o["occupancy"][:, :, 0].max() > 448 and np.all(o["n_selected"] == N)


STATES = {
    # domains of several mask words, more nodes than lanes
    "wide": ((Pool(POOL_CPU, 900, 300), Pool(POOL_GPU, 320, 8)), 10_000, 1.0),
    # one core per domain: every grant of more spans domains, more domains than lanes
    "spanning": ((Pool(POOL_CPU, 40, 1), Pool(POOL_GPU, 6, 2), Pool(POOL_CPU, 33, 11)), 10_000, 1.0),
    # live state in global memory; a window shorter than a round, a concurrency limit
    "global": ((Pool(POOL_CPU, 6000, 60), Pool(POOL_API, 3, 0, 4_000), Pool(POOL_API, 4, 0, 0), Pool(POOL_GPU, 16, 4)), 10_000, 1.0),
    # times beyond 32 bits: a step between two candidates that has to be decided exactly
    "long": ((Pool(POOL_CPU, 6, 3), Pool(POOL_GPU, 8, 8)), 4_000_000, 2e4),
    # round lengths around the ones whose reciprocal is used
    "round": ((Pool(POOL_CPU, 24, 8), Pool(POOL_GPU, 8, 8)), (1 << 22) - 1, 20.0),
    "rounds": ((Pool(POOL_CPU, 24, 8), Pool(POOL_GPU, 8, 8)), 1 << 22, 20.0),
}


@pytest.mark.parametrize("name", STATES)
def test_replay_state_layouts_match_oracle(oracle, name):
    pools, round_us, scale = STATES[name]
    w, a = random_round(sum(map(ord, name)), 12, 150, pools, small_durations=0.1, busy_fraction=0.2, max_mult=6)
    a["s_us"] = (a["s_us"] * scale).astype(np.int64)
    a["p_us"] = (a["p_us"] * scale).astype(np.int64)
    a["level_mask"] |= 1                            # (no head of the queue that never fits)
    rng = np.random.default_rng(len(name))
    a["arrival_us"] = np.cumsum(rng.integers(0, int(6000 * scale), a["pool"].shape), axis=1).astype(np.int64)
    for max_rounds in (3000, 60):                   # (60: cut off with actions waiting and running)
        o = oracle.replay_trace(pools, a, depth=2, round_us=round_us, max_rounds=max_rounds)
        assert_same(o, gpu_replay(pools, a, 2, round_us, max_rounds))
    assert o["n_selected"].sum() > 0


@pytest.mark.parametrize("policy", [0, 1])
def test_grants_of_calls_in_bursts_match_oracle(oracle, policy):
    # a quota and a concurrency pool, up to 90 calls a burst: many of a round are granted at once, 32 at a time, and every
    # offset is what was in use before; bursts of one and two elastic calls among them
    import torch
    from paper_2603_13019_b200 import binding
    pools = (Pool(POOL_API, 120, 0, 50_000), Pool(POOL_API, 90, 0, 0), Pool(POOL_CPU, 8, 4))
    S, N = 8, 600
    rng = np.random.default_rng(40 + policy)
    burst = np.stack([np.repeat(np.arange(N), rng.choice([1, 2, 40, 90], N))[:N] for _ in range(S)])
    a = dict(pool=rng.choice(3, (S, N), p=[0.5, 0.45, 0.05]).astype(np.uint8), unit=rng.integers(1, 4, (S, N)).astype(np.uint8),
             level_mask=np.where((rng.random((S, N)) < 0.5) | (burst % 2 == 0), 1, 0b1011).astype(np.uint32),
             s_us=rng.integers(0, 30_000, (S, N)), p_us=rng.integers(0, 60_000, (S, N)), arrival_us=burst * 7_000,
             n_actions=np.full(S, N, np.int32), gpu_busy=None)
    o = oracle.replay_trace(pools, a, round_us=10_000, max_rounds=3000, policy=policy)
    rnd = binding.Round(S, N, pools, round_us=10_000, max_rounds=3000)
    g = rnd.replay_trace(binding.to_device(a), policy=policy)
    torch.cuda.synchronize()
    assert_same(o, {k: v.cpu().numpy() for k, v in g.items()})
    assert np.all(o["n_selected"] == N) and (o["place_off"][a["pool"] == 0] > 40).any()
    rnd.destroy()


def test_rounds_of_different_sizes_replay_from_two_threads(oracle):
    # their replays take about 110 KB and 25 KB of shared memory per block of the same kernel; few actions, so that the host
    # calls set the pace
    import threading
    import torch
    from paper_2603_13019_b200 import binding
    jobs = []
    for N, pools in ((2000, (Pool(POOL_CPU, 24, 8),)), (32, (Pool(POOL_CPU, 6, 3),))):
        w, a = random_round(N, 1, N, pools, small_durations=0.2, max_mult=4)
        a["arrival_us"] = np.cumsum(np.random.default_rng(N).integers(0, 6000, a["pool"].shape), axis=1).astype(np.int64)
        a["n_actions"][:] = 1
        rnd = binding.Round(1, N, pools, round_us=10_000, max_rounds=4)
        jobs.append((rnd, binding.to_device(a), rnd.new_result(replay=True), torch.cuda.Stream(),
                     oracle.replay_trace(pools, a, depth=2, round_us=10_000, max_rounds=4)))
    torch.cuda.synchronize()
    failed = []

    def work(rnd, dev, out, stream, want):
        call, args = rnd._lib.tangram_replay_trace, (rnd._h, rnd._actions(dev), rnd._result(out), rnd._stream(stream))
        for k in range(300):
            failed.extend(filter(None, [call(*args) for _ in range(64)]))    # (a loop that is mostly in the library)
            stream.synchronize()
    threads = [threading.Thread(target=work, args=j) for j in jobs]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    torch.cuda.synchronize()
    assert not failed, (len(failed), failed[0])
    for rnd, _, out, _, want in jobs:
        assert_same(want, {k: v.cpu().numpy() for k, v in out.items()})
        rnd.destroy()


def test_first_replay_of_a_round_can_be_captured(oracle):
    import torch
    from paper_2603_13019_b200 import binding
    pools = POOLSETS[0]
    w, a = random_round(77, 3, 60, pools, small_durations=0.2, max_mult=4)
    a["arrival_us"] = np.cumsum(np.random.default_rng(7).integers(0, 6000, a["pool"].shape), axis=1).astype(np.int64)
    rnd, dev = binding.Round(3, 60, pools, round_us=10_000, max_rounds=300), binding.to_device(a)
    out, graph = rnd.new_result(replay=True), torch.cuda.CUDAGraph()
    torch.cuda.synchronize()
    with torch.cuda.graph(graph):
        rnd.replay_trace(dev, out)
    graph.replay()
    torch.cuda.synchronize()
    assert_same(oracle.replay_trace(pools, a, depth=2, round_us=10_000, max_rounds=300), {k: v.cpu().numpy() for k, v in out.items()})
    rnd.destroy()


@pytest.mark.parametrize("cores,group", [(2700, 60), (6000, 60)])
@pytest.mark.parametrize("policy", [0, 2])
def test_running_sets_in_global_memory_match_oracle(oracle, cores, group, policy):
    # a block's shared memory has no room for the 4000 actions that may run here, nor for more than 1600 that wait (most of
    # them do, behind GPUs that are taken); live state in shared and in global memory, with and without a sorted queue
    import torch
    from paper_2603_13019_b200 import binding
    pools = (Pool(POOL_CPU, cores, group), Pool(POOL_API, 1500, 0, 3_000_000), Pool(POOL_GPU, 32, 8))
    S, N = 3, 4000
    rng = np.random.default_rng(cores + policy)
    elastic = rng.random((S, N)) < 0.02
    pool = rng.choice(3, (S, N), p=[0.7, 0.28, 0.02]).astype(np.uint8)
    a = dict(pool=pool, unit=np.where(pool == 0, rng.integers(1, 4, (S, N)), 1).astype(np.uint8),
             level_mask=np.where(elastic, 0xB, 1).astype(np.uint32), s_us=rng.integers(200_000, 2_500_000, (S, N)).astype(np.int64),
             p_us=np.where(elastic, rng.integers(0, 900_000, (S, N)), 0).astype(np.int64),
             arrival_us=np.cumsum(rng.integers(0, 400, (S, N)), axis=1).astype(np.int64), n_actions=np.full(S, N, np.int32), gpu_busy=None)
    o = oracle.replay_trace(pools, a, round_us=10_000, max_rounds=2500, policy=policy)
    rnd = binding.Round(S, N, pools, round_us=10_000, max_rounds=2500)
    g = rnd.replay_trace(binding.to_device(a), policy=policy)
    torch.cuda.synchronize()
    assert_same(o, {k: v.cpu().numpy() for k, v in g.items()})
    assert np.all(o["n_selected"] == N)
    rnd.destroy()


@pytest.mark.parametrize("cores", [60, 300, 1500])
@pytest.mark.parametrize("policy", [0, 1])
def test_replays_of_many_scenarios_match_oracle(oracle, cores, policy):
    # 1160 scenarios, eight blocks on an SM: running actions and live state in shared memory, the state only, neither; up to
    # 300 actions wait, more than such a block keeps in shared memory (160 at most)
    import torch
    from paper_2603_13019_b200 import binding
    pools = (Pool(POOL_CPU, cores, 60), Pool(POOL_GPU, 8, 4))
    S, N, copies = 4, 300, 290
    w, a = random_round(cores + policy, S, N, pools, small_durations=0.1, max_mult=6)
    a["level_mask"] |= 1
    a["arrival_us"] = np.cumsum(np.random.default_rng(cores).integers(0, 200, (S, N)), axis=1).astype(np.int64)
    o = oracle.replay_trace(pools, a, round_us=10_000, max_rounds=1000, policy=policy)
    rnd = binding.Round(S * copies, N, pools, round_us=10_000, max_rounds=1000)
    many = {k: None if v is None else np.tile(v, (copies,) + (1,) * (v.ndim - 1)) for k, v in a.items()}
    g = rnd.replay_trace(binding.to_device(many), policy=policy)
    torch.cuda.synchronize()
    assert_same({k: np.tile(o[k], (copies,) + (1,) * (o[k].ndim - 1)) for k in KEYS}, {k: v.cpu().numpy() for k, v in g.items()})
    assert o["n_selected"].sum() > 0 and np.all(o["status"] == 0)
    rnd.destroy()


def test_running_and_candidates_around_256_match_oracle(oracle):
    # up to 270 one-core actions run; a few elastic ones are decided beside them all the time, with few cores to spare
    pools = (Pool(POOL_CPU, 270, 270),)
    S, N = 4, 1500
    rng = np.random.default_rng(256)
    elastic = rng.random((S, N)) < 0.4
    a = dict(pool=np.zeros((S, N), np.uint8), unit=np.ones((S, N), np.uint8), level_mask=np.where(elastic, 0xB, 1).astype(np.uint32),
             s_us=np.where(elastic, rng.integers(0, 20_000, (S, N)), rng.integers(0, 2_500_000, (S, N))),
             p_us=np.where(elastic, rng.integers(0, 400_000, (S, N)), 0), arrival_us=np.cumsum(rng.integers(0, 4_500, (S, N)), axis=1),
             n_actions=np.full(S, N, np.int32), gpu_busy=None)
    o = oracle.replay_trace(pools, a, depth=2, round_us=10_000, max_rounds=3000)
    assert_same(o, gpu_replay(pools, a, 2, 10_000, 3000))
    busy = o["occupancy"][:, :, 0]
    assert np.all(o["n_selected"] == N) and (busy > 258).sum() > 100 and ((busy > 200) & (busy < 254)).sum() > 100


@pytest.mark.parametrize("policy", [0, 1, 2])
@pytest.mark.parametrize("scenarios", [2, 1160])
def test_queues_that_stay_long_match_oracle(oracle, policy, scenarios):
    # actions arrive in bursts, faster than they run, more than a block keeps in shared memory: the part of the queue in global memory moves on, is drained and
    # fills again; evictions leave gaps in the prefix; a call for most of a concurrency pool holds long prefixes up
    import torch
    from paper_2603_13019_b200 import binding
    pools = (Pool(POOL_CPU, 48, 16), Pool(POOL_API, 40, 0, 0), Pool(POOL_GPU, 8, 8))
    S, N = 2, 2600
    w, a = random_round(60 + policy, S, N, pools, ragged=False, max_mult=4, small_durations=0.5, inelastic=0.5)
    a["level_mask"] |= 1
    a["unit"] = np.where((a["pool"] == 1) & (np.random.default_rng(1).random((S, N)) < 0.01), 38, a["unit"]).astype(np.uint8)
    gap = np.where(np.arange(N) % 1300 < 1200, 40, 90_000)
    a["arrival_us"] = np.cumsum(np.random.default_rng(2).integers(0, gap, (S, N)), axis=1).astype(np.int64)
    o = oracle.replay_trace(pools, a, round_us=10_000, max_rounds=9000, policy=policy)
    copies = scenarios // S
    rnd = binding.Round(scenarios, N, pools, round_us=10_000, max_rounds=9000)
    many = {k: None if v is None else np.tile(v, (copies,) + (1,) * (v.ndim - 1)) for k, v in a.items()}
    out = rnd.replay_trace(binding.to_device(many), policy=policy)
    torch.cuda.synchronize()
    for k in KEYS:
        g = out[k].cpu().numpy()
        assert np.array_equal(o[k], g[:S]) and np.array_equal(g, np.tile(g[:S], (copies,) + (1,) * (g.ndim - 1))), k
    assert np.all(o["status"] == 0) and np.all(o["n_selected"] > 2500)
    rnd.destroy()
