"""Performance cases of the scheduling library: what its users have it do, over the sizes they do it at.

A case is a dict of plain values:
  call      the entry point: round, ordered, pinned, host, static (single rounds), replay, replay_pinned
  cluster   the pools and the mix of actions (CLUSTERS below)
  scenarios, actions   independent scenarios per call, row length of every per-action array
  ragged    queues hold between half and all of `actions` records instead of all of them
  arrivals  single rounds: arrival times are passed, so that the predicted ACT includes the wait so far
  busy      share of the GPUs that earlier work still occupies
  policy    queue order: 0 first come first served, 1 shortest, 2 longest, 3 earliest arrival first

All inputs are drawn on the GPU from the seed, with the distributions of the `workloads` package.
"""
from __future__ import annotations

import math

import torch

from paper_2603_13019_b200 import binding
from paper_2603_13019_b200.binding import POOL_API, POOL_CPU, POOL_GPU, UNIT_GANG, PoolDesc

_CPU_NUMA = 64
_MIXED = dict(sigma_s=1.5, sigma_p=1.5, inelastic=0.20, outliers=0.0)
CLUSTERS = {
    # one machine and one GPU server: code sandboxes and reward models, everything elastic
    "node": dict(pools=(PoolDesc(POOL_CPU, 256, _CPU_NUMA), PoolDesc(POOL_GPU, 8, 8)), mix=(0.5, 0.5), max_level=8,
                 sigma_s=1.0, sigma_p=1.2, inelastic=0.0, outliers=0.0),
    # a rack: 4096 cores, 8 x 8 GPUs, one quota-limited API
    "rack": dict(pools=(PoolDesc(POOL_CPU, 4096, _CPU_NUMA), PoolDesc(POOL_GPU, 64, 8), PoolDesc(POOL_API, 512, 0, 1_000_000)),
                 mix=(0.60, 0.25, 0.15), max_level=16, **_MIXED),
    # a large site: 8192 cores, 16 x 8 GPUs, two API quotas, heavy-tailed durations
    "site": dict(pools=(PoolDesc(POOL_CPU, 8192, _CPU_NUMA), PoolDesc(POOL_GPU, 128, 8), PoolDesc(POOL_API, 1000, 0, 1_000_000),
                        PoolDesc(POOL_API, 200, 0, 1_000_000)),
                 mix=(0.50, 0.25, 0.15, 0.10), max_level=32, sigma_s=2.0, sigma_p=2.0, inelastic=0.35, outliers=0.01),
    # a site whose core actions also ask for memory and some of whose GPU actions take an API token
    "site_memory": dict(pools=(PoolDesc(POOL_CPU, 8192, _CPU_NUMA), PoolDesc(POOL_GPU, 128, 8),
                               PoolDesc(POOL_API, 1000, 0, 1_000_000), PoolDesc(POOL_API, 200, 0, 1_000_000),
                               PoolDesc(POOL_API, 2048, 0, 0)),
                        mix=(0.50, 0.25, 0.15, 0.10, 0.0), max_level=32, sigma_s=2.0, sigma_p=2.0, inelastic=0.35,
                        outliers=0.01, side_costs=2, mem_pool=4, mem_max=32, token_pool=3, token_fraction=0.3),
    # a rack whose GPUs remember two of the service instances they served (24 instances, 0.5 .. 4 s to restore)
    "rack_cache": dict(pools=(PoolDesc(POOL_CPU, 4096, _CPU_NUMA), PoolDesc(POOL_GPU, 64, 8), PoolDesc(POOL_API, 512, 0, 1_000_000)),
                       mix=(0.60, 0.25, 0.15), max_level=16, cache_slots=2, n_services=6, restore=(500_000, 4_000_000),
                       cache_fill=0.67, **_MIXED),
    # reward-model GPUs only: 64 x 8, replicas of chunks of 1 / 2 / 4 / 8
    "gpu_farm": dict(pools=(PoolDesc(POOL_GPU, 512, 8),), sizes=(0.4, 0.3, 0.2, 0.1), max_replicas=4, sigma_s=1.0, sigma_p=1.2),
    # CPU nodes with a scheduler each beside a GPU pool; trajectories live on one node
    "cpu_nodes": dict(pools=tuple(PoolDesc(POOL_CPU, 512, _CPU_NUMA) for _ in range(4)) + (PoolDesc(POOL_GPU, 64, 8),),
                      mix=(0.75, 0.0, 0.0, 0.0, 0.25), max_level=16, mem_max=16, node_mem=20_000, **_MIXED),
    # traces: code executions (Pareto) and elastic reward models on one GPU server, Poisson arrivals
    "trace": dict(pools=(PoolDesc(POOL_CPU, 256, _CPU_NUMA), PoolDesc(POOL_GPU, 8, 8)), rate=50.0, cpu_fraction=0.70,
                  reward="gpu"),
    # traces: code executions and parallelisable reward calculations on one core pool
    "trace_cores": dict(pools=(PoolDesc(POOL_CPU, 256, _CPU_NUMA),), rate=110.0, cpu_fraction=0.80, reward="cores"),
    # traces of trajectories, each of which stays on one of three CPU nodes while it has actions
    "trace_nodes": dict(pools=tuple(PoolDesc(POOL_CPU, 128, _CPU_NUMA) for _ in range(3)) + (PoolDesc(POOL_GPU, 8, 8),),
                        rate=50.0, cpu_fraction=0.70, reward="gpu", mem_max=16, node_mem=600),
}
_ROUND_US = 10_000
_ACTIONS_PER_TRAJECTORY = 4


def _case(name, call, cluster, scenarios, actions, ragged=False, arrivals=False, busy=0.0, policy=0):
    c = dict(call=call, cluster=cluster, scenarios=scenarios, actions=actions, ragged=ragged, arrivals=arrivals, busy=busy,
             policy=policy)
    return dict(c, name=name) if name else c


def listed():
    return [
        # the scheduler's own tick: one cluster, a few dozen pending actions; latency is what the user sees
        _case("round_1x64", "round", "node", 1, 64),
        # the tick of a program that may not allocate device memory
        _case("static_16x500", "static", "rack", 16, 500),
        # a few dozen what-if scenarios of a cluster with per-node CPU schedulers: pin the trajectories, then the round
        _case("pinned_48x300", "pinned", "cpu_nodes", 48, 300, ragged=True, arrivals=True, busy=0.3),
        # batched rounds of a rack
        _case("round_4096x1024", "round", "rack", 4096, 1024),
        # topology-constrained reward-model GPUs, three in ten of them occupied
        _case("topology_1024x2048", "round", "gpu_farm", 1024, 2048, busy=0.3),
        # the largest batch: 67 M pending actions
        _case("round_16384x4096", "round", "site", 16384, 4096),
        # memory and tokens beside the key resource
        _case("cost_vectors_2048x4096", "round", "site_memory", 2048, 4096),
        # placement that prefers GPUs with the service still loaded
        _case("cache_4096x1024", "round", "rack_cache", 4096, 1024),
        # another queue order, ragged queues of an odd length
        _case("shortest_first_3000x2001", "ordered", "site", 3000, 2001, ragged=True, arrivals=True, policy=1),
        # a batch that lives in host memory: copies in and out are part of the call
        _case("host_1500x3000", "host", "site", 1500, 3000, arrivals=True),
        # trace replay: 400 s of arrivals, 10 ms rounds
        _case("replay_256x20000", "replay", "trace", 256, 20000),
        # replay of trajectories that are pinned to CPU nodes on arrival, shortest action first
        _case("replay_pinned_60x4000", "replay_pinned", "trace_nodes", 60, 4000, policy=1),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    call = rng.choice(("round", "round", "round", "round", "ordered", "pinned", "host", "static", "replay", "replay_pinned"))
    if call in ("replay", "replay_pinned"):
        cluster = "trace_nodes" if call == "replay_pinned" else rng.choice(("trace", "trace_cores"))
        # traces of up to the listed lengths; the sorted queues take longer per action
        policy = rng.choice((0, 0, 1, 2))
        most = 4000 if cluster != "trace" else 12000 if policy else 20000
        return _case(None, call, cluster, _log_int(rng, 1, 256), _log_int(rng, 200, most), ragged=rng.random() < 0.3,
                     policy=policy)
    if call == "static":
        return _case(None, call, rng.choice(("node", "rack")), _log_int(rng, 1, 64), _log_int(rng, 64, 1024),
                     ragged=rng.random() < 0.5, arrivals=rng.random() < 0.5, busy=rng.choice((0.0, 0.3)))
    if call == "pinned":
        cluster = "cpu_nodes"
    elif call == "round":
        cluster = rng.choice(("node", "rack", "site", "site_memory", "rack_cache", "gpu_farm"))
    else:
        cluster = rng.choice(("node", "rack", "site"))
    actions = _log_int(rng, 64, 4096)
    total = (1 << 24) if call == "host" else 5 << 23      # records per call at most
    scenarios = _log_int(rng, 1, min(16384 if cluster != "gpu_farm" else 1024, max(1, total // actions)))
    return _case(None, call, cluster, scenarios, actions, ragged=rng.random() < 0.5, arrivals=rng.random() < 0.5,
                 busy=0.3 if cluster == "gpu_farm" else rng.choice((0.0, 0.3)),
                 policy=rng.choice((1, 2, 3)) if call == "ordered" else 0)


# ------------------------------------------------------------------------------------------ inputs
class _Draws:
    """Columns of random [scenarios, actions] fields, drawn in one fixed order from one generator on the GPU."""

    def __init__(self, seed, shape):
        self.gen = torch.Generator(device="cuda")
        self.gen.manual_seed(seed)
        self.shape = shape

    def uniform(self, shape=None):
        return torch.rand(shape or self.shape, generator=self.gen, device="cuda", dtype=torch.float32)

    def integers(self, lo, hi, shape=None, dtype=torch.int64):        # lo .. hi - 1
        return torch.randint(lo, hi, shape or self.shape, generator=self.gen, device="cuda", dtype=dtype)

    def lognormal_us(self, median, sigma):
        v = torch.empty(self.shape, device="cuda", dtype=torch.float32)
        v.log_normal_(math.log(median), sigma, generator=self.gen)
        return v.clamp_(max=float(1 << 40)).to(torch.int64)

    def choose(self, probs):
        edges = torch.tensor([sum(probs[:k + 1]) for k in range(len(probs) - 1)], device="cuda", dtype=torch.float32)
        return torch.bucketize(self.uniform(), edges, out_int32=True, right=True).to(torch.uint8)


def _pow2_mask(max_level):
    return sum(1 << ((1 << k) - 1) for k in range(6) if (1 << k) <= max_level)


def _signed32(v):
    return v - (1 << 32) if v >= 1 << 31 else v


def _mixed(d, c):
    """Pending actions over core, GPU (gang) and quota pools; elastic levels are powers of two."""
    pools = c["pools"]
    pool = d.choose(c["mix"])
    index = pool.long()
    tops = [1 if p.type == POOL_API else min(c["max_level"], 8 if p.type == POOL_GPU else c["max_level"]) for p in pools]
    full = torch.tensor([_signed32(_pow2_mask(t)) for t in tops], device="cuda", dtype=torch.int32)[index]
    n_levels = torch.tensor([int(math.log2(t)) + 1 for t in tops], device="cuda", dtype=torch.int32)[index]
    level = torch.minimum((d.uniform() * n_levels).to(torch.int32), n_levels - 1)          # the level of an inelastic action
    one = torch.tensor([_signed32(1 << ((1 << k) - 1)) for k in range(6)], device="cuda", dtype=torch.int32)[level.long()]
    del level, n_levels
    mask = torch.where(d.uniform() < c["inelastic"], one, full)
    unit = torch.tensor([1 | UNIT_GANG if p.type == POOL_GPU else 1 for p in pools], device="cuda", dtype=torch.uint8)[index]
    del index, one, full
    s, p = d.lognormal_us(20_000.0, c["sigma_s"]), d.lognormal_us(200_000.0, c["sigma_p"])
    if c["outliers"]:
        scale = torch.where(d.uniform() < c["outliers"], 100, 1)
        s, p = (s * scale).clamp_(max=1 << 40), (p * scale).clamp_(max=1 << 40)
    return dict(pool=pool, unit=unit, level_mask=mask, s_us=s, p_us=p)


def _replicas(d, c):
    """Requests for 1 .. max_replicas chunks of 1 / 2 / 4 / 8 GPUs on one GPU pool."""
    unit = torch.tensor([1, 2, 4, 8], device="cuda", dtype=torch.uint8)[d.choose(c["sizes"]).long()]
    return dict(pool=torch.zeros(d.shape, device="cuda", dtype=torch.uint8), unit=unit,
                level_mask=torch.full(d.shape, (1 << c["max_replicas"]) - 1, device="cuda", dtype=torch.int32),
                s_us=d.lognormal_us(20_000.0, c["sigma_s"]), p_us=d.lognormal_us(200_000.0, c["sigma_p"]))


def _trace(d, c):
    """Poisson arrivals of one-core code executions (Pareto 1.3, at least 5 ms) and elastic reward calculations."""
    gap = (-torch.log(d.uniform().clamp_(min=1e-9)) * (1e6 / c["rate"])).to(torch.int64)
    reward = d.uniform() >= c["cpu_fraction"]
    t_exec = (5_000.0 * d.uniform().clamp_(min=1e-9).double() ** (-1.0 / 1.3)).clamp_(max=float(1 << 40)).to(torch.int64)
    nodes = [j for j, p in enumerate(c["pools"]) if p.type == POOL_CPU]
    if c["reward"] == "gpu":                               # 50 .. 800 ms on 1 .. 8 GPUs of one server, a fifth of it serial
        t = d.integers(50_000, 800_000)
        s, pool, unit, mask = t // 5, len(nodes), 1 | UNIT_GANG, _pow2_mask(8)
    else:                                                  # median 4 s on 1 .. 32 cores, a twentieth of it serial
        t = d.lognormal_us(4_000_000.0, 1.0)
        s, pool, unit, mask = t // 20, 0, 1, _signed32(_pow2_mask(32))
    return dict(pool=torch.where(reward, pool, 0).to(torch.uint8), unit=torch.where(reward, unit, 1).to(torch.uint8),
                level_mask=torch.where(reward, mask, 1).to(torch.int32), s_us=torch.where(reward, s, t_exec),
                p_us=torch.where(reward, t - s, 0), arrival_us=torch.cumsum(gap, dim=1))


def _busy_gpus(d, pools, scenarios, share):
    """Every aligned block of 8, 4, 2 and 1 GPUs of a node is taken with one probability; `share` of the GPUs end up busy."""
    nodes = sum(p.capacity // p.group for p in pools if p.type == POOL_GPU)
    if nodes == 0:
        return None
    busy = torch.zeros((scenarios, nodes), device="cuda", dtype=torch.uint8)
    if share > 0.0:
        taken = d.uniform((scenarios, nodes, 15)) < 1.0 - (1.0 - share) ** 0.25
        blocks = [(((1 << z) - 1) << at) for z in (8, 4, 2, 1) for at in range(0, 8, z)]
        for k, bits in enumerate(blocks):
            busy |= taken[:, :, k].to(torch.uint8) * bits
    return busy


def _trajectories(d, c, a, pinned):
    """Consecutive actions of interleaved trajectories; some already live on a node, the last action of each is marked."""
    S, N = d.shape
    T = max(1, N // _ACTIONS_PER_TRAJECTORY)
    nodes = [j for j, p in enumerate(c["pools"]) if p.type == POOL_CPU]
    group = torch.arange(N, device="cuda") // (4 * _ACTIONS_PER_TRAJECTORY)       # four trajectories are in flight at a time
    traj = torch.clamp(group * 4 + d.integers(0, 4), max=T - 1).to(torch.int32)
    mem = d.integers(0, c["mem_max"] + 1, (S, T), dtype=torch.int32)
    last = torch.zeros((S, T), device="cuda", dtype=torch.int64)
    at = torch.arange(N, device="cuda").expand(S, N)
    last.scatter_reduce_(1, traj.long(), at, "amax")
    a["trajectory"] = traj
    a["traj_mem"] = torch.gather(mem, 1, traj.long())
    a["traj_last"] = (torch.gather(last, 1, traj.long()) == at).to(torch.uint8)
    a["traj_node"] = torch.where(d.uniform((S, T)) < pinned, d.integers(0, len(nodes), (S, T)), -1).to(torch.int32)
    a["node_mem_free"] = torch.full((S, len(c["pools"])), c["node_mem"], device="cuda", dtype=torch.int64)


def _extras(d, c, a):
    pool = a["pool"]
    if c.get("side_costs"):
        cpu, gpu = pool == 0, pool == 1
        mem = torch.where(cpu, d.integers(1, c["mem_max"] + 1), 0)
        token = gpu & (d.uniform() < c["token_fraction"])
        a["side_pool"] = torch.stack([torch.where(cpu, c["mem_pool"], 0xFF), torch.where(token, c["token_pool"], 0xFF)]).to(torch.uint8)
        a["side_units"] = torch.stack([mem, token.to(torch.int64)]).to(torch.int16)
    if c.get("cache_slots"):
        S, K = d.shape[0], c["cache_slots"]
        nodes = sum(p.capacity // p.group for p in c["pools"] if p.type == POOL_GPU)
        a["service"] = d.integers(0, c["n_services"], dtype=torch.int16)
        a["restore_us"] = d.integers(*c["restore"])
        # a node's GPUs start with the same instances (what whole-node or aligned runs left behind)
        tag = d.integers(0, c["n_services"], (S, nodes, 1, K)) * 8 + d.integers(0, 4, (S, nodes, 1, K)) + 1
        tag = torch.where(d.uniform((S, nodes, 1, K)) < c["cache_fill"], tag, 0)
        use = -d.integers(0, 1_000_000, (S, nodes, 1, K))
        a["cache_tag"] = tag.to(torch.int32).expand(S, nodes, 8, K).reshape(S, -1).contiguous()
        a["cache_use"] = use.expand(S, nodes, 8, K).reshape(S, -1).contiguous()


def _max_rounds(case, c):
    seconds = case["actions"] / c["rate"]
    return int(seconds * (1.5 if c["reward"] == "gpu" else 3.3) * 1e6 / _ROUND_US) + 1000


def prepare(case, seed):
    c, S, N = CLUSTERS[case["cluster"]], case["scenarios"], case["actions"]
    replay = case["call"].startswith("replay")
    d = _Draws(seed, (S, N))
    a = _trace(d, c) if replay else _replicas(d, c) if "sizes" in c else _mixed(d, c)
    if case["ragged"]:
        a["n_actions"] = d.integers((N + 1) // 2, N + 1, (S,), dtype=torch.int32)
    else:
        a["n_actions"] = torch.full((S,), N, device="cuda", dtype=torch.int32)
    a["gpu_busy"] = _busy_gpus(d, c["pools"], S, case["busy"])
    now = 0
    if not replay:
        a["arrival_us"] = None
        if case["arrivals"]:                               # everything queued within the last ten seconds
            now = 10_000_000
            a["arrival_us"] = torch.sort(d.integers(0, now), dim=1)[0].contiguous()
        _extras(d, c, a)
    if case["call"] in ("pinned", "replay_pinned"):
        _trajectories(d, c, a, 0.0 if replay else 0.5)
    state = dict(case=case, cluster=c, now=now, actions=a)
    if case["call"] == "static":
        wide, narrow = torch.int64, torch.int32            # there is no Round to ask for result tensors
        kinds = dict(alloc_units=narrow, place_node=narrow, place_off=narrow, act_us=wide)
        state["result"] = {k: torch.empty((S, N), dtype=t, device="cuda") for k, t in kinds.items()}
        kinds = dict(total_act_us=wide, n_selected=narrow, status=narrow)
        state["result"].update({k: torch.empty((S,), dtype=t, device="cuda") for k, t in kinds.items()})
        return state
    host = case["call"] == "host"
    if host:
        state["actions"] = {k: None if v is None else v.cpu().pin_memory() for k, v in a.items()}
    state["round"] = binding.Round(S, N, c["pools"], host_buffers=host, round_us=_ROUND_US,
                                   max_rounds=_max_rounds(case, c) if replay else 0,
                                   cache_slots=c.get("cache_slots", 0), side_costs=c.get("side_costs", 0))
    state["result"] = state["round"].new_result(replay=replay)
    torch.cuda.empty_cache()                               # what drawing the inputs took goes back
    return state


def run(state):
    case, a, res, now = state["case"], state["actions"], state["result"], state["now"]
    call = case["call"]
    if call == "static":
        rc = binding.schedule_batch_static(state["cluster"]["pools"], a, res, now_us=now)
        if rc != 0:
            raise RuntimeError(f"schedule_batch_static: {rc}")
        return res
    rnd = state["round"]
    if call in ("round", "host"):
        out = rnd.schedule_batch(a, now, res)
        if "cache_tag" in a:                               # the caches are carried from round to round
            out = dict(out, cache_tag=a["cache_tag"], cache_use=a["cache_use"])
        return out
    if call == "ordered":
        return rnd.schedule_batch_ordered(a, case["policy"], now, res)
    if call == "replay":
        return rnd.replay_trace(a, res, policy=case["policy"])
    # a what-if call: the live pins and free memory stay as they are
    b = dict(a, traj_node=a["traj_node"].clone(), node_mem_free=a["node_mem_free"].clone())
    pins = dict(traj_node=b["traj_node"], node_mem_free=b["node_mem_free"])
    if call == "replay_pinned":
        return dict(rnd.replay_trace_pinned(b, policy=case["policy"], result=res), **pins)
    pin = rnd.pin_trajectories(b)
    out = rnd.schedule_batch(dict(b, pool=pin["pool"], n_actions=pin["n_admitted"]), now, res)
    return dict(out, pool=pin["pool"], n_admitted=pin["n_admitted"], **pins)


def work(case):
    """Every input that the call cannot do without read once, every output written once.  The records (pool 1, unit 1, mask 4,
    s 8, p 8 B) up to the queue's length; the outputs (units, node, offset 4 B each, ACT 8 B) over the whole row."""
    c, S, N = CLUSTERS[case["cluster"]], case["scenarios"], case["actions"]
    replay = case["call"].startswith("replay")
    per_in = 22 + (8 if replay or case["arrivals"] else 0) + 3 * c.get("side_costs", 0) + (10 if c.get("cache_slots") else 0)
    per_out = 20
    per_scenario = 4 + 16                                  # queue length; total, count, status
    nodes = sum(p.capacity // p.group for p in c["pools"] if p.type == POOL_GPU)
    per_scenario += nodes * (1 + 2 * 12 * 8 * c.get("cache_slots", 0))
    if case["call"] in ("pinned", "replay_pinned"):
        per_in += 8 + (1 if replay else 0)
        per_out += 1
        per_scenario += 8 * (N // _ACTIONS_PER_TRAJECTORY) + 16 * len(c["pools"])
    if replay:
        per_scenario += 4 * _max_rounds(case, c) * len(c["pools"]) + 4
    queued = 0.75 * N if case["ragged"] else float(N)
    return {"bytes": S * (per_in * queued + per_out * N + per_scenario), "flops": 0}


def tolerance(case):
    return "exact"                                         # whole microseconds, units and positions
