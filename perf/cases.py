"""Cases of the NetKV scoring path: what a scheduler that uses this library has it do.

A case is one pass through the public one-step API (``pipeline.Scorer``) over inputs that
are made on the GPU from a seed: a cluster tree, telemetry rows, request streams with
block-hash chains, and decode caches that hold prefixes of the same shared roots.  The
distributions are those of the workloads in ``synth``: lognormal lengths and outputs,
Poisson arrivals, roots shared by a uniform fraction of a request, telemetry read from
rows refreshed every 100 ms.

Kinds of pass (``kind``):

- ``step``     prefix match and greedy of a batch of streams against resident caches;
- ``host``     the same from pinned host buffers, results read back to the host;
- ``refresh``  the cache index rebuilt from key lists, then a batch matched against it;
- ``evolving`` LRU caches set from key lists, hits and greedy in one walk that updates
               them, and the caches it leaves;
- ``oracle``   the network cost matrix and level bottlenecks of telemetry snapshots.
"""
from __future__ import annotations

import math
from collections import OrderedDict

import numpy as np
import torch

from paper_2606_03910_gb300 import netkv
from paper_2606_03910_gb300.pipeline import Scorer, StepInputs, weights_tensor

TIER_BW = (900e9, 400e9, 200e9, 100e9)   # bytes/s per level
TIER_LAT = (1e-6, 3e-6, 6e-6, 10e-6)     # seconds per tier
BYTES_PER_TOKEN = 81_920                 # Llama-3-70B fp16 at TP=4, per shard
CAP_TOKENS = 549_316                     # 45 GB of free HBM per decode
THETA = float(np.float32(1e-6))          # seconds of queueing per active token
KV_BYTES = 10e9                          # payload of the cost matrix
TBT_US = 13_000                          # time between tokens
INFLIGHT_CAP = 16
LOAD_MODEL = dict(t_a_s=float(np.float32(0.012)), t_b_s=float(np.float32(0.0004)), beta_max=64,
                  m_min_bytes=10 ** 9, m0_bytes=45 * 10 ** 9)
GROUP = 64                               # decodes per cache index

_BASE = dict(kind="step", fanout="1,2,2,4", roles="segregated", streams=1, requests=1000,
             rate=5.0, tokens=8192, max_tokens=131_072, fixed=False, roots=50, root_min=8192,
             root_max=8192, share="frac", keys=200_000, shared=False, greedy="fused",
             telemetry="links", snapshots=0)


def _case(name=None, **kw):
    c = dict(_BASE, **kw)
    return dict(c, name=name) if name else c


def listed():
    tree = dict(fanout="1,8,8,80", roles="mod5", shared=True, rate=400.0)
    return [
        # one arriving request of a 64-GPU cluster: the latency a router adds to a request
        _case("one_decision", requests=1),
        # a 64-GPU cluster's trace of 1,000 requests, level bottlenecks built first
        _case("single_stream", greedy="plain"),
        # 1,024 independent 64-GPU clusters side by side: weight sweeps, fleets of clusters
        _case("replicas", streams=1024),
        # a smaller fleet whose requests arrive in host memory and whose results go back
        _case("host_replicas", kind="host", streams=32),
        # one large cluster of 4,096 decodes, 16 scheduling streams over shared caches
        _case("large_cluster", **dict(tree, streams=16, requests=2000)),
        # prefix-heavy long context: 131,072-token requests over 8 shared roots, 1,024 decodes
        _case("long_context", fanout="1,8,8,20", roles="mod5", shared=True, rate=5.0, streams=64,
              requests=128, tokens=131_072, fixed=True, roots=8, root_min=256, root_max=7680,
              share="root", keys=65_536),
        # a ragged mid-size pool (262 decodes) under the queue and batch model, per-tier maps
        _case("load_model", fanout="3,5,5,7", roles="alternate", shared=True, rate=60.0,
              streams=24, requests=700, tokens=4096, keys=50_000, greedy="load",
              telemetry="tiers"),
        # self-contention on a fleet of 64-GPU clusters with directed links
        _case("self_contention", streams=256, greedy="inflight", telemetry="directed"),
        # caches that change with every dispatch, from key lists to the caches they leave
        _case("evolving_caches", kind="evolving", streams=32, requests=300, keys=60_000),
        # one telemetry refresh of a 2,048 x 8,192 cost matrix
        _case("oracle_refresh", kind="oracle", fanout="1,8,8,160", roles="mod5", snapshots=1),
        # the cost matrices of a trace of snapshots (sensitivity sweeps)
        _case("oracle_sweep", kind="oracle", fanout="1,8,8,160", roles="mod5", snapshots=32),
        # the cache index of 256 decodes rebuilt from their key lists, 4,096 requests matched
        _case("index_refresh", kind="refresh", fanout="1,8,8,5", roles="mod5", shared=True,
              rate=100.0, streams=4, requests=1024, keys=50_000, root_min=4096, root_max=4096),
    ]


# ---------------------------------------------------------------- draws
def _log_int(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def _tree(rng, d_lo, d_hi):
    """A random tree whose decode count lies in [d_lo, d_hi]."""
    while True:
        roles = rng.choice(["segregated", "mod5", "alternate"])
        want = _log_int(rng, d_lo, d_hi)
        f0, f1, f2 = rng.choice([1, 1, 1, 2, 3]), rng.randint(1, 8), rng.randint(2, 8)
        n = want * (1.25 if roles == "mod5" else 2.0)
        f3 = max(1, int(round(n / (f0 * f1 * f2))))
        c = dict(fanout="%d,%d,%d,%d" % (f0, f1, f2, f3), roles=roles)
        role = _roles(c)
        D = int(role.sum())
        if d_lo <= D <= d_hi and D < len(role):
            return c, D


def draw(rng):
    kind = rng.choice(["step"] * 6 + ["oracle", "refresh", "host", "evolving"])
    if kind == "oracle":
        tree, D = _tree(rng, 8, 8192)
        P = len(_roles(tree)) - D
        return _case(kind=kind, telemetry=rng.choice(["links", "links", "directed", "tiers"]),
                     snapshots=_log_int(rng, 1, max(1, min(2000, 2 ** 29 // (P * D)))), **tree)
    small = rng.random() < 0.5
    wide = {"evolving": 300, "refresh": 1024}.get(kind, 4096)
    tree, D = _tree(rng, 3, 16) if small else _tree(rng, 17, wide)
    c = dict(tree, kind=kind, rate=round(0.1 * D * math.exp(rng.uniform(0, 2)), 3),
             tokens=_log_int(rng, 1024, 16_384), roots=rng.randint(4, 60))
    c["root_min"] = c["root_max"] = rng.choice([1024, 4096, 8192])
    c["telemetry"] = rng.choice(["links", "links", "directed", "tiers"])
    c["greedy"] = rng.choice(["fused", "plain", "inflight", "load"])
    if c["greedy"] == "fused":
        c["telemetry"] = "links"
    if kind == "evolving":
        c["greedy"] = "plain"
        c["keys"] = _log_int(rng, 10_000, 100_000)
        c["streams"] = _log_int(rng, 1, max(1, min(64, 256 // D)))
        c["requests"] = _log_int(rng, 10, 300)
        return _case(**c)
    c["shared"] = bool(D > 64 or rng.random() < 0.3)
    c["keys"] = _log_int(rng, 10_000, max(20_000, min(200_000, 2 ** 28 // D)))
    if kind == "refresh":
        c["keys"] = _log_int(rng, 10_000, max(10_001, min(200_000, 2 ** 23 // D)))
    own = 256 if D <= 16 else 16                    # streams with an index of their own
    c["streams"] = _log_int(rng, 1, 256 if c["shared"] else own)
    most = min(2 ** 17, 2 ** 26 // D, 2 ** 17 * 8192 // c["tokens"]) // c["streams"]
    c["requests"] = _log_int(rng, 1, max(2, min(2000, most)))
    if kind == "host":
        c["requests"] = max(1, min(c["requests"], 32_000 // c["streams"]))
    return _case(**c)


# ---------------------------------------------------------------- inputs
_M1, _M2, _G = (np.uint64(x).astype(np.int64).item() for x in
                (0xBF58476D1CE4E5B9, 0x94D049BB133111EB, 0x9E3779B97F4A7C15))


def _mix(z):
    """SplitMix64's output function on int64 bits (logical shifts)."""
    z = (z ^ ((z >> 30) & ((1 << 34) - 1))) * _M1
    z = (z ^ ((z >> 27) & ((1 << 37) - 1))) * _M2
    return z ^ ((z >> 31) & ((1 << 33) - 1))


def _rows(key_a, key_b, split, lens, out):
    """Rows of block hashes, one after another: block j of row i is a function of
    (key_a[i] where j < split[i], else key_b[i], j)."""
    ends = torch.cumsum(lens, 0)
    total, i, n = int(ends[-1]), 0, len(lens)
    marks = torch.arange(1, total // (1 << 25) + 2, device=lens.device) * (1 << 25)
    cuts = sorted(set(torch.searchsorted(ends, marks, right=True).tolist()) | {n})
    for j in cuts:
        j = min(j, n)
        if j <= i:
            continue
        ln = lens[i:j]
        base = int(ends[i] - lens[i])
        row = torch.repeat_interleave(torch.arange(j - i, device=lens.device), ln)
        pos = torch.arange(len(row), device=lens.device) - (ends[i:j] - ln - base)[row]
        key = torch.where(pos < split[i:j][row], key_a[i:j][row], key_b[i:j][row])
        h = _mix(key + (pos + 1) * _G)
        out[base:base + len(row)] = torch.where(h == 0, torch.full_like(h, _G), h)
        i = j
    return out


def _fanout(case):
    return [int(x) for x in case["fanout"].split(",")]


def _roles(case):
    f0, f1, f2, f3 = _fanout(case)
    i = np.arange(f0 * f1 * f2 * f3)
    if case["roles"] == "segregated":
        return (((i // (f0 * f1)) % f2) >= f2 // 2).astype(np.uint8)
    if case["roles"] == "mod5":
        return (i % 5 != 0).astype(np.uint8)
    return (i % 2 == 1).astype(np.uint8)


def _n_links(case):
    f0, f1, f2, f3 = _fanout(case)
    return f3 * (1 + f2 * (1 + f1 * (1 + f0)))


def _n_sets(case):
    return 1 if case["shared"] else case["streams"]


def _telemetry(case, n_snap, g):
    def row(n):
        return torch.rand((n_snap, n), generator=g, device="cuda") * 0.9
    if case["telemetry"] == "tiers":
        return row(4), None
    L = _n_links(case)
    return row(L), row(L) if case["telemetry"] == "directed" else None


def _inputs(case, seed):
    """Everything a pass reads, as tensors on the GPU, and what it was built from."""
    dev = torch.device("cuda")
    g = torch.Generator(device=dev).manual_seed(int(seed))
    role = _roles(case)
    D, P = int(role.sum()), int((role == 0).sum())
    S, n = case["streams"], case["requests"]
    R, G, K = S * n, _n_sets(case), case["roots"]

    def uniform(*shape):
        return torch.rand(shape, generator=g, device=dev, dtype=torch.float64)

    def lognormal(median, lo, hi):
        z = torch.randn((S, n), generator=g, device=dev, dtype=torch.float64)
        return (median * torch.exp(z)).round().clamp(lo, hi).long()

    def keys(*shape):
        return torch.randint(-2 ** 63, 2 ** 63 - 1, shape, generator=g, device=dev)

    length = lognormal(case["tokens"], min(512, case["tokens"]), case["max_tokens"])
    if case["fixed"]:
        length = torch.full_like(length, case["tokens"])
    out_tokens = lognormal(256.0, 1, 4096)
    arrival = torch.cumsum((-torch.log1p(-uniform(S, n)) / case["rate"] * 1e6).round().long(), 1)
    depart = arrival + out_tokens * TBT_US
    prefill = torch.randint(0, P, (S, n), generator=g, device=dev)
    root = torch.randint(0, K, (S, n), generator=g, device=dev)
    nb = length // 16
    rl = torch.linspace(case["root_min"], case["root_max"], K, device=dev,
                        dtype=torch.float64).round().long()
    share = torch.floor(0.9 * uniform(S, n) * nb).long() if case["share"] == "frac" else nb
    share = torch.minimum(share, rl[root])
    # events by (time, departures first, request)
    t = torch.cat([depart * 2, arrival * 2 + 1], 1)
    order = torch.sort(t, dim=1, stable=True).indices
    dep = order < n
    code = torch.where(dep, order, order - n) + n * torch.arange(S, device=dev)[:, None]
    events = (code - dep.long() * 2 ** 31).to(torch.int32).reshape(-1)
    # telemetry refreshed every 100 ms and read 50 ms stale
    n_snap = int((n + 4 * math.sqrt(n) + 4) / case["rate"] * 10) + 1  # the trace's length
    snap = ((arrival - 50_000) // 100_000).clamp(0, n_snap - 1)
    if not case["shared"]:
        snap = snap + n_snap * torch.arange(S, device=dev)[:, None]
        n_snap *= S
    util, util_down = _telemetry(case, n_snap, g)
    # decode caches: the first depth blocks of every root, then blocks of no request
    depth = torch.floor(uniform(G, D, K) * (rl + 1)).long()
    tot = depth.sum(2, keepdim=True)
    depth = torch.where(tot > case["keys"], depth * case["keys"] // tot.clamp(min=1), depth)
    root_key, fill_key, tail_key = keys(G, K), keys(G, D), keys(R)
    weight = torch.linspace(0.1, 2.0, 16, device=dev)[
        torch.randint(0, 16, (S, 3), generator=g, device=dev)]
    return dict(D=D, P=P, R=R, role=role, n_snap=n_snap, util=util, util_down=util_down,
                length=length.reshape(-1), prefill=prefill.reshape(-1), root=root.reshape(-1),
                share=share.reshape(-1), nb=nb.reshape(-1), snap=snap.reshape(-1),
                arrival=arrival.reshape(-1), events=events, depth=depth, root_key=root_key,
                fill_key=fill_key, tail_key=tail_key, weight=weight.cpu().numpy(),
                set_of=torch.arange(R, device=dev) // (R if case["shared"] else n))


def _chains(x):
    total = int(x["nb"].sum())
    out = torch.empty(total, dtype=torch.int64, device="cuda")
    return _rows(x["root_key"][x["set_of"], x["root"]], x["tail_key"], x["share"], x["nb"], out)


def _key_lists(case, x, g0, g1):
    """Key lists of table sets [g0, g1): decode by decode, root prefixes then filler."""
    depth = x["depth"][g0:g1]
    fill = case["keys"] - depth.sum(2, keepdim=True)
    lens = torch.cat([depth, fill], 2).reshape(-1)
    key = torch.cat([x["root_key"][g0:g1, None, :].expand(-1, x["D"], -1),
                     x["fill_key"][g0:g1, :, None]], 2).reshape(-1)
    out = torch.empty((g1 - g0) * x["D"] * case["keys"], dtype=torch.int64, device="cuda")
    return _rows(key, key, lens, lens, out)


def _key_offsets(case, lists):
    return torch.arange(lists + 1, device="cuda") * case["keys"]


def _log2_capacity(case, depth):
    """Index size for the most distinct hashes of any group of decodes."""
    most = 0
    for d0 in range(0, depth.shape[1], GROUP):
        part = depth[:, d0:d0 + GROUP]
        distinct = part.max(1).values.sum(1) + (case["keys"] - part.sum(2)).sum(1)
        most = max(most, int(distinct.max()))
    return netkv.index_log2_capacity(most)


def _step_inputs(case, x):
    S, n = case["streams"], case["requests"]
    off = torch.zeros(x["R"] + 1, dtype=torch.int64, device="cuda")
    off[1:] = torch.cumsum(x["nb"], 0)
    sets = [0, x["R"]] if case["shared"] else [n * s for s in range(S + 1)]
    return StepInputs(
        util=x["util"], chains=_chains(x), chain_off=off,
        set_off=torch.tensor(sets, dtype=torch.int32, device="cuda"),
        length=x["length"].to(torch.int32), prefill=x["prefill"].to(torch.int32),
        snap=x["snap"].to(torch.int32), events=x["events"],
        event_off=torch.arange(S + 1, device="cuda") * (2 * n),
        weights=weights_tensor(x["weight"], THETA, CAP_TOKENS, BYTES_PER_TOKEN),
        arrival_us=x["arrival"], util_down=x["util_down"])


def _scorer(case, x, log2_capacity, index=True):
    sc = Scorer(_fanout(case), x["role"], TIER_BW, TIER_LAT, _n_links(case), _n_sets(case),
                log2_capacity, index=index)
    sc.oracle_mode = "tiers" if case["telemetry"] == "tiers" else "links"
    sc.fuse_level_bottlenecks = case["greedy"] == "fused"
    sc.inflight_cap = INFLIGHT_CAP if case["greedy"] == "inflight" else 0
    if case["greedy"] == "load":
        sc.load_model = netkv.LoadModel(reserved=0, **LOAD_MODEL)
    return sc


def prepare(case, seed):
    if case["kind"] == "oracle":
        g = torch.Generator(device="cuda").manual_seed(int(seed))
        role = _roles(case)
        D, P = int(role.sum()), int((role == 0).sum())
        util, down = _telemetry(case, case["snapshots"], g)
        topo = netkv.netkv_topology_create(_fanout(case), role, TIER_BW, TIER_LAT, _n_links(case))
        return dict(case=case, topo=topo, util=util, down=down,
                    C=torch.empty((case["snapshots"], P, D), device="cuda"),
                    UB=torch.empty((case["snapshots"], P + D, 4), device="cuda"),
                    status=torch.zeros(1, dtype=torch.int32, device="cuda"))
    x = _inputs(case, seed)
    if case["kind"] == "evolving":
        sc = _scorer(case, x, 1, index=False)
        sc.lru_setup(case["streams"], case["keys"])
        G = _n_sets(case)
        lists = _key_lists(case, x, 0, G)
        if G < case["streams"]:  # every stream starts from the shared caches
            lists = lists.repeat(case["streams"])
        state = dict(keys=lists, key_off=_key_offsets(case, case["streams"] * x["D"]))
    else:
        sc = _scorer(case, x, _log2_capacity(case, x["depth"]))
        state = {}
        if case["kind"] == "refresh":
            state = dict(keys=_key_lists(case, x, 0, sc.n_sets),
                         key_off=_key_offsets(case, sc.n_sets * x["D"]))
        else:
            per = max(1, (1 << 27) // (x["D"] * case["keys"]))
            for g0 in range(0, sc.n_sets, per):
                g1 = min(sc.n_sets, g0 + per)
                sc.load_caches(_key_lists(case, x, g0, g1), _key_offsets(case, (g1 - g0) * x["D"]),
                               set0=g0, n_sets=g1 - g0)
    inp = _step_inputs(case, x)
    out = sc.alloc_outputs(inp.n_snap, inp.R, inp.n_streams)
    state.update(case=case, sc=sc, x=inp, out=out)
    if case["kind"] == "host":
        fields = {k: v for k, v in vars(inp).items() if isinstance(v, torch.Tensor)}
        state["xh"] = StepInputs(**{k: v.cpu().pin_memory() if isinstance(v, torch.Tensor) else v
                                    for k, v in vars(inp).items()})
        # the chains are read in place from host memory: the device copies are the rest's
        state["x"] = StepInputs(**dict(vars(inp), chains=fields["chains"][:0]))
        state["res"] = {k: torch.empty_like(getattr(out, k), device="cpu").pin_memory()
                        for k in ("dec", "best", "second", "load_final")}
    return state


# ---------------------------------------------------------------- one pass
def run(state):
    case = state["case"]
    if case["kind"] == "oracle":
        args = (case["snapshots"], KV_BYTES, state["C"], state["UB"], state["status"])
        if case["telemetry"] == "tiers":
            netkv.netkv_oracle_build_tiers(state["topo"], state["util"], *args)
        elif case["telemetry"] == "directed":
            netkv.netkv_oracle_build_directed(state["topo"], state["util"], state["down"], *args)
        else:
            netkv.netkv_oracle_build(state["topo"], state["util"], *args)
        return {k: state[k] for k in ("C", "UB", "status")}
    sc, x, out = state["sc"], state["x"], state["out"]
    if case["kind"] == "refresh":
        sc.load_caches(state["keys"], state["key_off"])
        sc.prefix_match(x, out)
        return dict(M=out.M, status=out.status, build_status=sc.status)
    if case["kind"] == "host":
        sc.step_host(state["xh"], x, out, state["res"], zero_copy=("chains",))
        return dict(state["res"], M=out.M, status=out.status)
    got = {}
    if case["kind"] == "evolving":
        sc.lru_reset(state["keys"], state["key_off"])
        sc.step(x, out)
        got["caches"], got["cache_len"] = sc.lru_export()
    else:
        sc.step(x, out)
    got.update(M=out.M, dec=out.dec, best=out.best, second=out.second,
               load_final=out.load_final, status=out.status)
    if case["greedy"] != "fused":
        got["UB"] = out.UB
    if case["greedy"] == "inflight":
        got["xfer_us"] = out.xfer_us
    if case["greedy"] == "load":
        got["held_final"] = out.held_final
    return got


# ---------------------------------------------------------------- work and tolerance
def work(case):
    role = _roles(case)
    D, P = int(role.sum()), int((role == 0).sum())
    rows = 4 if case["telemetry"] == "tiers" else _n_links(case)
    rows *= 2 if case["telemetry"] == "directed" else 1
    if case["kind"] == "oracle":
        s = case["snapshots"]
        return dict(bytes=4 * s * (P * D + rows + 4 * (P + D)), flops=2 * s * P * D)
    R = case["streams"] * case["requests"]
    blocks = (case["tokens"] if case["fixed"] else 1.55 * case["tokens"]) / 16
    # the blocks up to the last decode's first miss
    seen = min(case["root_max"] if case["share"] == "root" else 0.45 * blocks, blocks) + 1
    # the snapshots that arrivals read (at most one a request), each row once
    span = case["requests"] / case["rate"] * 10
    snaps = min(span, case["requests"]) * (1 if case["shared"] else case["streams"])
    keys = 8 * case["keys"] * D
    if case["kind"] == "refresh":
        return dict(bytes=keys * _n_sets(case) + R * (8 * seen + 2 * D),
                    flops=case["keys"] * D * _n_sets(case))
    b = R * (8 * seen + 2 * D + 4 * 5 + 12) + 4 * rows * snaps + 8 * case["streams"] * D
    if case["kind"] == "evolving":  # lists in, lists out, every chain block used once
        b += 2 * keys * case["streams"] + R * 8 * blocks
    return dict(bytes=b, flops=10 * R * D)


def tolerance(case):
    if case["kind"] == "refresh":  # prefix hits are whole numbers
        return "exact"
    if case["kind"] == "oracle":  # against 64 bits: rel 5.8e-8, max 1.5e-7
        return {"rel": 2.5e-7, "max": 6e-7}
    # Single-precision scores.  Two candidates' scores can round to a tie, a decision then
    # goes to another decode, and the loads that follow from it differ: against 64 bits most
    # cases show rel 6e-8 and no such decision, fleets of many streams rel 5.6e-4, max 0.066
    # and up to 0.9% of decisions after the first tie.
    return {"rel": 2.2e-3, "max": 0.26, "differ": 0.01}


# ---------------------------------------------------------------- 64-bit results
def _coordinates(case):
    f0, f1, f2, f3 = _fanout(case)
    i = torch.arange(f0 * f1 * f2 * f3, device="cuda")
    N = len(i)
    node, leaf, pod = i // f0, i // (f0 * f1), i // (f0 * f1 * f2)
    links = torch.stack([i, N + node, N + N // f0 + leaf, N + N // f0 + N // (f0 * f1) + pod], 1)
    role = torch.from_numpy(_roles(case)).cuda()
    pre, dec = i[role == 0], i[role == 1]

    def same(v):
        return v[pre][:, None] == v[dec][None, :]
    three = torch.full((len(pre), len(dec)), 3, device="cuda")
    tau = torch.where(same(node), 0, torch.where(same(leaf), 1, torch.where(same(pod), 2, three)))
    return links, role, pre, dec, tau


def _level_bottlenecks(case, util, down, geo):
    """[n, N, 4] float64: the residual bandwidth of an instance's first k + 1 links."""
    links, role = geo[:2]
    bw = torch.tensor(TIER_BW, device="cuda", dtype=torch.float64)
    u = util.double()
    if case["telemetry"] == "tiers":
        return (bw * (1 - u))[:, None, :].expand(-1, len(role), -1)
    u = u[:, links]
    if down is not None:
        u = torch.where((role == 1)[None, :, None], down.double()[:, links], u)
    return torch.cummin(bw * (1 - u), 2).values


def _greedy(case, x, M, UB, geo):
    """Algorithm 1 in 64 bits, every stream one event at a time, side by side: (best,
    second score, decode) of every request."""
    _, _, pre, dec_inst, tau_pd = geo
    S, n, D = case["streams"], case["requests"], x["D"]
    dev, f64 = "cuda", torch.float64
    inf = torch.tensor(math.inf, device=dev, dtype=f64)
    lat = torch.tensor(TIER_LAT, device=dev, dtype=f64)
    w = torch.from_numpy(x["weight"]).to(dev).double()
    greedy = case["greedy"]
    lm = LOAD_MODEL
    load = torch.full((S, D), lm["m0_bytes"] if greedy == "load" else 0, device=dev)
    held = torch.zeros((S, D), device=dev, dtype=torch.int64)
    best = torch.full((x["R"],), math.inf, device=dev, dtype=f64)
    second = best.clone()
    chosen = torch.full((x["R"],), -1, device=dev)
    taken = torch.zeros((x["R"],), device=dev, dtype=torch.int64)
    count = torch.zeros((S, x["P"] * 4), device=dev, dtype=torch.int64)
    never = 2 ** 62
    done = torch.full((S, n), never, device=dev)          # completion of each request
    done_key = torch.zeros((S, n), device=dev, dtype=torch.int64)
    rows = torch.arange(S, device=dev)
    ev = x["events"].long().reshape(S, 2 * n)
    for e in range(2 * n):
        leave = ev[:, e] < 0
        r = ev[:, e] & 0x7FFFFFFF
        gone = leave & (chosen[r] >= 0)
        at = chosen[r].clamp(min=0)
        back = torch.where(gone, taken[r], 0)
        load[rows, at] += back if greedy == "load" else -back
        held[rows, at] -= gone.long()
        l, p, k = x["length"][r], x["prefill"][r], x["snap"][r]
        tau = tau_pd[p]
        ub_p = torch.gather(UB[k, pre[p]], 1, tau)
        ub_d = UB[k[:, None], dec_inst[None, :], tau]
        s_eff = (l[:, None] - 16 * M(r)) * BYTES_PER_TOKEN
        T = s_eff / torch.minimum(ub_p, ub_d)
        if greedy == "inflight":
            now = x["arrival"][r]
            due = (done <= now[:, None]) & ~leave[:, None]
            lower = torch.zeros_like(count).scatter_add_(1, done_key, due.long())
            count = (count - lower).clamp(min=0)
            done = torch.where(due, never, done)
            T = T * (1 + count.gather(1, p[:, None] * 4 + tau))
        T = T + lat[tau]
        miss = s_eff / BYTES_PER_TOKEN / l[:, None]
        if greedy == "load":
            beta = held.clamp(max=lm["beta_max"])
            queue = ((held - beta) - (lm["beta_max"] - beta)).clamp(min=0)
            term = queue * (lm["t_a_s"] + lm["t_b_s"] * beta) + lm["t_a_s"] + \
                lm["t_b_s"] * (beta + 1)
            feasible = load >= s_eff + lm["m_min_bytes"]
        else:
            term = THETA * load
            feasible = load + l[:, None] <= CAP_TOKENS
        score = w[:, :1] * T + w[:, 1:2] * miss + w[:, 2:] * term
        score = torch.where(feasible, score, inf)
        b, d = score.min(1)
        d = (score == b[:, None]).long().argmax(1)          # the lowest rank of a tie
        score[rows, d] = math.inf
        go = ~leave & torch.isfinite(b)
        cost = s_eff[rows, d] if greedy == "load" else l
        load[rows, d] += torch.where(go, -cost if greedy == "load" else cost, 0)
        held[rows, d] += go.long()
        a = r[~leave]
        best[a], second[a] = b[~leave], score.min(1).values[~leave]
        chosen[r[go]], taken[r[go]] = d[go], cost[go]
        if greedy == "inflight":
            key = p * 4 + tau[rows, d]
            bump = go & (count[rows, key] < INFLIGHT_CAP)
            count[rows, key] += bump.long()
            end = now + (T[rows, d] * 1e6).round().long()
            done[rows[go], (r % n)[go]] = end[go]
            done_key[rows[go], (r % n)[go]] = key[go]
    return best, second, chosen.to(torch.int32)


def _evolving(case, x, UB, geo):
    """Algorithm 1 with LRU caches held as ordered dictionaries, oldest block first."""
    _, _, pre, dec_inst, tau_pd = geo
    S, n, D, cap = case["streams"], case["requests"], x["D"], case["keys"]
    lists = _key_lists(case, x, 0, _n_sets(case)).cpu().numpy().reshape(-1, D, cap)
    chains = _chains(x).cpu().numpy()
    off = np.concatenate([[0], np.cumsum(x["nb"].cpu().numpy())])
    UB, pre, dec_inst, tau_pd = (v.cpu().numpy() for v in (UB, pre, dec_inst, tau_pd))
    length, prefill, snap = (x[k].cpu().numpy() for k in ("length", "prefill", "snap"))
    ev = x["events"].cpu().numpy().astype(np.int64).reshape(S, 2 * n)
    w, lat = x["weight"].astype(np.float64), np.array(TIER_LAT)
    best, second, took = np.full(x["R"], np.inf), np.full(x["R"], np.inf), {}
    for s in range(S):
        caches = [OrderedDict.fromkeys(reversed(lists[s % len(lists), d].tolist()))
                  for d in range(D)]
        load, chosen = np.zeros(D, np.int64), {}
        for code in ev[s].tolist():
            r = code & 0x7FFFFFFF
            if code < 0:
                if r in chosen:
                    load[chosen[r]] -= length[r]
                continue
            chain = chains[off[r]:off[r + 1]].tolist()
            M = np.zeros(D, np.int64)
            for d, c in enumerate(caches):
                M[d] = next((i for i, b in enumerate(chain) if b not in c), len(chain))
            tau = tau_pd[prefill[r]]
            bott = np.minimum(UB[snap[r], pre[prefill[r]], tau], UB[snap[r], dec_inst, tau])
            left = length[r] - 16 * M
            score = w[s, 0] * (left * BYTES_PER_TOKEN / bott + lat[tau]) + \
                w[s, 1] * (left / length[r]) + w[s, 2] * (THETA * load)
            score[load + length[r] > CAP_TOKENS] = np.inf
            d = int(score.argmin())
            best[r] = score[d]
            second[r] = np.delete(score, d).min() if D > 1 else np.inf
            if np.isfinite(best[r]):
                chosen[r] = took[r] = d
                load[d] += length[r]
                c = caches[d]
                for b in reversed(chain):
                    c[b] = None
                    c.move_to_end(b)
                while len(c) > cap:
                    c.popitem(last=False)
    dec = np.full(x["R"], -1, np.int32)
    dec[list(took)] = list(took.values())
    return torch.from_numpy(best), torch.from_numpy(second), torch.from_numpy(dec)


def exact(case, seed):
    kind = case["kind"]
    if kind == "refresh":  # whole numbers only
        return None
    geo = _coordinates(case)
    if kind == "oracle":
        g = torch.Generator(device="cuda").manual_seed(int(seed))
        util, down = _telemetry(case, case["snapshots"], g)
        UB = _level_bottlenecks(case, util, down, geo)
        _, _, pre, dec_inst, tau = geo
        lat = torch.tensor(TIER_LAT, device="cuda", dtype=torch.float64)[tau]
        C = torch.empty((len(util), len(pre), len(dec_inst)), device="cuda", dtype=torch.float64)
        for s in range(len(util)):
            bott = torch.minimum(torch.gather(UB[s, pre], 1, tau),
                                 torch.gather(UB[s, dec_inst], 1, tau.T).T)
            C[s] = KV_BYTES / bott + lat
        return dict(C=C, UB=UB.contiguous(), status=None)
    R, D = case["streams"] * case["requests"], int(_roles(case).sum())
    if kind == "evolving":
        hashed = R * (D + 3) * case["tokens"] / 16 + case["streams"] * D * case["keys"] * 3
        if hashed > 1.1e8:
            return None
    elif case["requests"] * max(1e3, case["streams"] * D / 50) > 1e7:
        return None
    x = _inputs(case, seed)
    UB = _level_bottlenecks(case, x["util"], x["util_down"], geo)
    if kind == "evolving":
        best, second, dec = _evolving(case, x, UB, geo)
    else:
        # a request's leading run of cached blocks, by construction of the key lists
        def hits(r):
            cached = x["depth"][x["set_of"][r], :, x["root"][r]]
            return torch.minimum(x["share"][r][:, None], cached)
        best, second, dec = _greedy(case, x, hits, UB, geo)
    got = dict(best=best, second=second, dec=dec)
    if kind in ("step", "evolving") and case["greedy"] != "fused":
        got["UB"] = UB.contiguous()
    return got
