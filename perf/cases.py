"""Performance cases of the library: the calls an engine makes, from one block to the largest index.

A case is one of these uses of the public entry points (``paper_2608_14624_b200.binding``):

``decide``    what a scheduler step needs before it moves anything: ``observe_invocations`` for the step's
              invocations, then ``select_step`` (victims of both tiers and prefetch candidates) over the block index
``select``    one list alone: ``select_victims`` or ``select_prefetch`` (an engine under memory pressure, a very
              large index)
``score``     ``score_blocks``: the reuse score of every entry (diagnostics, an engine with a policy of its own)
``observe``   a long batch of invocations, then the learner's state read back (warm start from a log, checkpoint)
``survival``  ``exact_survival``: the table of the alternative scorer
``compact``   ``compact_blocks``: scattered blocks moved inside the device
``link``      ``offload_blocks`` / ``prefetch_blocks`` / ``exchange_blocks`` between the pool and the pinned host tier
``step``      the whole scheduler step as one ``step`` call: decisions, compaction and both transfers

The clock moves on with every pass and the invocations come from a long trace, as in an engine.  The clock runs over
a window of 16 steps and the trace repeats after 64 batches, so that the age distribution and the transition model
stay what they are in a live cache however many passes are made.
"""
import math

import numpy as np
import torch

import paper_2608_14624_b200.binding as cs

DEV = "cuda:0"
NOW0 = 100_000
CLOCK_WINDOW = 16
N_BATCHES = 64
MIB = 1 << 20


def listed():
    return [
        # the smallest configuration: 4 agents, 512-block pool and 2,048-block host tier, one invocation per step;
        # launches and host work decide
        dict(name="decide_2560", kind="decide", n=2560, gpu_share=0.2, agents=4, chains=1, events=1, k_victims=32, k_prefetch=64,
             host_victims=True, tokens=True, anchors=True, prefer_copy=0, all_chains=False),
        # the decisions of every scheduler step at the 8B KV shape: 20,000 + 60,000 blocks, 12 agents, 64 sessions
        dict(name="decide_80000", kind="decide", n=80_000, gpu_share=0.25, agents=12, chains=64, events=5, k_victims=256,
             k_prefetch=384, host_victims=True, tokens=True, anchors=True, prefer_copy=0, all_chains=False),
        # metadata scale: an index shared by many workers, 256 agents, long lists, no host-tier victims
        dict(name="decide_1000000", kind="decide", n=1_000_000, gpu_share=0.5, agents=256, chains=16, events=64,
             k_victims=10_000, k_prefetch=2_000, host_victims=False, tokens=True, anchors=True, prefer_copy=0, all_chains=False),
        # the largest index: one victim list, where the metadata no longer fits the L2 cache
        dict(name="victims_64000000", kind="select", n=64_000_000, gpu_share=0.5, agents=256, chains=16, events=64, k=10_000,
             prefetch=False, tier=0, tokens=True, anchors=True, prefer_copy=0),
        # scores of the 8B index, as a monitoring thread or a custom policy reads them; explicit sources
        dict(name="score_80000", kind="score", n=80_000, gpu_share=0.25, agents=12, chains=64, events=5, sources=3, tokens=True),
        # and of the largest one, all bandwidth
        dict(name="score_64000000", kind="score", n=64_000_000, gpu_share=0.5, agents=256, chains=16, events=64, sources=0,
             tokens=True),
        # a day's invocation log replayed into a fresh learner, state exported as for a checkpoint
        dict(name="observe_20000", kind="observe", agents=12, chains=64, events=20_000, warmup=0.05, all_chains=False),
        # the exact scorer's table at the largest agent count the benchmark uses
        dict(name="survival_256", kind="survival", agents=256, chains=16, steps=4),
        # a step's compaction: 256 scattered 2 MiB blocks into a packed staging pool
        dict(name="compact_256", kind="compact", blocks=256, slots=512, layers=32, heads=8, head_dim=128, block_tokens=16,
             elem_bytes=2, src_layout=0, dst_layout=1),
        # one evicted 2 MiB block on its way to the host tier: the latency of the smallest transfer
        dict(name="offload_1", kind="link", off=1, pre=0, slots=64, layers=32, heads=8, head_dim=128, block_tokens=16, elem_bytes=2,
             gpu_layout=0, host_layout=1),
        # both directions of the host link at a step's 2:3 proportion
        dict(name="exchange_170_256", kind="link", off=170, pre=256, slots=512, layers=32, heads=8, head_dim=128, block_tokens=16,
             elem_bytes=2, gpu_layout=0, host_layout=1),
        # the whole step of the smallest configuration: decisions, compaction and both transfers of 512 KiB blocks
        dict(name="step_2560", kind="step", gpu_blocks=512, host_blocks=2048, agents=4, chains=1, events=1, k_victims=32,
             k_prefetch=64, layers=8, heads=8, head_dim=128, block_tokens=16, elem_bytes=2),
    ]


# ---- drawn cases ---------------------------------------------------------------------------------------------------
def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _agents(rng, hi=1024):
    return _log(rng, 2, hi)


def _block_bytes(shape):
    return 2 * shape["layers"] * shape["heads"] * shape["head_dim"] * shape["block_tokens"] * shape["elem_bytes"]


def _shape(rng):
    """A KV shape: grouped-query head counts, 16- or 32-token blocks, bf16 or 8-bit elements."""
    return dict(layers=rng.choice([8, 16, 28, 32, 48, 80]), heads=rng.choice([1, 2, 4, 8]), head_dim=rng.choice([64, 96, 128, 256]),
                block_tokens=rng.choice([16, 16, 32]), elem_bytes=rng.choice([1, 2, 2]))


def draw(rng):
    kind = rng.choice(["decide", "decide", "decide", "decide", "select", "select", "score", "score", "observe", "survival",
                       "compact", "compact", "link", "link", "link", "step"])
    if kind == "decide":
        n = _log(rng, 1_500, 4_000_000)
        return dict(kind=kind, n=n, gpu_share=round(rng.uniform(0.2, 0.6), 3), agents=_agents(rng), chains=_log(rng, 4, 512),
                    events=_log(rng, 1, 256), k_victims=max(1, min(_log(rng, 8, 20_000), n // 16)),
                    k_prefetch=max(1, min(_log(rng, 8, 4_000), n // 16)), host_victims=rng.random() < 0.7,
                    tokens=rng.random() < 0.7, anchors=rng.random() < 0.7, prefer_copy=int(rng.random() < 0.25),
                    all_chains=rng.random() < 0.2)
    if kind == "select":
        n = _log(rng, 2_000, 60_000_000)
        prefetch = rng.random() < 0.4
        return dict(kind=kind, n=n, gpu_share=round(rng.uniform(0.2, 0.6), 3), agents=_agents(rng), chains=_log(rng, 4, 512), events=16,
                    k=max(1, min(_log(rng, 1, 20_000), n // 16)), prefetch=prefetch, tier=1 if prefetch else rng.randrange(2),
                    tokens=rng.random() < 0.7, anchors=rng.random() < 0.7, prefer_copy=int(rng.random() < 0.25))
    if kind == "score":
        return dict(kind=kind, n=_log(rng, 500, 60_000_000), gpu_share=0.25, agents=_agents(rng), chains=_log(rng, 4, 512), events=16,
                    sources=rng.choice([0, 0, 1, 2, 7]), tokens=rng.random() < 0.7)
    if kind == "observe":
        return dict(kind=kind, agents=_agents(rng), chains=_log(rng, 8, 2048), events=_log(rng, 257, 20_000),
                    warmup=rng.choice([0.0, 0.05]), all_chains=rng.random() < 0.2)
    if kind == "survival":
        return dict(kind=kind, agents=_log(rng, 4, 400), chains=16, steps=rng.randint(2, 6))
    shape = _shape(rng)
    while kind == "step" and _block_bytes(shape) > 4 * MIB:
        shape = _shape(rng)
    block = _block_bytes(shape)
    if kind == "compact":
        blocks = min(_log(rng, 1, 1024), max(1, 500 * MIB // block))
        return dict(kind=kind, blocks=blocks, slots=2 * blocks + 3, src_layout=rng.randrange(2), dst_layout=rng.randrange(2), **shape)
    if kind == "link":
        way = rng.choice(["off", "pre", "both"])
        total = min(_log(rng, 2, 1024), max(2, 500 * MIB // block))
        share = {"off": 1.0, "pre": 0.0, "both": rng.uniform(0.2, 0.8)}[way]
        off = min(max(int(round(total * share)), 0), total) if way != "both" else min(max(int(round(total * share)), 1), total - 1)
        return dict(kind=kind, off=off, pre=total - off, slots=total + 5, gpu_layout=rng.randrange(2), host_layout=rng.randrange(2), **shape)
    gpu_blocks = max(64, min(_log(rng, 128, 4096), 512 * MIB // block))
    k_victims = max(1, min(_log(rng, 4, 128), gpu_blocks // 8))
    return dict(kind="step", gpu_blocks=gpu_blocks, host_blocks=gpu_blocks + _log(rng, 16, max(17, gpu_blocks)), agents=_agents(rng, 64),
                chains=_log(rng, 1, 64), events=_log(rng, 1, 32), k_victims=k_victims, k_prefetch=max(1, min(_log(rng, 4, 128), gpu_blocks // 8)),
                **shape)


# ---- inputs --------------------------------------------------------------------------------------------------------
def _gen(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(seed)
    return g


def _ints(g, lo, hi, n, dtype):
    return torch.randint(lo, hi, (n,), generator=g, device=DEV, dtype=torch.int32).to(dtype)


def _trace(rng, n_agents, n_chains, n_events):
    """Invocations of live sessions, one per chain, each following a sparse (or, for few agents, Dirichlet) transition
    matrix; a session ends after about eight invocations.  Returns chain u32 and agent u16 arrays."""
    if n_agents <= 16:
        p = rng.dirichlet(np.full(n_agents, 0.5), size=n_agents)
        nxt = None
    else:
        nnz = 8 if n_agents > 64 else 4
        nxt = (np.arange(n_agents)[:, None] + 1 + np.argsort(rng.random((n_agents, n_agents - 1)), axis=1)[:, :nnz]) % n_agents
        p = rng.dirichlet(np.ones(nnz), size=n_agents)
    cum = np.cumsum(p, axis=1)
    live = min(n_chains, max(1, n_events))
    rounds = -(-n_events // live)
    cur = rng.integers(0, n_agents, size=live)
    chain = np.empty((rounds, live), np.int32)
    agent = np.empty((rounds, live), np.int16)
    for t in range(rounds):
        pick = np.minimum((cum[cur] < rng.random(live)[:, None]).sum(axis=1), cum.shape[1] - 1)
        follow = pick if nxt is None else nxt[cur, pick]
        cur = np.where(rng.random(live) < 0.125, rng.integers(0, n_agents, size=live), follow)
        chain[t] = rng.permutation(live) if live > 1 else 0
        agent[t] = cur[chain[t]]
    return chain.reshape(-1)[:n_events].copy(), agent.reshape(-1)[:n_events].copy()


def _index(g, n, n_agents, gpu_share, tokens, anchors, block_tokens=16, gpu_blocks=None, free_slots=0):
    """Metadata of n cached blocks: references on 10 %, 2 % pinned, 30 % with a copy on the other tier; half of the ages
    below 64 steps, 30 % up to 1,024, the rest up to 65,536; 95 % full blocks.  Ids [0, gpu_blocks) are the GPU tier."""
    u = torch.rand(n, generator=g, device=DEV)
    age = torch.where(u < 0.5, _ints(g, 0, 64, n, torch.int32),
                      torch.where(u < 0.8, _ints(g, 64, 1024, n, torch.int32), _ints(g, 1024, 65536, n, torch.int32)))
    last_access = NOW0 - age
    del u, age
    ref = torch.where(torch.rand(n, generator=g, device=DEV) < 0.9, 0, _ints(g, 1, 5, n, torch.uint8)).to(torch.uint8)
    flags = (torch.rand(n, generator=g, device=DEV) < 0.98).to(torch.uint8) * cs.CS_FLAG_VALID
    flags |= (torch.rand(n, generator=g, device=DEV) < 0.02).to(torch.uint8) * cs.CS_FLAG_PINNED
    flags |= (torch.rand(n, generator=g, device=DEV) < 0.30).to(torch.uint8) * cs.CS_FLAG_OTHER_COPY
    flags[int(round(n * gpu_share)) if gpu_blocks is None else gpu_blocks:] |= cs.CS_FLAG_TIER_HOST
    if free_slots:
        flags[:free_slots] = 0                                    # GPU slots that hold nothing: prefetched blocks go there
    n_tokens = None
    if tokens:
        full = torch.rand(n, generator=g, device=DEV) < 0.95
        n_tokens = torch.where(full, block_tokens, _ints(g, 1, max(2, block_tokens), n, torch.uint8)).to(torch.uint8)
    return cs.DeviceIndex(agent=_ints(g, 0, n_agents, n, torch.int16), depth=_ints(g, 0, 512, n, torch.int16), ref_count=ref, flags=flags,
                          last_access=last_access, n_tokens=n_tokens,
                          anchor_blocks=_ints(g, 128, 385, n_agents, torch.int16) if anchors else None)


def _learner(case, seed, max_blocks, block_tokens=16):
    """A context whose learner has seen a history, and the batches the passes will feed it."""
    A, chains, events = case["agents"], case["chains"], case.get("events", 1)
    rng = np.random.default_rng([seed, 1])
    history = min(100 * A, 4_000 * min(chains, 64), 50_000)
    chain, agent = _trace(rng, A, chains, history + N_BATCHES * events)
    chain, agent = torch.from_numpy(chain).to(DEV), torch.from_numpy(agent).to(DEV)
    c = cs.CacheScout(cs.make_params(A, n_chains=chains, max_blocks=max_blocks, block_tokens=block_tokens,
                                     prefer_other_copy=case.get("prefer_copy", 0)), DEV)
    if case.get("all_chains"):
        cs.cs_set_survival_sources(c.ctx, cs.CS_SOURCES_ALL_CHAINS)
    for at in range(0, history, 256):
        c.observe_invocations(chain[at:min(at + 256, history)], agent[at:min(at + 256, history)])
    batches = [(chain[at:at + events], agent[at:at + events]) for at in range(history, history + N_BATCHES * events, events)]
    return c, batches


def _pool(g, slots, case, layout, host=False, first_id=0):
    """A paged pool of bf16 N(0, 1) values (raw bytes to the mover), pinned when it is the host tier."""
    words = slots * _block_bytes(case) // 2
    buf = torch.empty(words, dtype=torch.bfloat16, device=DEV).normal_(generator=g)
    if host:
        pinned = torch.empty(words, dtype=torch.bfloat16, pin_memory=True)
        pinned.copy_(buf)
        buf = pinned
    return cs.KVPool(buf, slots, layout, case["layers"], case["heads"], case["head_dim"], case["block_tokens"], case["elem_bytes"], first_id)


def _slots(g, total, n):
    return torch.randperm(total, generator=g, device=DEV)[:n].to(torch.int32)


def _ids(k):
    return torch.zeros(max(k, 4), dtype=torch.int32, device=DEV)


def prepare(case, seed):
    kind, g = case["kind"], _gen(seed)
    s = dict(case=case, kind=kind, i=0)
    if kind in ("decide", "select", "score"):
        s["c"], s["batches"] = _learner(case, seed, case["n"])
        s["idx"] = _index(g, case["n"], case["agents"], case["gpu_share"], case["tokens"], case.get("anchors", False))
        if kind == "decide":
            kv, kp = case["k_victims"], case["k_prefetch"]
            host = (_ids(kv), _ids(1)) if case["host_victims"] else (None, None)
            s["lists"] = (_ids(kv), _ids(1)) + host + (_ids(kp), _ids(1))
        elif kind == "select":
            s["lists"] = (_ids(case["k"]), _ids(1))
        else:
            s["scores"] = torch.empty(case["n"], dtype=torch.float32, device=DEV)
            s["sources"] = _slots(g, case["agents"], min(case["sources"], case["agents"])).to(torch.int16) if case["sources"] else None
    elif kind == "observe":
        A, rng = case["agents"], np.random.default_rng([seed, 2])
        chain, agent = _trace(rng, A, case["chains"], case["events"])
        s["chain"], s["agent"] = torch.from_numpy(chain).to(DEV), torch.from_numpy(agent).to(DEV)
        s["evflags"] = torch.from_numpy((rng.random(case["events"]) < case["warmup"]).astype(np.uint8)).to(DEV) if case["warmup"] else None
        s["c"] = cs.CacheScout(cs.make_params(A, n_chains=case["chains"]), DEV)
        if case["all_chains"]:
            cs.cs_set_survival_sources(s["c"].ctx, cs.CS_SOURCES_ALL_CHAINS)
        s["model"] = dict(C_out=torch.zeros(A, A, dtype=torch.int32, device=DEV), P_out=torch.zeros(A, A, device=DEV),
                          amax_out=torch.zeros(A, dtype=torch.int16, device=DEV), hops_out=torch.zeros(A, dtype=torch.int16, device=DEV),
                          fsurv_out=torch.zeros(A, device=DEV), R_out=torch.zeros(1, device=DEV),
                          cur_out=torch.zeros(case["chains"], dtype=torch.int16, device=DEV),
                          last_agent_out=torch.zeros(1, dtype=torch.int16, device=DEV))
    elif kind == "survival":
        s["c"], _ = _learner(case, seed, 1)
        s["psurv"], s["fsurv"] = (torch.zeros(case["agents"], device=DEV) for _ in range(2))
    elif kind == "compact":
        s["c"] = cs.CacheScout(cs.make_params(1), DEV)
        s["src"] = _pool(g, case["slots"], case, case["src_layout"])
        s["dst"] = _pool(g, case["blocks"], case, case["dst_layout"])
        s["src_slots"], s["dst_slots"] = _slots(g, case["slots"], case["blocks"]), _slots(g, case["blocks"], case["blocks"])
    elif kind == "link":
        s["c"] = cs.CacheScout(cs.make_params(1), DEV)
        s["gpu"] = _pool(g, case["slots"], case, case["gpu_layout"])
        s["host"] = _pool(g, case["slots"], case, case["host_layout"], host=True)
        n = case["off"] + case["pre"]
        gpu, host = _slots(g, case["slots"], n), _slots(g, case["slots"], n)
        s["off"] = (gpu[:case["off"]].clone(), host[:case["off"]].clone())
        s["pre"] = (host[case["off"]:].clone(), gpu[case["off"]:].clone())
    else:                                                          # step
        G, H, kv, kp = case["gpu_blocks"], case["host_blocks"], case["k_victims"], case["k_prefetch"]
        s["c"], s["batches"] = _learner(case, seed, G + H, case["block_tokens"])
        s["idx"] = _index(g, G + H, case["agents"], 0.0, True, True, case["block_tokens"], gpu_blocks=G, free_slots=kp)
        s["gpu"], s["host"] = _pool(g, G, case, 0), _pool(g, H, case, 1, host=True, first_id=G)
        s["stage"], s["stage_slots"] = _pool(g, kv, case, 1), _slots(g, kv, kv)
        s["free"] = torch.arange(kp, dtype=torch.int32, device=DEV)
        s["lists"] = (_ids(kv), _ids(1), _ids(kv), _ids(1), _ids(kp), _ids(1))
        s["side"] = torch.cuda.Stream(DEV)
    return s


# ---- one pass ------------------------------------------------------------------------------------------------------
def run(s):
    case, kind, c = s["case"], s["kind"], s["c"]
    i = s["i"]
    s["i"] = i + 1
    now = NOW0 + i % CLOCK_WINDOW
    if kind == "decide":
        chain, agent = s["batches"][i % N_BATCHES]
        c.observe_invocations(chain, agent)
        c.select_step(s["idx"], now, case["k_victims"], case["k_prefetch"], *s["lists"])
        return s["lists"]
    if kind == "select":
        if case["prefetch"]:
            return c.select_prefetch(s["idx"], now, case["k"], *s["lists"])
        return c.select_victims(s["idx"], now, case["tier"], case["k"], *s["lists"])
    if kind == "score":
        return c.score_blocks(s["idx"], now, s["sources"], s["scores"])
    if kind == "observe":
        c.observe_invocations(s["chain"], s["agent"], s["evflags"])
        cs.cs_get_model(c.ctx, **s["model"])
        return s["model"]
    if kind == "survival":
        cs.cs_exact_survival(c.ctx, cs.CS_AGENT_NONE, case["steps"], s["psurv"], s["fsurv"])
        return s["psurv"], s["fsurv"]
    if kind == "compact":
        c.compact_blocks(s["src"], s["dst"], s["src_slots"], s["dst_slots"])
        return s["dst"].buf.view(torch.int64)
    if kind == "link":
        if case["off"] and case["pre"]:
            c.exchange_blocks(s["gpu"], s["host"], *s["off"], *s["pre"])
            return s["gpu"].buf.view(torch.int64), s["host"].buf.view(torch.int64)
        if case["off"]:
            c.offload_blocks(s["gpu"], s["host"], *s["off"])
            return s["host"].buf.view(torch.int64)
        c.prefetch_blocks(s["host"], s["gpu"], *s["pre"])
        return s["gpu"].buf.view(torch.int64)
    chain, agent = s["batches"][i % N_BATCHES]
    c.step(s["idx"], now, chain, agent, None, case["events"], case["k_victims"], case["k_prefetch"], *s["lists"], s["gpu"], s["host"],
           s["free"], s["stage"], s["stage_slots"], side=s["side"], join_main=True)
    return s["lists"] + tuple(p.buf.view(torch.int64) for p in (s["gpu"], s["host"], s["stage"]))


# ---- what a pass cannot do without -----------------------------------------------------------------------------------
def _metadata_bytes(case, prefetch):
    """Per entry: agent 2, last_access 4, flags 1, ref_count 1, and n_tokens 1 when given; depth 2 for a prefetch list
    with anchors."""
    return 8 + (1 if case["tokens"] else 0) + (2 if prefetch and case["anchors"] else 0)


def work(case):
    kind = case["kind"]
    if kind == "decide":
        A, lists = case["agents"], (2 if case["host_victims"] else 1)
        return {"bytes": case["n"] * _metadata_bytes(case, True) + 4 * (lists * case["k_victims"] + case["k_prefetch"]) + 8 * A * A,
                "flops": 2 * case["n"] * (lists + 1) + 4 * A * A}
    if kind == "select":
        return {"bytes": case["n"] * _metadata_bytes(case, case["prefetch"]) + 4 * case["k"], "flops": 2 * case["n"]}
    if kind == "score":
        return {"bytes": case["n"] * (10 + (1 if case["tokens"] else 0)), "flops": 2 * case["n"]}
    if kind == "observe":
        A = case["agents"]
        return {"bytes": case["events"] * (7 if case["warmup"] else 6) + 8 * A * A, "flops": case["events"] + 4 * A * A}
    if kind == "survival":
        A = case["agents"]
        return {"bytes": 4 * A * A + 8 * A, "flops": 2 * A * A * A * (case["steps"] - 1)}
    block = _block_bytes(case)
    if kind == "compact":
        return {"bytes": 2 * case["blocks"] * block, "flops": 0}
    if kind == "link":
        return {"bytes": 2 * (case["off"] + case["pre"]) * block, "flops": 0}
    n = case["gpu_blocks"] + case["host_blocks"]
    # a victim is read once and written twice (host tier, staging pool)
    return {"bytes": 11 * n + (3 * case["k_victims"] + 2 * case["k_prefetch"]) * block, "flops": 6 * n}


def tolerance(case):
    """Lists, counts and bytes are exact.  Scores and the rows of the transition matrix are defined operation by
    operation in fp32 and come out the same; R and the exact table are sums of fp64 terms rounded to fp32 once, where
    another order of the sum may move the last bit (6e-8)."""
    if case["kind"] in ("observe", "survival"):
        return {"rel": 2.5e-7, "max": 2.5e-7}
    return "exact"
