"""The work that is measured: prefix-cache steps and probes as a scheduler calls them.

A case is one pool in its steady state (filled, evicting) and one pass is one
call on the next batch of a ring of ragged batches.  The ring's new blocks
turn the pool over before a batch comes round again, so its once-only prompts
miss every time, as new prompts do, while its shared prefixes hit.

Traffic follows the synthetic traces of ``paper_2608_01657_gb300.workloads``:

* a *hot* group repeats a few documents (zipf 1.1) with a short new suffix;
* a *flood* group sends only new prompts of lognormal length (it runs into
  admission debt);
* a *chat* group extends conversations: a shared system prompt, then the turns
  so far, so each request is the last one plus a turn.

``mix`` says which groups are what: "pollution" (half hot, half flood),
"chat" (all chat), "scale" (an eighth hot, an eighth flood, the rest chat).
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2608_01657_gb300 import binding as B

VOCAB = 32000
SUFFIX = 128        # new tokens after a hot document (the hot groups' ragged suffix averages this)
TURNS = 8           # requests of one conversation
ARRAYS = ("hit_blocks", "admitted_blocks", "admitted_offsets", "admitted_ids", "evicted_ids",
          "invalidated_ids", "counts", "debt_raw", "debt_norm")


def case(name, **kw):
    c = dict(entry="step", policy="prefixshield", queues=False, mix="scale", groups=64, pool=1 << 20,
             block=16, requests=4096, docs=64, doc=4096, fresh=4096, contracts=1, prefixes=False)
    c.update(kw)
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # One request at a time into a small pool: an engine that admits requests as they come.  Latency only.
        case("single", mix="pollution", groups=2, pool=511, requests=1, docs=4, doc=1536, fresh=1536),
        # The tiny pollution trace: 16 requests a step, a pool smaller than a step's demand.
        case("tiny", mix="pollution", groups=2, pool=256, requests=16, docs=1, doc=512, fresh=1024),
        # The 4096-block pollution trace: 8 requests a step under the recency baseline, 64 under the debt policy.
        case("pollution-lru", policy="lru", mix="pollution", groups=2, pool=4096, requests=8, docs=8, doc=2048,
             fresh=2048),
        case("pollution", mix="pollution", groups=2, pool=4096, requests=64, docs=8, doc=2048, fresh=2048),
        # The chat-shaped mix on a 65,536-block pool: the S3-FIFO baseline.
        case("chat-s3fifo", policy="s3fifo", mix="chat", groups=16, pool=65536, requests=256, docs=32, doc=2048,
             fresh=200),
        # The same kind of traffic from host buffers, with service contracts and explicit prefix ids: the
        # synchronous call of a scheduler whose batches live on the host.  Odd pool size, 32-token blocks.
        case("chat-host", entry="host", mix="chat", groups=23, pool=50021, block=32, requests=301, docs=32, doc=4096,
             fresh=200, contracts=3, prefixes=True),
        # Equal partitions per tenant, small blocks.
        case("quota", policy="staticquota", groups=16, pool=100003, block=8, requests=200, docs=16, doc=2048,
             fresh=2048),
        # The read-only probe: a router asks how much of each prompt is cached.
        case("probe", entry="probe", groups=32, pool=1 << 18, requests=1024, docs=32),
        # The scale trace (64 groups, 1,048,576 blocks, 4096 requests, about 12 M tokens a step): the benchmark's
        # workload with the debt policy, then with S3-FIFO, then end to end from page-locked host buffers with
        # two steps in flight.
        case("scale"),
        case("scale-s3fifo", policy="s3fifo"),
        case("scale-async", entry="async"),
        # A pool of 4 M blocks, victims from the indexed queues.
        case("scale-queues", queues=True, pool=1 << 22),
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def draw(rng):
    """Any batch from one request to the scale trace's, any policy, entry point, block size and option."""
    mix = rng.choice(["pollution", "chat", "scale"])
    policy = rng.choice(["prefixshield", "prefixshield", "prefixshield", "lru", "s3fifo", "staticquota"])
    entry = rng.choice(["step", "step", "step", "step", "host", "async", "probe"])
    requests = max(1, round(_log(rng, 1, 4096)))
    block = rng.choice([8, 16, 16, 16, 32, 64])
    groups = max({"pollution": 2, "chat": 1, "scale": 8}[mix], round(_log(rng, 2, 96)))
    tokens = _log(rng, 128, 4096)
    # at most about half a million blocks a step, as the largest listed batches have
    tokens = min(tokens, 2300 * 4096 / requests, 520000 * block / requests)
    doc = max(2 * block, round(tokens * rng.uniform(0.7, 1.5)))
    fresh = max(block, round(tokens * rng.uniform(0.7, 1.5)))
    docs = rng.choice([1, 4, 8, 16, 32, 64]) if mix == "pollution" else rng.choice([16, 32, 48])
    per_step = max(1.0, requests * tokens / block)
    # from pools that one step fills to pools of twelve steps' blocks.  The published S3-FIFO loop is one eviction
    # at a time where a step empties its main queue, so large pools of that policy hold a few steps at least.
    few = 3.0 if policy == "s3fifo" and per_step > 4000 else 0.6
    pool = int(min(1 << 20, max(64, per_step * _log(rng, few, 12.0))))
    pool = max(pool, 8 * groups)
    return case(None, entry=entry, policy=policy, queues=policy != "s3fifo" and rng.random() < 0.2, mix=mix,
                groups=groups, pool=pool, block=block, requests=requests, docs=docs, doc=doc, fresh=fresh,
                contracts=rng.choice([1, 1, 3]), prefixes=rng.random() < 0.25)


# ---- traffic -----------------------------------------------------------------
def _roles(c):
    """0 hot, 1 flood, 2 chat, per group."""
    G = c["groups"]
    if c["mix"] == "chat":
        return np.full(G, 2)
    if c["mix"] == "pollution":
        return np.arange(G) % 2
    r = np.full(G, 2)
    r[: max(1, G // 8)] = 0
    r[max(1, G // 8): 2 * max(1, G // 8)] = 1
    return r


def _zipf(n):
    w = 1.0 / np.arange(1, n + 1) ** 1.1
    return w / w.sum()


def _turn_ends(c, rng):
    """Lengths of a conversation's successive prompts [G, docs, TURNS]: ragged, growing, at most a document."""
    G, D, L = c["groups"], c["docs"], c["doc"]
    return np.sort(rng.integers(max(1, L // 8), L + 1, size=(G, D, TURNS)), axis=2)


def _batch(c, rng, t, roles, zipf, ends):
    """Batch t of the ring: per request the group, the document (or -1), its shared and its new tokens."""
    R, D = c["requests"], c["docs"]
    g = rng.integers(0, c["groups"], size=R)
    role = roles[g]
    hot = rng.choice(D, size=R, p=zipf)
    age = rng.integers(0, TURNS, size=R)
    conv = (t + (TURNS - 1 - age)) % D        # a window of eight conversations slides by one a batch
    doc = np.where(role == 0, hot, np.where(role == 2, conv, -1))
    shared = np.where(role == 0, c["doc"], np.where(role == 2, ends[g, conv, age], 0))
    flood = np.clip(np.round(rng.lognormal(math.log(c["fresh"]), 0.6, size=R)), c["fresh"] / 8, c["fresh"] * 6)
    suffix = rng.integers(1, 2 * SUFFIX, size=R)
    new = np.where(role == 0, suffix, np.where(role == 1, flood, 0)).astype(np.int64)
    return g.astype(np.int32), doc.astype(np.int64), shared.astype(np.int64), new


def _budget(c):
    """The scheduler's tokens a step (max_tokens): a quarter above the largest of a few batches of this kind."""
    rng = np.random.default_rng([0, 2])
    roles, zipf, ends = _roles(c), _zipf(c["docs"]), _turn_ends(c, rng)
    most = max(int(np.sum(shared + new)) for _, _, shared, new in (_batch(c, rng, t, roles, zipf, ends) for t in range(4)))
    return -(-max(most * 5 // 4, c["doc"] + 2 * SUFFIX, 3 * c["fresh"]) // 4096) * 4096


def _ring(c, seed):
    """Batches whose new blocks turn the pool over (4 to 64 of them), each cut to the token budget."""
    rng = np.random.default_rng([int(seed), 1])
    roles, zipf, ends = _roles(c), _zipf(c["docs"]), _turn_ends(c, rng)
    budget = _budget(c)
    batches, blocks, t = [], 0.0, 0
    while t < 4 or (t < 64 and blocks < 1.6 * c["pool"]):
        g, doc, shared, new = _batch(c, rng, t, roles, zipf, ends)
        left = np.maximum(budget - (np.cumsum(shared + new) - (shared + new)), 0)  # the last requests of a long batch
        shared = np.minimum(shared, left)
        new = np.minimum(new, left - shared)
        b = (g, doc, shared, new)
        role = roles[g]
        # a conversation's prompt is mostly the last one's; a turn of it is new
        blocks += float(np.sum(np.where(role == 2, b[2] / TURNS, b[3]))) / c["block"]
        batches.append(b)
        t += 1
    return batches


def prepare(case, seed):
    """A pool that the ring has gone through once (it is full and evicting), and the ring's batches in the memory
    the entry point takes them from: device tensors, or page-locked host arrays."""
    c = case
    dev = torch.device("cuda", torch.cuda.current_device())
    gen = torch.Generator(device=dev)
    gen.manual_seed(int(seed))
    G, D, L, C = c["groups"], c["docs"], c["doc"], c["contracts"]
    batches = _ring(c, seed)
    docs = torch.randint(0, VOCAB, (G, D, L), dtype=torch.int32, device=dev, generator=gen)
    sys_len = max(1, L // 8)  # conversations of a group start with one of four system prompts
    for j in range(4, D) if c["mix"] != "pollution" else ():
        docs[:, j, :sys_len] = docs[:, j % 4, :sys_len]
    host = c["entry"] in ("host", "async")
    rows = docs.view(G * D, L)
    steps = []
    for t, (g, doc, shared, new) in enumerate(batches):
        off = np.zeros(len(g) + 1, np.int64)
        np.cumsum(shared + new, out=off[1:])
        T = int(off[-1])
        offsets = torch.from_numpy(off).to(dev)
        row = torch.from_numpy(np.maximum(g * np.int64(D) + doc, 0)).to(dev)
        tokens = torch.randint(0, VOCAB, (T,), dtype=torch.int32, device=dev, generator=gen)
        req = torch.repeat_interleave(torch.arange(len(g), device=dev), offsets[1:] - offsets[:-1], output_size=T)
        pos = torch.arange(T, device=dev) - offsets[req]
        is_shared = pos < torch.from_numpy(shared).to(dev)[req]
        tokens = torch.where(is_shared, rows[row[req], torch.clamp(pos, max=L - 1)], tokens)
        contracts = torch.from_numpy((g % C).astype(np.int32)) if C > 1 else None
        # a logical prefix id: the document's, or one of the request's own
        own = 1 + G * D + t * len(g) + np.arange(len(g), dtype=np.int64)
        prefixes = torch.from_numpy(np.where(doc >= 0, 1 + g * np.int64(D) + doc, own)) if c["prefixes"] else None
        one = [torch.from_numpy(g), offsets, tokens, contracts, prefixes]
        if host:
            one = [None if x is None else x.cpu().pin_memory().numpy() for x in one]
        else:
            one = [None if x is None else x.to(dev) for x in one]
        steps.append(one)
        del req, pos, is_shared
    per_group = sum(int(s[1][-1]) for s in steps) / c["block"] / len(steps) / G
    rho = max(16.0, 0.4 * per_group)  # most groups stay within their refill, the floods do not
    tiers = [1.0, 40 / 64, 16 / 64][:C]
    cache = B.Cache(c["pool"], c["block"], G, c["policy"],
                    B.Params(rho=[rho * x for x in tiers], beta=[3 * rho * x for x in tiers],
                             flags=B.PS_FLAG_INDEXED_QUEUES if c["queues"] else 0),
                    max_requests=c["requests"], max_tokens=_budget(c))
    for x in cache.out.values():
        x.zero_()  # id lists are compared whole; a step writes the counts' worth of them
    state = dict(case=c, cache=cache, steps=steps, at=0, now=0, slots=[None, None])
    if host:
        state["out"] = [B.host_outputs(c["requests"], cache.max_blocks, G, pinned=True) for _ in range(2)]
        for o in state["out"]:
            for k in ARRAYS:
                o[k][:] = 0
    if c["entry"] == "probe":
        state["found"] = torch.zeros(c["requests"], dtype=torch.int32, device=dev)
        state["status"] = torch.zeros(1, dtype=torch.int32, device=dev)
    for k in range(len(steps)):  # fill the pool
        if host:
            out = _host(state, k)
            bad = out["rc"]
        else:
            bad = _device(state, k)
        if bad:
            raise RuntimeError("a filling step failed: %d" % bad)
    torch.cuda.synchronize()
    status = int(state["out"][0]["counts"][3]) if host else int(cache.out["counts"][3])
    if status:
        raise RuntimeError("a filling step's status is %d" % status)
    return state


def _device(state, k):
    g, o, t, c, p = state["steps"][k]
    state["now"] += 1
    return state["cache"].step(state["now"], g, o, t, contracts=c, prefixes=p)


def _host(state, k):
    g, o, t, c, p = state["steps"][k]
    state["now"] += 1
    return state["cache"].step_host(state["now"], g, o, t, contracts=c, prefixes=p, out=state["out"][0])


def run(state):
    """One call on the ring's next batch."""
    k = state["at"] % len(state["steps"])
    state["at"] += 1
    cache, entry = state["cache"], state["case"]["entry"]
    if entry == "step":
        rc = _device(state, k)
        out = cache.out
    elif entry == "probe":
        g, o, t, _, _ = state["steps"][k]
        cache.cached_prefix(g, o, t, out=state["found"], status=state["status"])
        return {"cached": state["found"], "status": state["status"]}
    elif entry == "host":
        out = _host(state, k)
        rc = out["rc"]
    else:  # two steps in flight: a slot's last step is waited for before the slot is used again
        slot = state["at"] % 2
        if state["slots"][slot]:
            rc = cache.step_host_wait(slot)
            if rc:
                raise RuntimeError("step_host_wait: %d" % rc)
        g, o, t, c, p = state["steps"][k]
        state["now"] += 1
        out = state["out"][slot]
        rc = cache.step_host_async(slot, state["now"], g, o, t, out, contracts=c, prefixes=p)
        state["slots"][slot] = True
    if rc:
        raise RuntimeError("the step failed: %d" % rc)
    return {a: out[a] for a in ARRAYS}


def work(case):
    """Bytes of an average batch: its tokens and descriptors read once, one 16-byte table entry a full block, 48
    bytes (table entry and block record) written for a new block and 32 read of the block it replaces, 16 a hit
    block's access record, and the outputs."""
    c = case
    rng = np.random.default_rng([0, 1])
    roles, zipf, ends = _roles(c), _zipf(c["docs"]), _turn_ends(c, rng)
    T = new = 0.0
    n = 4
    for t in range(n):
        g, _, shared, fresh = _batch(c, rng, t, roles, zipf, ends)
        T += float(np.sum(shared + fresh))
        new += float(np.sum(np.where(roles[g] == 2, shared / TURNS, fresh)))
    T, blocks = T / n, T / n / c["block"]
    new = min(new / n / c["block"], float(c["pool"]))
    R = c["requests"]
    if c["entry"] == "probe":
        return {"bytes": 4 * T + 12 * R + 16 * blocks + 4 * R, "flops": 0.0}
    hit = max(0.0, blocks - new)
    return {"bytes": 4 * T + 12 * R + 16 * blocks + (48 + 32) * new + 16 * hit + 8 * new + 12 * R + 16 * c["groups"],
            "flops": 0.0}


def tolerance(case):
    """Block ids, counts and debts are whole numbers (debts in fixed point): the same every time."""
    return "exact"


def exact(case, seed):
    """Whole numbers that follow from every earlier step of the pool: they have no 64-bit value to round from, and
    are compared for equality."""
    return None
