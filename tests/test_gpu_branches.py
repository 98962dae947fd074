"""The step's size-dependent branches against the oracle, at the sizes where
each begins, ends or leaves a remainder.  Every output, the exported state and
the statistics are whole numbers: the tolerance is zero.
"""
import ctypes

import numpy as np
import pytest

import oracle as O
from paper_2608_01657_gb300 import workloads as W
from _util import compare_outputs, compare_state, ctl_word, device_layout

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _pair(N, bs, G, policy, params_kw, max_requests, max_tokens):
    from paper_2608_01657_gb300 import binding as B
    gpu = B.Cache(N, bs, G, policy, B.Params(**params_kw), max_requests=max_requests, max_tokens=max_tokens)
    return gpu, O.OracleCache(N, bs, G, policy, O.Params(**params_kw))


def _run(gpu, orc, steps, state_every=8, label=""):
    dev = torch.device("cuda")
    for k, st in enumerate(steps):
        g = torch.from_numpy(st.groups).to(dev)
        o = torch.from_numpy(st.offsets).to(dev)
        t = torch.from_numpy(st.tokens if st.num_tokens else np.zeros(4, np.int32)).to(dev)
        c = None if st.contracts is None else torch.from_numpy(st.contracts).to(dev)
        p = None if st.prefixes is None else torch.from_numpy(st.prefixes.view(np.int64)).to(dev)
        assert gpu.step(st.now, g, o, t, c, p) == 0, f"{label} step {k}"
        want = orc.step(st.now, st.groups, st.offsets, st.tokens, st.contracts, st.prefixes)
        compare_outputs(gpu.fetch(st.num_requests), want, f"{label} step {k}")
        if k % state_every == state_every - 1 or k == len(steps) - 1:
            compare_state(gpu.export(), orc.export(), f"{label} step {k}", s3=gpu.policy == "s3fifo")
    assert np.array_equal(gpu.stats(), orc.stats()), f"{label}: stats differ"
    return orc.stats()


def _evicted(stats):
    return int(stats[:, O.STAT_NAMES.index("evicted_blocks")].sum())


def _prompts(lengths, groups, seed, docs=None):
    """One step's prompts: `lengths` tokens each, the first from documents."""
    rng = np.random.default_rng(seed)
    pieces = []
    for k, n in enumerate(lengths):
        if docs is not None and k % 2 == 0:
            d = docs[k % len(docs)]
            pieces.append(np.concatenate([d[:n], rng.integers(0, W.VOCAB, size=max(0, n - len(d)), dtype=np.int32)]))
        else:
            pieces.append(rng.integers(0, W.VOCAB, size=n, dtype=np.int32))
    off = np.concatenate([[0], np.cumsum([len(p) for p in pieces])]).astype(np.int64)
    toks = np.concatenate(pieces).astype(np.int32) if pieces else np.zeros(0, np.int32)
    return np.asarray(groups, np.int32), off, toks


@pytest.mark.parametrize("policy,N,G,beta", [
    ("prefixshield", 511, 1, 4.0), ("prefixshield", 4096, 2, 40.0), ("prefixshield", 4097, 2, 40.0),
    ("prefixshield", 2000, 32, 8.0), ("prefixshield", 2000, 33, 8.0), ("prefixshield", 31, 3, 1e6),
    ("lru", 2048, 2, 8.0), ("lru", 2049, 2, 8.0), ("lru", 1, 1, 8.0)])
def test_small_pool_select(policy, N, G, beta):
    """The one-CTA select and lists, at and past the largest pool and number
    of groups; large balances (no debt) leave every victim to the fallback."""
    steps = W.fuzz_steps(N + G, G, 12, 40, docs_per_group=2, doc_blocks=max(2, N // 24), now_stride=2,
                         fresh_max_blocks=max(2, N // 16), empty_every=11)
    gpu, orc = _pair(N, 16, G, policy, dict(rho=(1.0,), beta=(beta,)), 12, 12 * 16 * (N // 24 + N // 16 + 8))
    assert _evicted(_run(gpu, orc, steps, label=f"{policy}/{N}/{G}")) > 0


@pytest.mark.parametrize("N", [8191, 8192, 8193, 16400])
@pytest.mark.parametrize("policy", ["lru", "staticquota"])
def test_id_lists_at_chunk_edges(policy, N):
    """Free, evicted and invalidated ids over one chunk of 8192 ids, a last
    partial word, and a second chunk."""
    steps = W.fuzz_steps(N, 2, 8, 24, docs_per_group=2, doc_blocks=N // 16, fresh_max_blocks=N // 12, now_stride=2)
    gpu, orc = _pair(N, 16, 2, policy, dict(rho=(2.0,), beta=(64.0,)), 8, 8 * 16 * (N // 16 + N // 12 + 2))
    assert _evicted(_run(gpu, orc, steps, label=f"lists/{policy}/{N}")) > 0


@pytest.mark.parametrize("per_sm,more", [(1, 0), (1, 1), (2, 0), (2, 1), (4, 0), (4, 1)])
@pytest.mark.parametrize("bs", [8, 16, 32])
def test_hashing_widths_and_chunk_edges(bs, per_sm, more):
    """CTAs of one, two, four and eight hashing warps, at both sides of each
    switch (the handle's largest number of chunks against the SMs), with
    prompts of 0 to 130 blocks around the half (32) and the chunk (64), at
    every offset of a prompt's first token in its 16-byte word."""
    blocks = [0, 1, 2, 31, 32, 33, 63, 64, 65, 96, 127, 128, 129, 130]
    chunks = per_sm * torch.cuda.get_device_properties(0).multi_processor_count + more
    max_blocks = 64 * (chunks - len(blocks) - 1)  # chunks = max_blocks / 64 + requests + 1
    assert max_blocks >= sum(blocks)
    rng = np.random.default_rng(bs)
    docs = [rng.integers(0, W.VOCAB, size=130 * bs, dtype=np.int32) for _ in range(2)]
    steps = []
    for k in range(4):
        lengths = [b * bs + int(rng.integers(0, bs)) for b in blocks]
        g, o, t = _prompts(lengths, [i % 2 for i in range(len(blocks))], 10 * bs + k, docs)
        steps.append(W.Step(k, k, g, o, t, None, None))
    gpu, orc = _pair(2500, bs, 2, "prefixshield", dict(rho=(1.0,), beta=(50.0,)), len(blocks), max_blocks * bs)
    _run(gpu, orc, steps, 1, f"hash/{bs}/{chunks}")


@pytest.mark.parametrize("R,max_blocks", [(300, 4), (64, 8), (5, 512)])
def test_more_requests_than_blocks(R, max_blocks):
    """Claims and history entries share the insertion's threads: more requests
    than blocks in a step, and the other way round, most of them empty or hits."""
    rng = np.random.default_rng(R)
    doc = rng.integers(0, W.VOCAB, size=max_blocks * 16, dtype=np.int32)
    steps = []
    for k in range(12):
        n = int(rng.integers(1, max_blocks + 1))
        lengths = [0] * R
        lengths[int(rng.integers(0, R)) & ~1] = n * 16
        g, o, t = _prompts(lengths, rng.integers(0, 3, size=R), k, [doc])
        steps.append(W.Step(k, k, g, o, t, None, None))
    gpu, orc = _pair(max_blocks + 2, 16, 3, "prefixshield", dict(rho=(1.0,), beta=(2.0,)), R, max_blocks * 16)
    _run(gpu, orc, steps, 1, f"R/{R}")


@pytest.mark.parametrize("max_blocks", [1, 5, 8, 9, 10, 11, 12, 17, 19, 4099])
def test_claim_map_holds_a_full_step_of_new_blocks(max_blocks):
    """Every block of the largest step is new, at sizes just past a power of
    two times the claim map's four ways a bucket."""
    steps = []
    for k in range(3):
        g, o, t = _prompts([(max_blocks - 1) * 2, 2], [0, 1], 100 * max_blocks + k)
        steps.append(W.Step(k, k, g, o, t, None, None))
    gpu, orc = _pair(max_blocks + 1, 2, 2, "prefixshield", dict(rho=(1.0,), beta=(3.0,)), 2, max_blocks * 2)
    _run(gpu, orc, steps, 1, f"claims/{max_blocks}")


@pytest.mark.parametrize("G,contracts", [(2, 1), (40, 3), (1000, 3)])
def test_many_indebted_groups(G, contracts):
    """The water-filling's search with one, some and a thousand groups in debt
    (a thread a group), whole groups taken and partial ones."""
    steps = W.fuzz_steps(G, G, 64, 24, docs_per_group=1, doc_blocks=6, fresh_max_blocks=12,
                         with_contracts=contracts if contracts > 1 else 0, now_stride=2)
    rho, beta = (0.5, 1.0, 2.0)[:contracts], (1.0, 3.0, 2.0)[:contracts]
    kw = dict(rho=rho, beta=beta, contract_of_group=[g % contracts for g in range(G)])
    gpu, orc = _pair(4500, 16, G, "prefixshield", kw, 64, 64 * 16 * 19)
    assert _evicted(_run(gpu, orc, steps, label=f"debt/{G}")) > 0


def _aged(policy, old, new, need, gap, N=None):
    """A pool of `old` blocks, `gap` stamps, then `new` blocks, and a prompt
    that takes `need` victims among the old ones: a handle that served other
    prompts in between, as the recency counter tells it.  Returns the length
    of the select's split list."""
    N = N or old + new
    rng = np.random.default_rng(old + need)
    seq = [rng.integers(0, W.VOCAB, size=n * 2, dtype=np.int32) for n in (old, new, need + N - old - new)]
    gpu, orc = _pair(N, 2, 2, policy, dict(rho=(1.0,), beta=(0.0,)), 1, 2 * max(len(t) for t in seq))
    dev = torch.device("cuda")
    for k, t in enumerate(seq):
        if k == 1:
            ctl_word(gpu, "stamp_base", torch.int64).add_(gap)
        g, o = np.zeros(1, np.int32), np.array([0, len(t)], np.int64)
        assert gpu.step(k, torch.from_numpy(g).to(dev), torch.from_numpy(o).to(dev), torch.from_numpy(t).to(dev)) == 0
        want = orc.step(k, g, o, t)
        compare_outputs(gpu.fetch(1), want, f"aged/{policy}/{old}/{need}/{gap} step {k}")
        if k == 2:
            assert len(want["evicted_ids"]) == need
    listed = int(ctl_word(gpu, "lst_n", torch.int64).item())
    got, want = gpu.export(), orc.export()
    assert int(got["stamp"].max()) > gap  # the counter did jump
    for e in (got, want):  # the stamps' order is what has to agree
        e["stamp"] = np.unique(e["stamp"], return_inverse=True)[1]
    compare_state(got, want, f"aged/{policy}/{old}/{need}/{gap}")
    return listed


# Old blocks that fill the first bucket of the range, so the list holds all of
# them: bitmaps of the bucket rank more than 128 of them where it is at most
# 32768 stamps wide, counting ranks up to 512, byte digits the rest (up to 8192
# in shared memory).
@pytest.mark.parametrize("n,log2gap", [
    (128, 24),                                                                # counting
    (129, 24), (1024, 24), (1025, 24), (8192, 24), (16384, 29), (20000, 30),  # bitmaps: 5 to 1024 words
    (129, 40), (512, 40),                                                     # no room for a bitmap: counting
    (513, 40), (8192, 40),                                                    # digits, shared memory
    (8193, 40), (20000, 31)])                                                 # digits, global memory
@pytest.mark.parametrize("policy", ["lru", "prefixshield"])
def test_list_finish(policy, n, log2gap):
    """The split list at the edges of each way to finish it."""
    for need in (1, n // 2, n):
        listed = _aged(policy, n, max(3000, 5000 - n), need, 1 << log2gap)
        assert policy != "lru" or listed == n  # (a debt phase's list is reset for its fallback)


@pytest.mark.parametrize("policy", ["lru", "prefixshield"])
@pytest.mark.parametrize("gap,most", [(1 << 22, 1 << 11), (1 << 24, 1 << 13), (1 << 26, 1 << 11), (1 << 27, 1 << 12)])
def test_aged_range_is_cut_finely(policy, gap, most):
    """Old blocks beside new ones much later: past 2^25 stamps the range is cut
    into 65536 buckets, so the list stays a few thousand long (4096 buckets
    would put all 20,000 old blocks on it from 2^27 on)."""
    for need in (1, 9000, 20000):
        listed = _aged(policy, 20000, 3000, need, gap)
        assert policy != "lru" or 1 <= listed <= most  # (a debt phase's list is reset for its fallback)


@pytest.mark.parametrize("policy", ["staticquota", "prefixshield"])
@pytest.mark.parametrize("N,G", [(4096, 64), (4097, 64), (9000, 65), (9000, 64)])
def test_wide_buckets_at_the_rule_s_edges(policy, N, G):
    """Groups that select over ranges of mixed widths, at the largest pool
    without and the smallest with 65536 buckets, and at 64 and 65 groups."""
    steps = W.fuzz_steps(N + G, G, 64, 30, docs_per_group=2, doc_blocks=max(2, N // G // 2), now_stride=2,
                         fresh_max_blocks=max(2, N // G // 2), block_size=2)
    gpu, orc = _pair(N, 2, G, policy, dict(rho=(2.0,), beta=(4.0,)), 64, 64 * 2 * (2 * (N // G) + 4))
    dev = torch.device("cuda")
    base = ctl_word(gpu, "stamp_base", torch.int64)
    for k, st in enumerate(steps):
        base.add_((0, 1 << 13, 1 << 24, 1 << 25, 1 << 33)[k % 5])
        assert gpu.step(st.now, *(torch.from_numpy(x).to(dev) for x in (st.groups, st.offsets, st.tokens))) == 0
        want = orc.step(st.now, st.groups, st.offsets, st.tokens)
        compare_outputs(gpu.fetch(st.num_requests), want, f"wide/{policy}/{N}/{G} step {k}")
    assert _evicted(orc.stats()) > 0


@pytest.mark.parametrize("N,blocks", [(64, 12), (2000, 400)])
def test_s3fifo_ghost_readmission(N, blocks):
    """Keys evicted and asked for again: ghost hits, and keys found in the ghost
    that the same step's pushes trim before their block is inserted; some of
    the step's new blocks are shared by its requests."""
    steps = W.fuzz_steps(N, 2, 5, 40, docs_per_group=3, doc_blocks=blocks, fresh_max_blocks=blocks // 4, now_stride=2)
    params, limits = dict(rho=(2.0,), beta=(6.0,)), (5, 5 * 16 * (2 * blocks + 2))
    gpu, orc = _pair(N, 16, 2, "s3fifo", params, *limits)
    _run(gpu, orc, steps, label=f"ghost/{N}")
    again = O.OracleCache(N, 16, 2, "s3fifo", O.Params(**params))
    hits = trimmed = 0
    for st in steps:
        ghost = set(zip(*(x.tolist() for x in again.export()["ghost"][:2])))
        new = again.step(st.now, st.groups, st.offsets, st.tokens)["admitted_ids"]
        e = again.export()
        for b in new:
            if (int(e["group"][b]), int(e["key"][b])) in ghost:
                hits += int(e["s3q"][b] == 1)
                trimmed += int(e["s3q"][b] == 0)
    assert hits > 0 and trimmed > 0
    assert int(orc.stats()[:, O.STAT_NAMES.index("instep_hit_blocks")].sum()) > 0


def _queue_steps(gpu, orc, steps, before=None):
    """Steps against the oracle; returns the entry buffers seen after them
    (two: a compaction ran)."""
    dev, buffers = torch.device("cuda"), set()
    for k, st in enumerate(steps):
        if before:
            before()
        assert gpu.step(st.now, *(torch.from_numpy(x).to(dev) for x in (st.groups, st.offsets, st.tokens))) == 0
        compare_outputs(gpu.fetch(st.num_requests), orc.step(st.now, st.groups, st.offsets, st.tokens), f"step {k}")
        buffers.add(int(ctl_word(gpu, "lg_buf", torch.int32).item()))
    return buffers


@pytest.mark.parametrize("policy", ["lru", "prefixshield", "staticquota"])
def test_queue_logs_fill_and_compact(policy):
    """Indexed queues whose logs run full again and again."""
    steps = W.fuzz_steps(3, 3, 8, 300, docs_per_group=3, doc_blocks=6, fresh_max_blocks=1, now_stride=2)
    gpu, orc = _pair(40, 16, 3, policy, dict(rho=(2.0,), beta=(6.0,), flags=O.FLAG_INDEXED_QUEUES), 8, 4096)
    assert _queue_steps(gpu, orc, steps) == {0, 1}
    compare_state(gpu.export(), orc.export(), f"queues/{policy}")
    assert np.array_equal(gpu.stats(), orc.stats()) and _evicted(orc.stats()) > 0


def test_queue_barrier_starts_from_any_count():
    """The compaction's barrier does not depend on what an earlier launch left
    in its counter."""
    steps = W.fuzz_steps(3, 3, 8, 120, docs_per_group=3, doc_blocks=6, fresh_max_blocks=1, now_stride=2)
    gpu, orc = _pair(40, 16, 3, "lru", dict(rho=(2.0,), beta=(6.0,), flags=O.FLAG_INDEXED_QUEUES), 8, 4096)
    bar = ctl_word(gpu, "bar", torch.int64)
    assert _queue_steps(gpu, orc, steps, lambda: bar.fill_(17)) == {0, 1}


def test_queue_error_is_kept_until_reset():
    """A live count that disagrees with its log is found by the next
    compaction: that step and every later one report it (ps_clear_status does
    not help), and no later one changes the pool, until ps_reset."""
    steps = W.fuzz_steps(3, 3, 8, 300, docs_per_group=3, doc_blocks=6, fresh_max_blocks=1, now_stride=2)
    kw = dict(rho=(2.0,), beta=(6.0,), flags=O.FLAG_INDEXED_QUEUES)
    gpu, orc = _pair(40, 16, 3, "lru", kw, 8, 4096)
    dev = torch.device("cuda")
    _queue_steps(gpu, orc, steps[:5])
    at = device_layout()["DevState", "lg_live"]  # the handle starts with its DevState
    live = int.from_bytes(ctypes.string_at(gpu._h.value + at, 8), "little") - gpu.workspace.data_ptr()
    live += 8 * 3 * 3  # the global log
    gpu.workspace[live:live + 8].view(torch.int64).add_(1)
    status = []
    for st in steps[5:]:
        if len(status) == 3:
            break
        if status:
            gpu.clear_status()
            before = gpu.export()
        assert gpu.step(st.now, *(torch.from_numpy(x).to(dev) for x in (st.groups, st.offsets, st.tokens))) == 0
        if status:
            compare_state(gpu.export(), before, "a refused step")
        if status or gpu.fetch(st.num_requests)["status"]:
            status.append(gpu.fetch(st.num_requests)["status"])
    assert status == [-6] * 3  # PS_ERR_DEVICE_STATUS
    assert gpu.reset() == 0
    assert _queue_steps(gpu, O.OracleCache(40, 16, 3, "lru", O.Params(**kw)), steps[:120]) == {0, 1}


@pytest.mark.parametrize("R", [1, 7, 600])
def test_probe_edges(R):
    """Prompts without a full block count 0 whatever the output held; a call
    with an invalid request reports it and leaves the outputs untouched."""
    rng = np.random.default_rng(R)
    lengths = [int(n) for n in rng.choice([0, 5, 16, 40, 100 * 16 + 3], size=R)]
    g, o, t = _prompts(lengths, rng.integers(0, 2, size=R), R, [rng.integers(0, W.VOCAB, size=1700, dtype=np.int32)])
    gpu, orc = _pair(9000, 16, 2, "lru", dict(rho=(1.0,), beta=(1.0,)), R, max(64, len(t)))
    dev = torch.device("cuda")
    half = slice(0, max(1, R // 2))
    n = len(g[half])
    first = (g[half], o[:n + 1], t[:o[n]])
    gg, oo, tt = (torch.from_numpy(np.ascontiguousarray(x)).to(dev) for x in (g, o, t if len(t) else np.zeros(4, np.int32)))
    assert gpu.step(0, gg[:n], oo[:n + 1], tt) == 0
    compare_outputs(gpu.fetch(n), orc.step(0, *first), "first")
    out = torch.full((R,), -7, dtype=torch.int32, device=dev)
    _, status = gpu.cached_prefix(gg, oo, tt, out=out)
    assert int(status.item()) == 0
    assert np.array_equal(out.cpu().numpy(), orc.cached_prefix(g, o, t))
    bad = gg.clone()
    bad[R - 1] = 2
    out.fill_(-7)
    _, status = gpu.cached_prefix(bad, oo, tt, out=out)
    assert int(status.item()) == O.ERR_INVALID_ARG and bool((out == -7).all())


@pytest.mark.parametrize("tokens_pinned,outputs_pinned,shift", [
    (True, True, 0), (True, True, 1), (True, False, 0), (False, True, 0), (False, False, 3)])
def test_step_host_buffers(tokens_pinned, outputs_pinned, shift):
    """Page-locked buffers (read and written by kernels), pageable ones
    (copied), mixtures, and token buffers off a 16-byte boundary."""
    from paper_2608_01657_gb300 import binding as B
    steps = W.fuzz_steps(61, 3, 5, 16, docs_per_group=3, doc_blocks=6, with_contracts=2, with_prefixes=True, empty_every=7)
    kw = dict(rho=(2.0, 1.0), beta=(6.0, 3.0), contract_of_group=[0, 1, 0])
    gpu, orc = _pair(40, 16, 3, "prefixshield", kw, 5, 2048)

    def host(x, by=0):
        buf = torch.empty(len(x) + by + 4, dtype=torch.from_numpy(x[:0]).dtype, pin_memory=tokens_pinned).numpy()
        buf[by:by + len(x)] = x
        return buf[by:by + len(x)]

    for st in steps:
        out = B.host_outputs(5, gpu.max_blocks, 3, pinned=outputs_pinned)
        R = st.num_requests
        res = gpu.step_host(st.now, host(st.groups), host(st.offsets), host(st.tokens, shift), host(st.contracts),
                            host(st.prefixes.view(np.int64)), out=out)
        assert res["rc"] == 0
        cnt = out["counts"]
        got = {"status": int(cnt[3]), "hit_blocks": out["hit_blocks"][:R], "admitted_blocks": out["admitted_blocks"][:R],
               "admitted_offsets": out["admitted_offsets"][:R + 1], "admitted_ids": out["admitted_ids"][:cnt[0]],
               "evicted_ids": out["evicted_ids"][:cnt[1]], "invalidated_ids": out["invalidated_ids"][:cnt[2]],
               "debt_raw": out["debt_raw"], "debt_norm": out["debt_norm"]}
        compare_outputs(got, orc.step(st.now, st.groups, st.offsets, st.tokens, st.contracts, st.prefixes), f"step {st.index}")


@pytest.mark.parametrize("tokens", [1 << 21, (1 << 21) + 1])
def test_step_host_tokens_at_the_kernel_s_limit(tokens):
    """Page-locked tokens of 8 MB are read by a kernel, more are copied."""
    from paper_2608_01657_gb300 import binding as B
    rng = np.random.default_rng(tokens)
    t = torch.from_numpy(rng.integers(0, W.VOCAB, size=tokens, dtype=np.int32)).pin_memory().numpy()
    cut = tokens // 3
    g = torch.zeros(2, dtype=torch.int32, pin_memory=True).numpy()
    o = torch.tensor([0, cut, tokens], dtype=torch.int64).pin_memory().numpy()
    gpu, orc = _pair(20000, 64, 2, "lru", dict(rho=(1.0,), beta=(1.0,)), 2, tokens)
    for now in range(2):  # the second step hits what the first left
        out = B.host_outputs(2, gpu.max_blocks, 2, pinned=True)
        assert gpu.step_host(now, g, o, t, out=out)["rc"] == 0
        cnt = out["counts"]
        got = {"status": int(cnt[3]), **{k: out[k][:m] for k, m in (
            ("hit_blocks", 2), ("admitted_blocks", 2), ("admitted_offsets", 3), ("admitted_ids", cnt[0]),
            ("evicted_ids", cnt[1]), ("invalidated_ids", cnt[2]), ("debt_raw", 2), ("debt_norm", 2))}}
        compare_outputs(got, orc.step(now, g, o, t), f"step {now}")


@pytest.mark.parametrize("which", ["tokens", "admitted_ids"])
def test_step_host_array_that_leaves_page_locked_memory(which):
    """An array of which only the first pages are page-locked goes to the copy
    calls, which refuse it; the next call is as if that one had not been made
    (a refused input) or had only lost its outputs."""
    from paper_2608_01657_gb300 import binding as B
    bs, n = 2, 1 << 18
    rng = np.random.default_rng(5)
    docs = [rng.integers(0, W.VOCAB, size=n, dtype=np.int32) for _ in range(2)]
    gpu, orc = _pair(n // bs, bs, 2, "lru", dict(rho=(1.0,), beta=(1.0,)), 1, n)
    cudart = torch.cuda.cudart()
    raw = np.zeros(4 * n + (1 << 17), np.uint8)
    at = -raw.ctypes.data % (1 << 16)
    part = raw[at:at + 4 * n].view(np.int32)[:n if which == "tokens" else n // bs]

    def pinned(x):
        return torch.from_numpy(x).pin_memory().numpy()

    g, o = np.zeros(1, np.int32), np.array([0, n], np.int64)
    out = B.host_outputs(1, gpu.max_blocks, 2, pinned=True)
    assert int(cudart.cudaHostRegister(part.ctypes.data, 1 << 16, 0)) == 0
    try:
        if which == "tokens":
            part[:] = docs[0]
            res = gpu.step_host(0, pinned(g), pinned(o), part, out=out)
        else:
            orc.step(0, g, o, docs[0])
            res = gpu.step_host(0, pinned(g), pinned(o), pinned(docs[0]), out=dict(out, admitted_ids=part))
        assert res["rc"] == -4  # PS_ERR_CUDA
    finally:
        torch.cuda.synchronize()
        cudart.cudaHostUnregister(part.ctypes.data)
    res = gpu.step_host(1, pinned(g), pinned(o), pinned(docs[1]), out=out)
    assert res["rc"] == 0
    cnt = out["counts"]
    got = {"status": int(cnt[3]), **{k: out[k][:m] for k, m in (
        ("hit_blocks", 1), ("admitted_blocks", 1), ("admitted_offsets", 2), ("admitted_ids", cnt[0]),
        ("evicted_ids", cnt[1]), ("invalidated_ids", cnt[2]), ("debt_raw", 2), ("debt_norm", 2))}}
    compare_outputs(got, orc.step(1, g, o, docs[1]), which)
    compare_state(gpu.export(), orc.export(), which)
