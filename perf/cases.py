"""The cases that the performance of this package is measured on.

Each case is one call, or one short run of calls, that a program analysing
request traces makes through the package's public entry points: the whole path
from tokens to curves on traces of all four shapes that the repository's trace
generator knows (tiny, chat, agentic coding, mixed day), at several block
sizes, with and without session labels, from device and from host memory; the
five stages called one by one; the reuse analysis of a block trace that has no
prefix structure; and the analyses that start from a trace's ids or previous
uses (semantics variants, trace statistics, Belady's optimum, session-level
eviction).

Traces are drawn here with the parameters of tracegen's workloads, the request
plan in numpy and the tokens on the GPU.  A case fixes its sessions (turns,
lengths, system prompts), so that every seed's trace has the same size; the
seed decides when they arrive, and with that the order of all requests, and
the tokens.  Every result is a whole number and exact.
"""
import numpy as np
import torch

import paper_2609_28870_gb300 as ptc

VOCAB = 151_936
NONE = 0xFFFFFFFF

# append medians (user or tool, reply), system prompts (count, shortest,
# longest, Zipf), seconds of arrivals per session
_CHAT = dict(append=(300.0, 600.0), prompts=(50, 1024, 4096), window=5.9)
_TINY = dict(append=(200.0, 400.0), prompts=(10, 512, 2048), window=8.1)
_AGENT = dict(append=(2048.0, 500.0), prompts=(10, 2048, 8192), window=31.4)
_CONTEXT = 131_072  # an agentic context drops its oldest turns beyond this


def listed():
    return [
        # A look at a few minutes of traffic: 60 short conversations, no
        # labels, a 16-point grid.  Launches and waits are most of the time.
        _pipeline("small window", shape="tiny", chats=60, caps=16),
        # The conversational workload (5,600 sessions, 150M tokens).
        _pipeline("chat trace", shape="chat", chats=5600, caps=64, sessions=True),
        # The agentic coding workload (560 sessions, 2 billion tokens), with
        # labels: its id table does not fit in L2.
        _pipeline("agentic trace", shape="agentic", agents=560, caps=64, sessions=True),
        # A window of it in blocks of 64 tokens, without labels, where the
        # window starts at any token of a longer buffer; App. C's linear cost.
        _pipeline("agentic window B64", shape="agentic", agents=190, caps=64, B=64, lead=3, cost=ptc.PTC_COST_LINEAR),
        # Half a day of the mixed workload (5 billion tokens), 128 capacities.
        _pipeline("mixed half day", shape="mixed", chats=89_000, agents=650, caps=128, sessions=True),
        # The chat workload in page-locked host memory, as it comes from a
        # reader: the copy to the device is part of the call.
        dict(_pipeline("chat from host", shape="chat", chats=5600, caps=64, sessions=True), kind="host"),
        # The five calls one by one with every intermediate kept (keys too),
        # then the exact check of the ids; blocks of 24 tokens.
        dict(_pipeline("five calls B24", shape="chat", chats=2100, caps=33, B=24), kind="stages"),
        # A block trace without prefix structure (storage or key-value
        # traffic, the paper's secondary traces): ids given, requests of 1 to
        # 8 blocks, popularity near Zipf.
        {"name": "block trace", "kind": "blocks", "accesses": 12_000_000, "objects": 3_000_000, "caps": 65},
        # The chat workload under the simulator's whole-request residency with
        # blocks freed leaf first.
        dict(_pipeline("leaf-first residency", shape="chat", chats=5600, caps=64), kind="variant",
             order=ptc.PTC_TOUCH_LEAF_FIRST, residency=ptc.PTC_RESIDENCY_REQUEST),
        # Lifetimes, reuse intervals, popularity and reach of the chat workload.
        dict(_pipeline("trace statistics", shape="chat", chats=5600, caps=64), kind="stats"),
        # The offline optimum and the session-granularity curves of the chat
        # workload, for every capacity of its grid.
        dict(_pipeline("Belady curves", shape="chat", chats=5600, caps=64), kind="belady"),
        dict(_pipeline("session eviction", shape="chat", chats=5600, caps=64), kind="session"),
    ]


def _pipeline(name, shape, caps, chats=0, agents=0, B=16, sessions=False, lead=0, cost=ptc.PTC_COST_MEASURED):
    return {"name": name, "kind": "pipeline", "shape": shape, "chats": chats, "agents": agents, "B": B, "caps": caps,
            "sessions": sessions, "lead": lead, "cost": cost}


def _log_int(rng, lo, hi):
    return int(round(lo * (hi / lo) ** rng.random()))


def draw(rng):
    """One more case: a kind, then sizes spread over the logarithm of its range."""
    kind = rng.choice(["pipeline"] * 6 + ["host", "stages", "blocks", "variant", "stats", "belady", "session"])
    caps = rng.choice([1, 7, 16, 26, 64, 65, 100, 128])
    if kind == "blocks":
        n = _log_int(rng, 20_000, 24_000_000)
        return {"kind": kind, "accesses": n, "objects": max(100, int(n * rng.uniform(0.05, 0.8))), "caps": caps}
    shape = rng.choice(["tiny", "chat", "agentic", "mixed"])
    chats, agents = 0, 0
    if shape in ("tiny", "chat"):
        chats = _log_int(rng, 20, 5600)
    elif shape == "agentic":
        agents = _log_int(rng, 5, 560)
    else:
        agents = _log_int(rng, 5, 300)
        chats = agents * rng.randint(40, 137)
    B = rng.choice([16] * 6 + [1, 12, 24, 32, 48, 64, 100, 128, 256])
    if kind in ("belady", "session", "variant", "stats", "host", "stages"):
        # one analysis of a trace of the listed ones' size at most
        chats, agents, B = min(chats, 5600), min(agents, 30), max(B, 16)
        caps = min(caps, 64)
    elif B < 12:
        chats, agents = min(chats, 400), min(agents, 10)
    case = _pipeline("", shape, caps, chats, agents, B, rng.random() < 0.5, rng.choice([0, 0, 0, 1, 2, 3]),
                     rng.choice([ptc.PTC_COST_UNIFORM, ptc.PTC_COST_MEASURED, ptc.PTC_COST_MEASURED, ptc.PTC_COST_LINEAR]))
    del case["name"]
    case["kind"] = kind
    if kind == "variant":
        case["order"], case["residency"] = rng.choice([(0, 1), (1, 0), (1, 1)])
    return case


# ------------------------------------------------------------------ request plans
def _turns(u, shape):
    """Turn counts at the quantiles u of the shape's distribution."""
    if shape == "agentic":  # Zipf(1.2) on 1 .. 400
        cdf = np.cumsum(np.arange(1, 401) ** -1.2)
        return np.searchsorted(cdf / cdf[-1], u) + 1
    single, mean = (0.5, 6.0) if shape == "tiny" else (0.6, 4.0)
    v = np.clip((u - single) / (1.0 - single), 0.0, 1.0 - 1e-9)
    more = 2 + np.floor(np.log1p(-v) / np.log(mean / (1.0 + mean))).astype(np.int64)
    return np.where(u < single, 1, more)


def _half(rng, fixed, shape, S, window):
    """The requests of S sessions of one shape: per request the session, the
    time, the system prompt and its length, the place in the session's stream
    where the context after the prompt starts, and its length."""
    P = {"tiny": _TINY, "chat": _CHAT, "agentic": _AGENT}[shape]
    turns = fixed.permutation(_turns((np.arange(S) + 0.5) / S, shape))
    first = np.cumsum(turns) - turns
    ses = np.repeat(np.arange(S), turns)
    R = len(ses)
    append = sum(np.maximum(1, np.rint(m * np.exp(fixed.standard_normal(R)))).astype(np.int64) for m in P["append"])
    end = np.cumsum(append)
    begin = end - append                      # of each turn, in one stream of all sessions
    base = begin[first][ses]
    count, lo, hi = P["prompts"]
    length = fixed.integers(lo, hi + 1, count)
    if shape == "chat":
        weight = 1.0 / np.arange(1, count + 1)
        prompt = fixed.choice(count, S, p=weight / weight.sum())
    else:
        prompt = fixed.integers(0, count, S)
    prompt, plen = prompt[ses], length[prompt][ses]
    start = base
    if shape == "agentic":  # drop the oldest turns beyond the context length
        start = begin[np.minimum(np.searchsorted(begin, end - (_CONTEXT - plen)), np.arange(R))]
        start = np.maximum(start, base)
    body = np.minimum(end - start, _CONTEXT - plen)
    if shape == "agentic":
        gap = rng.uniform(5.0, 20.0, R)
    elif shape == "chat":
        gap = 45.0 * np.exp(0.3 * rng.standard_normal(R))
    else:
        gap = rng.uniform(27.0, 33.0, R)
    total = np.cumsum(gap)
    t = rng.uniform(0.0, window, S)[ses] + total - total[first][ses]
    return dict(ses=ses, t=t, prompt=prompt, plen=plen, start=start - base, body=body)


def _plan(case, seed):
    """All requests of a trace in time order."""
    rng, fixed = np.random.default_rng(seed), np.random.default_rng(0)
    shape, parts = case["shape"], []
    window = max(case["chats"] * (_TINY if shape == "tiny" else _CHAT)["window"], case["agents"] * _AGENT["window"])
    if shape == "mixed":
        window = max(case["agents"], case["chats"] / 137) * 66.0  # 86,400 s for 1,300 agentic sessions
    if case["chats"]:
        parts.append(_half(rng, fixed, "tiny" if shape == "tiny" else "chat", case["chats"], window))
    if case["agents"]:
        half = _half(rng, fixed, "agentic", case["agents"], window)
        half["ses"] = half["ses"] + case["chats"]
        half["prompt"] = half["prompt"] + 1000
        parts.append(half)
    p = {k: np.concatenate([h[k] for h in parts]) for k in parts[0]}
    at = np.lexsort((np.arange(len(p["t"])), p["t"]))
    p = {k: v[at] for k, v in p.items()}
    p["len"] = p["plen"] + p["body"]
    p["off"] = np.concatenate([[0], np.cumsum(p["len"])])
    p["n"] = int((p["len"] // case["B"]).sum())
    p["ts"] = (p["t"] * 1e6).astype(np.int64)
    p["key"] = rng.integers(1, 2**62)
    return p


def _tokens(p, lead):
    """The trace's tokens, on the GPU, after `lead` tokens of something else."""
    R, T = len(p["len"]), int(p["off"][-1])
    dev = {k: torch.from_numpy(np.ascontiguousarray(p[k])).cuda() for k in ("off", "plen", "len", "start", "ses", "prompt")}
    mult = 0x5851F42D4C957F2D
    prompt_key = (dev["prompt"] + 1) * mult + int(p["key"])
    session_key = (dev["ses"] + 100_000) * mult + int(p["key"])
    out = torch.empty(lead + T, dtype=torch.int32, device="cuda")
    a = 0
    while a < R:  # whole requests, about 2^26 tokens at a time
        b = max(a + 1, int(np.searchsorted(p["off"], p["off"][a] + (1 << 26))) - 1)
        lo, n = int(p["off"][a]), int(p["off"][b] - p["off"][a])
        r = torch.repeat_interleave(torch.arange(a, b, device="cuda"), dev["len"][a:b], output_size=n)
        k = torch.arange(lo, lo + n, device="cuda") - dev["off"][r]
        own = k - dev["plen"][r]
        h = torch.where(own < 0, prompt_key[r], session_key[r])
        h += torch.where(own < 0, k, own + dev["start"][r]) * 0x2545F4914F6CDD1D
        del r, k, own
        for s, m in ((31, 0x369DEA0F31A53F85), (29, 0x27BB2EE687B0B0FD), (32, 1)):
            h ^= (h >> s) & ((1 << (64 - s)) - 1)
            h *= m
        h &= 0x7FFFFFFF
        h *= VOCAB
        h >>= 31
        out[lead + lo: lead + lo + n] = h
        a = b
    return out[lead:]


def _grid(lo, hi, G):
    """G strictly ascending capacities, spread over the logarithm of lo .. hi."""
    lo, hi = max(1, lo), max(1, lo, hi)
    v = np.rint(lo * (hi / lo) ** (np.arange(G) / max(1, G - 1))).astype(np.int64)
    return (np.maximum.accumulate(v - np.arange(G)) + np.arange(G)).astype(np.uint64)


# ------------------------------------------------------------------ states
class _State:
    pass


def prepare(case, seed):
    s = _State()
    s.case = case
    if case["kind"] == "blocks":
        s.ids, s.D, s.blk_off = _block_trace(case, seed)
        s.caps = _grid(64, s.D, case["caps"])
        return s
    p = _plan(case, seed)
    s.n = p["n"]
    s.n_session = case["chats"] + case["agents"]
    tok = _tokens(p, case["lead"])
    off = torch.from_numpy(p["off"])
    ts = torch.from_numpy(p["ts"])
    ses = torch.from_numpy(p["ses"].astype(np.int32))
    B, cost = case["B"], case["cost"]
    s.caps = _grid(64, s.n // 2, case["caps"])
    if case["kind"] == "host":
        host = torch.empty(tok.numel(), dtype=torch.int32, pin_memory=True)
        host.copy_(tok)
        s.plan = ptc.HostPipelinePlan(host, off.pin_memory(), ts.pin_memory(), B, s.caps, cost,
                                      req_session=ses.pin_memory() if case["sessions"] else None,
                                      n_session=s.n_session)
        s.out = (s.plan.hits.view(np.int64), s.plan.saved.view(np.int64))
        return s
    s.tok, s.off, s.ts, s.ses = tok, off.cuda(), ts.cuda(), ses.cuda()
    if case["kind"] == "stages":
        return s
    # every per-access array goes to the caller
    room = max(1, tok.numel() // B)
    buf = {k: torch.empty(room, dtype=torch.int32, device="cuda") for k in ("ids", "prev", "next", "dist")}
    buf["req_blk_off"] = torch.empty(off.numel(), dtype=torch.int64, device="cuda")
    plan = ptc.PipelinePlan(tok, s.off, s.ts, B, s.caps, cost, outputs=buf,
                            req_session=s.ses if case["sessions"] else None, n_session=s.n_session)
    a = {k: v[: s.n] for k, v in buf.items() if k != "req_blk_off"}
    a["req_blk_off"] = buf["req_blk_off"]
    if case["kind"] == "pipeline":
        s.plan = plan
        s.out = (plan.hits.view(np.int64), plan.saved.view(np.int64), a)
        return s
    # the other analyses start from what the path leaves
    s.a = a
    s.D = plan.run().result()["n_distinct"]
    del plan, s.tok
    s.caps = _grid(64, s.D, case["caps"])
    if case["kind"] == "stats":
        s.plan = ptc.TraceStatsPlan(a["ids"], a["prev"], a["next"], s.D, a["req_blk_off"], s.ts, s.ses, s.n_session,
                                    a["dist"], s.caps)
        s.out = (s.plan.buf.view(np.int64), s.plan.reach.view(np.int64))
    return s


def _block_trace(case, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    n, objects = case["accesses"], case["objects"]
    u = torch.rand(n, device="cuda", generator=g, dtype=torch.float64)
    rank = torch.where(torch.rand(n, device="cuda", generator=g) < 0.7,
                       torch.exp(u * float(np.log(objects))), u * objects).long().clamp_(0, objects - 1)
    place = torch.randperm(objects, device="cuda", generator=g)
    distinct, ids = torch.unique(place[rank], return_inverse=True)
    lens = np.random.default_rng(0).integers(1, 9, n)
    off = np.minimum(np.concatenate([[0], np.cumsum(lens)]), n)
    off = off[: int(np.searchsorted(off, n)) + 1]
    return ids.int(), distinct.numel(), torch.from_numpy(off).cuda()


def _words(v):
    """128-bit sums as pairs of 64-bit words, low word first."""
    a = np.array([w for x in v for w in (x & (2**64 - 1), x >> 64)], dtype=np.uint64)
    return a.view(np.int64)


def run(s):
    case = s.case
    kind = case["kind"]
    if kind in ("pipeline", "host", "stats"):
        s.plan.run()
        return s.out
    if kind == "stages":
        o = ptc.pipeline(s.tok, s.off, s.ts, case["B"], s.caps, case["cost"])
        ptc.ptc_verify_ids(s.tok, s.off, o["req_blk_off"], case["B"], o["ids"], o["n_distinct"])
        return (np.array(o["hits"]), _words(o["saved"]),
                {k: o[k] for k in ("keys", "req_blk_off", "ids", "prev", "next", "dist")})
    if kind == "blocks":
        prev, nxt = ptc.ptc_reuse_indices(s.ids, s.D)
        dist = ptc.ptc_stack_distance(prev)
        c = ptc.ptc_curves(dist, s.blk_off, 16, s.caps, ptc.PTC_COST_UNIFORM)
        return np.array(c["hits"]), _words(c["saved"]), prev, nxt, dist
    a = s.a
    if kind == "variant":
        dist = ptc.ptc_stack_distance_variant(a["prev"], a["req_blk_off"], case["order"], case["residency"])
        c = ptc.ptc_curves(dist, a["req_blk_off"], case["B"], s.caps, case["cost"])
        return np.array(c["hits"]), _words(c["saved"]), dist
    if kind == "belady":
        c = ptc.ptc_belady_curves(a["prev"], a["req_blk_off"], case["B"], s.caps, case["cost"])
        return np.array(c["hits"]), _words(c["saved"]), np.array(c["raw_hits"])
    c = ptc.ptc_session_lru_curves(a["ids"], s.D, a["req_blk_off"], s.ses, s.n_session, case["B"], s.caps, case["cost"])
    return np.array(c["hits"]), _words(c["saved"])


def work(case):
    """Inputs read once, results written once."""
    out = 24 * case["caps"]
    if case["kind"] == "blocks":
        n = case["accesses"]
        return {"bytes": 16 * n + 8 * (n // 4.5) + out, "flops": 0}
    p = _plan(case, 0)
    T, n, R = int(p["off"][-1]), p["n"], len(p["len"])
    per_request = 16 * R + (4 * R if case["sessions"] else 0)
    if case["kind"] == "host":
        return {"bytes": 4 * T + per_request + out, "flops": 0}
    if case["kind"] == "pipeline":  # ids, prev, next, dist and block offsets
        return {"bytes": 4 * T + per_request + 8 * R + 16 * n + out, "flops": 0}
    if case["kind"] == "stages":    # keys too; the check reads the tokens
        return {"bytes": 4 * T + per_request + 8 * R + 32 * n + out, "flops": 0}
    if case["kind"] == "variant":   # prev, dist
        return {"bytes": 8 * n + 8 * R + out, "flops": 0}
    if case["kind"] == "stats":     # ids, prev, next, dist
        return {"bytes": 16 * n + 20 * R + out, "flops": 0}
    return {"bytes": 4 * n + 12 * R + out, "flops": 0}  # prev, or ids


def tolerance(case):
    return "exact"  # whole numbers


# ------------------------------------------------------------------ plain restatement
def _lru(ids):
    """prev, next and stack distance of every access, with -1 for none."""
    n = len(ids)
    at = np.argsort(ids, kind="stable")
    same = ids[at][1:] == ids[at][:-1]
    prev, nxt = np.full(n, -1, np.int64), np.full(n, -1, np.int64)
    prev[at[1:][same]] = at[:-1][same]
    nxt[at[:-1][same]] = at[1:][same]
    dist = np.full(n, -1, np.int64)
    tree = [0] * (n + 1)          # Fenwick tree over last touches

    def add(i, v):
        i += 1
        while i <= n:
            tree[i] += v
            i += i & -i

    live = 0
    for i, q in enumerate(prev.tolist()):
        if q >= 0:
            j, below = q + 1, 0
            while j:
                below += tree[j]
                j &= j - 1
            dist[i] = live - below + 1
            add(q, -1)
            live -= 1
        add(i, 1)
        live += 1
    return prev, nxt, dist


def _curves(dist, off, B, caps, kind):
    """Hits and compute saved at every capacity under the prefix rule."""
    far = np.where(dist < 0, NONE, dist)
    hits, saved = [0] * len(caps), [0] * len(caps)
    grid = [int(c) for c in caps]
    for a, b in zip(off[:-1].tolist(), off[1:].tolist()):
        for k, g in enumerate(np.searchsorted(grid, np.maximum.accumulate(far[a:b])).tolist()):
            if g < len(grid):
                seen = B * B * k + B * (B + 1) // 2
                hits[g] += 1
                saved[g] += (1, B * ptc.F_LIN + ptc.F_ATTN * seen, ptc.F_ATTN * seen)[kind]
    return np.cumsum(hits), _words([sum(saved[: g + 1]) for g in range(len(grid))])


def exact(case, seed):
    """The path in plain numpy and Python, for traces of up to 300,000 accesses."""
    i32 = lambda v: v.astype(np.uint32).view(np.int32)  # noqa: E731
    if case["kind"] == "blocks":
        if case["accesses"] > 300_000:
            return None
        ids, D, off = _block_trace(case, seed)
        prev, nxt, dist = _lru(ids.cpu().numpy())
        h, w = _curves(dist, off.cpu().numpy(), 16, _grid(64, D, case["caps"]), ptc.PTC_COST_UNIFORM)
        return h, w, i32(prev), i32(nxt), i32(dist)
    if case["kind"] not in ("pipeline", "host", "stages"):
        return None
    p, B = _plan(case, seed), case["B"]
    if p["n"] > 300_000:
        return None
    tok = _tokens(p, 0).cpu().numpy()
    blk_off = np.concatenate([[0], np.cumsum(p["len"] // B)])
    ids, seen = np.empty(p["n"], np.int64), {}
    for r in range(len(p["len"])):
        parent = -1
        for k in range(int(blk_off[r + 1] - blk_off[r])):
            at = int(p["off"][r]) + k * B
            parent = seen.setdefault((parent, tok[at: at + B].tobytes()), len(seen))
            ids[blk_off[r] + k] = parent
    prev, nxt, dist = _lru(ids)
    h, w = _curves(dist, blk_off, B, _grid(64, p["n"] // 2, case["caps"]), case["cost"])
    if case["kind"] == "host":
        return h, w
    a = {"ids": i32(ids), "prev": i32(prev), "next": i32(nxt), "dist": i32(dist), "req_blk_off": blk_off}
    return h, w, dict(a, keys=None) if case["kind"] == "stages" else a
