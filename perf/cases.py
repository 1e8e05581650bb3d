"""The calls that a user of this router makes, as cases to be timed.

Most cases are the serving loop of a rollout router in its steady state: a batch of requests
arrives, misat_route decides it, misat_commit applies the decisions, and misat_complete reports
the sessions that finished or released their protection meanwhile.  A state holds a ring of
batches that is long enough for the least recently used blocks to be evicted again before
their prompts return, and prepare() goes round it once, so every timed pass meets full
indexes, real evictions and partly resident prompts; one pass routes and commits the next
batch of the ring.  Each pass therefore depends on every commit, eviction and completion before
it: its decisions and its H matrix (longest cached prefix per request and instance) are wrong
when any of them was.  Other cases take the same loop from host memory (one call, or staged in
the delta layout), or hash blocks without the router.

Batches follow the repository's synthetic workloads: RLVR groups whose samples share a short
prompt, independent RLHF prompts, and agentic sessions whose prompt is the history so far plus
the new turn (several turns in a batch, and a session continues in the next batch).
"""

import math

import numpy as np
import torch

from paper_2608_11152_gb300 import misat

VOCAB = 151936
G = 0x9E3779B97F4A7C15

# Prompt lengths and session shapes (tokens, uniform ranges) of the repository's workloads.
MIXED = dict(rlvr_lo=64, rlvr_hi=1024, fanout=8, rlhf_lo=512, rlhf_hi=2048, first_lo=1000, first_hi=4000,
             add_lo=200, add_hi=1500, turns=5, life=2)
TINY = dict(rlvr_lo=128, rlvr_hi=512, fanout=4, rlhf_lo=512, rlhf_hi=1024, first_lo=1024, first_hi=4096,
            add_lo=100, add_hi=400, turns=4, life=2)


def listed():
    return [
        # a small deployment decides a handful of arrivals from host memory: latency of one call
        dict(TINY, name="online_host_4x2048_n24", kind="host", W=4, cap=2048, n=24, p_rlvr=0.5, p_rlhf=0.25,
             mode=0, index=0),
        # the tiny batch of the repository's first configuration, on device buffers
        dict(TINY, name="tiny_4x2048_n64", kind="route", W=4, cap=2048, n=64, p_rlvr=0.5, p_rlhf=0.25, mode=0,
             index=0),
        # medium mixed cluster with the default (global) prefix index
        dict(MIXED, name="medium_16x65536_n4096", kind="route", W=16, cap=65536, n=4096, p_rlvr=0.4, p_rlhf=0.3,
             mode=0, index=0),
        # RLVR-heavy: wide fan-out of short prompts, per-instance index
        dict(MIXED, name="rlvr_32x131072_n16384", kind="route", W=32, cap=131072, n=16384, p_rlvr=0.7, p_rlhf=0.15,
             mode=0, index=1, rlvr_hi=512, fanout=16),
        # long agentic sessions, one turn per batch, histories up to 128K tokens that stay resident
        dict(MIXED, name="agentic_64x131072_n9216", kind="route", W=64, cap=131072, n=9216, p_rlvr=0.445,
             p_rlhf=0.445, mode=0, index=0, first_lo=200, first_hi=120000, add_hi=2000, turns=1, life=4),
        # the throughput batch of the repository's benchmark
        dict(MIXED, name="stress_128x262144_n65536", kind="route", W=128, cap=262144, n=65536, p_rlvr=0.4,
             p_rlhf=0.3, mode=0, index=1),
        # many small instances, an ordinary batch: the index masks take two words
        dict(MIXED, name="wide_128x16384_n4096", kind="route", W=128, cap=16384, n=4096, p_rlvr=0.4, p_rlhf=0.3,
             mode=0, index=0),
        # class-agnostic session admission: the global caps bind; odd sizes throughout
        dict(MIXED, name="session_cap_23x50001_n6001", kind="route", W=23, cap=50001, n=6001, p_rlvr=0.4,
             p_rlhf=0.3, mode=2, index=1),
        # placement without admission control over close to the largest instance count
        dict(MIXED, name="placement_1000x3000_n3001", kind="route", W=1000, cap=3000, n=3001, p_rlvr=0.4,
             p_rlhf=0.3, mode=3, index=0),
        # a burst of very short prompts with the spatial quota: many requests, few tokens
        dict(MIXED, name="burst_64x131072_n131072", kind="route", W=64, cap=131072, n=131072, p_rlvr=0.4, p_rlhf=0.3,
             mode=1, index=1, rlvr_lo=8, rlvr_hi=96, rlhf_lo=16, rlhf_hi=128, first_lo=32, first_hi=160, add_lo=8,
             add_hi=48),
        # batches that arrive in pinned host memory in the delta layout, copied while the last one runs
        dict(MIXED, name="staged_delta_32x65536_n8192", kind="delta", W=32, cap=65536, n=8192, p_rlvr=0.4,
             p_rlhf=0.3, mode=0, index=1),
        # an engine hashes prompt blocks without allocating device memory
        dict(MIXED, name="block_hash_n20001", kind="hash", n=20001, p_rlvr=0.4, p_rlhf=0.3, life=1),
    ]


def draw(rng):
    """A case of the same ranges: any kind, instance counts, capacities, batch sizes, mixes and modes."""

    def log_int(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choices(["route", "host", "delta", "hash"], [12, 2, 2, 2])[0]
    hi = log_int(64, 3000)
    lo = rng.randint(1, hi)
    p1 = rng.uniform(0.1, 0.8)
    first = log_int(32, 8000)
    add = log_int(8, 2000)
    c = dict(kind=kind, n=log_int(1, 40000), p_rlvr=round(p1, 3), p_rlhf=round(rng.uniform(0.1, 0.9) * (1 - p1), 3),
             rlvr_lo=lo, rlvr_hi=hi, fanout=rng.choice([1, 2, 4, 8, 16]), rlhf_lo=rng.randint(1, hi), rlhf_hi=hi,
             first_lo=rng.randint(1, first), first_hi=first, add_lo=rng.randint(1, add), add_hi=add,
             turns=rng.randint(1, 6), life=1 if kind == "hash" else rng.choice([1, 2, 4]))
    while _tokens(c) > (2e7 if kind in ("host", "delta") else 1e8):
        c["n"] = max(1, c["n"] // 2)
    if kind != "hash":
        c["W"] = log_int(1, 700)
        c["cap"] = max(256, min(log_int(1000, 200000), 16_000_000 // c["W"]))
        # an H matrix no larger than the listed ones, a cache that holds a few batches
        while c["n"] > 1 and (c["W"] * c["n"] > 1 << 23 or _distinct(c) > 4 * c["W"] * c["cap"]):
            c["n"] //= 2
        c["mode"] = rng.choices([0, 1, 2, 3], [6, 2, 2, 2])[0]
        c["index"] = rng.randint(0, 1)
    return c


# ---- sizes that follow from a case


def _split(c):
    """Requests of each class, and agentic sessions per batch."""
    n1 = min(c["n"], int(round(c["n"] * c["p_rlvr"])))
    n2 = min(c["n"] - n1, int(round(c["n"] * c["p_rlhf"])))
    n3 = c["n"] - n1 - n2
    return n1, n2, n3, -(-n3 // c["turns"])


def _mean(c, k):
    return (c[k + "_lo"] + c[k + "_hi"]) / 2


def _tokens(c):
    """Expected prompt tokens of one batch."""
    n1, n2, n3, _ = _split(c)
    turns = (c["turns"] * c["life"] - 1) / 2  # turns appended before a turn, on average
    return n1 * _mean(c, "rlvr") + n2 * _mean(c, "rlhf") + n3 * (_mean(c, "first") + turns * _mean(c, "add"))


def _distinct(c):
    """Expected prompt tokens of one batch that no earlier request of the ring has sent."""
    n1, n2, n3, s = _split(c)
    return (-(-n1 // c["fanout"]) * _mean(c, "rlvr") + n2 * _mean(c, "rlhf") + s * _mean(c, "first") / c["life"] +
            n3 * _mean(c, "add"))


def _prior(c):
    """Blocks per session of each class before any has completed: mean prompt and median decode."""
    return (math.ceil((_mean(c, "rlvr") + 4096) / 16), math.ceil((_mean(c, "rlhf") + 1024) / 16),
            math.ceil((_mean(c, "first") + 256) / 16))


def _ring(c):
    """Batches in the ring: enough that their admitted sessions bring three times the capacity's worth of
    new blocks, within 32 batches and 24 GB of tokens; a multiple of a session's life."""
    if c["kind"] == "hash":
        return 1
    n1, n2, _, s = _split(c)
    blocks = sum(a * b for a, b in zip((n1, n2, s), _prior(c)))
    admitted = 1.0 if c["mode"] == 3 else min(1.0, 0.6 * c["W"] * c["cap"] / blocks)
    k = math.ceil(3 * c["W"] * c["cap"] * 16 / max(1.0, _distinct(c) * admitted))
    k = max(4, min(32, int(6e9 / _tokens(c)), k))
    return -(-k // c["life"]) * c["life"]


def _most_blocks(c):
    """Blocks of a batch of a hash case whose prompts all have their largest size."""
    n1, n2, n3, _ = _split(c)
    return max(1, (n1 * c["rlvr_hi"] + n2 * c["rlhf_hi"] + n3 * (c["first_hi"] + c["turns"] * c["add_hi"])) // 16)


def work(case):
    """Tokens and request fields read once, decisions and keys (or H rows) written once."""
    n, t = case["n"], _tokens(case)
    if case["kind"] == "hash":
        return {"bytes": 4 * t + 8 * n + 8 * t / 16, "flops": 0}
    sent = _distinct(case) if case["kind"] == "delta" else t
    out_h = 2 * n * case["W"] if case["kind"] == "route" else 0
    # the index: 16 bytes written for every block that no earlier request has sent
    return {"bytes": 4 * sent + 26 * n + out_h + _distinct(case), "flops": 0}


def tolerance(case):
    return "exact"  # every output is a whole number


# ---- inputs


def _uniform(gen, lo, hi, shape):
    return torch.randint(int(lo), int(hi) + 1, shape, generator=gen, device="cuda")


def _make_ring(c, seed):
    """The ring's batches on the GPU: (cls, session, tok_off, tokens, base, own) each, in arrival order.
    base / own: the delta layout's base request and own token count."""
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    n, K, t, life = c["n"], _ring(c), c["turns"], c["life"]
    n1, n2, n3, S = _split(c)
    dev = "cuda"
    # agentic sessions: slot j starts a new one every `life` batches (slots take turns); its
    # buffer holds the first prompt and every turn's addition, a turn's prompt is a prefix
    E = K // life
    slot = torch.arange(S, device=dev)
    first = _uniform(gen, c["first_lo"], c["first_hi"], (S, E, 1))
    adds = _uniform(gen, c["add_lo"], c["add_hi"], (S, E, t * life - 1))
    plen = torch.cat([first, adds], 2).cumsum(2).clamp_(max=(1 << 20) - 16)  # [S, E, t * life] prompt of each turn
    alen = plen[:, :, -1].reshape(-1)
    astart = (alen.cumsum(0) - alen).reshape(S, E)
    apool = torch.randint(0, VOCAB, (max(1, int(alen.sum())),), generator=gen, device=dev, dtype=torch.int32)
    sid0 = (seed % 4096 + 1) << 40
    g1 = -(-n1 // c["fanout"])
    grp = torch.arange(n1, device=dev) // c["fanout"]
    out = []
    for k in range(K):
        glen = _uniform(gen, c["rlvr_lo"], c["rlvr_hi"], (g1,))
        hlen = _uniform(gen, c["rlhf_lo"], c["rlhf_hi"], (n2,))
        plens = torch.cat([glen, hlen])
        pstart = plens.cumsum(0) - plens
        own_pool = torch.randint(0, VOCAB, (max(1, int(plens.sum())),), generator=gen, device=dev, dtype=torch.int32)
        pool = torch.cat([own_pool, apool])
        # the agentic slots' epoch and part of their life in this batch
        age = k + slot % life
        ep, part = (age // life) % E, age % life
        turn = part[:, None] * t + torch.arange(t, device=dev)
        al = plen[slot[:, None], ep[:, None], turn].reshape(-1)[:n3] if n3 else slot[:0]
        ast = (astart[slot, ep][:, None].expand(S, t).reshape(-1)[:n3] + own_pool.numel()) if n3 else slot[:0]
        asid = (sid0 + (1 << 38) + slot * E + ep)[:, None].expand(S, t).reshape(-1)[:n3] if n3 else slot[:0]
        lens = torch.cat([glen[grp], hlen, al])
        start = torch.cat([pstart[:g1][grp], pstart[g1:], ast])
        ses = torch.cat([sid0 + 1 + k * n + torch.arange(n1 + n2, device=dev), asid])
        cls = torch.cat([torch.full((n1,), 0, device=dev), torch.full((n2,), 1, device=dev),
                         torch.full((n3,), 2, device=dev)])
        # arrival order: random, a session's turns in order
        u = torch.rand(n1 + n2, generator=gen, device=dev, dtype=torch.float64)
        ua = torch.rand((S, t), generator=gen, device=dev, dtype=torch.float64).sort(1).values.reshape(-1)[:n3]
        order = torch.argsort(torch.cat([u, ua]))
        lens, start = lens[order], start[order]
        off = torch.zeros(n + 1, dtype=torch.int64, device=dev)
        off[1:] = lens.cumsum(0)
        total = int(off[-1])
        idx = torch.repeat_interleave(start - off[:-1], lens, output_size=total)
        idx += torch.arange(total, device=dev)
        tokens = torch.zeros(max(4, (total + 3) // 4 * 4), dtype=torch.int32, device=dev)
        tokens[:total] = pool[idx]
        del idx
        b = dict(n=n, n_tokens=total, cls=cls[order].to(torch.uint8), session=ses[order], tok_off=off, tokens=tokens)
        if c["kind"] == "delta":
            # a turn extends its session's last turn in the batch, a sample repeats its group's first
            place = torch.empty(n, dtype=torch.int64, device=dev)
            place[order] = torch.arange(n, device=dev)
            base = torch.full((n,), -1, dtype=torch.int64, device=dev)
            if n1:
                lead = torch.full((g1,), n, dtype=torch.int64, device=dev).scatter_reduce(0, grp, place[:n1], "amin")
                base[:n1] = torch.where(lead[grp] == place[:n1], -1, lead[grp])
            if n3:
                ap = place[n1 + n2:]
                prev = torch.cat([ap.new_full((1,), -1), ap[:-1]])
                prev[torch.arange(n3, device=dev) % t == 0] = -1
                base[n1 + n2:] = prev
            b["base"] = base[order].to(torch.int32)
        out.append(b)
    return out


def _completions(c, ring, seed):
    """After each batch: its RLVR and RLHF sessions and the agentic ones that end are done; half of
    the agentic sessions that go on release their protection (a tool call runs)."""
    rng = np.random.default_rng(seed)
    n1, n2, n3, S = _split(c)
    life, t = c["life"], c["turns"]
    out = []
    for k, b in enumerate(ring):
        ses = b["session"].cpu().numpy().view(np.uint64)
        cls = b["cls"].cpu().numpy()
        lens = np.diff(b["tok_off"].cpu().numpy())
        # the last request of each session
        last = len(ses) - 1 - np.unique(ses[::-1], return_index=True)[1]
        s, cl, ln = ses[last], cls[last], lens[last]
        done = np.ones(len(s), np.uint8)
        keep = np.ones(len(s), bool)
        ag = cl == 2
        if ag.any():
            K = len(ring)
            j = ((s[ag] - np.uint64(((seed % 4096 + 1) << 40) + (1 << 38))) // np.uint64(K // life)).astype(np.int64)
            going = (k + j % life) % life != life - 1
            done[ag] = ~going
            keep[ag] = ~going | (j % 4 < 2)
        decode = np.exp(rng.normal(0, 0.61, len(s))) * np.where(cl == 0, 4096, np.where(cl == 1, 1024, 256))
        decode = np.clip(decode, 1, 32768).astype(np.int64)
        out.append(tuple(a[keep] for a in (s, cl, (-(-(ln + decode) // 16)).astype(np.int32), decode * 25_000, done)))
    return out


class _Host:
    """A batch in pinned host memory, with the fields that the host calls read."""

    def __init__(self, b, fields):
        self.n = b["n"]
        self.n_tokens = b["n_tokens"]
        self._keep = {}
        for name in fields:
            t = b[name].cpu().pin_memory()
            self._keep[name] = t
            a = t.numpy()
            setattr(self, name, a.view(np.uint64) if name == "session" else a)


def _delta(b):
    """A ring batch in the delta layout, in pinned host memory."""
    off, base = b["tok_off"], b["base"].long()
    lens = off[1:] - off[:-1]
    skip = torch.where(base >= 0, lens[base.clamp(min=0)], 0)
    own = lens - skip
    doff = torch.zeros_like(off)
    doff[1:] = own.cumsum(0)
    total = int(doff[-1])
    idx = torch.repeat_interleave(off[:-1] + skip - doff[:-1], own, output_size=total)
    idx += torch.arange(total, device=idx.device)
    d = dict(n=b["n"], n_tokens=b["n_tokens"], cls=b["cls"], session=b["session"], base=b["base"], delta_off=doff,
             delta_tokens=b["tokens"][idx])
    return _Host(d, ("cls", "session", "base", "delta_off", "delta_tokens"))


def prepare(case, seed):
    c = case
    if c["kind"] == "hash":
        b = _make_ring(c, seed)[0]
        return dict(case=c, b=b, keys=torch.zeros(_most_blocks(c), dtype=torch.int64, device="cuda"))
    ring = _make_ring(c, seed)
    comp = _completions(c, ring, seed)
    rng = np.random.default_rng(seed + 7)
    W, n = c["W"], c["n"]
    r = misat.Router(np.full(W, c["cap"], np.int64), max_batch=n, max_tokens=max(b["n_tokens"] for b in ring),
                     max_sessions=len(ring) * n + 1024, mode=c["mode"], hold_delay_q=50_000_000, prior_kbar=_prior(c),
                     prefix_index=c["index"])
    rho1, rho2 = int(c["p_rlvr"] * 1_000_000), int(c["p_rlhf"] * 1_000_000)
    r.set_mixture([rho1, rho2, 1_000_000 - rho1 - rho2])
    # d_w: nanoseconds of queued prefill, 1/mu_w: nanoseconds per prompt token
    tokcost = rng.integers(20_000, 40_001, size=W, dtype=np.int64)
    backlog = [rng.integers(0, 20_000_000, size=W, dtype=np.int64) for _ in ring]
    r.set_instance_state(backlog[0], tokcost, np.zeros(W, np.int32))
    s = dict(case=c, r=r, comp=comp, backlog=backlog, k=0)
    if c["kind"] == "route":
        s["ring"] = ring
        s["out"] = r.alloc_decisions(n)
        s["H"] = torch.zeros(n * W, dtype=torch.int16, device="cuda")
    elif c["kind"] == "host":
        s["ring"] = [_Host(b, ("cls", "session", "tok_off", "tokens")) for b in ring]
    else:
        s["ring"] = [_delta(b) for b in ring]
        r.stage_host_delta(s["ring"][0], 0)
    for _ in ring:
        run(s)
    r.sync()
    return s


def run(state):
    """One batch of the serving loop (or one hash call)."""
    s = state
    kind = s["case"]["kind"]
    if kind == "hash":
        b = s["b"]
        misat.block_hash_noalloc(b["tok_off"], b["tokens"], b["n"], b["n_tokens"], s["keys"])
        return s["keys"]
    r, k = s["r"], s["k"]
    K = len(s["ring"])
    j = k % K
    s["k"] = k + 1
    # the engines' queue lengths at this batch
    r.set_instance_state(s["backlog"][j])
    if kind == "route":
        r.route(s["ring"][j], out=s["out"], out_H=s["H"])
        out = dict(s["out"], H=s["H"])
    elif kind == "host":
        out = r.route_host(s["ring"][j])
    else:
        # the next batch's copy overlaps this one
        r.stage_host_delta(s["ring"][(j + 1) % K], (k + 1) % 2)
        out = r.route_staged(k % 2)
    r.commit()
    r.complete(*s["comp"][j])
    return out


def exact(case, seed):
    """The block keys in plain 64-bit numpy; None for the router's decisions (a serial policy)."""
    if case["kind"] != "hash":
        return None
    b = _make_ring(case, seed)[0]
    off = b["tok_off"].cpu().numpy()
    tok = b["tokens"].cpu().numpy().view(np.uint32).astype(np.uint64)
    u = np.uint64
    nb = np.diff(off) // 16
    kb = np.cumsum(nb) - nb

    def mix(z):
        z = (z ^ (z >> u(30))) * u(0xBF58476D1CE4E5B9)
        z = (z ^ (z >> u(27))) * u(0x94D049BB133111EB)
        return z ^ (z >> u(31))

    keys = np.zeros(_most_blocks(case), u)
    a = np.full(len(nb), G, u)
    with np.errstate(over="ignore"):
        for j in range(int(nb.max(initial=0))):
            live = np.nonzero(nb > j)[0]
            p = off[live] + 16 * j
            c = np.zeros(len(live), u)
            for i in range(8):
                x = tok[p + 2 * i] | (tok[p + 2 * i + 1] << u(32))
                c ^= (x + u((i + 1) * G & (2**64 - 1))) * u(0x94D049BB133111EB)
            a[live] = a[live] * u(G) + mix(c)
            key = mix(a[live] ^ u(j + 1))
            keys[kb[live] + j] = key + u(2) * (key < u(2))
    return torch.from_numpy(keys.view(np.int64))
