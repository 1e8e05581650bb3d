"""The selection kernel at the sizes where its shape changes, against the CPU oracle (exact:
decisions, reasons, caps and protected counts): one CTA and clusters, batches just above a
shape's limit, several windows, instance counts whose price orders do not fit shared memory, an
Eq. (7) leader that has to give a proposal back, and ties between a cached instance and others."""

import itertools

import numpy as np
import pytest

from paper_2608_11152_gb300 import workload as wl
from tests.gpu_helpers import compare_state, make_router, route_both
from tests.helpers import make_oracle

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    import __graft_entry__

    __graft_entry__.build()


def _batch(rng, cls, session, lens, shared=0):
    """Prompts of the given lengths; `shared` leading tokens are the same in all of them."""
    off = np.zeros(len(lens) + 1, np.int64)
    np.cumsum(lens, out=off[1:])
    tok = rng.integers(0, wl.VOCAB, size=int(off[-1]), dtype=np.int32)
    for r in range(len(lens)):
        m = min(shared, int(lens[r]))
        tok[off[r]:off[r] + m] = np.arange(m)
    return wl.Batch(cls=np.asarray(cls, np.uint8), session=np.asarray(session, np.uint64),
                    group=np.zeros(len(lens), np.uint64), tok_off=off, tokens=tok)


def _scenario(W, cap, mode, backlog, tokcost, contraction, batches, hold=0):
    sc = wl.Scenario(name="selection", W=W, cap_blocks=np.asarray(cap, np.int64), rho_ppm=(400000, 300000, 300000),
                     prior_kbar=(4, 4, 4), prior_T_us=1_000_000, backlog_q=np.asarray(backlog, np.int64),
                     tokcost_q=np.asarray(tokcost, np.int64), contraction=np.asarray(contraction, np.int32),
                     hold_delay_q=hold, mode=mode)
    sc.max_batch = max(b.n for b in batches)
    sc.max_tokens = max(b.n_tokens for b in batches)
    return sc


@pytest.mark.parametrize("n,W,mode", [
    (256, 7, 0), (257, 7, 1), (512, 31, 0),                    # one CTA of 256 and 512 threads
    (513, 31, 1), (33, 32, 2), (1, 40, 0), (256, 40, 0), (257, 40, 1), (1024, 7, 2), (1025, 33, 0),  # clusters
    (4096, 100, 2), (4097, 100, 0), (8193, 64, 1),             # 256, 512 and 1024 threads a CTA
    (16500, 12, 0), (40000, 24, 2),                            # two and three windows
    (3000, 1000, 0), (9000, 513, 2),                           # price orders read from global memory
    (700, 1, 0), (500, 1024, 3),
])
def test_selection_shapes_match_the_oracle(n, W, mode):
    rng = np.random.default_rng(n + W)
    per = max(2, n // (2 * W))  # about half of the leaders find headroom
    ses = np.arange(1, n + 1, dtype=np.uint64)
    cls = rng.integers(0, 3, n)
    b0 = _batch(rng, cls, ses, rng.integers(0, 60, n), shared=16)
    # half of the sessions come again, some after a release (continuations and Eq. 7 leaders)
    ses1 = np.where(rng.random(n) < 0.5, ses, ses + np.uint64(n))
    cls1 = np.where(ses1 <= n, cls, rng.integers(0, 3, n))
    b1 = _batch(rng, cls1, ses1, rng.integers(0, 60, n), shared=16)
    # few distinct costs, so that ties go by the index
    sc = _scenario(W, rng.integers(4 * per, 6 * per + 8, W), mode, rng.integers(0, 4, W) * 1000,
                   rng.integers(1, 5, W) * 100, rng.integers(0, 2, W), [b0, b1], hold=300)
    r, o = make_router(sc, max_sessions=4 * n), make_oracle(sc)
    try:
        for b in (b0, b1):
            route_both(r, o, b, W, check_H=False, check_keys=False)
            r.commit()
            o.commit()
            compare_state(r, o, W, index=False)
            pick = ses[rng.random(n) < 0.4]
            z = [np.zeros(len(pick), t) for t in (np.uint8, np.int32, np.int64, np.uint8)]
            ids = dict(zip(b.session.tolist(), b.cls.tolist()))
            z[0][:] = [ids.get(s, 0) for s in pick.tolist()]
            for x in (r, o):
                x.complete(pick, *z)
    finally:
        r.close()


@pytest.mark.parametrize("tail", [1, 40, 1500])
def test_a_leader_that_must_wait_gives_its_proposal_back(tail):
    """Leader i (released, cached on the slow instance 0) is cheapest on instance 1 as long as
    instance 0 has headroom, and waits once it has none (Eq. 7).  The last headroom of
    instance 0 goes to an earlier leader only after that one was refused by instance 2, so i
    has proposed to 1 by then; a later leader gets that place."""
    rng = np.random.default_rng(tail)
    first = _batch(rng, [2], [7], [400], shared=256)
    lens = np.concatenate([[32, 32, 1600], np.full(tail, 32)])
    ses = np.concatenate([[101, 102, 7], 200 + np.arange(tail)])
    second = _batch(rng, np.full(len(lens), 2), ses, lens)
    second.tokens[64:64 + 400] = first.tokens  # i continues session 7
    W = 3
    sc = _scenario(W, [64] * W, 2, [0, 50_000, 60_000], [1, 1, 1], [13] * W, [first, second])  # K_w = 1
    r, o = make_router(sc), make_oracle(sc)
    try:
        route_both(r, o, first, W)
        for x in (r, o):
            x.commit()
            x.complete([7], [2], [0], [0], [0])
            x.set_instance_state(np.array([0, 50_000, 0]), np.array([100, 1, 0]), None)
        out = route_both(r, o, second, W)
        assert out["inst"][:4].cpu().tolist() == [2, 0, -1, 1]
        assert int(out["reason"][2]) == 19  # HOLD_PREFER_CACHE
        for x in (r, o):
            x.commit()
        compare_state(r, o, W)
    finally:
        r.close()


def _load(x, prompts, inst):
    """Makes the full blocks of prompts[i] resident on instance inst[i]."""
    off = np.concatenate([[0], np.cumsum([len(p) for p in prompts])]).astype(np.int64)
    n = len(prompts)
    x.load_chains(off, np.concatenate(prompts).astype(np.int32), np.asarray(inst, np.int32), np.zeros(n, np.uint64),
                  np.arange(n, dtype=np.uint32), np.full(n, 1 << 16, np.int32))


@pytest.mark.parametrize("slow,cheap,cached", list(itertools.permutations(range(3))))
def test_a_tie_with_a_cached_instance_goes_to_the_lower_index(slow, cheap, cached):
    """At the start of its price cell (992 tokens) `slow` and `cheap` cost the same; 8 tokens on, `cheap`
    costs what `cached` does with its 400 tokens, and `slow` 16 more."""
    rng = np.random.default_rng(1)
    back, cost = np.zeros(3, np.int64), np.zeros(3, np.int64)
    back[slow], cost[slow] = 3016, 7
    back[cheap], cost[cheap] = 5000, 5
    back[cached], cost[cached] = 6400, 6
    b = _batch(rng, [0], [1], [1000])
    sc = _scenario(3, [1000] * 3, 3, back, cost, [0] * 3, [b])
    r, o = make_router(sc), make_oracle(sc)
    try:
        for x in (r, o):
            _load(x, [b.tokens[:400]], [cached])
        out = route_both(r, o, b, 3)
        assert int(out["inst"][0]) == min(cheap, cached)
    finally:
        r.close()


def _tie_costs(rng, W, length, hits):
    """(d_w, 1/mu_w): most instances without a cached prefix cost the same at the start of the prompt's
    price cell, and the cheapest a token of them what one or two cached ones do with their prefix."""
    start = length >> (length.bit_length() - 5) << (length.bit_length() - 5)
    cost = rng.integers(2, 7, W)
    back = np.where(hits > 0, 40 * length - (length - 16 * hits) * cost,
                    40 * length - (length - start) * cost.min() - start * cost)
    return back + np.where(rng.random(W) < np.where(hits > 0, 1 - 2 / W, 0.2), rng.integers(1, 20, W), 0), cost


@pytest.mark.parametrize("W,mode,length", [(6, 3, 47), (20, 3, 70), (20, 0, 1000), (200, 2, 1000), (1000, 3, 5003)])
def test_ties_between_cached_and_other_instances(W, mode, length):
    rng = np.random.default_rng(W + length)
    n = 300 if mode == 3 else 30 * W  # more than the instances take
    b = _batch(rng, rng.integers(0, 3, n), np.arange(1, n + 1), np.full(n, length), shared=length)
    hits = np.where(rng.random(W) < 0.4, rng.integers(1, length // 16 + 1, W), 0)
    sc = _scenario(W, [1000 if mode == 3 else 100] * W, mode, np.zeros(W), np.ones(W), rng.integers(0, 2, W), [b])
    r, o = make_router(sc), make_oracle(sc)
    try:
        on = np.flatnonzero(hits)
        for x in (r, o):
            for at in np.array_split(on, -(-len(on) // 100)):
                _load(x, [b.tokens[:16 * h] for h in hits[at]], at)
        for _ in range(12):
            back, cost = _tie_costs(rng, W, length, hits)
            for x in (r, o):
                x.set_instance_state(back, cost, None)
            route_both(r, o, b, W)
    finally:
        r.close()
