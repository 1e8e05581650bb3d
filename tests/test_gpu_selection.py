"""The selection kernel at the sizes where its shape changes, against the CPU oracle (exact:
decisions, reasons, caps and protected counts): one CTA and clusters, batches just above a
shape's limit, several windows, instance counts whose price orders do not fit shared memory, and
an Eq. (7) leader that has to give a proposal back."""

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
    (256, 40, 0), (257, 40, 1), (1024, 7, 2), (1025, 33, 0),   # one CTA; the smallest cluster
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
