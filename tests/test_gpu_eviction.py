"""Eviction at the shapes where its selection changes (exact, against the oracle): whole and sampled
tables, more instances than SMs, a table that stays sparse after it was far over capacity, long prompts
in one tick, equal ticks that only the key decides, holes in runs of full buckets."""

import numpy as np
import pytest

from tests.gpu_helpers import compare_state, make_router, route_both
from tests.helpers import make_oracle
from tests.test_gpu_selection import _batch, _scenario

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    import __graft_entry__

    __graft_entry__.build()


@pytest.mark.parametrize("W,cap,n,hi,index", [
    (3, 50, 40, 300, 0),        # tables of a few buckets, whole in the sample
    (2, 4000, 60, 9000, 1),     # 2,048 buckets: the largest table that is
    (2, 4200, 60, 9000, 0),     # 4,096: sampled
    (200, 60, 500, 400, 0),     # more instances than SMs
    (1, 40000, 250, 16000, 1),  # thousands of candidates
])
def test_eviction_over_table_sizes(W, cap, n, hi, index):
    rng = np.random.default_rng(W + cap)
    caps = rng.integers(cap - cap // 8, cap + 1, W)
    ses = iter(range(1, 1 << 20))
    batches = []
    for k in range(5):
        lens = rng.integers(0, hi, n)
        # the first batch floods one instance: its table grows and is sparse afterwards
        batches.append(_batch(rng, rng.integers(0, 3, n), [next(ses) for _ in range(n)], lens, shared=32 * (k % 2)))
    sc = _scenario(W, caps, 3, rng.integers(0, 5, W), rng.integers(1, 4, W), np.zeros(W), batches)
    r, o = make_router(sc, max_sessions=8 * n, prefix_index=index), make_oracle(sc)
    try:
        for k, b in enumerate(batches):
            back = rng.permutation(W).astype(np.int64) * (10_000_000 if k == 0 else 1000)
            for x in (r, o):
                x.set_instance_state(back, None, None)
            route_both(r, o, b, W, check_H=False, check_keys=False)
            r.commit()
            o.commit()
            compare_state(r, o, W)
    finally:
        r.close()


@pytest.mark.parametrize("n,cap", [(70, 30), (3000, 1000), (20000, 7777)])
def test_equal_ticks_go_by_the_key(n, cap):
    rng = np.random.default_rng(n)
    keys = np.unique(rng.integers(2, 1 << 63, size=n, dtype=np.uint64))
    metas = np.full(len(keys), (5 << 36) | (7 << 16) | (65535 - 3), np.uint64)
    metas[::7] = (4 << 36) | (1 << 16) | 65535  # older ones among them
    b = _batch(rng, [0], [1], [16])
    sc = _scenario(1, [cap], 3, [0], [1], [0], [b])
    for index in (0, 1):
        r, o = make_router(sc, prefix_index=index), make_oracle(sc)
        try:
            for x in (r, o):
                x.load_entries(0, keys, metas)
            gk, gm = r.dump_index(0)
            ok_, om = o.dump_index(0)
            assert np.array_equal(gk, ok_) and np.array_equal(gm, om)
        finally:
            r.close()
