"""Eviction at the shapes where its selection changes (exact, against the oracle): whole and sampled
tables, more instances than SMs, a table that stays sparse after it was far over capacity, long prompts
in one tick, equal ticks that only the key decides, holes in runs of full buckets, ticks beyond those
that the sample of a table meets."""

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


@pytest.mark.parametrize("n,cap", [(9, 5), (600, 64), (600, 599), (3000, 2100), (7000, 4200)])
def test_the_largest_ticks(n, cap):
    """Sequence numbers, arrivals and depths up to the limits of their fields, in whole and in sampled
    tables, with the last entry to leave among the smallest, the middle and the largest."""
    rng = np.random.default_rng(n + cap)
    keys = np.unique(rng.integers(2, 1 << 63, size=n, dtype=np.uint64))
    b = _batch(rng, [0], [1], [16])
    sc = _scenario(1, [cap], 3, [0], [1], [0], [b])
    for old in (0.05, 0.5, 0.95):  # share of small sequence numbers
        seq = np.where(rng.random(len(keys)) < old, rng.integers(0, 3, len(keys)), (1 << 28) - 1 - rng.integers(0, 3, len(keys)))
        arr = rng.choice([0, 1, 77, 1 << 19, (1 << 20) - 1], len(keys))
        metas = seq.astype(np.uint64) << np.uint64(36) | arr.astype(np.uint64) << np.uint64(16)
        metas |= np.uint64(65535) - rng.choice([0, 1, 300, 65534], len(keys)).astype(np.uint64)
        r, o = make_router(sc), make_oracle(sc)
        try:
            for x in (r, o):
                x.load_entries(0, keys, metas)
            gk, gm = r.dump_index(0)
            ok_, om = o.dump_index(0)
            assert np.array_equal(gk, ok_) and np.array_equal(gm, om)
        finally:
            r.close()


GOLD = 0x9E3779B97F4A7C15
BUCKETS_LOG2 = 12  # an instance of 4,097 to 8,192 blocks; its even buckets are the sample


def _keys_at_home(rng, odd, taken):
    """One key per entry of `odd`, home in an odd or an even bucket of the table as it says, at most four
    to a bucket (so that every entry stays in its home bucket)."""
    out = np.zeros(len(odd), np.uint64)
    left = {0: list(np.flatnonzero(~odd)), 1: list(np.flatnonzero(odd))}
    while left[0] or left[1]:
        for k in np.unique(rng.integers(2, 1 << 63, size=20000, dtype=np.uint64)).tolist():
            home = ((k * GOLD) & (2**64 - 1)) >> (64 - BUCKETS_LOG2)
            todo = left[home & 1]
            if todo and taken.get(home, 0) < 4:
                taken[home] = taken.get(home, 0) + 1
                out[todo.pop()] = k
    return out


def _load_and_compare(keys, metas, cap, index):
    b = _batch(np.random.default_rng(0), [0], [1], [16])
    sc = _scenario(1, [cap], 3, [0], [1], [0], [b])
    r, o = make_router(sc, prefix_index=index), make_oracle(sc)
    try:
        assert r.table_buckets(0) == 1 << BUCKETS_LOG2
        for x in (r, o):
            x.load_entries(0, keys, metas)
        gk, gm = r.dump_index(0)
        ok_, om = o.dump_index(0)
        assert len(gk) == cap
        assert np.array_equal(gk, ok_) and np.array_equal(gm, om)
        assert r.table_buckets(0) == 1 << BUCKETS_LOG2
    finally:
        r.close()


@pytest.mark.parametrize("index", [0, 1])
@pytest.mark.parametrize("seed,n", [(0, 16), (1, 32), (2, 32)])
def test_an_arrival_beyond_the_sampled_ones(seed, n, index):
    """Eight commits of n requests (a power of two); the second has one more, whose few blocks, the only ones
    with so large an arrival, all lie in buckets that are not sampled.  The last entry to leave
    goes over that commit's end, through the larger arrival, and into the next commit."""
    rng = np.random.default_rng(seed)
    metas, late = [], []
    for seq in range(1, 9):
        for a in range(n + (seq == 2)):
            depths = int(rng.integers(1, 2 * 1100 // n)) if a < n - 1 else int(rng.integers(20, 40))
            metas += [(seq << 36) | (a << 16) | (65535 - d) for d in range(depths)]
            late += [a >= n] * depths
    metas, late = np.array(metas, np.uint64), np.array(late)
    keys = _keys_at_home(rng, np.where(late, True, rng.random(len(metas)) < 0.5), {})
    order = np.sort(metas)
    first, last = np.searchsorted(order, [(2 << 36) | (n << 16), 3 << 36])  # the larger arrival's entries
    for E in sorted({first - 60, first - 9, first - 1, first, first + 1, first + 8, last - 1, last, last + 1, last + 30}):
        _load_and_compare(keys, metas, len(metas) - int(E), index)


@pytest.mark.parametrize("n", [(6000, 500), (500, 6000)])
def test_a_sample_that_does_not_represent_the_table(n):
    """The sampled buckets hold the recent entries and the others the old ones (or few recent ones among
    many old), so that the bracket misses and the whole table is collected: equal and distinct
    ticks, thresholds in both parts."""
    rng = np.random.default_rng(n[0])
    seq = np.repeat([1, 9], n).astype(np.uint64)
    metas = (seq << np.uint64(36)) | (rng.integers(0, 50, sum(n)).astype(np.uint64) << np.uint64(16))
    metas |= np.uint64(65535) - rng.integers(0, 40, sum(n)).astype(np.uint64)
    keys = _keys_at_home(rng, seq == 1, {})
    for E in (1, 40, 499, 500, 501, 1000, 1600):
        _load_and_compare(keys, metas, sum(n) - E, 1)


@pytest.mark.parametrize("index", [0, 1])
def test_batches_of_changing_size(index):
    """A commit has a few more requests than a power of two, the ones before and behind it fewer."""
    rng = np.random.default_rng(5 + index)
    sizes = [31, 33, 32, 65, 64, 17, 129, 16, 33, 30, 35, 31]
    W, cap, ses, batches = 2, 4200, iter(range(1, 1 << 20)), []
    for n in sizes:
        lens = rng.integers(0, 2 * 6000 * 16 // n, n)
        lens[-2:] = rng.integers(16, 600, 2)  # few blocks at the largest arrivals
        batches.append(_batch(rng, rng.integers(0, 3, n), [next(ses) for _ in range(n)], lens))
    sc = _scenario(W, [cap, cap + 100], 3, np.zeros(W), np.ones(W), np.zeros(W), batches)
    r, o = make_router(sc, max_sessions=2000, prefix_index=index), make_oracle(sc)
    try:
        for k, b in enumerate(batches):
            back = np.array([0, 40_000]) if k % 2 else np.array([40_000, 0])
            for x in (r, o):
                x.set_instance_state(back, None, None)
            route_both(r, o, b, W, check_H=False, check_keys=False)
            r.commit()
            o.commit()
            compare_state(r, o, W)
    finally:
        r.close()
