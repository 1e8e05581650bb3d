"""Completion events: repeated sessions are refused before anything changes, wherever they stand among
the events, and the class histories are those of the serial reading (exact, against the oracle)."""

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _events(rng, n):
    # ids of a counter and of no pattern: neighbours share filter words, others collide by chance
    ids = np.arange(1, 2 * n + 1, dtype=np.uint64)
    ids[n:] = rng.integers(1, 1 << 63, size=n, dtype=np.uint64)
    ids = rng.permutation(np.unique(ids))[:n]
    return (ids, rng.integers(0, 3, n).astype(np.uint8), rng.integers(0, 5000, n).astype(np.int32),
            rng.integers(0, 1 << 30, n), (rng.random(n) < 0.7).astype(np.uint8))


@pytest.mark.parametrize("n,window", [(1, 4), (2, 1), (63, 16), (4097, 256), (70000, 4096)])
def test_repeated_sessions_and_histories(n, window):
    import __graft_entry__

    __graft_entry__.build()
    import oracle
    from paper_2608_11152_gb300 import misat

    rng = np.random.default_rng(n)
    cap = np.array([1 << 14, 1 << 15], np.int64)
    kw = dict(hist_window=window, prior_kbar=(4, 4, 4), prior_T_us=1000)
    r = misat.Router(cap, max_batch=max(4, n // 3), max_tokens=64, **kw)
    o = oracle.Oracle(cap, **kw)
    b = dict(n=1, n_tokens=16, cls=torch.zeros(1, dtype=torch.uint8, device="cuda"),
             session=torch.ones(1, dtype=torch.int64, device="cuda"),
             tok_off=torch.tensor([0, 16], device="cuda"), tokens=torch.zeros(16, dtype=torch.int32, device="cuda"))
    for only in (None, 1):  # all classes, then one class whose history alone moves
        s, c, tb, ru, dn = _events(rng, n)
        if only is not None:
            c[:] = only
        for i, j in ((0, n - 1), (n // 2, n // 2 + 1), (n - 2, n - 1)):
            if 0 <= i < j < n:
                bad = s.copy()
                bad[j] = bad[i]
                with pytest.raises(misat.MisatError) as e:
                    r.complete(bad, c, tb, ru, dn)
                assert e.value.code == misat.ERR_INVALID_ARG
        r.complete(s, c, tb, ru, dn)
        o.complete(s, c, tb, ru, dn)
        # a route estimates the classes from the histories
        r.route(b)
        o.route(np.zeros(1, np.uint8), np.ones(1, np.uint64), np.array([0, 16]), np.zeros(16, np.int32))
        got, ref = r.dump_caps(), o.caps()
        for k in ("K_w", "K_wb", "kbar_b", "T_b"):
            assert np.array_equal(got[k], ref[k]), k
    r.close()
