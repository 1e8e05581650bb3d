"""The eviction's packed ticks (host build of the header that the kernels include): their order, their
inverse and their bins, for ticks on both sides of the sampled arrivals and depths."""

import ctypes
import os
import subprocess

import numpy as np
import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2608_11152_gb300", "csrc")
SHIM = """
#include "tick_scale.h"
typedef unsigned long long u64;
extern "C" {
u64 ts_pack(int ab, int db, u64 m) { return misat::TickScale{ab, db}.pack(m); }
u64 ts_unpack(int ab, int db, u64 x) { return misat::TickScale{ab, db}.unpack(x); }
u64 ts_bin(u64 v, u64 range) { return v >> misat::bin_shift(range); }
}
"""


@pytest.fixture(scope="module")
def ts(tmp_path_factory):
    d = tmp_path_factory.mktemp("tick_scale")
    src, so = d / "shim.cpp", d / "shim.so"
    src.write_text(SHIM)
    subprocess.check_call(["g++", "-O1", "-std=c++17", "-shared", "-fPIC", "-I", CSRC, "-o", str(so), str(src)])
    lib = ctypes.CDLL(str(so))
    for f, args in ((lib.ts_pack, 2), (lib.ts_unpack, 2), (lib.ts_bin, 0)):
        f.restype = ctypes.c_uint64
        f.argtypes = [ctypes.c_int] * args + [ctypes.c_uint64] * (1 if args else 2)
    return lib


def _metas(ab, db):
    """Metas in order: sequence numbers, and arrivals and depths below, at and above the sampled ones."""
    top, deep = (1 << ab) - 1, (1 << db) - 1
    arrivals = sorted({a for a in (0, 1, top - 1, top, top + 1, top + 2, 2 * top + 1, (1 << 20) - 1) if 0 <= a < 1 << 20})
    depths = sorted({d for d in (0, 1, 2, 40, deep - 1, deep, deep + 1, 2 * deep + 2, 65534) if 0 <= d < 65535})
    return sorted((s << 36) | (a << 16) | (65535 - d)
                  for s in (0, 1, 2, 3, (1 << 27) + 5, (1 << 28) - 1) for a in arrivals for d in depths)


WIDTHS = [(0, 0), (0, 4), (1, 0), (4, 6), (5, 5), (6, 16), (13, 7), (20, 3), (20, 16)]


@pytest.mark.parametrize("ab,db", WIDTHS)
def test_the_order_of_ticks_is_kept(ts, ab, db):
    packed = [ts.ts_pack(ab, db, m) for m in _metas(ab, db)]
    assert packed == sorted(packed)


@pytest.mark.parametrize("ab,db", WIDTHS)
def test_unpack_is_the_smallest_tick_that_packs_so_high(ts, ab, db):
    for m in _metas(ab, db):
        x = ts.ts_pack(ab, db, m)
        lo = ts.ts_unpack(ab, db, x)
        assert lo <= m and ts.ts_pack(ab, db, lo) >= x
        assert lo == 0 or ts.ts_pack(ab, db, lo - 1) < x


@pytest.mark.parametrize("ab,db", WIDTHS)
def test_every_tick_of_a_bracket_has_a_bin(ts, ab, db):
    metas = _metas(ab, db)
    rng = np.random.default_rng(ab * 17 + db)
    for _ in range(200):
        i, j = sorted(rng.integers(0, len(metas), 2).tolist())
        base = ts.ts_pack(ab, db, metas[i])
        rng_hi = ts.ts_pack(ab, db, metas[j]) - base
        for m in metas[i:j + 1]:
            v = ts.ts_pack(ab, db, m) - base
            assert v >= 0 and ts.ts_bin(v & (2**64 - 1), rng_hi & (2**64 - 1)) < 4096


@pytest.mark.parametrize("seed", range(6))
def test_the_bin_of_the_target_holds_the_target(ts, seed):
    """The first pass of the exact selection restated: commits of up to 33 requests whose last one (arrival
    32) the sample misses; the candidates below the target's bin are all smaller than it."""
    rng = np.random.default_rng(seed)
    ab, db = 5, 6  # sampled: arrivals up to 31, depths up to 63
    metas = []
    for seq in range(1, 5):
        for a in range(33):
            n = int(rng.integers(1, 64)) if a < 32 else int(rng.integers(1, 64)) * (seq == 3)
            metas += [(seq << 36) | (a << 16) | (65535 - d) for d in range(n)]
    metas.sort()
    for _ in range(200):
        i, j = sorted(rng.integers(0, len(metas), 2).tolist())
        cand, want = metas[i:j + 1], int(rng.integers(0, j + 1 - i))
        base = ts.ts_pack(ab, db, cand[0])
        span = (ts.ts_pack(ab, db, cand[-1]) - base) & (2**64 - 1)
        bins = [ts.ts_bin((ts.ts_pack(ab, db, m) - base) & (2**64 - 1), span) for m in cand]
        below = sum(b < bins[want] for b in bins)
        assert below <= want < below + sum(b == bins[want] for b in bins)
        assert all(m < cand[want] for m, b in zip(cand, bins) if b < bins[want])
