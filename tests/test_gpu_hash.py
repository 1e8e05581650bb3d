"""Block keys at the lengths where the hash changes its split of the work (exact, against the oracle):
groups of short prompts, the first prompts hashed by a warp and by a CTA, ragged last chunks and
steps, every misalignment of a prompt's first token."""

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

EDGES = [0, 1, 15, 16, 17, 31 * 16, 32 * 16 - 1, 32 * 16, 33 * 16 + 2, 255 * 16 + 15, 256 * 16, 256 * 16 + 1]


def _lens(name, rng):
    if name == "edges":  # one request per warp; every length at every misalignment
        return np.concatenate([rng.permutation(EDGES * 4) + 0, [3, 1, 2, 5]])
    if name == "long":  # a CTA per prompt: one chunk, whole and ragged steps of eight, the longest prompt
        return np.array([256 * 16, 3, 257 * 16 + 1, 511 * 16, 512 * 16 + 5, 513 * 16, 2049 * 16 + 7, (1 << 20) - 1, 40])
    if name == "groups":  # 32 short prompts per group, empty ones and longer ones between them
        lens = rng.integers(0, 80, size=65536)
        lens[rng.random(65536) < 0.01] = 700
        lens[100:140] = 0
        return lens
    # groups of a few prompts whose blocks straddle the chunks
    lens = rng.integers(0, 512, size=9001)
    lens[::501] = 5000
    return lens


@pytest.mark.parametrize("name", ["edges", "long", "groups", "straddle"])
def test_keys_at_the_edges_of_the_split(name):
    import __graft_entry__

    __graft_entry__.build()
    import oracle
    from paper_2608_11152_gb300 import misat
    from paper_2608_11152_gb300 import workload as wl

    rng = np.random.default_rng(sum(map(ord, name)))
    lens = _lens(name, rng)
    n = len(lens)
    off = np.zeros(n + 1, np.int64)
    np.cumsum(lens, out=off[1:])
    b = wl.Batch(cls=np.zeros(n, np.uint8), session=np.arange(1, n + 1, dtype=np.uint64), group=np.zeros(n, np.uint64),
                 tok_off=off, tokens=rng.integers(0, wl.VOCAB, size=int(off[-1]), dtype=np.int32))
    ref = np.concatenate([oracle.hash_prompt(b.tokens[off[q]:off[q + 1]]) for q in range(n)])
    r = misat.Router(np.array([1 << 20]), max_batch=n, max_tokens=b.n_tokens)
    db = r.device_batch(b)
    r.route(db)
    torch.cuda.synchronize()
    assert np.array_equal(r.dump_keys(b.n_tokens // 16 + 1), ref)
    keys = torch.full((len(ref) + 3,), -1, dtype=torch.int64, device="cuda")
    misat.block_hash_noalloc(db["tok_off"], db["tokens"], n, b.n_tokens, keys)
    got = keys.cpu().numpy()
    assert np.array_equal(got[: len(ref)].view(np.uint64), ref)
    assert np.all(got[len(ref):] == -1)
    r.close()
