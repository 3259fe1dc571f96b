"""GPU parity of the one-launch radix sort through the library: hit counts
around a sort tile (2,048 keys: one block in shared memory, then several blocks
with grid barriers) up to many tiles per block, for the hit sort (keys) and the
record sort (keys and values)."""
import numpy as np
import pytest

from parity_util import canon, oracle_rows, run_gpu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("hits", [1, 31, 2047, 2048, 2049, 4097, 70_001])
def test_sort_sizes(hits):
    """K = 0 and one planted copy per hit: the text holds exactly `hits`."""
    rng = np.random.default_rng(900 + hits)
    pats = [np.frombuffer(b"GATTACAGG", np.uint8), np.frombuffer(b"CCTGATTGA", np.uint8)]
    text = np.frombuffer(b"T" * (hits * 16 + 40), np.uint8).copy()
    for i in range(hits):
        p = pats[int(rng.integers(0, 2))]
        o = 16 * i + int(rng.integers(0, 6))
        text[o:o + p.size] = p
    want = oracle_rows(pats, [0, 0], text)
    assert len(want) == hits
    for order in (1, 2):
        got, st = run_gpu(pats, [0, 0], text, cfg={"record_order": order})
        assert st["hits"] == hits and canon(got) == want
    ends, _ = run_gpu(pats, [0, 0], text, {"output": "ends"}, cfg={"graphs": 1})
    assert canon(ends) == oracle_rows(pats, [0, 0], text, mode="ends")


def test_sort_many_tiles_per_block():
    """A binary text and short patterns: millions of hits."""
    rng = np.random.default_rng(950)
    alphabet = np.arange(2, dtype=np.uint8)
    pats = [alphabet[rng.integers(0, 2, size=6)] for _ in range(3)]
    text = alphabet[rng.integers(0, 2, size=600_000)]
    got, st = run_gpu(pats, [2, 1, 2], text)
    assert st["hits"] > 2_000_000
    assert canon(got) == oracle_rows(pats, [2, 1, 2], text)
