"""GPU parity of small steps, which run everything after the scan in one launch:
around the text size and the pair count where they end, counts of hits and
records around a sort tile and the records that go straight to the host, windows
carried over many steps, and records that stay queued while later steps run."""
import numpy as np
import pytest

from paper_1712_03560_gb300 import binding as B
from paper_1712_03560_gb300 import workloads as W
from parity_util import canon, gpu_rows, oracle_rows, random_case, run_gpu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1, 2, 40, 5000, (8 << 20) - 1, 8 << 20, (8 << 20) + 1])
def test_text_sizes(n):
    rng = np.random.default_rng(1000 + n)
    pats = [W.DNA[rng.integers(0, 4, size=m)] for m in (8, 11, 20)]
    ks = [2, 1, 3]
    text = W.DNA[rng.integers(0, 4, size=n)]
    want = oracle_rows(pats, ks, text)
    for graphs in (0, 1):
        got, st = run_gpu(pats, ks, text, cfg={"graphs": graphs})
        assert canon(got) == want
    timed, st_t = run_gpu(pats, ks, text, cfg={"timing": 1})  # one launch per kernel class
    assert canon(timed) == want
    assert (st["launches"] / (st["steps"] + st["reruns"]) <
            st_t["launches"] / (st_t["steps"] + st_t["reruns"])) == (n <= 8 << 20)


@pytest.mark.parametrize("records", [4095, 4096, 4097, 9000])
def test_records_straight_to_the_host_or_copied(records):
    text = np.frombuffer(b"T" * (records * 12), np.uint8).copy()
    for i in range(records):
        text[12 * i:12 * i + 7] = np.frombuffer(b"GATTACA", np.uint8)
    got, _ = run_gpu([b"GATTACA"], [0], text)
    assert len(got) == records and canon(got) == oracle_rows([b"GATTACA"], [0], text)


def test_many_streams_and_rules_over_steps():
    """Streams cut at random, a step after each piece, all rules of one kind
    and the other; some queues are left to grow over several steps."""
    for rules in ({}, {"order": "per_start_best", "acc": "last", "cmp": "ge",
                       "replace": "same_end"}):
        rng = np.random.default_rng(1100 + len(rules))
        pats, ks, _ = random_case(rng, 4, 12, 5, 40, 10, kmax=4)
        texts = [random_case(rng, 4, 1, 6, 8, int(rng.integers(200, 4000)))[2] for _ in range(9)]
        for t in texts:
            for p, k in zip(pats, ks):
                W.plant(rng, t, W.edit_copy(rng, p, k, W.DNA))
        cuts = [np.split(t, np.sort(rng.integers(0, t.size, size=6))) for t in texts]
        ctx = B.oasm_create(pats, ks, rules or None, {"max_streams": 9})
        try:
            sids = [B.oasm_open_stream(ctx) for _ in texts]
            got = {s: [] for s in sids}
            for step in range(7):
                for s, c in zip(sids, cuts):
                    B.oasm_feed(ctx, s, c[step])
                    if step == 6:
                        B.oasm_end_stream(ctx, s)
                B.oasm_step(ctx)
                if step in (3, 6):
                    for r in B.oasm_drain(ctx):
                        got[int(r["stream_id"])].append(r)
            for s, t in zip(sids, texts):
                rows = gpu_rows(np.array(got[s], dtype=B.HIT_DTYPE))
                assert canon(rows) == oracle_rows(pats, ks, t, rules)
        finally:
            B.oasm_destroy(ctx)
