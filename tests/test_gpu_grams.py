"""GPU parity of the gram index (csrc/grams.cu): large steps look up grams of
the text that a piece of a pattern may appear as, and examine only the ends
they allow.  The records must equal the oracle's element by element, and those
of the forward scan alone (cfg.full_words = 1 and myers_only = 1 keep every
pattern on it), at sizes just above those from which the index runs; the
counts of steps that it served or was left for say that it did."""
import numpy as np
import pytest

from paper_1712_03560_gb300 import binding as B
from paper_1712_03560_gb300 import workloads as W
from parity_util import canon, gpu_rows, oracle_rows, run_gpu

pytestmark = pytest.mark.gpu

N_PAT = 1200  # with 100,000 symbols: a little more than the index's least work


def dictionary(rng, sigma, n_pat, mlo, mhi, n, kfun, copies=2):
    alphabet = np.frombuffer(b"ACGT", np.uint8) if sigma == 4 else \
        rng.permutation(256).astype(np.uint8)[:sigma]
    ms = rng.integers(mlo, mhi + 1, size=n_pat)
    ks = [int(kfun(int(m))) for m in ms]
    pats = [alphabet[rng.integers(0, sigma, size=int(m))] for m in ms]
    text = alphabet[rng.integers(0, sigma, size=n)]
    for p, k in zip(pats, ks):
        for cp in W.edit_copies(rng, p, rng.integers(0, k + 1, size=copies), alphabet):
            W.plant(rng, text, cp)
    return pats, ks, text


def runs_index(st, st_scan):
    """The index runs no bit-vector words for the patterns it serves."""
    return st["word_steps"] < 0.75 * st_scan["word_steps"]


# (alphabet, pattern lengths, threshold, text symbols): one to four words, 2-bit
# and byte text, whole pieces and pieces with an edit, the shortest to the
# longest grams, odd sizes
CASES = [(4, 8, 32, lambda m: m // 10, 130_003), (4, 24, 128, lambda m: m // 11, 110_007),
         (4, 16, 40, lambda m: 0, 100_001), (256, 16, 128, lambda m: min(8, m // 4), 100_013),
         (20, 33, 96, lambda m: 6, 105_019), (3, 30, 64, lambda m: 2, 100_151),
         (4, 12, 30, lambda m: 1 + m // 10, 140_009), (256, 16, 32, lambda m: 4, 100_057)]


@pytest.mark.parametrize("case", range(len(CASES)))
def test_index_equals_oracle_and_scan(case):
    sigma, mlo, mhi, kfun, n = CASES[case]
    rng = np.random.default_rng(800 + case)
    pats, ks, text = dictionary(rng, sigma, N_PAT, mlo, mhi, n, kfun)
    want = oracle_rows(pats, ks, text)
    got, st = run_gpu(pats, ks, text)
    scan, st_scan = run_gpu(pats, ks, text, cfg={"full_words": 1, "myers_only": 1})
    assert len(want) > 0 and canon(got) == canon(scan) == want
    assert runs_index(st, st_scan) and st["index_steps"] == 1 and st_scan["index_steps"] == 0
    dev, st = run_gpu(pats, ks, text, device_feed=True, cfg={"graphs": 1})
    assert canon(dev) == want and st["index_steps"] == 1


@pytest.mark.parametrize("mode,output", [("ends", "ends"), ("hits", "all_hits")])
def test_index_raw_outputs(mode, output):
    """Every end with D[e] <= K and every hit of Eq. 2: a missed end shows."""
    rng = np.random.default_rng(820)
    pats, ks, text = dictionary(rng, 4, N_PAT, 20, 60, 100_003, lambda m: m // 10)
    got, st = run_gpu(pats, ks, text, {"output": output})
    assert canon(got) == oracle_rows(pats, ks, text, mode=mode) and st["index_steps"] == 1


def test_index_over_steps_and_streams():
    """Stream cuts inside occurrences (each step rescans its stored tail),
    large steps with the index among small ones without it, and many streams
    of odd lengths in one step."""
    rng = np.random.default_rng(830)
    pats, ks, text = dictionary(rng, 4, N_PAT, 18, 70, 260_011, lambda m: m // 10, copies=6)
    want = oracle_rows(pats, ks, text)
    cuts = [88_001, 88_002, 88_040, 176_500]
    rows, st = run_gpu(pats, ks, text, splits=cuts)
    assert canon(rows) == want and (st["steps"], st["index_steps"]) == (6, 3)
    lens = [1, 5, 63, 64, 65, 127, 1000, 4099, 20_001, 90_000]
    ctx = B.oasm_create(pats, ks, None, {"max_streams": 16})
    try:
        parts = np.split(text[:sum(lens)], np.cumsum(lens)[:-1])
        sids = [B.oasm_open_stream(ctx) for _ in parts]
        for sid, t in zip(sids, parts):
            B.oasm_feed(ctx, sid, t)
            B.oasm_end_stream(ctx, sid)
        B.oasm_step(ctx)
        res = B.oasm_drain(ctx)
        for sid, t in zip(sids, parts):
            got = [(int(r["pattern_id"]), int(r["decided_at"]), int(r["k"]), int(r["start"]),
                    int(r["len"])) for r in res[res["stream_id"] == sid]]
            assert canon(got) == oracle_rows(pats, ks, t)
        assert B.oasm_get_routes(ctx)["index_steps"] == 1
    finally:
        B.oasm_destroy(ctx)


def test_index_gives_way_on_repetitive_text():
    """Every piece matches nearly everywhere: the suspects outgrow their
    buffer, the step is re-run on the forward scan, and so are the next
    32, then the index is tried again; symbols outside the patterns' alphabet
    match nothing."""
    rng = np.random.default_rng(840)
    unit = np.frombuffer(b"ACGGTCA", np.uint8)
    pats = [np.roll(np.tile(unit, 5), i % 7)[:25 + i % 9].copy() for i in range(N_PAT)]
    ks = [int(rng.integers(0, 3)) for _ in pats]
    text = np.tile(unit, 24_000)[:90_000].copy()
    text[rng.integers(0, text.size, size=400)] = ord("T")
    text[40_000:40_100] = ord("N")
    other = W.DNA[rng.integers(0, 4, size=100_000)]
    ctx = B.oasm_create(pats, ks)
    try:
        out, routes = [], []
        sid = B.oasm_open_stream(ctx)
        for part in np.split(text, [85_000]):
            B.oasm_feed(ctx, sid, part)
            out.append(B.oasm_flush(ctx, sid, end_of_stream=len(out) == 1))
        for part in 33 * [other] + [text[:85_000]]:
            B.oasm_feed(ctx, sid, part)
            B.oasm_flush(ctx, sid)
            r = B.oasm_get_routes(ctx)
            routes.append((r["index_steps"], r["index_left"]))
    finally:
        B.oasm_destroy(ctx)
    got = [(int(r["pattern_id"]), int(r["decided_at"]), int(r["k"]), int(r["start"]),
            int(r["len"])) for r in np.concatenate(out)]
    assert canon(got) == oracle_rows(pats, ks, text)
    assert routes[30:] == [(0, 1), (0, 1), (1, 1), (1, 2)]


@pytest.mark.parametrize("costs", [(1, 2, 2), (2, 3, 2), (1, 1, 1), (9, 5, 7)])
def test_index_under_edit_costs(costs):
    """K bounds the cost, so the edits are at most K over the cheapest cost."""
    rng = np.random.default_rng(850)
    pats, ks, text = dictionary(rng, 4, N_PAT, 10, 40, 100_003, lambda m: m // 7)
    got, st = run_gpu(pats, ks, text, costs=costs)
    assert canon(got) == oracle_rows(pats, ks, text, costs=costs) and st["index_steps"] == 1
    ends, st = run_gpu(pats, ks, text, {"output": "ends"}, costs=costs)
    assert canon(ends) == oracle_rows(pats, ks, text, mode="ends", costs=costs)
    assert st["index_steps"] == 1


def test_index_runs_of_one_symbol():
    """Pieces with repeated symbols, where several edits give one string: DNA
    patterns made of short runs, thresholds 1 to 3."""
    rng = np.random.default_rng(860)
    pats, ks = [], []
    for i in range(N_PAT):
        p = np.repeat(W.DNA[rng.integers(0, 4, size=60)], rng.integers(1, 4, size=60))
        pats.append(p[:int(rng.integers(26, 60))].copy())
        ks.append(1 + i % 3)
    n = 200_000
    text = np.repeat(W.DNA[rng.integers(0, 4, size=n)], rng.integers(1, 4, size=n))
    for p, k in zip(pats, ks):
        for cp in W.edit_copies(rng, p, np.full(4, k), W.DNA):
            W.plant(rng, text, cp)
    got, st = run_gpu(pats, ks, text)
    assert canon(got) == oracle_rows(pats, ks, text) and st["index_steps"] == 1


@pytest.mark.parametrize("piece", [1, 4])
def test_index_takes_the_piece_filters_patterns(piece):
    """A large step looks the piece filter's patterns up in the index too, or,
    with patterns that it leaves (a symbol that most of the pattern text is
    made of), runs the piece filter beside it; small steps of the same stream
    run the filter.  Half of the patterns have pieces too short for it."""
    rng = np.random.default_rng(870 + piece)
    pats, ks, text = dictionary(rng, 256, N_PAT // 2, 12, 100, 300_003, lambda m: min(8, m // 6))
    for _ in range(N_PAT // 2):
        p = rng.permutation(256).astype(np.uint8)[:int(rng.integers(30, 46))]
        pats, ks = pats + [p], ks + [p.size // 3 - 1]
        for cp in W.edit_copies(rng, p, rng.integers(0, ks[-1] + 1, size=2),
                                np.arange(256, dtype=np.uint8)):
            W.plant(rng, text, cp)
    assert B.oasm_piece_filter_choice(pats, ks, piece).sum() == N_PAT // 2
    cuts = [290_000, 290_500, 299_990]
    proposed = []
    for extra in (False, True):
        if extra:
            pats = pats + 400 * [np.full(128, text[0], np.uint8)]
            ks = ks + 400 * [1]
            text[200_000:200_300] = text[0]
        got, st = run_gpu(pats, ks, text, splits=cuts, cfg={"prefilter_piece": piece})
        assert canon(got) == oracle_rows(pats, ks, text)
        assert (st["steps"], st["index_steps"]) == (5, 1)
        proposed.append(st["prefilter_candidates"])
    assert 0 < 20 * proposed[0] < proposed[1]  # of the small steps; of the large one too


def test_index_of_a_few_long_patterns():
    """Fewer patterns than a warp has lanes, thresholds up to 15."""
    rng = np.random.default_rng(880)
    pats, ks, text = dictionary(rng, 256, 9, 60, 128, 1_000_003, lambda m: 3 + m // 11, copies=40)
    got, st = run_gpu(pats, ks, text)
    scan, st_scan = run_gpu(pats, ks, text, cfg={"full_words": 1})
    assert runs_index(st, st_scan) and st["index_steps"] == 1
    assert canon(got) == canon(scan) == oracle_rows(pats, ks, text)


@pytest.mark.parametrize("short", [33, 55, 64, 65, 97])
def test_short_patterns_of_three_errors_beside_the_index(short):
    """Patterns too short for the index, two a lane: one to two groups, a last
    lane with one pattern, lengths from K + 1 on."""
    rng = np.random.default_rng(860 + short)
    n = 130_003
    pats, ks, text = dictionary(rng, 4, 500, 40, 64, n, lambda m: 3)
    few = [np.frombuffer(b"ACGT", np.uint8)[rng.integers(0, 4, size=m)]
           for m in [4, 5] + [9 + j % 5 for j in range(short - 2)]]
    high = np.uint8(0x80 * (short & 1))  # symbols in either half of the table
    pats, ks = [p | high for p in few[:3] + pats + few[3:]], [3] * (short + 500)
    text = text | high
    want = oracle_rows(pats, ks, text)
    got, st = run_gpu(pats, ks, text)
    assert canon(got) == want
    assert st["word_steps"] == (short + 1) // 2 * n and st["index_steps"] == 1


@pytest.mark.parametrize("piece", [0, 1])
def test_the_set_of_ends_fits_each_step(piece):
    """Steps after a large one clear the part of the (end, pattern) set that
    their own text needs; a step that needs more runs again with more, and the
    ones after it start there."""
    import torch
    rng = np.random.default_rng(890 + piece)
    sigma = 256 if piece else 4
    pats, ks, text = dictionary(rng, sigma, N_PAT, 24, 90, 140_000, lambda m: m // 10)
    alphabet = np.unique(text)
    one = alphabet[rng.integers(0, alphabet.size, size=80)]  # a pattern many times over
    pats, ks = pats + [one] * 300, ks + [8] * 300
    dense = text.copy()
    for at in range(500, dense.size, 2_000):
        dense[at:at + one.size] = one
    big = torch.from_numpy(alphabet).cuda()[
        torch.randint(0, alphabet.size, (1 << 25,), device="cuda")]
    ctx = B.oasm_create(pats, ks, None, {"prefilter_piece": piece})

    def step(t):
        before = B.oasm_get_routes(ctx)["set_slots"], B.oasm_get_stats(ctx)["reruns"]
        sid = B.oasm_open_stream(ctx)
        (B.oasm_feed if isinstance(t, np.ndarray) else B.oasm_feed_device)(ctx, sid, t)
        B.oasm_end_stream(ctx, sid)
        B.oasm_step(ctx)
        rows = gpu_rows(B.oasm_drain(ctx))
        B.oasm_close_stream(ctx, sid)
        return rows, B.oasm_get_routes(ctx)["set_slots"] - before[0], \
            B.oasm_get_stats(ctx)["reruns"] - before[1]

    try:
        step(big)
        step(big)
        assert step(big)[1] >= 1 << 21
        want, want_dense = oracle_rows(pats, ks, text), oracle_rows(pats, ks, dense)
        rows, slots, _ = step(text)
        assert canon(rows) == want and 0 < slots <= 1 << 19
        for _ in range(2):
            rows, slots, reruns = step(dense)
            assert canon(rows) == want_dense
        assert reruns == 0 and slots > 1 << 19
        assert step(big)[1] >= 1 << 21
    finally:
        B.oasm_destroy(ctx)


@pytest.mark.parametrize("piece,costs,scan", [(0, None, 0), (4, None, 0), (0, (1, 2, 2), 0),
                                              (0, None, 1)])
def test_memory_for_the_index_is_not_needed(piece, costs, scan):
    """Each device allocation of a context and its first steps fails in turn,
    once.  Those of the index only cost the index, and a step's own take its
    memory; a context that finds no room for anything else is not created, and
    a step of one without an index fails and is there to be run again."""
    rng = np.random.default_rng(895 + piece)
    pats, ks, text = dictionary(rng, 256 if piece else 4, N_PAT, 12, 70, 100_003,
                                lambda m: m // 10)
    want = oracle_rows(pats, ks, text, costs=costs)

    def run(fail_at):
        made = {"created": False, "failed_steps": 0}
        B.oasm_selftest_alloc(fail_at)
        try:
            ctx = B.oasm_create(pats, ks, None, {"prefilter_piece": piece, "full_words": scan},
                                costs=costs)
        except B.OasmError as e:
            assert e.code == B.OASM_ENOMEM
            return made
        try:
            made["created"] = True
            made["allocs"] = B.oasm_selftest_alloc(0)
            B.oasm_selftest_alloc(max(fail_at - made["allocs"], 0))
            sid, out = B.oasm_open_stream(ctx), []
            for part in np.split(text, [text.size // 50]):
                B.oasm_feed(ctx, sid, part)
                try:
                    out.append(B.oasm_flush(ctx, sid, end_of_stream=len(out) == 1))
                except B.OasmError as e:
                    assert e.code == B.OASM_ENOMEM
                    made["failed_steps"] += 1
                    out.append(B.oasm_flush(ctx, sid, end_of_stream=len(out) == 1))
            made["step_allocs"] = B.oasm_selftest_alloc(0)
            assert canon(gpu_rows(np.concatenate(out))) == want
            return made
        finally:
            B.oasm_selftest_alloc(0)
            B.oasm_destroy(ctx)

    whole = run(0)
    runs = [run(i) for i in range(1, whole["allocs"] + whole["step_allocs"] + 1)]
    needed = [r["created"] for r in runs].index(True)  # allocations that a context needs
    assert all(r["created"] for r in runs[needed:])
    if scan:
        assert needed == whole["allocs"] and any(r["failed_steps"] for r in runs)
    else:
        assert needed <= whole["allocs"] - 4 and not any(r["failed_steps"] for r in runs)


def test_a_first_step_sizes_its_buffers_in_few_runs():
    """Many slices of a step's text, each with more ends than the buffers hold
    at first: the counts of one run size them for the whole step."""
    rng = np.random.default_rng(899)
    pats, ks, text = dictionary(rng, 4, N_PAT, 24, 60, 1_500_000, lambda m: m // 10)
    one = W.DNA[rng.integers(0, 4, size=40)]
    pats, ks = pats + [one] * 300, ks + [4] * 300
    for at in range(500, text.size - 100, 2_000):
        text[at:at + one.size] = one
    scan, _ = run_gpu(pats, ks, text, cfg={"full_words": 1, "myers_only": 1})
    ctx = B.oasm_create(pats, ks)
    try:
        B.oasm_selftest_limits(ctx, gram_slice=1 << 15)
        sid = B.oasm_open_stream(ctx)
        B.oasm_feed(ctx, sid, text)
        rows = gpu_rows(B.oasm_flush(ctx, sid, end_of_stream=True))
        st = B.oasm_get_stats(ctx)
    finally:
        B.oasm_destroy(ctx)
    assert canon(rows) == canon(scan)
    # suspects; ends and their set, 31 times what there was room for, twice (8
    # times at most); hits; records
    assert st["candidates"] > 1_000_000 and st["reruns"] <= 5


def test_index_gives_way_to_a_text_of_one_shared_key():
    """Every piece of every pattern starts with the same four symbols, and the
    text repeats those: thousands of entries to compare at each of their
    places, and no suspect."""
    rng = np.random.default_rng(897)
    a = np.frombuffer(b"ABCDEF", np.uint8)
    pats = [np.concatenate([np.concatenate([a[:4], a[4 + rng.integers(0, 2, 4)]])
                            for _ in range(4)]) for _ in range(2048)]
    ks = [3] * len(pats)
    text = np.tile(a[:4], 50_000)
    text[1_000:1_032] = pats[7]
    text[150_000:150_032] = pats[8]
    ctx = B.oasm_create(pats, ks)
    try:
        sid = B.oasm_open_stream(ctx)
        out, routes = [], []
        for part in np.split(text, [140_000]):
            B.oasm_feed(ctx, sid, part)
            out.append(B.oasm_flush(ctx, sid, end_of_stream=len(out) == 1))
            r = B.oasm_get_routes(ctx)
            routes.append((r["index_steps"], r["index_left"]))
    finally:
        B.oasm_destroy(ctx)
    want = oracle_rows(pats, ks, text)
    assert canon(gpu_rows(np.concatenate(out))) == want and {r[0] for r in want} >= {7, 8}
    assert routes == [(0, 1), (0, 1)]
