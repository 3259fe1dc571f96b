"""The work that a user has the matcher do, as timed cases.

Every case goes through the public binding: a context over a pattern set, text
fed to streams (host or device memory), steps, and the decided records back in
host arrays.  Sizes, pattern sets and planting densities are those of
``workloads.py`` and of the benchmark, at lengths that a pass of well under a
second allows.  All results are whole numbers: records of pattern, level,
start, length, stream and decision point, in canonical order.

A case holds
  kind     search: one text as one stream, ended (feed, flush, close)
           chunks: one stream fed and flushed chunk by chunk, as it arrives
           texts:  many texts, one stream each, one batched step
           served: many packet streams, two batches of packets, a step each
  alpha    dna (iid ACGT) or zipf (bytes whose ranks follow Zipf(1.1))
  n_pat, mlo, mhi, spread   pattern count and lengths (uniform or log-uniform)
  k        a threshold, or "m//10", or "zipf" (uniform in 1..min(8, m // 4)),
           or "long" (uniform in 4..15)
  n        text symbols in all; per_sym: planted copies per text symbol
  feed     host (ordinary memory) or device
  output   filtered, ends or all_hits
  piece    prefilter_piece of the context; graphs: steps as CUDA graphs
  costs    "" or "sub,ins,del"
"""
import numpy as np
import torch

from paper_1712_03560_gb300 import binding as B
from paper_1712_03560_gb300 import workloads as W

MIB = 1 << 20


def _case(name=None, **kw):
    c = {"kind": "search", "alpha": "dna", "n_pat": 1, "mlo": 8, "mhi": 8, "spread": "uniform",
         "k": "2", "n": MIB, "per_sym": 2e-4, "feed": "device", "output": "filtered", "piece": 0,
         "graphs": 0, "costs": "", "streams": 1, "chunk": 0}
    c.update(kw)
    if name:
        c["name"] = name
    return c


# densities of planted copies per text symbol, as in workloads.py
DICT, ZIPF, MANY = 1024 * 1000 / (256 * MIB), 4096 * 500 / (1024 * MIB), 2.6e-5


def listed():
    return [
        # one motif searched in one short buffer from host memory: the smallest
        # call, where launches and latency count
        _case("short_text", n=1500, feed="host"),
        # one DNA motif over a million symbols (the plain configuration)
        _case("plain_dna_1m", n=1_000_000),
        # the same over a long text: the output-heavy one-pattern search
        _case("plain_dna_256m", n=256 * MIB),
        # 1,024 miRNA-sized motifs, K = m // 10, over a genome-like text
        _case("dictionary_dna_64m", n_pat=1024, mhi=32, k="m//10", n=64 * MIB, per_sym=DICT),
        # unfiltered Less Naive ends of an odd dictionary over an odd text that
        # comes from host memory
        _case("dictionary_ends_3m", n_pat=700, mhi=32, k="m//10", n=3_000_017, per_sym=DICT,
              feed="host", output="ends"),
        # 4,096 byte signatures of 16..128 symbols over Zipf bytes (the
        # benchmark's default dictionary), every pattern on the forward scan
        _case("bytes_zipf_32m", alpha="zipf", n_pat=4096, mlo=16, mhi=128, spread="log",
              k="zipf", n=32 * MIB, per_sym=ZIPF),
        # the same signatures with the automatic piece filter
        _case("bytes_zipf_piece_128m", alpha="zipf", n_pat=4096, mlo=16, mhi=128, spread="log",
              k="zipf", n=128 * MIB, per_sym=ZIPF, piece=1),
        # a dozen long signatures with high thresholds: fewer patterns than a
        # warp has lanes
        _case("few_long_8m", alpha="zipf", n_pat=12, mlo=40, mhi=128, k="long", n=8 * MIB,
              per_sym=2e-5, feed="host"),
        # many DNA texts of log-normal lengths against 512 motifs in one step
        _case("many_texts_64m", kind="texts", n_pat=512, mlo=12, mhi=48, k="3", n=64_000_000,
              per_sym=MANY, streams=160),
        # the DNA dictionary under integer edit costs
        _case("dictionary_weighted_16m", n_pat=1024, mhi=32, k="m//10", n=16 * MIB, per_sym=DICT,
              costs="1,2,2"),
        # a loaded server's steps: 4,096 packet streams against 2,000 signatures
        _case("served_batch_8m", kind="served", alpha="zipf", n_pat=2000, mlo=8, mhi=64, k="2",
              n=8 * MIB, per_sym=1.3e-5, feed="host", piece=1, graphs=1, streams=4096),
        # online matching of one stream: small chunks, results after each
        _case("online_chunks", kind="chunks", n_pat=64, mhi=32, k="m//10", n=16 * 4096,
              per_sym=DICT, feed="host", chunk=4096),
    ]


def draw(rng):
    """One more case of the same ranges."""
    def size(lo, hi):
        return int(round(lo * (hi / lo) ** rng.random()))

    what = rng.choice(["plain", "dictionary", "zipf", "zipf_piece", "few_long", "texts", "weighted",
                       "served", "chunks"])
    if what == "plain":
        return _case(n=size(1500, 256 * MIB), mlo=(m := rng.randint(8, 32)), mhi=m,
                     k=str(rng.randint(1, 2)), feed=rng.choice(["host", "device"]))
    if what == "dictionary":
        return _case(n_pat=size(40, 1024), mhi=32, k="m//10", n=size(100_000, 64 * MIB),
                     per_sym=DICT, output=rng.choice(["filtered", "filtered", "ends", "all_hits"]),
                     feed=rng.choice(["host", "device"]), graphs=rng.randint(0, 1))
    if what in ("zipf", "zipf_piece"):
        return _case(alpha="zipf", n_pat=size(100, 4096), mlo=16, mhi=128, spread="log", k="zipf",
                     n=size(100_000, 32 * MIB if what == "zipf" else 128 * MIB), per_sym=ZIPF,
                     piece=0 if what == "zipf" else 1, feed=rng.choice(["host", "device"]))
    if what == "few_long":
        return _case(alpha="zipf", n_pat=rng.randint(2, 31), mlo=40, mhi=128, k="long",
                     n=size(50_000, 8 * MIB), per_sym=2e-5, feed="host")
    if what == "texts":
        n_texts = size(4, 160)
        return _case(kind="texts", n_pat=size(48, 512), mlo=12, mhi=48, k="3", n=n_texts * 400_000,
                     per_sym=MANY, streams=n_texts)
    if what == "weighted":
        return _case(n_pat=size(40, 1024), mhi=32, k="m//10", n=size(50_000, 16 * MIB),
                     per_sym=DICT, costs=rng.choice(["1,2,2", "2,3,1", "1,1,1"]))
    if what == "served":
        return _case(kind="served", alpha="zipf", n_pat=size(200, 2000), mlo=8, mhi=64, k="2",
                     n=size(100_000, 8 * MIB), per_sym=1.3e-5, feed="host", piece=1, graphs=1,
                     streams=size(64, 4096))
    chunk = size(256, 16384)
    return _case(kind="chunks", n_pat=size(4, 256), mhi=32, k="m//10", n=12 * chunk, per_sym=DICT,
                 feed="host", chunk=chunk)


# ------------------------------------------------------------------- inputs
def _patterns(case, rng, perm):
    n, lo, hi = case["n_pat"], case["mlo"], case["mhi"]
    if case["spread"] == "log":
        ms = np.exp(rng.uniform(np.log(lo), np.log(hi + 1), size=n)).astype(np.int64).clip(lo, hi)
    else:
        ms = rng.integers(lo, hi + 1, size=n)
    if case["k"] == "m//10":
        ks = ms // 10
    elif case["k"] == "zipf":
        ks = 1 + (rng.random(n) * np.minimum(8, ms // 4)).astype(np.int64)
    elif case["k"] == "long":
        ks = rng.integers(4, 16, size=n)
    else:
        ks = np.full(n, int(case["k"]))
    if case["alpha"] == "dna":
        flat = W.iid_dna(rng, int(ms.sum()))
    else:
        flat = W.zipf_bytes(rng, int(ms.sum()), perm)
    return np.split(flat, np.cumsum(ms)[:-1]), ms, ks


def _edited_copies(rng, pats, ms, ks, count, lo_edits, alphabet):
    """count copies of patterns drawn uniformly, each with lo_edits(k)..k
    edits (substitution, insertion or deletion at a uniform place)."""
    width = int(ms.max() + ks.max() + 1)
    rows = np.zeros((len(pats), width), np.uint8)
    for i, p in enumerate(pats):
        rows[i, :p.size] = p
    dev = torch.device("cuda")
    own = rng.integers(0, len(pats), size=count)
    lo = np.minimum(lo_edits(ks[own]), ks[own])
    edits = lo + (rng.random(count) * (ks[own] - lo + 1)).astype(np.int64)
    buf = torch.from_numpy(rows).to(dev)[torch.from_numpy(own).to(dev)]
    ln = torch.from_numpy(ms[own]).to(dev)
    left = torch.from_numpy(edits).to(dev)
    col = torch.arange(width, device=dev)[None, :]
    for step in range(int(edits.max(initial=0))):
        op = torch.from_numpy(rng.integers(0, 3, size=count)).to(dev)
        op = torch.where(ln <= 1, torch.ones_like(op), op)
        u = torch.from_numpy(rng.random(count)).to(dev)
        sym = torch.from_numpy(alphabet[rng.integers(0, alphabet.size, size=count)]).to(dev)
        pos = (u * (ln + (op == 1))).long()[:, None]
        ins = torch.where(col < pos, buf, torch.where(col == pos, sym[:, None], buf.roll(1, 1)))
        dele = torch.where(col < pos, buf, buf.roll(-1, 1))
        sub = torch.where(col == pos, sym[:, None], buf)
        new = torch.where((op == 0)[:, None], sub, torch.where((op == 1)[:, None], ins, dele))
        act = left > step
        buf = torch.where(act[:, None], new, buf)
        ln = ln + act * ((op == 1).long() - (op == 2).long())
    return buf, ln


def _plant(rng, text, buf, ln):
    """Overwrites the text with the copies, each in a slot of its own."""
    width = buf.shape[1]
    slots = text.numel() // width
    count = min(buf.shape[0], slots // 2)
    if count == 0:
        return
    dev = text.device
    g = torch.Generator(device=dev).manual_seed(int(rng.integers(1 << 62)))
    at = torch.randperm(slots, generator=g, device=dev)[:count] * width
    room = (width - ln[:count] + 1).double()
    at = at + (torch.rand(count, generator=g, device=dev, dtype=torch.float64) * room).long()
    col = torch.arange(width, device=dev)[None, :]
    keep = col < ln[:count, None]
    text[(at[:, None] + col)[keep]] = buf[:count][keep]


def _text(case, rng, pats, ms, ks, perm):
    n, dev = case["n"], torch.device("cuda")
    g = torch.Generator(device=dev).manual_seed(int(rng.integers(1 << 62)))
    if case["alpha"] == "dna":
        table, alphabet = W.DNA, W.DNA
    else:
        table, alphabet = W.zipf_table(perm), perm
    cells = torch.from_numpy(np.ascontiguousarray(table)).to(dev)
    text = torch.empty(n, dtype=torch.uint8, device=dev)
    for a in range(0, n, 1 << 25):
        b = min(n, a + (1 << 25))
        text[a:b] = cells[torch.randint(0, cells.numel(), (b - a,), generator=g, device=dev)]
    count = max(1, int(n * case["per_sym"]))
    # exactly K edits in the DNA dictionary, 1..K in the byte one, 0..K otherwise
    lo = {"m//10": lambda k: k, "zipf": lambda k: np.ones_like(k)}.get(case["k"], np.zeros_like)
    buf, ln = _edited_copies(rng, pats, ms, ks, count, lo, alphabet)
    _plant(rng, text, buf, ln)
    return text


class _State:
    pass


def prepare(case, seed):
    rng = W.rng_for(seed)
    perm = rng.permutation(256).astype(np.uint8)
    pats, ms, ks = _patterns(case, rng, perm)
    text = _text(case, rng, pats, ms, ks, perm)
    costs = tuple(int(c) for c in case["costs"].split(",")) if case["costs"] else None
    s = _State()
    s.kind = case["kind"]
    s.mt = B.Matcher(pats, ks, {"output": case["output"]}, costs,
                     max_streams=max(4, case["streams"]), prefilter_piece=case["piece"],
                     graphs=case["graphs"])
    s.device = case["feed"] == "device"
    host = None if s.device else text.cpu().numpy()
    if case["kind"] == "search":
        s.text = text if s.device else host
    elif case["kind"] == "chunks":
        s.chunks = np.split(host, range(case["chunk"], case["n"], case["chunk"]))
    elif case["kind"] == "texts":
        # log-normal lengths, as in workloads.many_texts, scaled to the total
        w = np.exp(rng.normal(np.log(1e5), 1.75, size=case["streams"])).clip(1e3, 1e7)
        cuts = np.floor(np.cumsum(w) / w.sum() * case["n"]).astype(np.int64)
        s.texts = [t for t in torch.tensor_split(text, torch.from_numpy(cuts[:-1]))]
    else:
        s.packets = []
        s.n_streams = case["streams"]
        lens = rng.integers(64, 1501, size=max(2, case["n"] // 782)).astype(np.uint32)
        ends = np.cumsum(lens.astype(np.uint64))
        lens = lens[ends <= case["n"]]
        offs = (np.cumsum(lens.astype(np.uint64)) - lens).astype(np.uint64)
        owner = rng.integers(0, case["streams"], size=lens.size)
        s.payload = host
        half = lens.size // 2
        for sl in (slice(0, half), slice(half, lens.size)):
            s.packets.append((owner[sl], offs[sl], lens[sl]))
    # the caller's array for the records, with room to spare
    s.out = np.zeros(4096 + 3 * _records(case), dtype=B.HIT_DTYPE)
    torch.cuda.synchronize()
    return s


# ---------------------------------------------------------------------- run
def _result(s, count):
    """The record count and the caller's array, as whole numbers: pattern and
    level, start, length and stream, decision point (a view, no copy)."""
    return {"count": count, "records": s.out.view(np.int64).reshape(-1, 4)}


def run(s):
    ctx, n = s.mt.ctx, 0
    if s.kind == "search":
        sid = B.oasm_open_stream(ctx)
        if s.device:
            B.oasm_feed_device(ctx, sid, s.text)
        else:
            B.oasm_feed(ctx, sid, s.text)
        B.oasm_end_stream(ctx, sid)
        B.oasm_step(ctx)
        n = B.oasm_drain(ctx, s.out).size
        B.oasm_close_stream(ctx, sid)
    elif s.kind == "chunks":
        sid = B.oasm_open_stream(ctx)
        for i, c in enumerate(s.chunks):
            B.oasm_feed(ctx, sid, c)
            hits = B.oasm_flush(ctx, sid, end_of_stream=i + 1 == len(s.chunks))
            s.out[n:n + hits.size] = hits
            n += hits.size
        B.oasm_close_stream(ctx, sid)
    elif s.kind == "texts":
        sids = B.oasm_open_streams(ctx, len(s.texts))
        for sid, t in zip(sids.tolist(), s.texts):
            B.oasm_feed_device(ctx, sid, t)
        B.oasm_end_streams(ctx, sids)
        B.oasm_step(ctx)
        n = B.oasm_drain(ctx, s.out).size
        B.oasm_close_streams(ctx, sids)
    else:
        sids = B.oasm_open_streams(ctx, s.n_streams)
        for i, (owner, offs, lens) in enumerate(s.packets):
            B.oasm_feed_many(ctx, sids[owner], s.payload, offs, lens)
            if i + 1 == len(s.packets):
                B.oasm_end_streams(ctx, sids)
            B.oasm_step(ctx)
            n += B.oasm_drain(ctx, s.out[n:]).size
        B.oasm_close_streams(ctx, sids)
    return _result(s, n)


def _records(case):
    """Records expected: the planted copies, and the matches of random text
    where they are many."""
    n = case["n"]
    records = n * case["per_sym"]
    if case["alpha"] == "dna" and case["n_pat"] == 1:
        # chance of a random match of a pattern of this length (0.0107 at m = 8, K = 2)
        records += n * min(0.05, 0.0107 * 4.0 ** (8 - case["mlo"]) * case["mlo"] / 8)
    elif case["kind"] == "texts":
        records += n * 0.034 * case["n_pat"] / 512
    elif case["alpha"] == "dna":
        records += n * 0.0035 * case["n_pat"] / 1024
    return int(records)


def work(case):
    """The text read once and the records (32 bytes each) written once.  The
    path has no floating-point work."""
    return {"bytes": case["n"] + 32 * _records(case), "flops": 0}


def tolerance(case):
    """Records are whole numbers and fully determined by the rules."""
    return "exact"


def exact(case, seed):
    """No output is a rounded number: nothing to compare in 64 bits."""
    return None
