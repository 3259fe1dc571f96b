"""GPU parity of the copies into the text arena: device pieces of every length
and alignment around the 16-byte vectors, the warp- and block-sized copies and
their chunk length; short patterns at K = 0 find nearly every symbol, so a
wrong byte shows in the ends."""
import numpy as np
import pytest

from paper_1712_03560_gb300 import binding as B
from paper_1712_03560_gb300 import workloads as W
from parity_util import canon, gpu_rows, oracle_rows

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("lens", [list(range(1, 70)), [15, 16, 17, 31, 32, 33, 47, 48, 4095, 4096],
                                  [4097, 3, 65535, 65536, 65537, 1, 100_003]])
def test_pieces_of_any_alignment(lens):
    import torch
    rng = np.random.default_rng(970 + len(lens))
    text = W.DNA[rng.integers(0, 4, size=sum(lens))]
    pats = [W.DNA[rng.integers(0, 4, size=3)] for _ in range(24)]
    want = oracle_rows(pats, [0] * len(pats), text, mode="ends")
    for start in (0, 1, 7, 15):
        ctx = B.oasm_create(pats, [0] * len(pats), {"output": "ends"})
        try:
            sid = B.oasm_open_stream(ctx)
            keep, pos = [], 0
            for i, n in enumerate(lens):  # each piece at its own offset in its own buffer
                off = (start + 5 * i) % 16
                buf = torch.zeros(n + off, dtype=torch.uint8, device="cuda")
                buf[off:] = torch.from_numpy(text[pos:pos + n].copy()).cuda()
                keep.append(buf)
                B.oasm_feed_device(ctx, sid, buf[off:])
                pos += n
            torch.cuda.synchronize()
            got = gpu_rows(B.oasm_flush(ctx, sid, end_of_stream=True))
        finally:
            B.oasm_destroy(ctx)
        assert canon(got) == want
