"""fc_decode_attention where its blocks' shares of the rows meet the sequences' edges: more sequences than a warp has
lanes, empty ones in between, sequences of one tile, one sequence over all blocks, more heads than SMs, tails only."""
import numpy as np
import pytest
import torch

from oracle import flashcache_oracle as O

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("lens,tails,H,G", [
    ([0] * 3 + [1, 64, 65, 0, 128] * 14 + [700], None, 2, 2),     # 74 sequences, 32 at a time
    ([9600], None, 1, 8),                                          # one sequence, one head: 150 tiles over every block
    ([64 * 149], None, 1, 1),
    ([130, 70], None, 160, 1),                                     # more heads than blocks
    ([0, 0, 5], [3, 0, 64], 3, 9),                                 # tails only, and behind a partial tile
    ([1000, 0, 3000] * 12, [1, 65, 0] * 12, 2, 16)])
def test_decode_shares_at_sequence_edges(lens, tails, H, G):
    from paper_2511_16786_b200 import binding as fc
    g = torch.Generator().manual_seed(len(lens) + H)
    offs, B = [0] + [int(x) for x in np.cumsum(lens)], len(lens)
    rows = max(offs[-1], 1)
    q = torch.randn((B, H * G, 128), generator=g).to(torch.bfloat16)
    ck, cv = (torch.randn((rows, H, 128), generator=g).to(torch.bfloat16) for _ in range(2))
    tk = tv = tl = None
    if tails:
        tk, tv = (torch.randn((B, 80, H, 128), generator=g).to(torch.bfloat16) for _ in range(2))
        tl = torch.tensor(tails, dtype=torch.int32)
    h = fc.fc_create(0, 64)
    try:
        dev = [t.cuda() if t is not None else None for t in (q, ck, cv, torch.tensor(offs), tk, tv, tl)]
        most = max(n + (tails[b] if tails else 0) for b, n in enumerate(lens))
        args = fc.make_decode_args(*dev[:4], most, *dev[4:])
        ws = torch.empty(fc.fc_decode_workspace_bytes(h, args), dtype=torch.uint8, device="cuda")
        out = torch.full(q.shape, float("nan"), dtype=q.dtype, device="cuda")
        for _ in range(2):                                          # the second call finds the first one's workspace
            fc.fc_decode_attention(h, args, out, ws)
        assert fc.fc_last_device_status(h) == 0
        got = out.double().cpu().numpy()
    finally:
        fc.fc_destroy(h)
    extra = (tk.double().numpy(), tv.double().numpy(), tails) if tails else ()
    want = O.decode_attention(q.double().numpy(), ck.double().numpy(), cv.double().numpy(), offs, *extra)
    scale = np.maximum(np.abs(want).max(axis=-1, keepdims=True), 1e-6)
    assert (np.abs(got - want) / scale).max() <= 2e-2
    for b in range(B):
        if lens[b] + (tails[b] if tails else 0) == 0:
            assert not got[b].any()
