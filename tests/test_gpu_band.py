"""Scoring in the kept band (16-bit inputs whose kept band a grid of a quarter to half of the tokens holds) at the edges of its
windows, grids and dispatch rule, against the fp64 oracle."""
import math

import numpy as np
import pytest
import torch

from oracle import flashcache_oracle as O

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def fc():
    if not torch.cuda.is_available():
        pytest.fail("GPU tests need a CUDA device")
    from paper_2511_16786_b200 import binding
    return binding


def _kv(T, H, d, dtype, seed):
    g = torch.Generator().manual_seed(seed)
    t = torch.arange(T, dtype=torch.float32)[:, None, None] / T
    far = torch.rand((T, H, 1), generator=g) < 0.1
    out = []
    for a in (2.5, 7.0):
        n = torch.randn((T, H, d), generator=g)
        trend = 3.0 * torch.cos(a * t + torch.randn((1, H, d), generator=g))
        out.append(torch.where(far, 5.0 * n, trend + 0.1 * n).to(dtype))
    return out


def _score(fc, k, v, cu, gamma, repeat=1):
    """scores [H, T] and energies [B, 4] of one layer, the same in every repetition"""
    H, d, T = k.shape[1], k.shape[2], cu[-1]
    h = fc.fc_create(0, max(cu[b + 1] - cu[b] for b in range(len(cu) - 1)))
    try:
        ws = torch.empty(fc.fc_score_workspace_bytes(h, k, v, cu), dtype=torch.uint8, device="cuda")
        got = []
        for i in range(repeat):
            ws.fill_(255 if i % 2 else 0)
            s = torch.full((H, T), -1.0, dtype=torch.float32, device="cuda")
            e = torch.full((len(cu) - 1, 4), -1.0, dtype=torch.float64, device="cuda")
            fc.fc_score_layer(h, k, v, cu, gamma, s, e, ws)
            assert fc.fc_last_device_status(h) == 0
            got.append((s.cpu(), e.cpu()))
    finally:
        fc.fc_destroy(h)
    for s, e in got[1:]:
        assert torch.equal(s, got[0][0]) and torch.equal(e, got[0][1])
    return got[0]


def _check(k, v, cu, gamma, scores, energy):
    d = k.shape[2]
    for b in range(len(cu) - 1):
        sums = np.zeros(4)
        for h in range(k.shape[1]):
            kk, vv = (x[cu[b]:cu[b + 1], h].double().numpy() for x in (k, v))
            o, _ = O.score_head(kk, vv, gamma, "fft")
            g = scores[h, cu[b]:cu[b + 1]].double().numpy()
            # A residual is z - base, the base a sum of fp32 products: its error per element is bounded by a small
            # multiple (here 24) of 2^-24 times the head's values, and a score, the mean of the squares of 2d residuals,
            # moves by at most twice its own root times that (plus the error's square).
            eps = 24 * 2.0 ** -24 * math.sqrt(((kk ** 2).sum(1) + (vv ** 2).sum(1)).max() / d)
            bound = 2 * np.sqrt(o) * eps + eps * eps + 1e-6 * o
            assert (np.abs(g - o) <= bound).all(), "%d tokens, head %d: %.2f of the bound" % (
                cu[b + 1] - cu[b], h, (np.abs(g - o) / bound).max())
            rk, rv = kk - O.base_kv(kk, gamma, "fft")[0], vv - O.base_kv(vv, gamma, "fft")[0]
            sums += [(rk ** 2).sum(), (kk ** 2).sum(), (rv ** 2).sum(), (vv ** 2).sum()]
        assert np.allclose(energy[b].numpy(), sums, rtol=2e-6, atol=1e-12)


# the smallest and largest sequences, every transform length, whole and broken ratios of tokens to grid points, lengths
# around the 128-token and 16-point steps, cutoffs from none to beyond what the form takes, head widths of one to four tiles
@pytest.mark.parametrize("N,H,d,gamma,dtype", [
    (513, 3, 128, 0.2, torch.bfloat16), (767, 1, 64, 0.1, torch.float16), (1023, 2, 128, 0.3, torch.bfloat16), (1025, 2, 64, 0.2, torch.float16), (1151, 1, 192, 0.15, torch.bfloat16),
    (1281, 2, 128, 0.0, torch.bfloat16), (2047, 2, 128, 0.2, torch.float16), (2048, 1, 256, 0.3, torch.bfloat16),
    (2500, 2, 128, 0.39, torch.bfloat16), (3072, 2, 64, 0.25, torch.float16), (4096, 2, 128, 0.2, torch.bfloat16),
    (4097, 2, 128, 0.2, torch.bfloat16), (5119, 3, 128, 0.1, torch.float16), (8192, 2, 64, 0.2, torch.bfloat16),
    (10164, 2, 128, 0.2, torch.bfloat16), (16384, 1, 128, 0.3, torch.float16), (32768, 1, 128, 0.3, torch.bfloat16),
    (53602, 1, 128, 0.2, torch.float16), (65535, 1, 64, 0.2, torch.bfloat16), (65536, 1, 128, 0.2, torch.bfloat16),
    (65536, 1, 64, 0.45, torch.bfloat16), (2200, 2, 128, 0.3, torch.bfloat16), (4200, 1, 128, 0.26, torch.float16)])
def test_band_scores(fc, N, H, d, gamma, dtype):
    k, v = _kv(N, H, d, dtype, N)
    s, e = _score(fc, k.cuda(), v.cuda(), [0, N], gamma, repeat=3)
    _check(k, v, [0, N], gamma, s, e)


def test_band_is_taken_where_the_rule_says(fc):
    # 16-bit rows of 513 .. 65536 tokens, not 1024, heads of up to 512 channels, where a grid of a power of two points M holds
    # the band (256 <= M <= 16384, N/4 <= M <= N/2, omega <= 0.8 M) and 128 tokens with the kernel's ends lie within 24 aligned quads
    # of it, which keeps N just above 2 M with the widest kernels out (1100 tokens, 0.37)
    h = fc.fc_create(0, 131072)
    try:
        form = lambda N, gamma, dtype=torch.bfloat16, d=128: tuple(fc.fc_scoring_form(h, N, dtype, d, gamma).values())
        for N, gamma, want in [
                (512, 0.2, ("short", 512)), (513, 0.2, ("band", 256)), (599, 0.3, ("band", 256)), (767, 0.1, ("band", 256)),
                (1023, 0.3, ("padded", 2048)), (1024, 0.2, ("short", 1024)), (1025, 0.2, ("band", 512)), (1100, 0.37, ("padded", 2560)),
                (1281, 0.0, ("band", 512)), (1100, 0.3, ("band", 512)), (2047, 0.2, ("band", 512)), (2048, 0.3, ("band", 1024)), (2048, 0.39, ("band", 1024)),
                (2500, 0.39, ("padded", 5120)), (4096, 0.2, ("band", 1024)), (4097, 0.2, ("band", 2048)), (4200, 0.26, ("band", 2048)),
                (16384, 0.3, ("band", 8192)), (32768, 0.2, ("band", 8192)), (32768, 0.45, ("direct", 32768)), (32769, 0.2, ("band", 16384)),
                (65535, 0.2, ("band", 16384)), (65536, 0.2, ("band", 16384)), (65536, 0.45, ("direct", 65536))]:
            assert form(N, gamma) == want, (N, gamma)
            assert form(N, gamma, torch.float16) == want, (N, gamma)
            assert form(N, gamma, torch.float32)[0] != "band"
        assert form(2048, 0.2, d=512)[0] == "band" and form(2048, 0.2, d=576)[0] == "direct"
        assert form(131072, 0.2)[0] == "generic"
    finally:
        fc.fc_destroy(h)


def test_band_ragged_batch_strided_views_and_neighbours(fc):
    # sequences of every form side by side, rows and heads strided, and non-finite rows of one sequence next to another's
    lens = [1100, 300, 1100, 4096, 2311]
    cu = [0] + [int(x) for x in np.cumsum(lens)]
    k, v = _kv(cu[-1], 3, 64, torch.bfloat16, 5)
    wide = [torch.full((cu[-1], 5, 80), float("nan"), dtype=torch.bfloat16, device="cuda") for _ in range(2)]
    kd, vd = (w[:, 1:4, :64] for w in wide)
    kd.copy_(k)
    vd.copy_(v)
    s, e = _score(fc, kd, vd, cu, 0.2, repeat=2)
    _check(k, v, cu, 0.2, s, e)
    bad = k.clone()
    bad[cu[2]:cu[2] + 40, 1, 3] = float("nan")
    bad[cu[3] - 1, 1, 60] = float("inf")
    kd.copy_(bad)
    s2, _ = _score(fc, kd, vd, cu, 0.2)
    assert torch.isnan(s2[1, cu[2]:cu[3]]).all()
    s2[1, cu[2]:cu[3]] = s[1, cu[2]:cu[3]]
    assert torch.equal(s, s2)


def test_band_heads_before_tokens(fc):
    # [H, T, d] storage seen as [T, H, d]: the head stride is the larger one
    k, v = _kv(1500, 3, 128, torch.float16, 7)
    kd, vd = (x.transpose(0, 1).contiguous().cuda().transpose(0, 1) for x in (k, v))
    s, e = _score(fc, kd, vd, [0, 1500], 0.2)
    _check(k, v, [0, 1500], 0.2, s, e)


def test_band_calls_agree_however_the_work_is_grouped(fc):
    # many layers in one call (internal streams, several launch groups), one call per layer (the caller's stream), small
    # launch groups, and a replayed capture, whose tables are built anew: the same bits
    L, lens, H, d = 9, [2311, 1100], 2, 128
    cu = [0] + [int(x) for x in np.cumsum(lens)]
    K, V = zip(*(_kv(cu[-1], H, d, torch.bfloat16, 20 + l) for l in range(L)))
    K, V = [k.cuda() for k in K], [v.cuda() for v in V]
    ref_s, ref_e = zip(*(_score(fc, K[l], V[l], cu, 0.2) for l in range(L)))
    for group_bytes in (None, 1 << 16):
        comp = fc.Compressor(L, H, d, cu, torch.bfloat16, 0.2, 0.2, group_bytes=group_bytes)
        comp.compress(K, V)
        comp.check_device_status()
        got = [comp.scores.clone(), comp.energy.clone()]
        graph = comp.capture(K, V)
        comp.scores.zero_()
        comp.energy.zero_()
        graph.replay()
        comp.check_device_status()
        for s, e in (got, [comp.scores, comp.energy]):
            for l in range(L):
                assert torch.equal(s[l].cpu(), ref_s[l]) and torch.equal(e[l].cpu(), ref_e[l])
        del graph
        comp.close()


def test_band_scales(fc):
    # rows whose channels differ by many powers of two: a channel's values are scaled by themselves
    k, v = _kv(2048, 1, 128, torch.bfloat16, 11)
    f = torch.exp2(torch.arange(128) % 61 - 30.0)
    k, v = (k.float() * f).to(torch.bfloat16), (v.float() * f.flip(0)).to(torch.bfloat16)
    k[:, 0, 5] = 0.0
    s, e = _score(fc, k.cuda(), v.cuda(), [0, 2048], 0.2)
    _check(k, v, [0, 2048], 0.2, s, e)


@pytest.mark.parametrize("lens", [[1500], [2048, 1100, 300]])
def test_band_deferred_calls_of_broken_lengths_are_complete_in_stream_order(fc, lens):
    # fc_set_score_overlap defers the join only where every sequence is short or a power of two long: whatever the caller's
    # stream reads after such a call is final, with enough layers that the call uses the internal streams
    L, H, d = 28, 4, 128
    cu = [0] + [int(x) for x in np.cumsum(lens)]
    K, V = zip(*(_kv(cu[-1], H, d, torch.bfloat16, 40 + l) for l in range(L)))
    K, V = [k.cuda() for k in K], [v.cuda() for v in V]
    h = fc.fc_create(0, max(lens))
    try:
        ws = torch.empty(fc.fc_score_layers_workspace_bytes(h, K[0], V[0], cu, L), dtype=torch.uint8, device="cuda")
        s = torch.empty((L, H, cu[-1]), dtype=torch.float32, device="cuda")
        e = torch.empty((L, len(lens), 4), dtype=torch.float64, device="cuda")
        fc.fc_score_layers(h, K, V, cu, 0.2, s, e, ws)
        ref = s.clone(), e.clone()
        assert fc.fc_last_device_status(h) == 0
        fc.fc_set_score_overlap(h, True)
        busy = torch.randn((4096, 4096), device="cuda")
        for _ in range(5):
            busy = torch.tanh(busy @ busy)                # the call is enqueued whole while the stream works on this
            s.fill_(-1.0)
            e.fill_(-1.0)
            fc.fc_score_layers(h, K, V, cu, 0.2, s, e, ws)
            got = s.clone(), e.clone()                    # by the caller's stream, without a joining call
            s.fill_(-2.0)
            assert torch.equal(got[0], ref[0]) and torch.equal(got[1], ref[1])
        assert fc.fc_last_device_status(h) == 0
    finally:
        fc.fc_destroy(h)


@pytest.mark.parametrize("N,d,gamma,dtype", [(599, 128, 0.3, torch.bfloat16), (3540, 128, 0.2, torch.bfloat16),
                                             (8192, 128, 0.3, torch.float16), (9144, 64, 0.3, torch.bfloat16),
                                             (32768, 128, 0.2, torch.bfloat16), (38863, 128, 0.3, torch.float16)])
def test_band_single_scores_are_as_exact_as_fp32_passes(fc, N, d, gamma, dtype):
    # Single scores, small ones as much as large ones: the relative error of the three fp32 passes over lengths, cutoffs and
    # widths like these (10 % of the rows far from a smooth trend) is 3.2e-7 .. 6.2e-7 in the root mean square, that of sums
    # cut off at 24 bits and of two-term matrices 7.8e-7 .. 1.05e-6.
    g = torch.Generator().manual_seed(N)
    i, m = torch.arange(N, dtype=torch.float64)[:, None], torch.arange(8, dtype=torch.float64)[None, :]
    basis = torch.cos(math.pi / (2 * N) * m * (2 * i + 1)).float()
    far = torch.rand((N, 2, 1), generator=g) < 0.1
    k, v = (torch.where(far, 5.0 * n, (basis @ torch.randn((8, 2 * d), generator=g)).view(N, 2, d) + 0.1 * n).to(dtype)
            for n in (torch.randn((N, 2, d), generator=g) for _ in range(2)))
    s, _ = _score(fc, k.cuda(), v.cuda(), [0, N], gamma)
    for h in range(2):
        o, _ = O.score_head(k[:, h].double().numpy(), v[:, h].double().numpy(), gamma, "fft")
        rel = (s[h].double().numpy() - o) / o
        assert math.sqrt((rel ** 2).mean()) <= 6.2e-7
        assert abs(rel).max() <= 1e-5


@pytest.mark.parametrize("L,H,lens,most", [(28, 4, [32768], 300e6), (28, 4, [8192], 300e6), (32, 32, [16384], 300e6), (1, 4, [2048], 20e6)])
def test_band_workspace_is_bounded(fc, L, H, lens, most):
    # two groups of at most four times 32 MiB and, at powers of two, a few hundred KB of tables; all intermediates where
    # those are less: 2 streams x 4 heads x 256 channels x 1024 values of 4 bytes = 8.4 MB for one layer of 2048 tokens
    h = fc.fc_create(0, max(lens))
    try:
        k = torch.empty((lens[0], H, 128), dtype=torch.bfloat16, device="cuda")
        assert 0 < fc.fc_score_layers_workspace_bytes(h, k, k, [0, lens[0]], L) <= most
    finally:
        fc.fc_destroy(h)


def test_band_tables_are_kept_evicted_and_rebuilt(fc):
    # one handle over calls whose tables fill what it keeps, displace one another, do not fit at all or are more than it counts:
    # the same bits as from a handle that has seen nothing else; one sequence (the caller's stream) and several (internal
    # streams, deferred or not) by turns on one workspace
    H, d = 2, 64
    calls = [[517, 1999, 4096, 2311], [1500], [1500, 1100, 2500], [517, 1999, 4096, 2311], [3000, 2700, 4095], [2048], [2311],
             [600, 700, 800, 900, 1000, 1100, 1200, 1300, 1400, 1700], [1100, 300, 1100], [4096, 2048], [4095], [1999, 1500]]
    data, ref = {}, {}
    for lens in calls:
        cu = [0] + [int(x) for x in np.cumsum(lens)]
        k, v = (x.cuda() for x in _kv(cu[-1], H, d, torch.float16, sum(lens)))
        data[tuple(lens)] = (cu, k, v)
        ref[tuple(lens)] = _score(fc, k, v, cu, 0.2)
    h = fc.fc_create(0, 4096)
    try:
        ws = torch.empty(max(fc.fc_score_workspace_bytes(h, k, v, cu) for cu, k, v in data.values()), dtype=torch.uint8, device="cuda")
        for rnd in range(4):
            fc.fc_set_score_overlap(h, rnd % 2 == 1)
            got = []
            for i, lens in enumerate(calls if rnd < 2 else calls[::-1]):
                cu, k, v = data[tuple(lens)]
                s = torch.full((H, cu[-1]), -1.0, dtype=torch.float32, device="cuda")
                e = torch.full((len(lens), 4), -1.0, dtype=torch.float64, device="cuda")
                fc.fc_score_layer(h, k, v, cu, 0.2, s, e, ws)
                got.append((lens, s, e))
            assert fc.fc_last_device_status(h) == 0
            for lens, s, e in got:
                assert torch.equal(s.cpu(), ref[tuple(lens)][0]) and torch.equal(e.cpu(), ref[tuple(lens)][1]), lens
    finally:
        fc.fc_destroy(h)


def test_band_more_layers_than_one_launch_spans(fc):
    # 35 layers in one call against one call each, on a length whose work fits the caller's stream chunk by chunk and one whose does not
    H, d, L = 1, 64, 35
    for lens in ([640], [2500, 1030]):
        cu = [0] + [int(x) for x in np.cumsum(lens)]
        K, V = zip(*(_kv(cu[-1], H, d, torch.bfloat16, 70 + l) for l in range(L)))
        K, V = [k.cuda() for k in K], [v.cuda() for v in V]
        h = fc.fc_create(0, max(lens))
        try:
            ws = torch.empty(fc.fc_score_layers_workspace_bytes(h, K[0], V[0], cu, L), dtype=torch.uint8, device="cuda")
            s = torch.empty((L, H, cu[-1]), dtype=torch.float32, device="cuda")
            e = torch.empty((L, len(lens), 4), dtype=torch.float64, device="cuda")
            fc.fc_score_layers(h, K, V, cu, 0.2, s, e, ws)
            assert fc.fc_last_device_status(h) == 0
            for l in range(L):
                one_s, one_e = _score(fc, K[l], V[l], cu, 0.2)
                assert torch.equal(s[l].cpu(), one_s) and torch.equal(e[l].cpu(), one_e)
        finally:
            fc.fc_destroy(h)
        _check(K[34].cpu(), V[34].cpu(), cu, 0.2, s[34].cpu(), e[34].cpu())


# wide heads: an odd number of 64-channel halves (K and V share a tile), and the widest that the form takes
@pytest.mark.parametrize("N,H,d,dtype", [(1100, 2, 320, torch.bfloat16), (2048, 1, 448, torch.float16), (2311, 1, 512, torch.bfloat16),
                                         (1500, 1, 576, torch.bfloat16)])
def test_band_wide_heads(fc, N, H, d, dtype):
    k, v = _kv(N, H, d, dtype, N + d)
    s, e = _score(fc, k.cuda(), v.cuda(), [0, N], 0.2, repeat=2)
    if d <= 512:
        _check(k, v, [0, N], 0.2, s, e)
    else:                                     # on the passes: their own tolerance
        for h in range(H):
            o, _ = O.score_head(k[:, h].double().numpy(), v[:, h].double().numpy(), 0.2, "fft")
            assert np.allclose(s[h].double().numpy(), o, rtol=1e-3, atol=1e-9)
