"""Spectrum, selection and short-sequence scoring at the edges of their dispatch rules and tiles, against the fp64 oracle
(selection: exactly)."""
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
    k = 0.3 * torch.randn((T, H, d), generator=g) + torch.cos(2.5 * t + torch.randn((1, H, d), generator=g))
    v = 0.3 * torch.randn((T, H, d), generator=g) + t
    return k.to(dtype), v.to(dtype)


# the generic kernels (512), every direct shape, and chirp lengths just inside a transform length of every first factor,
# with rows of 32 to 512 points; heads in one launch and in several, a head in column groups
@pytest.mark.parametrize("lens,H,d,dtype", [((512, 1024, 2048, 640, 641), 2, 64, torch.float32),
                                            ((4096, 8192, 897, 1793), 3, 128, torch.float16),
                                            ((16384, 10000), 4, 128, torch.bfloat16),
                                            ((65536, 24577, 36865), 1, 64, torch.float32),
                                            ((65535, 57345), 1, 128, torch.bfloat16)])
def test_power_spectrum_at_its_edges(fc, lens, H, d, dtype):
    cu = [0] + [int(x) for x in np.cumsum(lens)]
    k, v = _kv(cu[-1], H, d, dtype, cu[-1])
    h = fc.fc_create(0, max(lens))
    try:
        kd, vd = k.cuda(), v.cuda()
        ws = torch.empty(fc.fc_power_spectrum_workspace_bytes(h, kd, vd, cu), dtype=torch.uint8, device="cuda")
        got = []
        for _ in range(2):                                    # the second call finds its tables kept
            spec = torch.full((cu[-1], 2), -1.0, dtype=torch.float64, device="cuda")
            fc.fc_power_spectrum(h, kd, vd, cu, spec, ws)
            assert fc.fc_last_device_status(h) == 0
            got.append(spec.cpu())
            ws.fill_(255)
    finally:
        fc.fc_destroy(h)
    assert torch.equal(got[0], got[1])
    want = O.power_spectrum(k.double().numpy(), v.double().numpy(), cu, "fft")
    for b in range(len(lens)):
        w, g = want[cu[b]:cu[b + 1]], got[0][cu[b]:cu[b + 1]].numpy()
        for j in range(2):
            err = np.abs(g[:, j] - w[:, j]) / np.maximum(w[:, j], 1e-6 * w[:, j].max())
            assert err.max() <= 2e-3, "%d tokens: %.3e" % (lens[b], err.max())


# powers of two the small kernel runs directly, padded lengths around each of its transforms, and head dims whose
# blocks make a cluster (or do not: 192)
@pytest.mark.parametrize("d", [64, 128, 192, 256])
def test_short_sequences_at_their_edges(fc, d):
    lens = (1, 2, 32, 33, 63, 64, 65, 128, 129, 256, 257, 512, 513, 1024)
    cu = [0] + [int(x) for x in np.cumsum(lens)]
    k, v = _kv(cu[-1], 2, d, torch.float32, d)
    h = fc.fc_create(0, max(lens))
    try:
        kd, vd = k.cuda(), v.cuda()
        scores = torch.full((2, cu[-1]), -1.0, device="cuda")
        energy = torch.empty((len(lens), 4), dtype=torch.float64, device="cuda")
        ws = torch.empty(fc.fc_score_workspace_bytes(h, kd, vd, cu), dtype=torch.uint8, device="cuda")
        fc.fc_score_layer(h, kd, vd, cu, 0.2, scores, energy, ws)
        assert fc.fc_last_device_status(h) == 0
        scores, energy = scores.cpu().numpy(), energy.cpu().numpy()
    finally:
        fc.fc_destroy(h)
    for b, n in enumerate(lens):
        ks, vs = k[cu[b]:cu[b + 1]].double().numpy(), v[cu[b]:cu[b + 1]].double().numpy()
        tot = 0.0
        for hd in range(2):
            want, en = O.score_head(ks[:, hd], vs[:, hd], 0.2, "fft")
            ebar = ((ks[:, hd] ** 2).sum(1) + (vs[:, hd] ** 2).sum(1)).mean() / d
            err = np.abs(scores[hd, cu[b]:cu[b + 1]] - want) / np.maximum(want, 1e-6 * ebar)
            assert err.max() <= 1e-3, "%d tokens: %.3e" % (n, err.max())
            tot += np.asarray(en)[1]
        np.testing.assert_allclose(energy[b, 1], tot, rtol=1e-5)


# lengths around what one block, and a cluster of two, four and eight, hold; budgets at both ends; scores that leave the
# threshold's bin with few keys (finished directly), with many distinct ones (every digit), and with one value for all
@pytest.mark.parametrize("per_layer", [False, True])
@pytest.mark.parametrize("n", [2047, 4097, 16384, 16385, 32769, 65537, 131072])
def test_selection_at_its_edges(fc, n, per_layer):
    rng = np.random.default_rng(n)
    H, d = 3, 64
    g = torch.Generator().manual_seed(n)
    k, v = torch.randn((n, H, d), generator=g).half(), torch.randn((n, H, d), generator=g).half()
    spread = (rng.integers(0, 1 << 17, (H, n)) * 2.0 ** -17).astype(np.float32)          # sums over heads are exact
    near = (1.0 + rng.integers(0, 4096, (H, n)) * 2.0 ** -20).astype(np.float32)
    same = np.full((H, n), 0.25, np.float32)
    h = fc.fc_create(0, 131072)
    try:
        kd, vd, cu = k.cuda(), v.cuda(), [0, n]
        ws = torch.empty(fc.fc_select_workspace_bytes(h, kd, vd, cu), dtype=torch.uint8, device="cuda")
        for scores in (spread, near, same):
            for budget in (1, n // 5, n - 1, n):
                out_k = torch.zeros((budget, H, d), dtype=k.dtype, device="cuda")
                out_v, idx = torch.zeros_like(out_k), torch.full((H, budget), -1, dtype=torch.int32, device="cuda")
                bd = torch.tensor([budget], dtype=torch.int32, device="cuda")
                of = torch.tensor([0, budget], dtype=torch.int64, device="cuda")
                fc.fc_select_compact_ex(h, kd, vd, cu, torch.from_numpy(scores).cuda(), bd, of, out_k, out_v, idx, ws,
                                        per_layer=per_layer)
                assert fc.fc_last_device_status(h) == 0
                for hd in range(H):
                    got = idx[hd].cpu().numpy()
                    dev = scores.astype(np.float64)
                    np.testing.assert_array_equal(got, O.select_topk(O.layer_score(dev) if per_layer else dev[hd], budget))
                    at = torch.from_numpy(got.astype(np.int64)).cuda()
                    assert torch.equal(out_k[:, hd], kd[at, hd]) and torch.equal(out_v[:, hd], vd[at, hd])
    finally:
        fc.fc_destroy(h)


# short sequences in more blocks than SMs (smaller blocks that share an SM), around the lengths they hold
@pytest.mark.parametrize("lens", [(1024, 1, 0, 300), (1025, 2048, 7), (2049, 64, 4096), (4097, 100, 1000)])
def test_selection_of_many_short_sequences(fc, lens):
    rng = np.random.default_rng(sum(lens))
    H, d, cu = 256, 64, [0] + [int(x) for x in np.cumsum(lens)]
    budgets = [(n + 3) // 4 for n in lens]
    offs = [0] + [int(x) for x in np.cumsum(budgets)]
    g = torch.Generator().manual_seed(sum(lens))
    k = torch.randn((cu[-1], H, d), generator=g).half().cuda()
    scores = (rng.integers(0, 1 << 12, (H, cu[-1])) * 2.0 ** -9).astype(np.float32)
    h = fc.fc_create(0, 8192)
    try:
        ws = torch.empty(fc.fc_select_workspace_bytes(h, k, k, cu), dtype=torch.uint8, device="cuda")
        out_k = torch.zeros((offs[-1], H, d), dtype=k.dtype, device="cuda")
        out_v, idx = torch.zeros_like(out_k), torch.full((H, offs[-1]), -1, dtype=torch.int32, device="cuda")
        fc.fc_select_compact_ex(h, k, k, cu, torch.from_numpy(scores).cuda(),
                                torch.tensor(budgets, dtype=torch.int32, device="cuda"),
                                torch.tensor(offs, dtype=torch.int64, device="cuda"), out_k, out_v, idx, ws)
        assert fc.fc_last_device_status(h) == 0
        for hd in range(H):
            for b in range(len(lens)):
                got = idx[hd, offs[b]:offs[b + 1]].cpu().numpy()
                np.testing.assert_array_equal(got, O.select_topk(scores[hd, cu[b]:cu[b + 1]].astype(np.float64), budgets[b]))
            at = torch.cat([idx[hd, offs[b]:offs[b + 1]].long() + cu[b] for b in range(len(lens))])
            assert torch.equal(out_k[:, hd], k[at, hd]) and torch.equal(out_v[:, hd], k[at, hd])
    finally:
        fc.fc_destroy(h)


# every token kept by clusters of two, four and eight blocks, more of them than run at a time: no digit is counted, so
# nothing but its own barrier lets a block write into its neighbours' memory
@pytest.mark.parametrize("n,batch,per_layer", [(300, 200, True), (16385, 60, False), (32769, 24, True), (65537, 10, False)])
def test_selection_that_keeps_every_token_in_clusters(fc, n, batch, per_layer):
    H, d, cu = 2, 64, [i * n for i in range(batch + 1)]
    g = torch.Generator(device="cuda").manual_seed(n)
    k = torch.randn((cu[-1], H, d), generator=g, device="cuda").half()
    scores = torch.rand((H, cu[-1]), generator=g, device="cuda")
    h = fc.fc_create(0, 131072)
    try:
        ws = torch.empty(fc.fc_select_workspace_bytes(h, k, k, cu), dtype=torch.uint8, device="cuda")
        out_k = torch.zeros_like(k)
        out_v, idx = torch.zeros_like(k), torch.full((H, cu[-1]), -1, dtype=torch.int32, device="cuda")
        fc.fc_select_compact_ex(h, k, k, cu, scores, torch.full((batch,), n, dtype=torch.int32, device="cuda"),
                                torch.tensor(cu, dtype=torch.int64, device="cuda"), out_k, out_v, idx, ws,
                                per_layer=per_layer)
        assert fc.fc_last_device_status(h) == 0
        assert torch.equal(idx, torch.arange(n, dtype=torch.int32, device="cuda").repeat(H, batch))
        assert torch.equal(out_k, k) and torch.equal(out_v, k)
    finally:
        fc.fc_destroy(h)


# more sequences than clusters run at a time (and than one launch describes), short and long in turn, so that clusters start
# while others end: every block may write to its cluster's first one only once that has started
def test_cutoff_of_many_sequences(fc):
    rng = np.random.default_rng(3)
    lens = [int(n) for n in rng.integers(1, 9000, 150)]
    lens[7] = lens[80] = 0
    cu = [0] + [int(x) for x in np.cumsum(lens)]
    P = rng.random((cu[-1], 2)) * np.exp(-rng.random((cu[-1], 1)) * 6.0)
    h = fc.fc_create(0, 9000)
    try:
        om = torch.full((150,), -7, dtype=torch.int32, device="cuda")
        ga = torch.full((150,), -7.0, dtype=torch.float64, device="cuda")
        fc.fc_cutoff_from_spectrum(h, torch.from_numpy(P).cuda(), cu, 0.7, om, ga)
        assert fc.fc_last_device_status(h) == 0
        om, ga = om.cpu().numpy(), ga.cpu().numpy()
    finally:
        fc.fc_destroy(h)
    for b, n in enumerate(lens):
        if n == 0:
            assert om[b] == 0 and ga[b] == 0.0
            continue
        seg = P[cu[b]:cu[b + 1]]
        wo, wg = O.cutoff_for_energy_share(seg, 0.7)
        if om[b] != wo:                                      # only where rounding of the running sum decides
            c, tot = np.cumsum(seg.sum(1)), seg.sum()
            assert abs(c[min(om[b], wo)] - 0.7 * tot) <= 1e-12 * tot
        else:
            assert ga[b] == wg


# few (sequence, head) pairs: one, two and four blocks each by length, around the numbers of pairs whose clusters fit
# at once (33 pairs of 4, 65 of 2 on 148 SMs do not)
@pytest.mark.parametrize("n", [2048, 2049, 4096, 4097, 8193, 16384, 16385])
@pytest.mark.parametrize("H", [1, 32, 33, 64, 65])
def test_selection_of_few_heads_takes_clusters(fc, n, H):
    rng = np.random.default_rng(n + H)
    d = 64
    scores = (rng.integers(0, 1 << 11, (H, n)) * 2.0 ** -9).astype(np.float32)          # many ties
    g = torch.Generator(device="cuda").manual_seed(n)
    k = torch.randn((n, H, d), generator=g, device="cuda").half()
    budget, cu = n // 3, [0, n]
    h = fc.fc_create(0, 16385)
    try:
        ws = torch.empty(fc.fc_select_workspace_bytes(h, k, k, cu), dtype=torch.uint8, device="cuda")
        out_k = torch.zeros((budget, H, d), dtype=k.dtype, device="cuda")
        out_v, idx = torch.zeros_like(out_k), torch.full((H, budget), -1, dtype=torch.int32, device="cuda")
        fc.fc_select_compact_ex(h, k, k, cu, torch.from_numpy(scores).cuda(),
                                torch.tensor([budget], dtype=torch.int32, device="cuda"),
                                torch.tensor([0, budget], dtype=torch.int64, device="cuda"), out_k, out_v, idx, ws)
        assert fc.fc_last_device_status(h) == 0
        for hd in {0, H // 2, H - 1}:
            np.testing.assert_array_equal(idx[hd].cpu().numpy(), O.select_topk(scores[hd].astype(np.float64), budget))
            at = idx[hd].long()
            assert torch.equal(out_k[:, hd], k[at, hd]) and torch.equal(out_v[:, hd], k[at, hd])
    finally:
        fc.fc_destroy(h)
