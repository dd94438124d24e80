"""Scoring of several layers in one call, and the padded form at the edges of its transform lengths, against the fp64
oracle and against one call per layer."""
import numpy as np
import pytest
import torch

from oracle import flashcache_oracle as O

pytestmark = pytest.mark.gpu

TOL = {torch.float32: 1e-3, torch.float16: 2e-2, torch.bfloat16: 2e-2}


@pytest.fixture(scope="module")
def fc():
    if not torch.cuda.is_available():
        pytest.fail("GPU tests need a CUDA device")
    from paper_2511_16786_b200 import binding
    return binding


def _kv(T, H, d, dtype, seed):
    g = torch.Generator().manual_seed(seed)
    t = torch.arange(T, dtype=torch.float32)[:, None, None] / T
    k = 0.3 * torch.randn((T, H, d), generator=g) + 3.0 * torch.cos(2.5 * t + torch.randn((1, H, d), generator=g))
    v = 0.3 * torch.randn((T, H, d), generator=g) + 2.0 * t
    return k.to(dtype), v.to(dtype)


def _score_layers(fc, layers, cu, gamma):
    L, H, T = len(layers), layers[0][0].shape[1], cu[-1]
    h = fc.fc_create(0, max(cu[b + 1] - cu[b] for b in range(len(cu) - 1)))
    try:
        K, V = [k.cuda() for k, _ in layers], [v.cuda() for _, v in layers]
        scores = torch.full((L, H, T), -1.0, dtype=torch.float32, device="cuda")
        energy = torch.full((L, len(cu) - 1, 4), -1.0, dtype=torch.float64, device="cuda")
        ws = torch.empty(fc.fc_score_layers_workspace_bytes(h, K[0], V[0], cu, L), dtype=torch.uint8, device="cuda")
        fc.fc_score_layers(h, K, V, cu, gamma, scores, energy, ws)
        assert fc.fc_last_device_status(h) == 0
        one_s, one_e = torch.empty_like(scores), torch.empty_like(energy)
        ws1 = torch.empty(fc.fc_score_workspace_bytes(h, K[0], V[0], cu), dtype=torch.uint8, device="cuda")
        for l in range(L):
            fc.fc_score_layer(h, K[l], V[l], cu, gamma, one_s[l], one_e[l], ws1)
        assert fc.fc_last_device_status(h) == 0
        return scores.cpu(), energy.cpu(), one_s.cpu(), one_e.cpu()
    finally:
        fc.fc_destroy(h)


def _check_head(k, v, score, gamma, dtype):
    o, _ = O.score_head(k.double().numpy(), v.double().numpy(), gamma, "fft")
    ebar = (k.double().square().sum(1) + v.double().square().sum(1)).mean().item() / k.shape[1]
    err = np.abs(score.double().numpy() - o) / np.maximum(o, 1e-6 * ebar)
    assert err.max() <= TOL[dtype], "score error %.3e" % err.max()


# more layers than one launch spans (32), lengths of every kind incl. an empty sequence
@pytest.mark.parametrize("L,lens,H,dtype", [(35, (1000, 0, 1024, 3), 2, torch.bfloat16), (3, (20500, 2048, 513), 3, torch.float16),
                                            (2, (65536, 40000), 1, torch.float32)])
def test_layers_in_one_call_equal_one_call_per_layer(fc, L, lens, H, dtype):
    cu = [0] + [int(x) for x in np.cumsum(lens)]
    layers = [_kv(cu[-1], H, 128, dtype, 7 * l + L) for l in range(L)]
    s, e, s1, e1 = _score_layers(fc, layers, cu, 0.2)
    assert torch.equal(s.view(torch.int32), s1.view(torch.int32)) and torch.equal(e.view(torch.int64), e1.view(torch.int64))
    for l in (0, L - 1):
        k, v = layers[l]
        for b, n in enumerate(lens):
            if n:
                _check_head(k[cu[b]:cu[b + 1], H - 1], v[cu[b]:cu[b + 1], H - 1], s[l, H - 1, cu[b]:cu[b + 1]], 0.2, dtype)


# 2N - 1 just below and just above a transform length of every first factor, the longest sequence, both band edges
@pytest.mark.parametrize("N,gamma", [(640, 0.2), (641, 0.2), (768, 0.2), (896, 0.0), (897, 0.2), (1280, 0.2), (1536, 1.0),
                                     (1792, 0.2), (1793, 0.3), (36865, 0.2), (49152, 0.1), (57345, 0.2), (65535, 0.2)])
def test_padded_lengths_at_their_edges(fc, N, gamma):
    k, v = _kv(N, 1, 64, torch.float32, N)
    s, e, _, _ = _score_layers(fc, [(k, v)], [0, N], gamma)
    _check_head(k[:, 0], v[:, 0], s[0, 0], gamma, torch.float32)
    _, eo = O.score_head(k[:, 0].double().numpy(), v[:, 0].double().numpy(), gamma, "fft")
    np.testing.assert_allclose(e[0, 0, [1, 3]].numpy(), np.asarray(eo)[[1, 3]], rtol=1e-5)


# one handle, one length, head dimensions that fill a cluster of the small kernel (128) and that do not (192, 256 at more
# than 256 tokens, 384): each finds a filter table of its own form
@pytest.mark.parametrize("N", [100, 300, 333, 500, 1000])
def test_head_dims_that_take_different_kernels_share_a_handle(fc, N):
    h = fc.fc_create(0, N)
    try:
        for d in (128, 192, 256, 384, 128, 192):
            k, v = _kv(N, 2, d, torch.float32, N + d)
            kd, vd = k.cuda(), v.cuda()
            scores = torch.full((2, N), -1.0, dtype=torch.float32, device="cuda")
            energy = torch.full((1, 4), -1.0, dtype=torch.float64, device="cuda")
            ws = torch.empty(fc.fc_score_workspace_bytes(h, kd, vd, [0, N]), dtype=torch.uint8, device="cuda")
            fc.fc_score_layer(h, kd, vd, [0, N], 0.2, scores, energy, ws)
            assert fc.fc_last_device_status(h) == 0
            for head in range(2):
                _check_head(k[:, head], v[:, head], scores[head].cpu(), 0.2, torch.float32)
    finally:
        fc.fc_destroy(h)


# calls left on the internal streams, one after the other, that put their buffers at different places of one workspace: the
# second waits for the first (the two pairs' sizes are such that a sum or exclusive-or of them does not tell them apart)
@pytest.mark.parametrize("N,first,second", [(2048, (31, 11, 64), (17, 5, 256)), (4096, (31, 11, 64), (17, 5, 256)),
                                            (8192, (2, 4, 128), (3, 2, 64))])
def test_deferred_calls_share_a_workspace(fc, N, first, second):
    cu = [0, N]
    h = fc.fc_create(0, N)
    try:
        calls = []
        for L, H, d in (first, second):
            layers = [_kv(N, H, d, torch.bfloat16, 100 * l + H) for l in range(L)]
            K, V = [k.cuda() for k, _ in layers], [v.cuda() for _, v in layers]
            need = fc.fc_score_layers_workspace_bytes(h, K[0], V[0], cu, L)
            calls.append((K, V, need, torch.empty((L, H, N), device="cuda"), torch.empty((L, 1, 4), dtype=torch.float64, device="cuda")))
        ws = torch.empty(max(c[2] for c in calls), dtype=torch.uint8, device="cuda")
        want = []
        for K, V, _, scores, energy in calls:
            fc.fc_score_layers(h, K, V, cu, 0.2, scores, energy, ws)
            want.append((scores.clone(), energy.clone()))
        fc.fc_set_score_overlap(h, True)
        for _ in range(3):
            for K, V, _, scores, energy in calls:
                scores.zero_()
                energy.zero_()
            for K, V, _, scores, energy in calls:
                fc.fc_score_layers(h, K, V, cu, 0.2, scores, energy, ws)
            assert fc.fc_last_device_status(h) == 0
            for (_, _, _, scores, energy), (ws_, we) in zip(calls, want):
                assert torch.equal(scores, ws_) and torch.equal(energy, we)
    finally:
        fc.fc_destroy(h)
