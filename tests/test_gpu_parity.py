"""GPU parity: the CUDA library (through its C ABI) against the fp64 CPU oracle on
the same seeded inputs, element by element.

Tolerances: score error |g-o| / max(o, 1e-6*e_bar) <= 1e-3
for fp32 inputs and <= 2e-2 for fp16/bf16 inputs, where e_bar is the head's mean
of (|k_x|^2+|v_x|^2)/d (so the gamma=1 case, whose true scores are 0, is still
testable); index sets identical except for tokens whose oracle score is within that
tolerance of the k-th largest; compacted rows bit-exact given the index set.
"""
import math

import numpy as np
import pytest
import torch

from oracle import flashcache_oracle as O
from paper_2511_16786_b200 import synth_kv as S

pytestmark = pytest.mark.gpu

TOL = {torch.float32: 1e-3, torch.float16: 2e-2, torch.bfloat16: 2e-2}


@pytest.fixture(scope="module")
def fc():
    if not torch.cuda.is_available():
        pytest.fail("GPU tests need a CUDA device")
    from paper_2511_16786_b200 import binding
    return binding


def _rand_kv(T, H, d, dtype, seed, smooth=True):
    g = torch.Generator().manual_seed(seed)
    k = torch.randn((T, H, d), generator=g)
    v = torch.randn((T, H, d), generator=g)
    if smooth and T > 1:
        t = torch.arange(T, dtype=torch.float32)[:, None, None] / T
        k = 0.3 * k + 3.0 * torch.cos(2.5 * t + torch.randn((1, H, d), generator=g))
        v = 0.3 * v + 2.0 * t + torch.randn((1, H, d), generator=g)
    return k.to(dtype), v.to(dtype)


def _gpu_scores(fc, k, v, cu, gamma, max_seqlen=None, group_bytes=None, band=None):
    T, H, d = k.shape
    seqlens = [cu[i + 1] - cu[i] for i in range(len(cu) - 1)]
    h = fc.fc_create(0, max_seqlen or max(1, max(seqlens, default=1)))
    try:
        if group_bytes:
            fc.fc_set_group_bytes(h, group_bytes)
        if band is not None:
            fc.fc_set_chirp_band(h, band)
        kd, vd = (k if k.is_cuda else k.cuda()), (v if v.is_cuda else v.cuda())
        scores = torch.full((H, max(T, 1)), -1.0, dtype=torch.float32, device="cuda")
        energy = torch.full((len(cu) - 1, 4), -1.0, dtype=torch.float64, device="cuda")
        need = fc.fc_score_workspace_bytes(h, kd, vd, cu)
        assert need > 0
        ws = torch.empty(need, dtype=torch.uint8, device="cuda")
        fc.fc_score_layer(h, kd, vd, cu, gamma, scores, energy, ws)
        assert fc.fc_last_device_status(h) == 0
        return scores.cpu().numpy().astype(np.float64)[:, :T], energy.cpu().numpy()
    finally:
        fc.fc_destroy(h)


def _score_errors(g, o, k, v, cu):
    """max over heads/tokens of |g-o| / max(o, 1e-6*e_bar)."""
    kk = k.double().numpy()
    vv = v.double().numpy()
    worst = 0.0
    for b in range(len(cu) - 1):
        s, e = cu[b], cu[b + 1]
        if e == s:
            continue
        for h in range(g.shape[0]):
            ebar = ((kk[s:e, h] ** 2).sum(1) + (vv[s:e, h] ** 2).sum(1)).mean() / kk.shape[2]
            den = np.maximum(o[h, s:e], 1e-6 * ebar)
            worst = max(worst, float((np.abs(g[h, s:e] - o[h, s:e]) / den).max()))
    return worst


def _check_layer(fc, k, v, cu, gamma, **kw):
    g, en = _gpu_scores(fc, k, v, cu, gamma, **kw)
    o, eo = O.score_layer(k.double().numpy(), v.double().numpy(), cu, gamma, "fft")
    err = _score_errors(g, o, k, v, cu)
    assert err <= TOL[k.dtype], "score error %.3e" % err
    assert np.all(g >= 0.0)
    for b in range(len(cu) - 1):
        if cu[b + 1] == cu[b]:
            assert not en[b].any()
            continue
        tol = 1e-4 if k.dtype == torch.float32 else 2e-2
        np.testing.assert_allclose(en[b, [1, 3]], eo[b, [1, 3]], rtol=1e-5)
        scale = eo[b, [1, 3]] * 1e-6
        assert np.all(np.abs(en[b, [0, 2]] - eo[b, [0, 2]]) <= tol * np.maximum(eo[b, [0, 2]], scale))
    return g, en


# ---------------------------------------------------------------- scores
@pytest.mark.parametrize("N", [16, 32, 64, 256, 1024, 4096])
@pytest.mark.parametrize("gamma", [0.2, 1.0])
def test_scores_power_of_two_fp32(fc, N, gamma):
    k, v = _rand_kv(N, 2, 128, torch.float32, N)
    _check_layer(fc, k, v, [0, N], gamma)


@pytest.mark.parametrize("N", [1, 2, 3, 5, 8, 17, 100, 257, 1000, 1500, 4099])
def test_scores_arbitrary_length_fp32(fc, N):
    k, v = _rand_kv(N, 2, 64, torch.float32, 100 + N)
    _check_layer(fc, k, v, [0, N], 0.2)


@pytest.mark.parametrize("gamma", [0.0, 0.0003, 0.1, 0.5, 0.77, 1.0])
def test_scores_cutoff_sweep(fc, gamma):
    k, v = _rand_kv(512, 1, 128, torch.float32, 7)
    _check_layer(fc, k, v, [0, 512], gamma)
    k, v = _rand_kv(300, 1, 128, torch.float32, 8)
    _check_layer(fc, k, v, [0, 300], gamma)


@pytest.mark.parametrize("dtype", [torch.float16, torch.bfloat16])
@pytest.mark.parametrize("N", [2048, 777])
def test_scores_16bit_inputs(fc, dtype, N):
    k, v = _rand_kv(N, 3, 128, dtype, 11)
    _check_layer(fc, k, v, [0, N], 0.2)


def test_scores_ragged_batch_with_empty_sequence(fc):
    lens = [64, 0, 300, 1024, 17, 2048]
    cu = [0] + list(np.cumsum(lens))
    cu = [int(x) for x in cu]
    k, v = _rand_kv(cu[-1], 2, 128, torch.bfloat16, 5)
    _check_layer(fc, k, v, cu, 0.2, max_seqlen=4096)


def test_scores_strided_view_and_small_groups(fc):
    # K and V live inside a wider buffer (extra heads, padded channels); tiny transform groups
    N, H, d = 1024, 4, 128
    big_k, big_v = _rand_kv(N, H + 2, d + 64, torch.float16, 3)
    k, v = big_k[:, 1:1 + H, :d], big_v[:, 1:1 + H, :d]
    kd, vd = big_k.cuda()[:, 1:1 + H, :d], big_v.cuda()[:, 1:1 + H, :d]
    assert not kd.is_contiguous()
    g1, e1 = _gpu_scores(fc, kd, vd, [0, N], 0.2)
    g2, e2 = _gpu_scores(fc, k.contiguous(), v.contiguous(), [0, N], 0.2, group_bytes=1 << 20)
    assert np.array_equal(g1, g2) and np.array_equal(e1, e2)
    o, _ = O.score_layer(k.double().numpy(), v.double().numpy(), [0, N], 0.2, "fft")
    assert _score_errors(g1, o, k, v, [0, N]) <= 2e-2


def test_scores_are_deterministic(fc):
    k, v = _rand_kv(4096, 2, 128, torch.bfloat16, 9)
    a = _gpu_scores(fc, k, v, [0, 4096], 0.2)
    b = _gpu_scores(fc, k, v, [0, 4096], 0.2)
    assert np.array_equal(a[0], b[0]) and np.array_equal(a[1], b[1])
    k, v = _rand_kv(1234, 2, 128, torch.bfloat16, 9)
    a = _gpu_scores(fc, k, v, [0, 1234], 0.2)
    b = _gpu_scores(fc, k, v, [0, 1234], 0.2)
    assert np.array_equal(a[0], b[0]) and np.array_equal(a[1], b[1])


@pytest.mark.parametrize("N", [8192, 32768, 65536, 131072])
def test_scores_long_sequences_sampled_head(fc, N):
    k, v = _rand_kv(N, 1, 128, torch.bfloat16, N)
    _check_layer(fc, k, v, [0, N], 0.2)


@pytest.mark.parametrize("N", [8192, 32768, 65536])
def test_scores_long_power_of_two_fp32_inputs(fc, N):
    # fp32 rows at the 1e-3 bar on the lengths whose twiddles are products of table values (up to three factors)
    k, v = _rand_kv(N, 1, 64, torch.float32, 7 + N)
    _check_layer(fc, k, v, [0, N], 0.2)


def test_scores_long_arbitrary_length(fc):
    N = 40961
    k, v = _rand_kv(N, 1, 64, torch.bfloat16, N)
    _check_layer(fc, k, v, [0, N], 0.2)


def test_scores_mixed_paths_in_one_call(fc):
    # power-of-two and other lengths alternate in one batch: the direct and the padded form of the three passes (two
    # internal streams, up to 81920 points) and a tiny sequence on the caller's stream; results match the oracle and do
    # not change from run to run
    lens = [5000, 4096, 3000, 8192, 33000, 7, 2048]
    cu = [0] + [int(x) for x in np.cumsum(lens)]
    k, v = _rand_kv(cu[-1], 4, 128, torch.bfloat16, 12)
    g1, e1 = _check_layer(fc, k, v, cu, 0.2, max_seqlen=65536)
    g2, e2 = _gpu_scores(fc, k, v, cu, 0.2, max_seqlen=65536)
    assert np.array_equal(g1, g2) and np.array_equal(e1, e2)


@pytest.mark.parametrize("dtype", [torch.float32, torch.float16])
def test_scores_131072_point_chirp_transform(fc, dtype):
    # 2N - 1 = 66001, just past a power of two (131072 points where only powers of two are padded to, 81920 here)
    N = 33001
    k, v = _rand_kv(N, 2, 128, dtype, 13)
    _check_layer(fc, k, v, [0, N], 0.2, band=False)


@pytest.mark.parametrize("N,gamma,d,group_bytes", [
    (2500, 0.2, 128, None),      # N + 2*omega + 1 = 3501 -> 4096 points instead of 8192
    (2500, 0.0, 64, None),       # band of one bin (the mean)
    (5000, 0.3, 128, None),      # 8001 -> 8192 instead of 16384
    (5000, 0.1, 192, 1),         # heads in column groups
    (1367, 0.25, 64, None),      # 2051 -> 4096: band form does not apply (same length), full form runs
    (33001, 0.2, 128, None),     # 46202 -> 65536 instead of 131072
    (46800, 0.2, 64, None),      # 65521 -> 65536: the longest sequence the band form shortens at this cutoff
])
def test_scores_chirp_band_form(fc, N, gamma, d, group_bytes):
    # The lengths at which a chirp transform of the band -omega .. omega would be shorter than one of all bins.  Every one
    # of them is scored by one padded convolution, whatever fc_set_chirp_band says: both settings match the oracle and
    # give the same values.  (The chirp form itself, which the entry point without allocation runs, is compared with this
    # one in test_zz_no_alloc.py.)
    k, v = _rand_kv(N, 2, d, torch.float32, 500 + N)
    g1, e1 = _check_layer(fc, k, v, [0, N], gamma, band=True, group_bytes=group_bytes)
    g2, e2 = _check_layer(fc, k, v, [0, N], gamma, band=False, group_bytes=group_bytes)
    np.testing.assert_allclose(g1, g2, rtol=2e-3, atol=1e-6 * float(g2.max()))
    np.testing.assert_allclose(e1, e2, rtol=1e-4)


@pytest.mark.parametrize("M", [5120, 6144, 7168, 10240, 12288, 14336, 20480, 24576, 28672, 40960, 49152, 57344,
                               81920, 98304, 114688])
def test_scores_chirp_lengths_with_an_odd_factor(fc, M):
    # N = M/2 - 1: 2N - 1 = M - 3 pads to M = 2^k * {5, 3, 7}, every shape the specialised kernels have for such lengths
    # (first-stage radix 10, 12, 14; rows of 32..512 points), against the oracle; fc_set_chirp_band changes nothing
    N = M // 2 - 1
    k, v = _rand_kv(N, 1, 64, torch.float32, 900 + M % 1000)
    g1, e1 = _check_layer(fc, k, v, [0, N], 0.2, band=False)
    g2, e2 = _check_layer(fc, k, v, [0, N], 0.2, band=True)
    np.testing.assert_allclose(g1, g2, rtol=2e-3, atol=1e-6 * float(g2.max()))


@pytest.mark.parametrize("N", [5118, 20478, 29255, 35107, 40958, 58513])
def test_scores_chirp_band_form_on_lengths_with_an_odd_factor(fc, N):
    # lengths whose band would fill a chirp transform with an odd factor; padded to 10240 ... 131072 points
    k, v = _rand_kv(N, 2, 128, torch.bfloat16, 30 + N % 100)
    _check_layer(fc, k, v, [0, N], 0.2)


def test_describe_plan_reports_the_convolution_length_in_use(fc):
    # powers of two: the transform in use; other lengths: the chirp lengths (form and size) it documents
    h = fc.fc_create(0, 65536)
    try:
        p = fc.fc_describe_plan(h, 32768, 0.2)
        assert (p["bluestein"], p["nfft"], p["n1"] * p["n2"]) == (False, 32768, 32768)
        p = fc.fc_describe_plan(h, 2500, 0.2)                    # 2500 + 1000 + 1 -> 4096
        assert (p["band_form"], p["nfft"], p["n1"] * p["n2"]) == (True, 4096, 4096)
        p = fc.fc_describe_plan(h, 35107, 0.2)                   # 35107 + 14042 + 1 = 49150 -> 49152 = 192 x 256
        assert (p["band_form"], p["nfft"], p["n1"], p["n2"]) == (True, 49152, 192, 256)
        p = fc.fc_describe_plan(h, 33001, 0.6)                   # band wider than the spectrum: 2N - 1 -> 81920
        assert (p["bluestein"], p["band_form"], p["nfft"], p["n1"], p["n2"]) == (True, False, 81920, 160, 512)
        fc.fc_set_chirp_band(h, False)
        p = fc.fc_describe_plan(h, 2500, 0.2)                    # 4999 -> 5120 = 160 x 32
        assert (p["band_form"], p["nfft"], p["n1"], p["n2"]) == (False, 5120, 160, 32)
        p = fc.fc_describe_plan(h, 300, 0.2)                     # short: a power of two
        assert (p["bluestein"], p["nfft"]) == (True, 1024)
    finally:
        fc.fc_destroy(h)


def test_scores_chirp_band_form_16bit_ragged(fc):
    lens = [2500, 1024, 5000, 40961, 300]
    cu = [0] + [int(x) for x in np.cumsum(lens)]
    k, v = _rand_kv(cu[-1], 4, 128, torch.bfloat16, 77)
    g1, e1 = _check_layer(fc, k, v, cu, 0.2, max_seqlen=65536)
    g2, e2 = _gpu_scores(fc, k, v, cu, 0.2, max_seqlen=65536)
    assert np.array_equal(g1, g2) and np.array_equal(e1, e2)


@pytest.mark.parametrize("d,group_bytes", [(128, 1), (128, 1 << 20), (192, 1), (64, 1), (256, 1)])
def test_scores_arbitrary_length_in_column_groups(fc, d, group_bytes):
    # a small cache budget makes a head of 128 or 256 channels go in two or four groups of 64 columns, whose contributions
    # are added to the score one after the other (64 channels, and 192, which does not halve to whole groups, go whole)
    N = 3000
    k, v = _rand_kv(N, 2, d, torch.float32, 40 + d)
    g1, _ = _check_layer(fc, k, v, [0, N], 0.2, group_bytes=group_bytes)
    g2, _ = _check_layer(fc, k, v, [0, N], 0.2)
    np.testing.assert_allclose(g1, g2, rtol=2e-3, atol=1e-6 * float(g2.max()))


# ---------------------------------------------------------------- power spectrum (Eq. 11)
@pytest.mark.parametrize("lens,H,d,dtype", [([16], 1, 64, torch.float32), ([1024], 2, 128, torch.float32),
                                            ([1, 2, 3, 8, 300, 0, 1000], 2, 64, torch.float32),
                                            ([4096, 777, 2048], 3, 128, torch.bfloat16),
                                            ([32768], 1, 128, torch.float16), ([5000], 2, 192, torch.float32)])
def test_power_spectrum_matches_oracle(fc, lens, H, d, dtype):
    cu = [0] + [int(x) for x in np.cumsum(lens)]
    T = cu[-1]
    k, v = _rand_kv(T, H, d, dtype, 77 + T)
    h = fc.fc_create(0, max(lens))
    try:
        kd, vd = k.cuda(), v.cuda()
        spec = torch.full((T, 2), -1.0, dtype=torch.float64, device="cuda")
        ws = torch.empty(fc.fc_power_spectrum_workspace_bytes(h, kd, vd, cu), dtype=torch.uint8, device="cuda")
        fc.fc_power_spectrum(h, kd, vd, cu, spec, ws)
        assert fc.fc_last_device_status(h) == 0
        got = spec.cpu().numpy()
        # the band sums are what fc_score_layer reports as energies
        scores = torch.empty((H, T), dtype=torch.float32, device="cuda")
        energy = torch.empty((len(lens), 4), dtype=torch.float64, device="cuda")
        ws2 = torch.empty(fc.fc_score_workspace_bytes(h, kd, vd, cu), dtype=torch.uint8, device="cuda")
        fc.fc_score_layer(h, kd, vd, cu, 0.2, scores, energy, ws2)
        assert fc.fc_last_device_status(h) == 0
        en = energy.cpu().numpy()
    finally:
        fc.fc_destroy(h)
    want = O.power_spectrum(k.double().numpy(), v.double().numpy(), cu, "fft")
    for b, n in enumerate(lens):
        if n == 0:
            continue
        s, e = cu[b], cu[b + 1]
        for j in range(2):
            # fp32 transforms: every bin carries an error proportional to the largest bins of the sequence
            floor = 1e-6 * want[s:e, j].max()
            err = np.abs(got[s:e, j] - want[s:e, j]) / np.maximum(want[s:e, j], floor)
            assert err.max() <= 2e-3, "sequence %d matrix %d: %.3e" % (b, j, err.max())
            np.testing.assert_allclose(got[s:e, j].sum(), want[s:e, j].sum(), rtol=1e-5)          # Parseval
        om = O.cutoff_index(n, 0.2)
        np.testing.assert_allclose(got[s + om + 1:e, 0].sum(), en[b, 0], rtol=2e-3, atol=1e-6 * en[b, 1])
        np.testing.assert_allclose(got[s + om + 1:e, 1].sum(), en[b, 2], rtol=2e-3, atol=1e-6 * en[b, 3])


@pytest.mark.parametrize("share", [0.0, 0.5, 0.9, 0.999, 1.0])
def test_cutoff_from_spectrum_matches_oracle(fc, share):
    # (a) on spectra given to both sides (exact integer agreement, sequences of every size incl. empty, zero energy,
    # longer than one bin per thread), (b) end to end: spectrum and cutoff on the device, then scoring at the
    # returned gamma uses exactly that omega
    rng = np.random.default_rng(int(share * 1000) + 3)
    lens = [1, 0, 7, 1000, 5000, 64, 131072]
    cu = [0] + [int(x) for x in np.cumsum(lens)]
    P = rng.random((cu[-1], 2)) * np.exp(-rng.random((cu[-1], 1)) * 8.0)
    P[cu[5]:cu[6]] = 0.0                                         # a sequence without energy
    P[cu[3]:cu[3] + 40] *= 1e4                                   # one with a dominant low band
    h = fc.fc_create(0, 131072)
    try:
        om = torch.full((len(lens),), -7, dtype=torch.int32, device="cuda")
        ga = torch.full((len(lens),), -7.0, dtype=torch.float64, device="cuda")
        fc.fc_cutoff_from_spectrum(h, torch.from_numpy(P).cuda(), cu, share, om, ga)
        assert fc.fc_last_device_status(h) == 0
        om, ga = om.cpu().numpy(), ga.cpu().numpy()
        for b, n in enumerate(lens):
            if n == 0:
                assert om[b] == 0 and ga[b] == 0.0
                continue
            wo, wg = O.cutoff_for_energy_share(P[cu[b]:cu[b + 1]], share)
            if om[b] != wo:                                      # only where rounding of the running sum decides
                tot = P[cu[b]:cu[b + 1]].sum()
                c = np.cumsum(P[cu[b]:cu[b + 1]].sum(1))
                assert abs(c[min(om[b], wo)] - share * tot) <= 1e-12 * tot
            else:
                assert ga[b] == wg
            assert O.cutoff_index(n, float(ga[b])) == om[b]
        # end to end on one layer
        k, v = _rand_kv(3000, 2, 128, torch.float32, 5)
        cu2 = [0, 1000, 3000]
        kd, vd = k.cuda(), v.cuda()
        spec = torch.empty((3000, 2), dtype=torch.float64, device="cuda")
        ws = torch.empty(fc.fc_power_spectrum_workspace_bytes(h, kd, vd, cu2), dtype=torch.uint8, device="cuda")
        fc.fc_power_spectrum(h, kd, vd, cu2, spec, ws)
        om2 = torch.empty(2, dtype=torch.int32, device="cuda")
        ga2 = torch.empty(2, dtype=torch.float64, device="cuda")
        fc.fc_cutoff_from_spectrum(h, spec, cu2, share, om2, ga2)
        assert fc.fc_last_device_status(h) == 0
        want = O.power_spectrum(k.double().numpy(), v.double().numpy(), cu2, "fft")
        for b in range(2):
            wo, _ = O.cutoff_for_energy_share(want[cu2[b]:cu2[b + 1]], share)
            seg = want[cu2[b]:cu2[b + 1]].sum(1)
            got = int(om2[b])
            if got != wo:                                        # fp32 spectrum against fp64: the kept share must still fit
                assert abs(np.cumsum(seg)[min(got, wo)] / seg.sum() - share) <= 2e-3
    finally:
        fc.fc_destroy(h)


# ---------------------------------------------------------------- budgets
def _gpu_budgets(fc, energy, cu, rho, min_keep):
    L, B = energy.shape[:2]
    h = fc.fc_create(0, 1024)
    try:
        e = torch.from_numpy(np.ascontiguousarray(energy)).cuda()
        budgets = torch.full((L, B), -7, dtype=torch.int32, device="cuda")
        offsets = torch.full((L, B + 1), -7, dtype=torch.int64, device="cuda")
        fc.fc_allocate_budgets(h, e, cu, rho, min_keep, budgets, offsets)
        assert fc.fc_last_device_status(h) == 0
        return budgets.cpu().numpy(), offsets.cpu().numpy()
    finally:
        fc.fc_destroy(h)


@pytest.mark.parametrize("seed", range(8))
def test_budgets_match_oracle(fc, seed):
    rng = np.random.default_rng(seed)
    L = int(rng.integers(1, 70))
    B = int(rng.integers(1, 6))
    lens = [int(x) for x in rng.integers(0, 5000, B)]
    cu = [0] + [int(x) for x in np.cumsum(lens)]
    energy = rng.random((L, B, 4))
    energy[..., 1] += energy[..., 0]
    energy[..., 3] += energy[..., 2]
    if seed % 3 == 0:
        energy[rng.integers(0, L), :, :] = 0.0
    rho = float(rng.choice([0.05, 0.1, 0.2, 0.6, 1.0]))
    min_keep = int(rng.choice([0, 1, 8]))
    gb, go = _gpu_budgets(fc, energy, cu, rho, min_keep)
    ob, oo = O.allocate_budgets(energy, lens, rho, min_keep)
    np.testing.assert_array_equal(gb, ob)
    np.testing.assert_array_equal(go, oo)


def test_budgets_special_cases(fc):
    e = np.zeros((4, 1, 4))
    gb, go = _gpu_budgets(fc, e, [0, 100], 0.5, 1)            # all-zero energy: uniform
    assert gb[:, 0].tolist() == [50, 50, 50, 50]
    e = np.ones((3, 1, 4))
    e[:, 0, 0] = [0.8, 0.1, 0.1]
    e[:, 0, 2] = 0.0
    gb, _ = _gpu_budgets(fc, e, [0, 100], 0.5, 1)             # upper cap binds, rest re-shared
    assert gb[:, 0].tolist() == [100, 25, 25]
    e = np.ones((1, 1, 4))
    gb, go = _gpu_budgets(fc, e, [0, 1024], 0.2, 1)           # one layer: floor(204.8+.5)
    assert gb.tolist() == [[205]] and go.tolist() == [[0, 205]]


# ---------------------------------------------------------------- selection + compaction
def _gpu_select(fc, k, v, cu, scores, budgets, offsets, capacity, per_layer=False, protect=None):
    T, H, d = k.shape
    h = fc.fc_create(0, 65536)
    try:
        kd, vd = k.cuda(), v.cuda()
        sc = torch.from_numpy(np.ascontiguousarray(scores, dtype=np.float32)).cuda()
        bd = torch.tensor(budgets, dtype=torch.int32, device="cuda")
        of = torch.tensor(offsets, dtype=torch.int64, device="cuda")
        out_k = torch.zeros((capacity, H, d), dtype=k.dtype, device="cuda")
        out_v = torch.zeros((capacity, H, d), dtype=k.dtype, device="cuda")
        out_idx = torch.full((H, capacity), -1, dtype=torch.int32, device="cuda")
        ws = torch.empty(fc.fc_select_workspace_bytes(h, kd, vd, cu), dtype=torch.uint8, device="cuda")
        if per_layer or protect is not None:
            pr = None if protect is None else torch.from_numpy(np.ascontiguousarray(protect, dtype=np.uint8)).cuda()
            fc.fc_select_compact_ex(h, kd, vd, cu, sc, bd, of, out_k, out_v, out_idx, ws, per_layer=per_layer,
                                    protect=pr)
        else:
            fc.fc_select_compact(h, kd, vd, cu, sc, bd, of, out_k, out_v, out_idx, ws)
        status = fc.fc_last_device_status(h)
        return out_k.cpu(), out_v.cpu(), out_idx.cpu().numpy(), status
    finally:
        fc.fc_destroy(h)


@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16])
def test_select_exact_on_given_scores(fc, dtype):
    rng = np.random.default_rng(0)
    lens = [1, 37, 0, 1024, 3000, 5]
    cu = [0] + [int(x) for x in np.cumsum(lens)]
    T, H, d = cu[-1], 3, 128
    k, v = _rand_kv(T, H, d, dtype, 1, smooth=False)
    scores = rng.integers(0, 50, (H, T)).astype(np.float32) / 7.0      # heavy ties
    scores[0, cu[3] + 5] = np.nan
    scores[1, cu[4]:cu[4] + 10] = np.inf
    scores[2, cu[4] + 100:cu[4] + 200] = 0.0
    budgets = [1, 11, 0, 205, 2999, 5]
    offsets = [0] + [int(x) for x in np.cumsum(budgets)]
    out_k, out_v, out_idx, status = _gpu_select(fc, k, v, cu, scores, budgets, offsets, offsets[-1] + 3)
    assert status == 0
    for h in range(H):
        for b, n in enumerate(lens):
            want = O.select_topk(scores[h, cu[b]:cu[b + 1]], budgets[b])
            got = out_idx[h, offsets[b]:offsets[b + 1]]
            np.testing.assert_array_equal(got, want)
            rows = slice(offsets[b], offsets[b + 1])
            assert torch.equal(out_k[rows, h].view(torch.uint8), k[cu[b] + want, h].contiguous().view(torch.uint8))
            assert torch.equal(out_v[rows, h].view(torch.uint8), v[cu[b] + want, h].contiguous().view(torch.uint8))
    assert (out_idx[:, offsets[-1]:] == -1).all()                          # nothing past the last row


@pytest.mark.parametrize("per_layer", [False, True])
@pytest.mark.parametrize("with_mask", [False, True])
@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16])
def test_select_options_exact_on_given_scores(fc, dtype, with_mask, per_layer):
    # scores are multiples of 1/8, so their sums over heads are exact in fp32 and the order is the oracle's
    rng = np.random.default_rng(3)
    lens = [1, 37, 0, 1024, 3000, 5, 20000]
    cu = [0] + [int(x) for x in np.cumsum(lens)]
    T, H, d = cu[-1], 3, 128
    k, v = _rand_kv(T, H, d, dtype, 4, smooth=False)
    scores = rng.integers(0, 50, (H, T)).astype(np.float32) / 8.0
    scores[0, cu[3] + 5] = np.nan
    scores[1, cu[4]:cu[4] + 10] = np.inf
    protect = None
    if with_mask:
        protect = (rng.random(T) < 0.02).astype(np.uint8)
        protect[cu[3]:cu[3] + 4] = 1                     # sinks
        protect[cu[4] - 16:cu[4]] = 1                    # a recent window
        protect[cu[1]:cu[2]] = 1                         # a whole sequence marked: more marked tokens than budget
    budgets = [1, 11, 0, 205, 2999, 5, 1234]
    offsets = [0] + [int(x) for x in np.cumsum(budgets)]
    out_k, out_v, out_idx, status = _gpu_select(fc, k, v, cu, scores, budgets, offsets, offsets[-1] + 3,
                                                per_layer=per_layer, protect=protect)
    assert status == 0
    for h in range(H):
        for b, n in enumerate(lens):
            dev = scores[:, cu[b]:cu[b + 1]].astype(np.float64)
            dev = O.layer_score(dev) if per_layer else dev[h]
            pr = None if protect is None else protect[cu[b]:cu[b + 1]]
            want = O.select_topk_protected(dev, budgets[b], pr)
            got = out_idx[h, offsets[b]:offsets[b + 1]]
            np.testing.assert_array_equal(got, want)
            rows = slice(offsets[b], offsets[b + 1])
            assert torch.equal(out_k[rows, h].view(torch.uint8), k[cu[b] + want, h].contiguous().view(torch.uint8))
            assert torch.equal(out_v[rows, h].view(torch.uint8), v[cu[b] + want, h].contiguous().view(torch.uint8))
    assert (out_idx[:, offsets[-1]:] == -1).all()


def test_compress_per_layer_with_protected_tokens_matches_oracle(fc):
    from paper_2511_16786_b200.binding import Compressor
    base = S.paper_configs()["cfg2"]
    cfg = S.scaled(base, "per_layer_small", num_layers=4, seqlens=(2048, 700), min_keep=24)
    L, cu = cfg.num_layers, cfg.cu_seqlens
    Ks, Vs = zip(*[S.make_layer(cfg, l, "cpu") for l in range(L)])
    protect = np.zeros(cu[-1], dtype=np.uint8)
    for b in range(2):
        protect[cu[b]:cu[b] + 4] = 1                     # sinks
        protect[cu[b + 1] - 16:cu[b + 1]] = 1            # recent window
    comp = Compressor(L, cfg.num_heads, cfg.head_dim, cu, cfg.torch_dtype, cfg.rho, cfg.gamma, cfg.min_keep,
                      per_layer=True, protect=torch.from_numpy(protect).cuda())
    comp.compress([k.cuda() for k in Ks], [v.cuda() for v in Vs])
    comp.check_device_status()
    budgets, offsets = comp.budgets.cpu().numpy(), comp.offsets.cpu().numpy()
    idx = comp.out_idx.cpu().numpy()
    tol = TOL[cfg.torch_dtype]
    for l in range(L):
        o, _ = O.score_layer(Ks[l].double().numpy(), Vs[l].double().numpy(), cu, cfg.gamma, "fft")
        for b, n in enumerate(cfg.seqlens):
            kb, off = int(budgets[l, b]), int(offsets[l, b])
            got = idx[l, 0, off:off + kb]
            for h in range(1, cfg.num_heads):
                np.testing.assert_array_equal(idx[l, h, off:off + kb], got)       # one index set per layer
            pr = protect[cu[b]:cu[b + 1]]
            assert set(np.flatnonzero(pr)) <= set(got.tolist())                    # 20 marked tokens, min_keep 24
            dev = O.layer_score(o[:, cu[b]:cu[b + 1]])
            want = O.select_topk_protected(dev, kb, pr)
            diff = np.setxor1d(got, want)
            if len(diff):
                tau = np.sort(dev[pr == 0])[::-1][kb - int(pr.sum()) - 1]
                assert np.all(np.abs(dev[diff] - tau) <= tol * tau)
            for h in range(cfg.num_heads):
                gk = comp.out_k[l][off:off + kb, h].cpu().view(torch.uint8)
                assert torch.equal(gk, Ks[l][cu[b] + got, h].contiguous().view(torch.uint8))
                gv = comp.out_v[l][off:off + kb, h].cpu().view(torch.uint8)
                assert torch.equal(gv, Vs[l][cu[b] + got, h].contiguous().view(torch.uint8))
    comp.close()


def test_select_capacity_overflow_is_reported_not_written(fc):
    k, v = _rand_kv(64, 1, 128, torch.float32, 2, smooth=False)
    scores = np.arange(64, dtype=np.float32)[None]
    _, _, out_idx, status = _gpu_select(fc, k, v, [0, 64], scores, [10], [0, 10], 4)
    assert status != 0
    assert (out_idx == -1).all()


# ---------------------------------------------------------------- whole pass
def _compare_compress(fc, cfg, layers=None, sample_heads=None, tier="fft"):
    from paper_2511_16786_b200.binding import Compressor
    L = cfg.num_layers
    Ks, Vs = [], []
    for l in range(L):
        k, v = S.make_layer(cfg, l, "cpu")
        Ks.append(k)
        Vs.append(v)
    comp = Compressor(L, cfg.num_heads, cfg.head_dim, cfg.cu_seqlens, cfg.torch_dtype, cfg.rho,
                      cfg.gamma, cfg.min_keep)
    Kd, Vd = [k.cuda() for k in Ks], [v.cuda() for v in Vs]
    comp.compress(Kd, Vd)
    comp.check_device_status()
    tol = TOL[cfg.torch_dtype]
    cu = cfg.cu_seqlens
    g_scores = comp.scores.cpu().numpy().astype(np.float64)
    g_energy = comp.energy.cpu().numpy()
    g_budgets = comp.budgets.cpu().numpy()
    g_offsets = comp.offsets.cpu().numpy()
    g_idx = comp.out_idx.cpu().numpy()
    o_energy = np.zeros_like(g_energy)
    o_scores = []
    for l in range(L):
        o, e = O.score_layer(Ks[l].double().numpy(), Vs[l].double().numpy(), cu, cfg.gamma, tier)
        o_scores.append(o)
        o_energy[l] = e
        assert _score_errors(g_scores[l], o, Ks[l], Vs[l], cu) <= tol
    ob, oo = O.allocate_budgets(o_energy, list(cfg.seqlens), cfg.rho, cfg.min_keep)
    # budgets: identical, or +-1 swaps where the largest-remainder fractions nearly tie
    assert g_budgets.sum(axis=0).tolist() == ob.sum(axis=0).tolist()
    assert np.abs(g_budgets - ob).max() <= 1
    # the device budgets are exactly what the oracle rule gives on the device's own energies
    ob2, oo2 = O.allocate_budgets(g_energy, list(cfg.seqlens), cfg.rho, cfg.min_keep)
    np.testing.assert_array_equal(g_budgets, ob2)
    np.testing.assert_array_equal(g_offsets, oo2)
    for l in range(L):
        for h in range(cfg.num_heads):
            for b, n in enumerate(cfg.seqlens):
                kb = int(g_budgets[l, b])
                got = g_idx[l, h, g_offsets[l, b]:g_offsets[l, b] + kb]
                assert np.all(np.diff(got) > 0) and (kb == 0 or (got[0] >= 0 and got[-1] < n))
                osc = o_scores[l][h, cu[b]:cu[b + 1]]
                want = O.select_topk(osc, kb)
                diff = np.setxor1d(got, want)
                if len(diff) and kb > 0:
                    tau = np.sort(osc)[::-1][kb - 1]
                    assert np.all(np.abs(osc[diff] - tau) <= tol * tau), "index sets differ away from the threshold"
                rows = slice(int(g_offsets[l, b]), int(g_offsets[l, b]) + kb)
                gk = comp.out_k[l][rows, h].cpu().view(torch.uint8)
                gv = comp.out_v[l][rows, h].cpu().view(torch.uint8)
                assert torch.equal(gk, Ks[l][cu[b] + got, h].contiguous().view(torch.uint8))
                assert torch.equal(gv, Vs[l][cu[b] + got, h].contiguous().view(torch.uint8))
    comp.close()
    return g_budgets


def test_config1_full(fc):
    cfg = S.paper_configs()["cfg1"]
    b = _compare_compress(fc, cfg, tier="literal")
    assert b.tolist() == [[205]]


def test_config2_shape_reduced(fc):
    base = S.paper_configs()["cfg2"]
    cfg = S.scaled(base, "cfg2_small", num_layers=6, seqlens=(2048,))
    b = _compare_compress(fc, cfg)
    assert len(set(b[:, 0].tolist())) > 1        # per-layer outlier fractions give different budgets


def test_config4_shape_reduced(fc):
    base = S.paper_configs()["cfg4"]
    cfg = S.scaled(base, "cfg4_small", num_layers=3, num_heads=8, seqlens=(1024,))
    _compare_compress(fc, cfg)


def test_config5_shape_reduced_ragged(fc):
    base = S.paper_configs()["cfg5"]
    cfg = S.scaled(base, "cfg5_small", num_layers=4, seqlens=(517, 1024, 64, 1999, 333, 4096, 100, 2311))
    _compare_compress(fc, cfg)


def test_overlapping_launches_give_the_same_results(fc):
    from paper_2511_16786_b200.binding import Compressor
    cfg = S.scaled(S.paper_configs()["cfg2"], "cfg2_overlap", num_layers=12, seqlens=(4096, 1000))
    Kd, Vd = zip(*(S.make_layer(cfg, l, "cuda") for l in range(cfg.num_layers)))
    res = []
    for overlap in (False, True):
        comp = Compressor(cfg.num_layers, cfg.num_heads, cfg.head_dim, cfg.cu_seqlens, cfg.torch_dtype, cfg.rho,
                          cfg.gamma, cfg.min_keep, select_overlap=overlap, score_overlap=overlap)
        comp.out_k = comp.out_v = comp.out_idx = None
        for _ in range(3):                                    # repeated passes reuse the output buffers
            comp.compress(Kd, Vd)
        comp.check_device_status()
        off = comp.offsets.cpu()
        rows = [int(off[l, -1]) for l in range(cfg.num_layers)]
        res.append(([comp.scores.cpu().view(torch.int32)], [comp.energy.cpu().view(torch.int32)],
                    [comp.budgets.cpu()]))
        res[-1] = res[-1] + ([comp.out_k[l, :rows[l]].cpu() for l in range(cfg.num_layers)],
                    [comp.out_v[l, :rows[l]].cpu() for l in range(cfg.num_layers)],
                    [comp.out_idx[l, :, :rows[l]].cpu() for l in range(cfg.num_layers)])
        comp.close()
    for a, b in zip(res[0], res[1]):
        for x, y in zip(a, b):
            assert torch.equal(x.view(torch.uint8) if x.dtype != torch.int32 else x,
                               y.view(torch.uint8) if y.dtype != torch.int32 else y)


@pytest.mark.parametrize("per_layer", [False, True])
def test_one_selection_launch_for_all_layers_is_bit_identical(fc, per_layer):
    # fc_select_compact_layers against one fc_select_compact_ex call per layer: same indices, same rows; more layers
    # than one launch takes (32) so the chunking is exercised, ragged batch with an empty sequence
    from paper_2511_16786_b200.binding import Compressor
    cfg = S.scaled(S.paper_configs()["cfg2"], "cfg2_layers", num_layers=35, seqlens=(1000, 0, 2048, 517))
    Kd, Vd = zip(*(S.make_layer(cfg, l, "cuda") for l in range(cfg.num_layers)))
    comp = Compressor(cfg.num_layers, cfg.num_heads, cfg.head_dim, cfg.cu_seqlens, cfg.torch_dtype, cfg.rho,
                      cfg.gamma, cfg.min_keep, per_layer=per_layer)
    comp.score(Kd, Vd)
    comp.allocate()
    res = []
    for one_launch in (False, True):
        comp.out_k.fill_(0)
        comp.out_v.fill_(0)
        comp.out_idx.fill_(-1)
        comp.select_compact(Kd, Vd, one_launch=one_launch)
        comp.check_device_status()
        res.append((comp.out_k.cpu().view(torch.uint8).clone(), comp.out_v.cpu().view(torch.uint8).clone(),
                    comp.out_idx.cpu().clone()))
    assert int(comp.offsets[:, -1].sum()) > 0
    for a, b in zip(res[0], res[1]):
        assert torch.equal(a, b)
    comp.close()


# ---------------------------------------------------------------- full-size shapes, sampled
def test_head_sharded_pass_equals_the_whole_pass(fc):
    # two shards of the KV heads, run one after the other on this GPU, with the energy sums added by hand
    # where the ranks would all-reduce them: budgets, indices and rows equal those of the unsharded pass
    from paper_2511_16786_b200.binding import Compressor
    from paper_2511_16786_b200.head_shard import HeadShardedCompressor, shard_heads
    base = S.paper_configs()["cfg2"]
    cfg = S.scaled(base, "shard_small", num_layers=4, seqlens=(2048, 500))
    L, H = cfg.num_layers, cfg.num_heads
    Kd = [S.make_layer(cfg, l, "cuda")[0] for l in range(L)]
    Vd = [S.make_layer(cfg, l, "cuda")[1] for l in range(L)]
    whole = Compressor(L, H, cfg.head_dim, cfg.cu_seqlens, cfg.torch_dtype, cfg.rho, cfg.gamma, cfg.min_keep)
    whole.compress(Kd, Vd)
    whole.check_device_status()
    shards = []
    for rank in range(2):
        h0, h1 = shard_heads(H, 2, rank)
        sc = HeadShardedCompressor(None, rank, 2, L, H, cfg.head_dim, cfg.cu_seqlens, cfg.torch_dtype, cfg.rho,
                                   cfg.gamma, cfg.min_keep)
        Kl = [k[:, h0:h1] for k in Kd]
        Vl = [v[:, h0:h1] for v in Vd]
        sc.local.score(Kl, Vl)
        shards.append((sc, Kl, Vl, h0, h1))
    torch.cuda.synchronize()
    total = shards[0][0].local.energy + shards[1][0].local.energy
    np.testing.assert_allclose(total.cpu().numpy(), whole.energy.cpu().numpy(), rtol=1e-12)
    for sc, Kl, Vl, h0, h1 in shards:
        sc.local.energy.copy_(total)
        sc.local.allocate()
        sc.local.select_compact(Kl, Vl)
        sc.local.check_device_status()
        assert torch.equal(sc.local.budgets, whole.budgets)
        off = whole.offsets.cpu()
        for l in range(L):
            r = int(off[l, -1])
            assert torch.equal(sc.local.out_idx[l, :, :r], whole.out_idx[l, h0:h1, :r])
            assert torch.equal(sc.local.out_k[l, :r].view(torch.uint8), whole.out_k[l, :r, h0:h1].contiguous().view(torch.uint8))
        sc.close()
    # one rank, no group: the wrapper is the plain pass
    one = HeadShardedCompressor(None, 0, 1, L, H, cfg.head_dim, cfg.cu_seqlens, cfg.torch_dtype, cfg.rho, cfg.gamma,
                                cfg.min_keep)
    one.compress(Kd, Vd)
    one.local.check_device_status()
    assert torch.equal(one.local.budgets, whole.budgets) and torch.equal(one.local.offsets, whole.offsets)
    one.close()
    whole.close()


def test_graph_replay_gives_the_same_results(fc):
    # the whole call sequence captured once into a CUDA graph; replays on new contents of the same
    # tensors must equal an eager pass on those contents, and eager calls must still work afterwards
    from paper_2511_16786_b200.binding import Compressor
    base = S.paper_configs()["cfg3"]
    cfg = S.scaled(base, "graph_small", num_layers=5, seqlens=(2048, 300, 4096))
    cfg2 = S.scaled(base, "graph_small_b", num_layers=5, seqlens=(2048, 300, 4096), seed=base.seed + 3)
    L = cfg.num_layers
    Kd = [S.make_layer(cfg, l, "cuda")[0] for l in range(L)]
    Vd = [S.make_layer(cfg, l, "cuda")[1] for l in range(L)]
    comp = Compressor(L, cfg.num_heads, cfg.head_dim, cfg.cu_seqlens, cfg.torch_dtype, cfg.rho, cfg.gamma,
                      cfg.min_keep)
    graph = comp.capture(Kd, Vd)

    def snapshot():
        torch.cuda.synchronize()
        return [t.clone() for t in (comp.scores, comp.energy, comp.budgets, comp.offsets, comp.out_idx)]

    def kept_rows_equal(a_k, b_k, offsets):
        for l in range(L):
            r = int(offsets[l, -1])
            if not torch.equal(a_k[l, :r].view(torch.uint8), b_k[l, :r].view(torch.uint8)):
                return False
        return True

    for contents in (cfg2, cfg):
        for l in range(L):
            k, v = S.make_layer(contents, l, "cuda")
            Kd[l].copy_(k)
            Vd[l].copy_(v)
        comp.compress(Kd, Vd)
        want = snapshot()
        want_k, want_v = comp.out_k.clone(), comp.out_v.clone()
        for t in (comp.scores, comp.out_idx, comp.out_k, comp.out_v):
            t.zero_()
        graph.replay()
        got = snapshot()
        for a, b in zip(got[:4], want[:4]):
            assert torch.equal(a, b)
        off = want[3].cpu()
        for l in range(L):
            r = int(off[l, -1])
            assert torch.equal(got[4][l, :, :r], want[4][l, :, :r])
        assert kept_rows_equal(comp.out_k, want_k, off) and kept_rows_equal(comp.out_v, want_v, off)
    comp.check_device_status()
    comp.close()


def _compare_sampled(fc, cfg, samples):
    """Whole pass at a benchmark configuration's own sizes (same Compressor, same launch
    configuration as bench.py); the oracle checks the sampled (layer, sequence, head) triples one by
    one, properties that hold at any size cover the rest."""
    from paper_2511_16786_b200.binding import Compressor
    L, H, d = cfg.num_layers, cfg.num_heads, cfg.head_dim
    Kd, Vd = zip(*(S.make_layer(cfg, l, "cuda") for l in range(L)))
    comp = Compressor(L, H, d, cfg.cu_seqlens, cfg.torch_dtype, cfg.rho, cfg.gamma, cfg.min_keep)
    comp.compress(Kd, Vd)
    comp.check_device_status()
    tol = TOL[cfg.torch_dtype]
    cu = cfg.cu_seqlens
    g_energy = comp.energy.cpu().numpy()
    g_budgets = comp.budgets.cpu().numpy()
    g_offsets = comp.offsets.cpu().numpy()
    # any size: Parseval totals, score/energy identity, the budget rule on the device's own energies
    for l in range(L):
        for b, n in enumerate(cfg.seqlens):
            ks, vs = Kd[l][cu[b]:cu[b + 1]].double(), Vd[l][cu[b]:cu[b + 1]].double()
            np.testing.assert_allclose(g_energy[l, b, 1], float((ks * ks).sum()), rtol=1e-5)
            np.testing.assert_allclose(g_energy[l, b, 3], float((vs * vs).sum()), rtol=1e-5)
            dev_sum = float(comp.scores[l][:, cu[b]:cu[b + 1]].double().sum()) * d
            np.testing.assert_allclose(g_energy[l, b, 0] + g_energy[l, b, 2], dev_sum, rtol=1e-4)
    ob, oo = O.allocate_budgets(g_energy, list(cfg.seqlens), cfg.rho, cfg.min_keep)
    np.testing.assert_array_equal(g_budgets, ob)
    np.testing.assert_array_equal(g_offsets, oo)
    for b, n in enumerate(cfg.seqlens):
        assert int(g_budgets[:, b].sum()) == O.total_budget(n, L, cfg.rho, cfg.min_keep)
    # sampled triples against the oracle
    for (l, b, h) in samples:
        n = cfg.seqlens[b]
        kh = Kd[l][cu[b]:cu[b + 1], h].cpu()
        vh = Vd[l][cu[b]:cu[b + 1], h].cpu()
        o, _ = O.score_head(kh.double().numpy(), vh.double().numpy(), cfg.gamma, "fft")
        g32 = comp.scores[l][h, cu[b]:cu[b + 1]].cpu().numpy()
        g = g32.astype(np.float64)
        ebar = ((kh.double().numpy() ** 2).sum(1) + (vh.double().numpy() ** 2).sum(1)).mean() / d
        err = float((np.abs(g - o) / np.maximum(o, 1e-6 * ebar)).max())
        assert err <= tol, "layer %d seq %d head %d: score error %.3e" % (l, b, h, err)
        kb = int(g_budgets[l, b])
        off = int(g_offsets[l, b])
        got = comp.out_idx[l, h, off:off + kb].cpu().numpy()
        # index work is exact on the fp32 scores both sides see ...
        np.testing.assert_array_equal(got, O.select_topk(g32, kb))
        # ... and agrees with the fp64 scores except within the tolerance of the threshold
        want = O.select_topk(o, kb)
        diff = np.setxor1d(got, want)
        if len(diff) and kb > 0:
            tau = np.sort(o)[::-1][kb - 1]
            assert np.all(np.abs(o[diff] - tau) <= tol * tau)
        rows = slice(off, off + kb)
        assert torch.equal(comp.out_k[l][rows, h].cpu().view(torch.uint8), kh[got].contiguous().view(torch.uint8))
        assert torch.equal(comp.out_v[l][rows, h].cpu().view(torch.uint8), vh[got].contiguous().view(torch.uint8))
    comp.close()


def test_config2_full_size_sampled(fc):
    cfg = S.paper_configs()["cfg2"]
    _compare_sampled(fc, cfg, [(0, 0, 0), (13, 0, 2), (27, 0, 3)])


def test_config3_full_size_sampled(fc):
    # every head of four layers against the oracle, the any-size properties on all 28
    cfg = S.paper_configs()["cfg3"]
    _compare_sampled(fc, cfg, [(l, 0, h) for l in (0, 9, 18, 27) for h in range(4)])


def test_config4_full_size_sampled(fc):
    # all 32 layers x 32 heads x 16384 tokens on the device; eight (layer, head) pairs against the oracle
    cfg = S.paper_configs()["cfg4"]
    _compare_sampled(fc, cfg, [(0, 0, 0), (3, 0, 17), (8, 0, 31), (13, 0, 5), (19, 0, 22), (24, 0, 9), (28, 0, 30),
                               (31, 0, 12)])


def test_config5_full_size_sampled(fc):
    # all 28 layers of the eight ragged sequences; the longest and the shortest sequence are among the samples
    cfg = S.paper_configs()["cfg5"]
    lens = list(cfg.seqlens)
    longest, shortest = lens.index(max(lens)), lens.index(min(lens))
    _compare_sampled(fc, cfg, [(0, longest, 0), (27, shortest, 3), (5, 0, 1), (11, 1, 2), (14, 2, 0), (17, 3, 3),
                               (21, 4, 1), (25, 5, 2), (9, 6, 0), (2, 7, 3)])


# ---------------------------------------------------------------- tensor-pipe stage (measurement aid)
def test_dft16_stage_on_both_pipes_matches_fp64(fc):
    # both variants against the 16-point DFT in fp64; the tensor form keeps about 21 bits per operand, which
    # carries through a whole transform at the 1e-3 score tolerance of fp32 inputs (here: 1e-5 of the column's norm)
    g = torch.Generator().manual_seed(4)
    ncols = 4096 + 8
    x = torch.randn((16, ncols, 2), generator=g) * torch.rand((1, ncols, 1), generator=g) * 10.0
    xc = x[..., 0].double().numpy() + 1j * x[..., 1].double().numpy()
    want = np.fft.fft(xc, axis=0)
    h = fc.fc_create(0, 1024)
    try:
        xd = x.cuda()
        for variant, tol in ((0, 2e-6), (1, 1e-5)):
            yd = torch.zeros_like(xd)
            fc.fc_proto_dft16_stage(h, xd, yd, variant)
            assert fc.fc_last_device_status(h) == 0
            y = yd.cpu().double().numpy()
            got = y[..., 0] + 1j * y[..., 1]
            err = np.abs(got - want).max(axis=0) / np.linalg.norm(xc, axis=0)
            assert err.max() <= tol, "variant %d: %.3e" % (variant, err.max())
        yd = torch.zeros_like(xd)
        fc.fc_proto_dft16_stage(h, xd, yd, 2)
        assert torch.equal(yd, xd)
    finally:
        fc.fc_destroy(h)


# ---------------------------------------------------------------- inputs
def test_generator_gives_the_same_bytes_on_cpu_and_gpu(fc):
    # "seed 0" names one tensor: the oracle side (CPU) and the bench side (GPU) see identical inputs
    for name, changes in (("cfg1", {}), ("cfg2", dict(num_layers=2, seqlens=(1000, 0, 333))),
                          ("cfg4", dict(num_layers=1, num_heads=3, seqlens=(2048,))),
                          ("cfg5", dict(num_layers=1, seqlens=(517, 4099)))):
        cfg = S.scaled(S.paper_configs()[name], name + "_bytes", **changes)
        for l in range(cfg.num_layers):
            kc, vc = S.make_layer(cfg, l, "cpu")
            kg, vg = S.make_layer(cfg, l, "cuda")
            assert torch.equal(kc.view(torch.uint8), kg.cpu().view(torch.uint8))
            assert torch.equal(vc.view(torch.uint8), vg.cpu().view(torch.uint8))


# ---------------------------------------------------------------- failure reporting
def test_bounded_wait_that_runs_out_is_reported(fc):
    # a wait nothing will ever satisfy gives up after its limit, the status word says so, and the handle and the
    # context go on working (no trap, no hang)
    h = fc.fc_create(0, 1024)
    try:
        assert fc.fc_last_device_status(h) == 0
        fc.fc_selftest_bounded_wait(h)
        assert fc.fc_last_device_status(h) == 5                     # FC_ERR_TIMEOUT
        assert fc.fc_last_device_status(h) == 0                     # reading clears it
    finally:
        fc.fc_destroy(h)
    k, v = _rand_kv(1024, 1, 128, torch.float32, 3)
    _check_layer(fc, k, v, [0, 1024], 0.2)


@pytest.mark.parametrize("N", [1024, 300])
def test_nonfinite_input_poisons_its_own_sequence_and_head_only(fc, N):
    # a NaN or Inf element makes every score of its (sequence, head) NaN, as in the fp64 definition (the transform
    # mixes all tokens of a column); other heads and other sequences are untouched; the selection then keeps the
    # first tokens by index for that head (NaN ranks as +inf, ties by index)
    k, v = _rand_kv(2 * N, 3, 128, torch.float32, 91)
    cu = [0, N, 2 * N]
    kc, vc = k.clone(), v.clone()
    k[N // 3, 1, 7] = float("nan")              # sequence 0, head 1
    v[N + 5, 2, 100] = float("inf")             # sequence 1, head 2
    g, en = _gpu_scores(fc, k, v, cu, 0.2)
    o, _ = O.score_layer(kc.double().numpy(), vc.double().numpy(), cu, 0.2, "fft")
    assert np.isnan(g[1, :N]).all() and np.isnan(g[2, N:]).all()
    ok = np.ones_like(g, dtype=bool)
    ok[1, :N] = False
    ok[2, N:] = False
    assert np.isfinite(g[ok]).all()
    np.testing.assert_allclose(g[ok], o[ok], rtol=2e-3, atol=1e-6 * o.mean())
    # the oracle agrees on which scores are lost
    on, _ = O.score_layer(k.double().numpy(), v.double().numpy(), cu, 0.2, "fft")
    assert np.array_equal(np.isnan(on), ~ok)
    scores = torch.from_numpy(g.astype(np.float32))
    got = _gpu_select(fc, k, v, cu, scores, [5, 7], [0, 5, 12], 12)[2]
    np.testing.assert_array_equal(got[1, 0:5], np.arange(5))
    np.testing.assert_array_equal(got[2, 5:12], np.arange(7))


# ---------------------------------------------------------------- ABI error paths (host-side checks only)
def test_abi_rejects_bad_arguments(fc):
    h = fc.fc_create(0, 1024)
    try:
        k, v = _rand_kv(128, 2, 128, torch.float32, 0)
        kd, vd = k.cuda(), v.cuda()
        scores = torch.empty((2, 128), dtype=torch.float32, device="cuda")
        energy = torch.empty((1, 4), dtype=torch.float64, device="cuda")
        ws = torch.empty(fc.fc_score_workspace_bytes(h, kd, vd, [0, 128]), dtype=torch.uint8, device="cuda")
        with pytest.raises(fc.FlashCacheError) as e:
            fc.fc_score_layer(h, kd, vd, [0, 128], 1.5, scores, energy, ws)          # gamma out of range
        assert e.value.code == 1
        with pytest.raises(fc.FlashCacheError) as e:
            fc.fc_score_layer(h, kd, vd, [0, 128], 0.2, scores, energy, ws[:64])     # workspace too small
        assert e.value.code == 3
        with pytest.raises(fc.FlashCacheError) as e:
            fc.fc_score_layer(h, kd, vd, [0, 200, 128], 0.2, scores, energy, ws)     # decreasing cu_seqlens
        assert e.value.code == 1
        k2, v2 = _rand_kv(2048, 1, 128, torch.float32, 0)
        assert fc.fc_score_workspace_bytes(h, k2.cuda(), v2.cuda(), [0, 2048]) == 0  # longer than max_seqlen
        k3, v3 = _rand_kv(64, 1, 96, torch.float32, 0)
        assert fc.fc_score_workspace_bytes(h, k3.cuda(), v3.cuda(), [0, 64]) == 0    # head_dim not a multiple of 64
        assert fc.fc_last_device_status(h) == 0
    finally:
        fc.fc_destroy(h)
    with pytest.raises(fc.FlashCacheError):
        fc.fc_create(0, 0)
