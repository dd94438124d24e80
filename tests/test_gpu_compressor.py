"""`Compressor` on tensors and buffers that change between calls: its marshalled arguments follow them."""
import pytest
import torch

pytestmark = pytest.mark.gpu

L, H, D, T, RHO = 2, 3, 64, 700, 0.25


@pytest.fixture(scope="module")
def fc():
    if not torch.cuda.is_available():
        pytest.fail("GPU tests need a CUDA device")
    from paper_2511_16786_b200 import binding
    return binding


def _compressor(fc, dtype=torch.float16):
    return fc.Compressor(L, H, D, [0, T], dtype, RHO)


def _tensors(seed, dtype=torch.float16):
    g = torch.Generator(device="cuda").manual_seed(seed)
    return [torch.randn((T, H, D), generator=g, device="cuda").to(dtype) for _ in range(2 * L)]


def _results(c):
    """Scores, budgets, offsets and every kept row and index (what lies behind a layer's rows is not written)."""
    c.check_device_status()
    off = c.offsets.cpu()
    out = [c.scores.clone(), c.budgets.clone(), c.offsets.clone()]
    for l in range(L):
        n = int(off[l, -1])
        out += [c.out_k[l, :n].clone(), c.out_v[l, :n].clone(), c.out_idx[l, :, :n].clone()]
    return out


def _fresh(fc, K, V):
    c = _compressor(fc)
    c.compress([k.contiguous() for k in K], [v.contiguous() for v in V])
    res = _results(c)
    c.close()
    return res


def _same(a, b):
    return all(torch.equal(x, y) for x, y in zip(a, b)) and len(a) == len(b)


def test_the_same_memory_in_another_layout(fc):
    mem = _tensors(1)
    tokens_first = [t for t in mem]
    heads_first = [t.view(H, T, D).transpose(0, 1) for t in mem]          # same addresses, other strides
    c = _compressor(fc)
    for K, V in ((tokens_first[:L], tokens_first[L:]), (heads_first[:L], heads_first[L:]),
                 (tokens_first[:L], tokens_first[L:])):
        c.compress(K, V)
        assert _same(_results(c), _fresh(fc, K, V))
    c.close()


def test_replaced_buffers_receive_the_results(fc):
    mem = _tensors(2)
    K, V = mem[:L], mem[L:]
    want = _fresh(fc, K, V)
    c = _compressor(fc)
    c.compress(K, V)
    for name in ("out_k", "out_v", "out_idx", "scores", "energy", "budgets", "offsets"):
        old = getattr(c, name)
        setattr(c, name, torch.zeros_like(old))
        kept = old.clone()
        old.zero_()
        c.compress(K, V)
        assert _same(_results(c), want), name
        assert not old.any() and kept.any(), name                          # nothing went to the old one
    c.close()


def test_tensors_that_do_not_fit_are_refused(fc):
    mem = _tensors(3)
    K, V = mem[:L], mem[L:]
    c = _compressor(fc)
    for bad in ([k.float() for k in K], [k[:T - 1] for k in K], [k[:, :1] for k in K], K[:1]):
        with pytest.raises(ValueError):
            c.compress(bad, bad)
    c.compress(K, V)
    assert _same(_results(c), _fresh(fc, K, V))
    c.close()


def test_layers_of_unlike_layouts(fc):
    # one layer token-major, one head-major: each is read by its own strides, in the selection too
    mem = _tensors(4)
    K = [mem[0], mem[1].view(H, T, D).transpose(0, 1)]
    V = [mem[2], mem[3].view(H, T, D).transpose(0, 1)]
    c = _compressor(fc)
    c.compress(K, V)
    assert _same(_results(c), _fresh(fc, K, V))
    # the entry points that describe all layers by one view refuse them
    cu = [0, T]
    with pytest.raises(ValueError):
        fc.fc_score_layers(c.handle, K, V, cu, 0.2, c.scores, c.energy, c._ws)
    with pytest.raises(ValueError):
        fc.fc_select_compact_layers(c.handle, K, V, cu, c.scores, c.budgets, c.offsets, c.out_k, c.out_v, c.out_idx, c._ws)
    c.close()
