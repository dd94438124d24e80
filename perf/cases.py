"""Workloads of the FlashCache library as its users run them, for timing and for comparing two builds.

Every case goes through the package's public entry points on tensors a program would hold anyway:

* ``prefill``   `Compressor.compress` (score every layer, allocate the budgets, keep and gather the rows) on device
                tensors; ``graph`` replays the captured call sequence instead, as a server of short prompts does.
* ``host``      `HostCompressor.compress`: K and V in page-locked host memory, the compacted caches back in host memory.
* ``decode``    `fc_decode_attention` for every layer of one decoding step, on kept rows and an uncompressed tail.
* ``spectrum``  `fc_power_spectrum` and `fc_cutoff_from_spectrum` for every layer: reading the cutoff off the energies.

Inputs follow the structure the method is made for: a smooth trend along the tokens (a few low cosines), small noise
and a share of rows far from the trend.  That share is near the cache ratio where rows are selected, since a ratio is
picked to hold the outliers.
"""
import math

import torch

from paper_2511_16786_b200 import binding as fc

_DTYPES = {"f32": torch.float32, "f16": torch.float16, "bf16": torch.bfloat16}
_BITS = {"f32": torch.int32, "f16": torch.int16, "bf16": torch.int16}
_COSINES = 8                      # low frequencies in the smooth trend
_MAX_ROWS = 12_000_000            # (layer, head, token) rows of a drawn prefill at head_dim 128


def _prefill(name, layers, heads, seqlens, dtype, rho, **more):
    case = dict(name=name, kind="prefill", layers=layers, heads=heads, dim=128, seqlens=seqlens, dtype=dtype, rho=rho,
                gamma=0.2, outliers=rho, per_layer=False, protect=False, graph=False)
    case.update(more)
    return case


def listed():
    return [
        # one layer of a short prompt in fp32: the smallest call, all launches and latency
        _prefill("prefill_1024_f32", 1, 4, "1024", "f32", 0.2),
        # a GQA model's image prompt
        _prefill("prefill_8192_bf16", 28, 4, "8192", "bf16", 0.2),
        # long multi-image context, the length the library is quoted on
        _prefill("prefill_32768_bf16", 28, 4, "32768", "bf16", 0.1),
        # multi-head attention (as many KV heads as query heads): the most bytes per token
        _prefill("prefill_16384_f16_mha", 32, 32, "16384", "f16", 0.2),
        # a batch of videos of unlike lengths, packed: no length is a power of two
        _prefill("prefill_ragged_long_bf16", 28, 4, "32092,26864,10164,8221,38158,13763,53602,6946", "bf16", 0.2),
        # a batch of ordinary requests, packed
        _prefill("prefill_ragged_short_bf16", 28, 4, "517,1024,64,1999,333,4096,100,2311", "bf16", 0.2),
        # one index set per layer, with text tokens, sinks and a recent window that must survive
        _prefill("prefill_layerwise_protect_f16", 28, 4, "12001,3072", "f16", 0.2, per_layer=True, protect=True),
        # a short prompt of a whole model, captured once and replayed
        _prefill("prefill_graph_1500_bf16", 28, 4, "1500", "bf16", 0.2, graph=True),
        # a decoding step on an uncompressed long cache: the largest read
        dict(name="decode_65536_bf16", kind="decode", layers=28, heads=4, q_heads=28, rows="65536", tails="", dtype="bf16"),
        # a decoding step of a small batch on kept rows with the tokens generated since: small reads, many launches
        dict(name="decode_kept_tails_f16", kind="decode", layers=28, heads=4, q_heads=28, rows="1638,205,3277,820",
             tails="17,64,1,100", dtype="f16"),
        # choosing the cutoff for a few layers of two prompts
        dict(name="spectrum_32768_10000_bf16", kind="spectrum", layers=4, heads=4, dim=128, seqlens="32768,10000",
             dtype="bf16", share=0.9, outliers=0.01),
        # the cache lives in host memory: copies in and out of the card are part of the call
        dict(name="host_8192_bf16", kind="host", layers=28, heads=4, dim=128, seqlens="8192", dtype="bf16", rho=0.2,
             gamma=0.2, outliers=0.2),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _length(rng, lo, hi):
    """A sequence length: spread over the logarithm, every third one a power of two."""
    n = _log_int(rng, lo, hi)
    return min(hi, 1 << int(round(math.log2(n)))) if rng.random() < 1 / 3 else n


def draw(rng):
    kind = rng.choices(("prefill", "decode", "spectrum", "host"), weights=(8, 3, 1, 1))[0]
    dtype = rng.choice(("bf16", "bf16", "f16", "f32"))
    if kind == "decode":
        batch = rng.choice((1, 1, 2, 4, 8))
        heads = rng.choice((1, 2, 4, 8, 32))
        group = 1 if heads == 32 else rng.choice((4, 7, 8))
        rows = [_log_int(rng, 64, 65536 // batch) for _ in range(batch)]
        tails = [rng.randint(0, 128) for _ in range(batch)] if rng.random() < 0.5 else []
        layers = max(1, min(_log_int(rng, 4, 32), 28 * 4 * 65536 // (heads * sum(rows))))
        return dict(kind="decode", layers=layers, heads=heads, q_heads=heads * group, rows=",".join(map(str, rows)),
                    tails=",".join(map(str, tails)), dtype="f16" if dtype == "f32" else dtype)
    batch = 1 if rng.random() < 0.5 else rng.randint(2, 8)
    top = {"prefill": 65536, "spectrum": 32768, "host": 8192}[kind]
    lens = [_length(rng, 64, top) for _ in range(batch)]
    dim = rng.choice((64, 128, 128))
    heads = rng.choice((1, 2, 4, 4, 8, 32))
    rows = _MAX_ROWS * 128 // dim // {"prefill": 1, "spectrum": 8, "host": 16}[kind]
    while heads > 1 and heads * sum(lens) > rows:
        heads //= 2
    layers = max(1, min(_log_int(rng, 1, 32), rows // (heads * sum(lens))))
    rho = rng.choice((0.1, 0.2, 0.4))
    case = dict(kind=kind, layers=layers, heads=heads, dim=dim, seqlens=",".join(map(str, lens)), dtype=dtype)
    if kind == "spectrum":
        case.update(share=0.9, outliers=0.01)
        return case
    case.update(rho=rho, gamma=rng.choice((0.1, 0.2, 0.2, 0.3)), outliers=rho)
    if kind == "prefill":
        case.update(per_layer=rng.random() < 0.2, protect=rng.random() < 0.2, graph=rng.random() < 0.2)
    return case


def _ints(text):
    return [int(x) for x in text.split(",")] if text else []


def _cu(lens):
    cu = [0]
    for n in lens:
        cu.append(cu[-1] + n)
    return cu


def _make_layer(case, lens, bases, gen):
    """K, V [T, H, d] of one layer on the GPU."""
    H, d, T = case["heads"], case["dim"], sum(lens)
    # rows far from the trend: per head, or common to the heads where a layer keeps one index set
    far = torch.rand((T, 1 if case.get("per_layer") else H, 1), generator=gen, device="cuda") < case["outliers"]
    kv = []
    for _ in range(2):
        noise = torch.randn((T, H, d), generator=gen, device="cuda")
        trend = torch.cat([b @ torch.randn((_COSINES, H * d), generator=gen, device="cuda") for b in bases])
        x = torch.where(far, noise * 5.0, trend.view(T, H, d).add_(noise, alpha=0.1))
        kv.append(x.to(_DTYPES[case["dtype"]]))
    return kv


def _make_layers(case, seed):
    gen = torch.Generator(device="cuda").manual_seed(seed)
    lens = _ints(case["seqlens"])
    bases = []
    for n in lens:
        i = torch.arange(n, dtype=torch.float64, device="cuda")[:, None]
        m = torch.arange(_COSINES, dtype=torch.float64, device="cuda")[None, :]
        bases.append(torch.cos(math.pi / (2.0 * n) * m * (2.0 * i + 1.0)).float())
    layers = [_make_layer(case, lens, bases, gen) for _ in range(case["layers"])]
    return lens, [k for k, _ in layers], [v for _, v in layers]


class _Prefill:
    def __init__(self, case, seed):
        lens, self.k, self.v = _make_layers(case, seed)
        cu, L, H, d = _cu(lens), case["layers"], case["heads"], case["dim"]
        protect, min_keep = None, 1
        if case["protect"]:              # sinks, a recent window and scattered text tokens: at most 32 a sequence
            protect, min_keep = torch.zeros(cu[-1], dtype=torch.uint8), 32
            for b, n in enumerate(lens):
                protect[cu[b]:cu[b] + 4] = 1
                protect[cu[b + 1] - 16:cu[b + 1]] = 1
                protect[cu[b] + n // 3:cu[b] + n // 3 + 12] = 1
            protect = protect.cuda()
        self.comp = c = fc.Compressor(L, H, d, cu, _DTYPES[case["dtype"]], case["rho"], case["gamma"], min_keep,
                                      per_layer=case["per_layer"], protect=protect)
        # the compressor's output buffers, cleared once: rows past a layer's last kept one are never written
        c.out_k = torch.zeros((L, c.capacity, H, d), dtype=_DTYPES[case["dtype"]], device="cuda")
        c.out_v = torch.zeros_like(c.out_k)
        c.out_idx = torch.zeros((L, H, c.capacity), dtype=torch.int32, device="cuda")
        self.bits = _BITS[case["dtype"]]
        self.graph = c.capture(self.k, self.v) if case["graph"] else None

    def run(self):
        c = self.comp
        if self.graph is not None:
            self.graph.replay()
        else:
            c.compress(self.k, self.v)
        # rows are copied bit for bit: compared as whole numbers
        return dict(scores=c.scores, energy=c.energy, budgets=c.budgets, offsets=c.offsets, idx=c.out_idx,
                    k=c.out_k.view(self.bits), v=c.out_v.view(self.bits))


class _Host:
    def __init__(self, case, seed):
        lens, k, v = _make_layers(case, seed)
        self.comp = fc.HostCompressor(case["layers"], case["heads"], case["dim"], _cu(lens), _DTYPES[case["dtype"]],
                                      case["rho"], case["gamma"])
        self.k, self.v = [self._pinned(t) for t in k], [self._pinned(t) for t in v]
        self.results = [self.comp.new_result(), self.comp.new_result()]      # in turn, as a serving loop holds them
        self.bits = _BITS[case["dtype"]]

    @staticmethod
    def _pinned(t):
        return torch.empty(t.shape, dtype=t.dtype, pin_memory=True).copy_(t)

    def run(self):
        r = self.results[0]
        self.results.reverse()
        self.comp.compress(self.k, self.v, r)
        return dict(k=r.out_k.view(self.bits), v=r.out_v.view(self.bits), idx=r.out_idx, budgets=r.budgets,
                    offsets=r.offsets, layer_rows=r.layer_rows)


class _Decode:
    def __init__(self, case, seed):
        gen = torch.Generator(device="cuda").manual_seed(seed)
        dt, L, H, Hq, d = _DTYPES[case["dtype"]], case["layers"], case["heads"], case["q_heads"], 128
        rows, tails = _ints(case["rows"]), _ints(case["tails"])
        B, offs = len(rows), _cu(rows)

        def normal(*shape):
            return torch.randn(shape, generator=gen, device="cuda").to(dt)

        self.handle = fc.fc_create(0, 1024)
        offsets = torch.tensor(offs, dtype=torch.int64, device="cuda")
        tail_len = torch.tensor(tails, dtype=torch.int32, device="cuda") if tails else None
        self.out = torch.empty((L, B, Hq, d), dtype=dt, device="cuda")
        self.args, self.keep = [], [offsets, tail_len]
        most = max(r + (tails[b] if tails else 0) for b, r in enumerate(rows))
        for _ in range(L):
            q, k, v = normal(B, Hq, d), normal(offs[-1], H, d), normal(offs[-1], H, d)
            tk, tv = (normal(B, 128, H, d), normal(B, 128, H, d)) if tails else (None, None)
            self.args.append(fc.make_decode_args(q, k, v, offsets, most, tk, tv, tail_len))
            self.keep += [q, k, v, tk, tv]
        self.ws = torch.empty(fc.fc_decode_workspace_bytes(self.handle, self.args[0]), dtype=torch.uint8, device="cuda")

    def run(self):
        for l, a in enumerate(self.args):
            fc.fc_decode_attention(self.handle, a, self.out[l], self.ws)
        return self.out

    def __del__(self):
        fc.fc_destroy(self.handle)


class _Spectrum:
    def __init__(self, case, seed):
        lens, self.k, self.v = _make_layers(case, seed)
        L, B, self.cu, self.share = case["layers"], len(lens), _cu(lens), case["share"]
        self.handle = fc.fc_create(0, max(lens))
        self.spectrum = torch.empty((L, self.cu[-1], 2), dtype=torch.float64, device="cuda")
        self.omega = torch.empty((L, B), dtype=torch.int32, device="cuda")
        self.gamma = torch.empty((L, B), dtype=torch.float64, device="cuda")
        self.ws = torch.empty(fc.fc_power_spectrum_workspace_bytes(self.handle, self.k[0], self.v[0], self.cu),
                              dtype=torch.uint8, device="cuda")

    def run(self):
        for l in range(len(self.k)):
            fc.fc_power_spectrum(self.handle, self.k[l], self.v[l], self.cu, self.spectrum[l], self.ws)
            fc.fc_cutoff_from_spectrum(self.handle, self.spectrum[l], self.cu, self.share, self.omega[l], self.gamma[l])
        return dict(spectrum=self.spectrum, omega=self.omega, gamma=self.gamma)

    def __del__(self):
        fc.fc_destroy(self.handle)


def prepare(case, seed):
    return {"prefill": _Prefill, "host": _Host, "decode": _Decode, "spectrum": _Spectrum}[case["kind"]](case, seed)


def run(state):
    return state.run()


def work(case):
    """Bytes: every input read once, every output written once.  Flops: one real-to-spectrum transform each way per
    column (2.5 n log2 n for each of K and V), whatever the length; attention: two products per row and query head."""
    es = 4 if case["dtype"] == "f32" else 2
    L, H = case["layers"], case["heads"]
    if case["kind"] == "decode":
        Hq, rows = case["q_heads"], sum(_ints(case["rows"])) + sum(_ints(case["tails"]))
        batch = len(_ints(case["rows"]))
        return dict(bytes=L * 128 * es * (2.0 * rows * H + 2.0 * batch * Hq), flops=L * 4.0 * 128 * rows * Hq)
    lens, d = _ints(case["seqlens"]), case["dim"]
    rows = float(L * H * sum(lens))
    points = L * H * d * sum(n * math.log2(n) for n in lens)
    if case["kind"] == "spectrum":
        return dict(bytes=rows * 2 * d * es + L * sum(lens) * 16.0, flops=5.0 * points)
    kept = case["rho"] * rows * (2 * d * es + 4)
    scores = 4.0 * rows if case["kind"] == "prefill" else 0.0
    return dict(bytes=rows * 2 * d * es + scores + kept, flops=10.0 * points)


def tolerance(case):
    if case["kind"] == "decode":          # 16-bit probabilities and outputs
        return {"rel": 1e-2}
    # fp32 transforms; a token may change places with another whose score is the same to fp32 rounding
    return {"rel": 1e-5, "max": 1e-4, "differ": 0.01}
