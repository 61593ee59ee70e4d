"""Sizes where the kernels' tiles, splits and fast paths begin and end.

Prompt encoding (the relative 2-norm error of the last row's logits against the
fp64 oracle).  K and V are rounded to fp16 (2^-11 of
their size each), everything else carries 16 bits or more, so the error of an
output is a few times 2^-11 of what attention contributes: bound 4 * 2^-11.
With large scores (S in magnitude) a score's own error, 2^-11 S, moves its
weight by as much: bound 4 * 2^-11 * (1 + S).

Such a bound lets one wrong row of a long prompt pass: attention is nearly uniform,
so a row of 514 is 0.2 % of it.  The cache that the prompt kernels leave is therefore
also compared with one that the decode kernel wrote, 16 rows at a time, through
forwards at positions around the ends of tiles and blocks.  Both round the same
K and V to fp16; sums in another order turn a rounding around here and there, by 2^-11
of one value, and an output averages over many: bound 2^-11 (measured 2e-4).  A wrong
row in the reference is seen by every later position that is tested.  With large
scores, if all hd elements of a key turned around, with random signs, a score would
move by 2^-11 S / sqrt(hd): bound 2^-11 * (1 + S / sqrt(hd)) (measured 2e-3 of 7e-3; an
accumulator that is not rescaled is off by 2^8).

Stand-alone projection: activations as bf16 pairs (2^-17 per element, in the
2-norm about half of that), 32-bit sums: bound 1e-5.  A row's result is the
same bits whatever rows come with it.

Sampling: with a nucleus of one token the draw is the argmax, for any
vocabulary, so sampled and greedy sequences are equal.  With any other
nucleus a drawn token has less than top_p of the mass above it (1e-5 for the
32-bit sums: a sum of at most 32768 values in trees of 32 + 10 additions is
within 42 * 2^-24 = 2.5e-6, on both sides), counting as above it only tokens
whose probability is larger by more than 32 bits can confuse (the exponent
x / T - max has an error of 2^-23 of its size, exp and the rounding to 1 a few
2^-24: at T = 1e4 many of 32000 probabilities are the same 32-bit number).  The
last tenth of the nucleus is drawn from.  High temperatures put most of the row into the list that the
threshold is searched in, top_p next to 1 takes the search down to zero.

Decode: forwards around the first segment's end (position 128), where
attention without partials takes over, and with K of one to four chunks
(the shortest splits): every row the same bits as alone.
"""
import numpy as np
import pytest

import oracle
import synth
from gpu_util import config_for, decoder

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

EPS = 2.0 ** -11


def model(heads=4, kv_heads=2, hd=64, d=256, ffn=688, vocab=512, layers=2):
    return synth.Workload("edges", layers, d, heads, kv_heads, hd, ffn, vocab, 16, 8, 4, 0, skip=[])


def prompt_error(w, hw, dw, P, seed, max_seq=None):
    import paper_2309_08168_gb300 as ssd
    max_seq = max_seq or P + 8
    prompt = synth.prompt(P, seed=seed, vocab=w.vocab)
    dec = ssd.Decoder(config_for(w, max_seq), dw, on_device=True)
    dec.prefill(prompt)
    got = dec.debug_forward(False, prompt[-1:], P - 1)[0].astype(np.float64)
    dec.close()
    orc = oracle.Oracle(w, hw, max_seq=max_seq)
    orc.prefill(prompt)
    ref = orc.forward(int(prompt[-1]), P - 1)
    orc.close()
    return np.linalg.norm(got - ref) / np.linalg.norm(ref)


EDGES = (1, 2, 15, 16, 17, 31, 32, 33, 63, 64, 65, 96, 127, 128, 129, 160, 191, 192, 193, 255, 256, 257, 258, 288, 384,
         511, 512)


class CachePair:
    """The prompt's cache by the prompt kernels and by the decode kernel, and the
    relative 2-norm distance of the logits at a position over the two."""

    def __init__(self, w, dw, P, seed):
        import paper_2309_08168_gb300 as ssd
        torch.cuda.synchronize()
        self.prompt = synth.prompt(P, seed=seed, vocab=w.vocab)
        self.new, self.ref = (ssd.Decoder(config_for(w, P + 8), dw, on_device=True) for _ in range(2))
        for i in range(0, P, 16):
            self.ref.debug_forward(False, self.prompt[i:i + 16], i)
        self.positions = sorted({p for p in EDGES if p < P} | {P - 1})

    def error(self, p):
        self.new.prefill(self.prompt)  # (the forward below writes row p)
        got, ref = (d.debug_forward(False, self.prompt[p:p + 1], p)[0].astype(np.float64) for d in (self.new, self.ref))
        return np.linalg.norm(got - ref) / np.linalg.norm(ref)

    def close(self):
        self.new.close()
        self.ref.close()


# token tiles of 32 .. 256 rows and their edges; GQA, an odd number of 128-row
# boxes of q / k / v, ffn not a multiple of the tile
@pytest.mark.parametrize("P", [18, 33, 34, 65, 66, 97, 161, 257, 258, 290, 514])
def test_prompt_token_tiles(P):
    w = model()
    hw = synth.host_weights(w, seed=21)
    assert prompt_error(w, hw, synth.host_to_device_weights(hw), P, seed=P) <= 4 * EPS


@pytest.mark.parametrize("P", [18, 33, 66, 161, 258, 514])
def test_prompt_rows(P):
    w = model()
    caches = CachePair(w, synth.host_to_device_weights(synth.host_weights(w, seed=21)), P, seed=P)
    for p in caches.positions:
        assert caches.error(p) <= EPS, p
    # the same with one row of the reference replaced by another token's
    row = P // 2
    caches.ref.debug_forward(False, [(caches.prompt[row] + 1) % w.vocab], row)
    for p in caches.positions:
        if p > row:
            assert caches.error(p) > EPS, p
    caches.close()


@pytest.mark.parametrize("heads,kv_heads,hd,d,ffn", [(1, 1, 128, 128, 64), (3, 3, 128, 384, 1040), (6, 2, 64, 640, 80),
                                                     (8, 1, 128, 1024, 2736)])
def test_prompt_shapes(heads, kv_heads, hd, d, ffn):
    w = model(heads, kv_heads, hd, d, ffn)
    hw = synth.host_weights(w, seed=22)
    dw = synth.host_to_device_weights(hw)
    assert prompt_error(w, hw, dw, 150, seed=5) <= 4 * EPS
    caches = CachePair(w, dw, 150, seed=5)
    for p in caches.positions:
        assert caches.error(p) <= EPS, p
    caches.close()


# scores large enough that the running maximum moves after the first key block
@pytest.mark.parametrize("P", [130, 260])
def test_prompt_attention_rescale(P):
    w = model(heads=4, kv_heads=4, hd=64)
    hw = synth.host_weights(w, seed=23)
    scale = 16.0  # q k^T / sqrt(hd): about 0.8 x scale^2 / 10 in the spread
    for layer in hw["layers"]:
        for name in ("wq", "wk"):
            layer[name] = synth.round_bf16_host(synth.bf16_bits_to_f64(layer[name]) * scale).reshape(layer[name].shape)
    S = 4 * (0.02 * scale) ** 2 * w.d_model
    dw = synth.host_to_device_weights(hw)
    assert prompt_error(w, hw, dw, P, seed=6) <= 4 * EPS * (1 + S)
    caches = CachePair(w, dw, P, seed=6)
    for p in caches.positions:
        assert caches.error(p) <= EPS * (1 + S / np.sqrt(w.head_dim)), p
    caches.close()


# clusters of 1, 2, 4 and 8 CTAs, more than one chunk of 1024 k, ends of rows,
# K blocks and row tiles
@pytest.mark.parametrize("M,K,N", [(1, 16, 1), (3, 48, 127), (8, 80, 129), (9, 272, 128), (16, 528, 300), (2, 1040, 257),
                                   (5, 4112, 640), (16, 4096, 8192), (1, 2064, 39000), (4, 4096, 20001), (7, 304, 100000)])
def test_linear_edges(M, K, N):
    import paper_2309_08168_gb300 as ssd
    g = torch.Generator(device="cuda").manual_seed(M * K + N)
    w = torch.empty(N, K, dtype=torch.bfloat16, device="cuda").normal_(0.0, 1.0, generator=g)
    x = torch.randn(M, K, device="cuda", generator=g)
    stream = torch.cuda.current_stream().cuda_stream

    def linear(rows):
        y = torch.full((rows.shape[0], N), float("nan"), device="cuda")
        ssd.ssd_linear_noalloc(w, rows, y, N, K, rows.shape[0], stream)
        return y

    y = linear(x)
    ref = x.double() @ w.double().T
    assert float((y.double() - ref).norm() / ref.norm()) <= 1e-5
    for m in range(0, M, 5):
        assert torch.equal(linear(x[m:m + 1].contiguous())[0], y[m])


def test_linear_overlapping_calls():
    """Calls on several streams share nothing."""
    import paper_2309_08168_gb300 as ssd
    M, K, N = 8, 4096, 2048
    jobs = []
    for i in range(4):
        g = torch.Generator(device="cuda").manual_seed(i)
        w = torch.empty(N, K, dtype=torch.bfloat16, device="cuda").normal_(0.0, 1.0, generator=g)
        jobs.append((w, torch.randn(M, K, device="cuda", generator=g), torch.empty(M, N, device="cuda"), torch.cuda.Stream()))
    torch.cuda.synchronize()
    for _ in range(5):
        for w, x, y, s in jobs:
            ssd.ssd_linear_noalloc(w, x, y, N, K, M, s.cuda_stream)
    torch.cuda.synchronize()
    for w, x, y, s in jobs:
        ref = x.double() @ w.double().T
        assert float((y.double() - ref).norm() / ref.norm()) <= 1e-5


@pytest.mark.parametrize("vocab", [3, 130, 1000, 2049, 31999, 32768])
def test_one_token_nucleus_is_greedy(vocab):
    import paper_2309_08168_gb300 as ssd
    w = model(vocab=vocab)
    hw = synth.host_weights(w, seed=25)
    dw = synth.host_to_device_weights(hw)
    torch.cuda.synchronize()
    dec = decoder(w, dw, 64, mask=[0, 1, 0, 0])
    prompt = synth.prompt(20, seed=8, vocab=vocab)
    greedy, _ = dec.generate(prompt, 24, 4)
    dec.set_sampling(1.0, 1e-6)
    sampled, st = dec.generate(None, 24, 4, mode=ssd.SSD_SAMPLE, seed=3)
    assert np.array_equal(greedy, sampled) and st["drafted"] > 0
    dec.close()


@pytest.mark.parametrize("vocab", [3, 300, 2049, 32000])
@pytest.mark.parametrize("temperature,top_p", [(1.0, 0.5), (1.0, 0.95), (40.0, 0.95), (1e4, 0.3), (1.0, 0.9995),
                                               (1.0, 0.99999994), (0.02, 0.99999994)])
def test_nucleus_cut(vocab, temperature, top_p):
    import paper_2309_08168_gb300 as ssd
    w = model(vocab=vocab)
    hw = synth.host_weights(w, seed=26)
    dw = synth.host_to_device_weights(hw)
    torch.cuda.synchronize()
    dec = decoder(w, dw, 64, mask=[0, 1, 0, 0])
    prompt = synth.prompt(20, seed=8, vocab=vocab)
    dec.set_sampling(temperature, top_p)
    dec.prefill(prompt)
    x = dec.debug_forward(False, prompt[-1:], len(prompt) - 1)[0].astype(np.float64) / temperature
    dec.prefill(prompt)
    n = 200
    drawn = np.array([dec.generate(None, 2, 1, mode=ssd.SSD_SAMPLE, seed=100 + i)[0][0] for i in range(n)])
    dec.close()
    pi = np.exp(x - x.max())
    pi /= pi.sum()
    order = np.argsort(-pi, kind="stable")
    above = np.empty(vocab)
    above[order] = np.concatenate([[0.0], np.cumsum(pi[order])[:-1]])
    p_min = pi[drawn].min() * (1 + (4 + np.abs(x).max()) * 2.0 ** -22)
    assert pi[pi > p_min].sum() < top_p + 1e-5
    last = (above >= 0.9 * top_p) & (above < top_p)
    if pi[last].sum() >= 0.05 * top_p:  # missed by 200 draws: 0.95 ** 200 = 4e-5
        assert (above[drawn] >= 0.9 * top_p).any()


@pytest.mark.parametrize("d,heads,hd,ffn", [(128, 2, 64, 64), (256, 2, 128, 384), (384, 6, 64, 400), (512, 4, 128, 528)])
@pytest.mark.parametrize("pos0,n_rows", [(126, 2), (125, 5), (127, 9), (128, 13), (120, 16)])
def test_rows_alone_around_first_segment(d, heads, hd, ffn, pos0, n_rows):
    w = model(heads, heads, hd, d, ffn)
    dw = synth.host_to_device_weights(synth.host_weights(w, seed=26))
    torch.cuda.synchronize()
    dec = decoder(w, dw, 160)
    dec.prefill(synth.prompt(pos0 + 1, seed=9, vocab=w.vocab))
    rows = synth.prompt(n_rows, seed=10 + n_rows, vocab=w.vocab)
    many = dec.debug_forward(False, rows, pos0)
    one = np.stack([dec.debug_forward(False, rows[r:r + 1], pos0 + r)[0] for r in range(n_rows)])
    assert np.array_equal(many.view(np.uint32), one.view(np.uint32))
    dec.close()
