"""Prompt attention where a key's fp16 value is infinite.

The first token's key overflows fp16 and every query has a negative component
against it, so that its scores are -inf: the other rows give it no weight, and the
first row, which sees nothing else, has no weights at all.  Its attention output is
zero, as with the value row of that key, which is zero too: the results are those
of the same model with a key that is finite and as far away, bit for bit.
"""
import numpy as np
import pytest

import synth
from gpu_util import config_for

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("hd", [64, 128])
@pytest.mark.parametrize("P", [20, 200])
def test_first_row_without_weights(hd, P):
    import paper_2309_08168_gb300 as ssd
    w = synth.Workload("inf", 2, 256, 4, 4, hd, 64, 64, 16, 8, 4, 0, skip=[])
    w.rope_theta = 1e30  # the last rotation pair does not turn
    first, j = 5, hd // 2 - 1
    g = torch.Generator().manual_seed(41)
    d, qd, V = w.d_model, w.n_heads * hd, w.vocab

    def mat(n, k):
        return torch.randn(n, k, generator=g) * k ** -0.5

    embed = torch.where(torch.rand(V, d, generator=g) < 0.5, -1.0, 1.0)
    embed[:, 0], embed[:, 1], embed[:, 2] = 1.0, 0.0, 1.0
    embed[first, 1], embed[first, 2] = 1.0, 0.0  # (every row has the same norm)
    layers = [{"wq": mat(qd, d), "wk": mat(qd, d), "wv": mat(qd, d), "wo": mat(d, qd), "attn_norm": torch.ones(d),
               "w_gate": mat(64, d), "w_up": mat(64, d), "w_down": mat(d, 64), "mlp_norm": torch.ones(d)} for _ in range(2)]
    q, k, v = layers[0]["wq"], layers[0]["wk"], layers[0]["wv"]
    # a weight with which the query's fp16 hi and lo parts are both negative, scaled
    # (as in the prompt kernel) or not, by more than q's own error of 2^-17
    x0 = 1.0 / np.sqrt((d - 1) / d + w.rms_eps)
    weight = next(-1 - i / 128 for i in range(128) if all(
        np.float32((-1 - i / 128) * x0 * f) - np.float32(np.float16((-1 - i / 128) * x0 * f)) < -5e-5 * f
        for f in (1.0, np.log2(np.e) / np.sqrt(hd))))
    q.zero_()
    q[j::hd, 0] = weight
    k.zero_()
    value = v[:, 2].clone()
    v.zero_()
    v[:, 2] = value  # zero for the first token

    def logits(key):
        k[j::hd, 1] = key  # the first token's, against zero for the others
        dw = {"embed": embed, "lm_head": head, "final_norm": torch.ones(d), "layers": layers}
        dw = {n: [{m: t.to(torch.bfloat16).cuda() for m, t in y.items()} for y in a] if n == "layers"
              else a.to(torch.bfloat16).cuda() for n, a in dw.items()}
        torch.cuda.synchronize()
        prompt = synth.prompt(P, seed=42, vocab=V)
        prompt[prompt == first] = first + 1
        prompt[0] = first
        dec = ssd.Decoder(config_for(w, P + 8), dw, on_device=True)
        dec.prefill(prompt)
        out = dec.debug_forward(False, prompt[-1:], P - 1)
        dec.close()
        return out

    head = mat(V, d)
    finite, infinite = logits(3e4), logits(1e5)
    assert np.isfinite(finite).all()
    assert np.array_equal(finite.view(np.uint32), infinite.view(np.uint32))
