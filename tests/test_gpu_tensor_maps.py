"""The prompt GEMMs' weight maps: whatever the addresses of the matrices and the form
of their maps, the same rows reach the same place of shared memory, so the results
are the same bits.

w_gate and w_up share one tensor map with the distance between them as a stride:
either may come first in memory (the epilogue swaps the halves), and with no
distance (one matrix as both) there is no such map.  Plain maps with boxes of 16
rows stand in where the folded ones do not exist; SSD_PLAIN_TMAPS=1 chooses them.
Shapes: 64- and 128-wide heads, an odd number of 128-row boxes of q / k / v, GQA,
ffn ending inside a tile and inside a box.
"""
import numpy as np
import pytest

import synth
from gpu_util import config_for

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

SHAPES = [(4, 2, 64, 256, 688), (6, 2, 64, 640, 80), (3, 3, 128, 384, 1040), (8, 1, 128, 1024, 2736)]
P = 150


def model(heads, kv_heads, hd, d, ffn):
    return synth.Workload("maps", 2, d, heads, kv_heads, hd, ffn, 512, 16, 8, 4, 0, skip=[])


def logits(w, dw):
    """Rows at positions over all of the prompt's cache."""
    import paper_2309_08168_gb300 as ssd
    torch.cuda.synchronize()
    prompt = synth.prompt(P, seed=31, vocab=w.vocab)
    dec = ssd.Decoder(config_for(w, P + 8), dw, on_device=True)
    out = []
    for pos in (1, 33, 127, P - 1):
        dec.prefill(prompt)
        out.append(dec.debug_forward(False, prompt[pos:pos + 1], pos)[0])
    dec.close()
    out = np.stack(out)
    assert np.isfinite(out).all()
    return out.view(np.uint32)


@pytest.mark.parametrize("shape", SHAPES)
@pytest.mark.parametrize("gap", [0, 48])
def test_gate_and_up_in_one_tensor_in_both_orders(shape, gap):
    w = model(*shape)
    dw = synth.host_to_device_weights(synth.host_weights(w, seed=32))
    expected = logits(w, dw)
    n = w.ffn * w.d_model
    for up_first in (False, True):
        for layer in dw["layers"]:
            both = torch.empty(2 * n + gap, dtype=torch.bfloat16, device="cuda")
            halves = [both[:n], both[n + gap:]]
            gate, up = halves[::-1] if up_first else halves
            gate.copy_(layer["w_gate"].view(torch.bfloat16).reshape(-1))
            up.copy_(layer["w_up"].view(torch.bfloat16).reshape(-1))
            layer["w_gate"], layer["w_up"] = gate, up
        assert np.array_equal(logits(w, dw), expected), up_first


@pytest.mark.parametrize("shape", SHAPES)
def test_one_matrix_as_gate_and_up(shape):
    w = model(*shape)
    dw = synth.host_to_device_weights(synth.host_weights(w, seed=33))
    for layer in dw["layers"]:
        layer["w_up"] = layer["w_gate"].clone()
    expected = logits(w, dw)
    for layer in dw["layers"]:
        layer["w_up"] = layer["w_gate"]
    assert np.array_equal(logits(w, dw), expected)


@pytest.mark.parametrize("shape", SHAPES)
def test_plain_maps(shape, monkeypatch):
    w = model(*shape)
    dw = synth.host_to_device_weights(synth.host_weights(w, seed=34))
    expected = logits(w, dw)
    monkeypatch.setenv("SSD_PLAIN_TMAPS", "1")
    assert np.array_equal(logits(w, dw), expected)
