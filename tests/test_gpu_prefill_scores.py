"""Prefill attention at large scores of either sign, against the fp64 oracle.

Each head's scores share a large constant: 16 columns of every input row are 1, and one rotation pair of the
head's q and k (the last, whose angle is below 1e-27 here, rope_theta = 2^100) reads them with weights A and B.
Every row has the same norm (entries +-1), so the constant is the same for all keys and the softmax is that of the
remaining columns' scores, a few units wide.  In units of log2 the constants are about +-8e3, +-2e4 and +-4e4: a
running maximum kept with 8 significant bits is off by up to 128 there, beyond the range of fp32 exponentials.

Tolerance: a score is summed in at most 24 tensor-core steps at a magnitude below 2^18, each within one fp32 step
of 2^-6, so after the scale of 1 / sqrt(head_dim) it is within 0.034.  The oracle with its scores moved at random by
up to that much gives next-layer rows within 6.3 % of their rms and logits within 2.3 % (equal weights for all keys:
200 % and 57 %); 10 % is asked for.
"""
import numpy as np
import pytest
import torch

import oracle
import paper_2510_22641_gb300 as lib
import synth
from tests.gpu_util import make_model

pytestmark = pytest.mark.gpu

D, CONST = 256, 16
# per head: weights of the constant columns in q and k (exact in bf16); constants in log2 units in the comments
HEADS = {64: [(32, 30), (-32, 31), (16, 11), (-16, 27)],    # 44319, -45796, 8125, -19944
         128: [(32, 39), (-32, 35), (-16, 16), (16, 38)]}   # 40740, -36561, -8357, 19848


@pytest.mark.parametrize("head_dim", [64, 128])
def test_large_scores_match_oracle(head_dim):
    shape = synth.ModelShape(2, D, 4, head_dim, 512, 1000, rope_theta=2.0 ** 100)
    w = synth.TINY.replace(shape=shape, draft_exit_k=1, in_hidden=256, n_vis=150, n_prompt=0, max_new=1, weight_std=0.05)
    bits = synth.make_weights(w)
    layer = bits["layers"][0]
    for h, weights in enumerate(HEADS[head_dim]):
        last = (h + 1) * head_dim - 1
        for name, a in zip(("wq", "wk"), weights):
            layer[name][[last - head_dim // 2, last]] = 0
            layer[name][last - head_dim // 2, :CONST] = synth.f32_to_bf16(np.array([a]))[0]
    layer["wo"] = synth.f32_to_bf16(8 * synth.bf16_to_f32(layer["wo"]))  # the attention dominates the next layer's rows
    rng = np.random.default_rng(5)
    rows = rng.choice([-1.0, 1.0], (w.n_vis, D))
    rows[:, :CONST] = 1.0
    vis = synth.f32_to_bf16(rows)
    m = oracle.model_from_bits(w, bits, synth.bf16_to_f64)
    cache = oracle.KVCache(m.cfg, 256)
    ref = oracle.prefill(m, cache, synth.bf16_to_f64(vis), np.zeros(0, dtype=np.int64))
    model, _, _ = make_model(w, bits, gamma_max=4, max_seq=256)
    logits = torch.full((1, shape.vocab), float("nan"), device="cuda")
    try:
        model.set_logits_capture(logits)
        model.prefill(lib.bf16_bits_to_device(vis), torch.zeros(0, dtype=torch.int32, device="cuda"))
        model.sync()
        k, v, _ = model.kv()
        for got, r in ((k, cache.k), (v, cache.v)):
            r = r[1, :, :w.n_vis]
            rms = float(np.sqrt(np.mean(r * r)))
            np.testing.assert_allclose(got[1, :, :w.n_vis].cpu().numpy(), r, rtol=0, atol=0.1 * rms)
        r = np.asarray(ref).reshape(-1, shape.vocab)[-1]
        rms = float(np.sqrt(np.mean(r * r)))
        np.testing.assert_allclose(logits[0].cpu().numpy(), r, rtol=0, atol=0.1 * rms)
    finally:
        model.set_logits_capture(None)
        model.close()
