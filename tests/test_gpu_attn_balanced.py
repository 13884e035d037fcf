"""The balanced unclustered attention (splits by the cached lengths) against
the oracle: lengths that need one and many splits, a sequence of a single
entry, slices that end inside a group of 16 entries, and steps that grow the
caches under the captured plan."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_2605_27255_gb300 import capi, synth

pytestmark = pytest.mark.gpu

S = synth.ModelShape("bal", H=512, L=2, n_q=8, n_kv=2, d_h=128, F=1408, V=4096, compressor="mlp", mtp_block=1,
                     dtype="bf16", rope_theta=1e6, tau=0.5)


@pytest.mark.parametrize("lens,balanced", [([3, 40, 2900], True), ([1500, 1, 17, 16, 2333, 40, 5], True),
                                           ([5] * 33 + [3000], True), ([900, 900, 900], False)])
def test_ragged_batch_matches_oracle(lens, balanced):
    B = len(lens)
    w = synth.gen_weights(S, seed=5)
    cap = max(lens) + 8
    g = capi.Pipo(S, w, max_batch=B, max_ctx=cap, debug=True)
    m = O.Model(S, w, max_ctx=cap)
    o = O.State(m, B)
    try:
        prompts = synth.gen_prompts(B, 2, S.V, seed=3).numpy()
        g.prefill(prompts)
        o.prefill(prompts, tau=S.tau)
        for b, n in enumerate(lens):
            K, V = (t.numpy() for t in synth.gen_kv_fill(S, n, seed=50 + b))
            g.load_cache(b, K, V)
            o.set_cache(b, K, V)
        pend = np.stack([prompts[:, 1], prompts[:, 0]], 1)
        for i in range(3):
            g.set_pending(pend)
            o.set_pending(pend)
            g.step()
            r = o.step(tau=S.tau)
            assert ("balanced" in g.describe()) == balanced, g.describe()
            d = g.debug()
            assert np.abs(d["logits_b"] - r["logits_b"]).max() < 2e-2
            assert np.abs(d["h_b"] - r["h_b"]).max() < 2e-2
            pend = np.stack([r["x_b"], np.full(B, -1)], 1).astype(np.int32)
    finally:
        g.close()
