"""Prefill chunks of more than 128 rows (the CTA-pair GEMM) against the
oracle: position tiles with remainders, one and several sequences, both chunk
attentions, and a projection whose K is not a multiple of 64 (F = 1376)."""
import pytest

from paper_2605_27255_gb300 import synth
from parity_util import run_forced_replay

pytestmark = pytest.mark.gpu

MID = synth.ModelShape("mid", H=512, L=3, n_q=8, n_kv=2, d_h=128, F=1376, V=5003,
                       compressor="mlp", mtp_block=1, dtype="bf16", rope_theta=1e6, tau=0.5)


@pytest.mark.parametrize("attn", ["rows", "tile"])
@pytest.mark.parametrize("rows,B,T,F,compressor", [(129, 1, 260, 1376, "mlp"), (300, 1, 700, 1408, "linear"),
                                                   (640, 3, 500, 1408, "mlp"), (4096, 2, 1100, 1408, "mlp"),
                                                   (512, 70, 31, 1408, "mlp")])
def test_tall_chunks_match_oracle(monkeypatch, attn, rows, B, T, F, compressor):
    monkeypatch.setenv("PIPO_PREFILL_ROWS", str(rows))
    monkeypatch.setenv("PIPO_PREFILL_ATTN", attn)
    s = MID.with_(F=F, compressor=compressor)
    w = synth.gen_weights(s, seed=3)
    prompts = synth.gen_prompts(B, T, s.V, seed=7).numpy()
    st = run_forced_replay(s, w, prompts, 3,
                           expect="attn_prefill_kernel" if attn == "tile" else "per-row attention")
    assert st.tok_checked >= 0.5 * st.tok_total
