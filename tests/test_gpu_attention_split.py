"""Key tiles of the prefill attention shared by the CTAs of a cluster: one to eight of them, groups whose rows fill the exchange
area and whose last rows lie behind it, token counts that leave a CTA of the cluster few rows or none."""
import pytest

from paper_2503_09387_b200 import synth
from tests.parity import Pair

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("Hq,Hkv,D,S", [(7, 1, 128, 1), (8, 1, 128, 1), (8, 1, 64, 2), (12, 4, 128, 1), (3, 3, 64, 1)])
def test_every_cluster_size(Hq, Hkv, D, S):
    d = Hq * D
    w = synth.workload("deep", n_layers=1, d_model=d, n_q_heads=Hq, n_kv_heads=Hkv, head_dim=D, tokens_per_frame=5, n_frames=2, bank_capacity=3,
                       prefix_len=3, question_len=0, decode_tokens=0, n_streams=S, frame_model="iid", seed=47)
    p = Pair(w, with_gain=True, with_bias=True, max_prefix=1100, max_text=160, max_step_tokens=128)
    ids = list(range(S))
    row = lambda tag, T, s: synth.normal_bf16(w.seed, synth.TAG_QUESTION, (T, d), 1.0, offset=(tag * 4 + s) * 128 * d)
    for i in range(8):                                        # keys of 1 to 17 tiles
        p.text(ids, [row(i, 128, s) for s in ids], f"prefix rows from {128 * i}")
    for t in range(2):
        p.frame(ids, [w.frame_hidden(t, s) for s in ids], f"frame {t}")
    for i, T in enumerate((2, 9, 15, 16, 17, 33)):
        p.text(ids, [row(8 + i, T, s) for s in ids], f"{T} rows")
    for s in ids:
        p.check_bank(s)
    p.close()
