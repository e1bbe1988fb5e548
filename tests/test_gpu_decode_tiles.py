"""Decode attention by KV head: key axes on either side of the tiles a warp walks (16 keys, eight warps, one to four rounds), so that the step's
own key lies in the first tile, in one that is fetched ahead or alone in its tile; both head sizes; a cluster of two."""
import pytest

from paper_2503_09387_b200 import synth
from tests.parity import Pair

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("H,D,S,prefixes", [(16, 64, 10, (1, 11, 12, 13, 123, 124, 125, 252, 381, 383)),
                                            (8, 128, 20, (1, 12, 13, 121, 123, 124, 125, 140, 155, 250, 251, 252, 253, 300, 363, 379, 380, 381, 507, 508)),
                                            (16, 64, 6, (2, 124, 251, 255, 380, 509))])
def test_keys_at_the_edges_of_tiles(H, D, S, prefixes):
    d = H * D
    w = synth.workload("deep", n_layers=1, d_model=d, n_q_heads=H, n_kv_heads=H, head_dim=D, tokens_per_frame=5, n_frames=4, bank_capacity=3,
                       prefix_len=3, question_len=0, decode_tokens=0, n_streams=S, frame_model="iid", seed=83)
    p = Pair(w, max_prefix=512, max_text=8, max_step_tokens=512)
    row = lambda tag, T, s: synth.normal_bf16(w.seed, synth.TAG_QUESTION, (T, d), 1.0, offset=(tag * 32 + s) * 512 * d)
    for s, n in enumerate(prefixes):
        p.text([s], [row(0, n, s)], f"prefix of {n}")
    ids = list(range(S))
    for t in range(4):                                        # the bank is full from the fourth on: 3 carriers and the free slot
        p.frame(ids, [w.frame_hidden(t, s) for s in ids], f"frame {t}")
    for i in range(5):
        p.text(ids, [row(1 + i, 1, s) for s in ids], f"token {i}")
    p.close()
