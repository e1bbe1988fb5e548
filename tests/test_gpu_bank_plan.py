"""A chunk's bank updates planned by one block: banks on either side of the block's 256 entries, chunks that fill the bank
and go on to evict, chunks that evict carriers of their own."""
import pytest

from paper_2503_09387_b200 import synth
from tests.parity import Pair

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("M,policy", [(1, 0), (5, 0), (255, 0), (256, 0), (257, 2), (300, 0)])
def test_chunks_across_the_fill_of_the_bank(M, policy):
    n_fill = max(M - 3, 0)
    w = synth.workload("long", d_model=128, n_q_heads=2, n_kv_heads=1, head_dim=64, tokens_per_frame=3, n_frames=n_fill + 21,
                       bank_capacity=M, prefix_len=5, question_len=0, decode_tokens=1)
    p = Pair(w, max_chunk_frames=7, evict_policy=policy)
    p.text([0], [w.prefix_hidden()], "prefix")
    shared = w.frame_shared()
    for t in range(n_fill):
        p.frame([0], [w.frame_hidden(t, shared=shared)], f"frame {t}", mode="carrier")
    for t in range(n_fill, w.n_frames, 7):
        p.frame_chunk(0, [w.frame_hidden(t + j, shared=shared) for j in range(7)], f"chunk at frame {t}")
        p.check_bank(0)
    assert p.ora[0].evictions == w.n_frames - M
    p.text([0], [w.decode_hidden(0)], "decode")
    p.close()


@pytest.mark.parametrize("M,L,heads", [(1, 1, 2), (2, 1, 9), (4, 2, 9), (5, 1, 17), (13, 2, 9), (140, 1, 9)])
def test_neighbours_scored_in_groups(M, L, heads):
    w = synth.workload("long" if L == 1 else "deep", n_layers=L, d_model=64 * heads, n_q_heads=heads, n_kv_heads=1 if heads < 9 else heads, head_dim=64, tokens_per_frame=3,
                       n_frames=M + 9, bank_capacity=M, prefix_len=2, question_len=0, decode_tokens=0, frame_model="iid", seed=53)
    p = Pair(w, evict_policy=1)
    p.text([0], [w.prefix_hidden()], "prefix")
    for t in range(w.n_frames):
        p.frame([0], [w.frame_hidden(t)], f"frame {t}", mode="full" if L > 1 or t + 3 > w.n_frames else "carrier")
        if t + 1 >= M:
            p.check_bank(0)
    p.close()
