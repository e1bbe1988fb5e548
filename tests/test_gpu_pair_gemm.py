"""The linear layers at the sizes where their tiling can go wrong: token counts around 16-token blocks, 32-token chunks and the
256-token tile, K splits with more shares than blocks, feature counts that leave a pair's second CTA empty."""
import pytest

from paper_2503_09387_b200 import synth
from tests.parity import Pair

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d,Hq,Hkv,D,d_ff,S,Ns", [(128, 2, 1, 64, 64, 1, (1, 15, 16, 31, 33)), (384, 3, 3, 128, 320, 2, (1, 7, 63, 127, 128)),
                                                  (640, 5, 1, 128, 0, 3, (85, 86, 170)), (1152, 18, 3, 64, 704, 1, (16, 47, 254, 255)),
                                                  (1280, 10, 2, 128, 7936, 4, (64, 200, 255))])
def test_frames_of_every_tiling(d, Hq, Hkv, D, d_ff, S, Ns):
    w = synth.workload("deep", n_layers=1, d_model=d, n_q_heads=Hq, n_kv_heads=Hkv, head_dim=D, tokens_per_frame=max(Ns), n_frames=len(Ns),
                       bank_capacity=2, prefix_len=3, question_len=0, decode_tokens=0, n_streams=S, frame_model="iid", seed=43)
    p = Pair(w, with_gain=True, with_bias=True, d_ff=d_ff, max_step_tokens=64)
    ids = list(range(S))
    p.text(ids, [w.prefix_hidden(s) for s in ids], "prefix")
    for t, N in enumerate(Ns):
        p.frame(ids, [w.frame_hidden(t, s)[:N] for s in ids], f"frame of {N}")
        for s in ids:
            p.check_bank(s)
    p.close()
