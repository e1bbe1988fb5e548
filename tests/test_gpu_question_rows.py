"""Questions on either side of the row counts at which the projection leaves room for the prefill attention (24, 32, 48 rows; over few keys and
over many), of one stream and of several, where K is deep enough to lose stages by it and where it is not."""
import pytest

from paper_2503_09387_b200 import binding, synth
from tests.parity import Pair

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d,Hq,Hkv,d_ff,L,more,affine", [(3584, 28, 4, 0, 1, 448, False), (1024, 16, 4, 704, 2, 128, True)])
def test_rows_around_the_rule(d, Hq, Hkv, d_ff, L, more, affine):
    w = synth.workload("deep", n_layers=L, d_model=d, n_q_heads=Hq, n_kv_heads=Hkv, head_dim=d // Hq, tokens_per_frame=5, n_frames=2, bank_capacity=1,
                       prefix_len=3, question_len=0, decode_tokens=0, n_streams=3, frame_model="iid", seed=89)
    p = Pair(w, with_gain=affine, with_bias=affine, max_prefix=64 + more, max_text=320, max_step_tokens=64, **({"d_ff": d_ff} if d_ff else {}))
    ids = [0, 1, 2]
    row = lambda tag, T, s: synth.normal_bf16(w.seed, synth.TAG_QUESTION, (T, d), 1.0, offset=(tag * 4 + s) * 64 * d)
    for s in ids:
        p.text([s], [row(0, 17, s)], "prefix of 17")
    for i in range(more // 64):                               # stream 0 alone has many keys
        p.text([0], [row(1 + i, 64, 0)], f"64 rows more of stream 0's prefix, {i}")
    for t in range(2):
        p.frame(ids, [w.frame_hidden(t, s) for s in ids], f"frame {t}")
    for i, T in enumerate((17, 24, 25, 32, 33, 48, 49)):
        for s in (0, 1):
            p.text([s], [row(16 + i, T, s)], f"{T} rows of stream {s}")
    for i, T in enumerate((8, 11, 16)):                       # 24, 33 and 48 rows
        p.text(ids, [row(24 + i, T, s) for s in ids], f"3 x {T} rows")
    for s in ids:
        p.check_bank(s, layer=L - 1)
    p.close()


def test_the_projection_beside_the_attention_takes_half_the_registers():
    regs = binding.load_library()._ZN2vs24few_row_linear_registersEv()
    assert 0 < regs and 2 * 320 * ((regs + 7) // 8 * 8) <= 65536          # ten warps; registers are given out eight a thread
