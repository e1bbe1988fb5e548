"""The persistent kernel for steps of a few token rows: row counts on either side of its tile shapes (8, 16 rows) and beyond them, widths
that are no multiple of a stage, both head sizes, cut tiles, keys split over CTAs, the attention path alone and full layers."""
import pytest

from paper_2503_09387_b200 import synth
from tests.parity import Pair
from tests.test_gpu_parity import _check_lm, _lm_case

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d,Hq,Hkv,D,d_ff,L,prefix", [(1152, 18, 3, 64, 0, 2, 17), (1152, 18, 3, 64, 704, 2, 17), (1280, 10, 2, 128, 0, 1, 300),
                                                    (1280, 10, 2, 128, 1856, 2, 140), (1536, 12, 12, 128, 0, 2, 17)])
def test_steps_of_every_tile_shape(d, Hq, Hkv, D, d_ff, L, prefix):
    w = synth.workload("deep", n_layers=L, d_model=d, n_q_heads=Hq, n_kv_heads=Hkv, head_dim=D, tokens_per_frame=5,
                       n_frames=5, bank_capacity=4, prefix_len=3, question_len=0, decode_tokens=0, n_streams=3, frame_model="iid",
                       seed=41)
    kw = {} if d_ff == 0 else dict(d_ff=d_ff)
    p = Pair(w, with_gain=True, with_bias=True, max_prefix=prefix, max_text=96, max_step_tokens=32, **kw)
    ids = [0, 1, 2]
    row = lambda tag, T, s: synth.normal_bf16(w.seed, synth.TAG_QUESTION, (T, d), 1.0, offset=(tag * 4 + s) * 32 * d)
    for at in range(0, prefix, 32):
        p.text([0], [row(8 + at // 32, min(32, prefix - at), 0)], f"prefix rows from {at}")
    p.text([1, 2], [row(0, 1, s) for s in (1, 2)], "two one-row prefixes")
    for t in range(w.n_frames):
        p.frame(ids, [w.frame_hidden(t, s) for s in ids], f"frame {t}")
    for tag, T in ((1, 1), (2, 2), (3, 3), (4, 10)):          # 3, 6, 9 and 30 rows
        p.text(ids, [row(tag, T, s) for s in ids], f"3 streams x {T}")
    p.text([1], [row(5, 32, 1)], "32 rows")
    p.text([2, 0], [row(6, 8, s) for s in (2, 0)], "16 rows")
    p.text([0], [row(7, 1, 0)], "one row")
    for s in ids:
        for layer in range(L):
            p.check_bank(s, layer=layer)
    p.close()


@pytest.mark.parametrize("d_ff,one_launch", [(704, [(1, 1), (2, 1), (1, 2), (1, 8), (3, 2)]), (0, [(1, 2), (1, 8), (1, 9), (3, 2), (3, 3)])])
def test_which_steps_are_one_launch(d_ff, one_launch):
    """Narrow layers (24 KB of projection an SM): single tokens of three streams on are launches, several tokens are not."""
    w = synth.workload("deep", n_layers=2, d_model=1152, n_q_heads=18, n_kv_heads=3, head_dim=64, tokens_per_frame=5, n_frames=1, bank_capacity=2,
                       prefix_len=3, question_len=0, decode_tokens=0, n_streams=3, frame_model="iid", seed=71)
    p = Pair(w, max_prefix=64, max_text=16, max_step_tokens=32, **({"d_ff": d_ff} if d_ff else {}))
    for n, T in ((1, 1), (2, 1), (3, 1), (1, 2), (1, 8), (1, 9), (3, 2), (3, 3), (1, 17)):
        p.gpu.profile_read()
        p.text(list(range(n)), [synth.normal_bf16(w.seed, synth.TAG_QUESTION, (T, 1152), 1.0, offset=(T * 4 + s) * 32 * 1152) for s in range(n)], f"{n} x {T}")
        launches = sum(v[2] for v in p.gpu.profile_read().values())
        assert (launches == 1) == ((n, T) in one_launch), (n, T, launches)
    p.close()


@pytest.mark.parametrize("d,vocab,rows,norm,gain,out_dtype", [(1152, 1280, 1, True, True, 1), (1088, 1280, 8, True, False, 0), (1088, 1280, 9, True, False, 0),
                                                              (1088, 1280, 32, False, False, 1)])
def test_lm_head_of_a_few_rows(d, vocab, rows, norm, gain, out_dtype):
    _check_lm(*_lm_case(d, vocab, rows, norm, gain, out_dtype), f"lm head {d} {vocab} {rows}")
