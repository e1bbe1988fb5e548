"""Where a step's rows may be written.  Single tokens of the attention path go to any element-aligned `out`, whichever kernel an
aligned one of that step is served by; every other call refuses an `out` (and `hidden`) that its kernels cannot store to."""
import numpy as np
import pytest
import torch

from paper_2503_09387_b200 import binding, synth
from tests.parity import Pair, assert_close, to_dev, to_f64

pytestmark = pytest.mark.gpu


def _shifted(shape, dtype, by=1):
    n = int(np.prod(shape))
    return torch.empty(n + 8, dtype=dtype, device="cuda")[by:by + n].view(shape)


@pytest.mark.parametrize("d,Hq,Hkv,D,L,S,out_dtype", [(256, 4, 2, 64, 1, 2, 1),           # by KV head
                                                      (1024, 8, 1, 128, 1, 5, 0),
                                                      (1152, 18, 3, 64, 2, 6, 1),         # the persistent kernel
                                                      (1536, 12, 12, 128, 2, 9, 0),
                                                      (256, 4, 2, 64, 1, 1, 0)])          # by query head
def test_single_tokens_to_any_address(d, Hq, Hkv, D, L, S, out_dtype):
    w = synth.workload("deep", n_layers=L, d_model=d, n_q_heads=Hq, n_kv_heads=Hkv, head_dim=D, tokens_per_frame=5, n_frames=2, bank_capacity=2,
                       prefix_len=130, question_len=0, decode_tokens=1, n_streams=S, frame_model="iid", seed=59)
    p = Pair(w, with_gain=True, out_dtype=out_dtype, max_text=4, max_step_tokens=130)
    ids = list(range(S))
    p.text(ids, [w.prefix_hidden(s) for s in ids], "prefix", compare=False)
    for t in range(w.n_frames):
        p.frame(ids, [w.frame_hidden(t, s) for s in ids], f"frame {t}")
    bits = [w.decode_hidden(0, s) for s in ids]
    x = to_dev(np.stack(bits))
    got = to_f64(p.gpu.decode_step(ids, x, out=_shifted((S, 1, p.gpu.out_width), p.gpu.out_torch_dtype)))
    for s in ids:
        want = p.ora[s].text_step(synth.bf16_bits_to_f64(bits[s]))
        if out_dtype == 1:
            assert_close(got[s], want, f"stream {s}")
        else:       # 2e-2 for the arithmetic and half a bf16 unit (at most 2^-8 of the value) for the rounding to the output type
            assert np.all(np.abs(got[s] - want) <= 2e-2 + 2.0 ** -8 * np.abs(want)), f"stream {s}"
        p.check_bank(s)
    p.close()


@pytest.mark.parametrize("d_ff,out_dtype", [(0, 1), (320, 0)])
def test_misaligned_rows_are_refused(d_ff, out_dtype):
    w = synth.workload("deep", n_layers=1, d_model=256, n_q_heads=4, n_kv_heads=2, head_dim=64, tokens_per_frame=5, n_frames=3, bank_capacity=2,
                       prefix_len=4, question_len=3, decode_tokens=1, seed=61)
    p = Pair(w, d_ff=d_ff, out_dtype=out_dtype, max_chunk_frames=2)
    E, dt = p.gpu.out_width, p.gpu.out_torch_dtype

    def refused(call, *a, **kw):
        with pytest.raises(binding.VsError) as err:
            call(*a, **kw)
        assert err.value.code == binding.VS_ERR_INVALID_ARG

    frames = to_dev(np.stack([w.frame_hidden(t) for t in range(2)]))
    refused(p.gpu.decode_step, [0], to_dev(w.prefix_hidden()[None]), out=_shifted((1, 4, E), dt))
    p.text([0], [w.prefix_hidden()], "prefix")
    refused(p.gpu.frame_prefill, [0], frames[:1], out=_shifted((1, 6, E), dt))
    moved = _shifted((1, 5, 256), torch.bfloat16)
    moved.copy_(frames[:1])
    refused(p.gpu.frame_prefill, [0], moved)
    refused(p.gpu.frame_prefill_chunk, 0, frames, out=_shifted((2, 6, E), dt))
    p.frame([0], [w.frame_hidden(0)], "frame 0")
    with pytest.raises(binding.VsError):
        binding.vs_bank_forward(p.gpu.handle, 0, _shifted((1, E), dt).data_ptr(), p.gpu._stream())
    if d_ff:
        refused(p.gpu.decode_step, [0], to_dev(w.decode_hidden(0)[None]), out=_shifted((1, 1, E), dt))
    p.text([0], [w.question_hidden()], "question")       # nothing of the refused calls was kept
    p.check_bank(0)
    p.close()
