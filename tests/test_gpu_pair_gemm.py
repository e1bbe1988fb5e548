"""The linear layers at the sizes where their tiling can go wrong: token counts around 16-token blocks, 32-token chunks and the
256-token tile, K splits with more shares than blocks, feature counts that leave a pair's second CTA empty."""
import ctypes as C

import pytest
import torch

from paper_2503_09387_b200 import binding, synth
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


class _Tiling(C.Structure):
    _fields_ = [(n, C.c_int) for n in ("tile_n", "n_tiles", "ksplit", "pairs")]


def test_pairs_with_an_empty_second_cta():
    """All four layers of a block on CTA pairs (asked of the library), with an odd number of 128-row weight tiles each."""
    d, Hq, Hkv, D, d_ff, S, N = 1920, 15, 5, 128, 2112, 5, 203
    lib = binding.load_library()
    lib._ZN2vs12choose_tilesEiiiiib.restype = _Tiling
    n_sms, pairs = torch.cuda.get_device_properties(0).multi_processor_count, lib._ZN2vs19pair_gemm_max_pairsEv()
    for K, E in ((d, (Hq + 2 * Hkv) * D), (d, d), (d, 2 * d_ff), (d_ff, d)):
        assert lib._ZN2vs12choose_tilesEiiiiib(K, E, n_sms, pairs, S * (N + 1), False).pairs and E // 128 % 2 == 1
    w = synth.workload("deep", n_layers=1, d_model=d, n_q_heads=Hq, n_kv_heads=Hkv, head_dim=D, tokens_per_frame=N, n_frames=1, bank_capacity=1,
                       prefix_len=3, question_len=0, decode_tokens=0, n_streams=S, frame_model="iid", seed=73)
    p = Pair(w, with_gain=True, with_bias=True, d_ff=d_ff)
    ids = list(range(S))
    p.text(ids, [w.prefix_hidden(s) for s in ids], "prefix")
    p.frame(ids, [w.frame_hidden(0, s) for s in ids], "frame")
    for s in ids:
        p.check_bank(s)
    p.close()
