"""Key tiles of the prefill attention shared by the CTAs of a cluster: every size of cluster that a group can have (the choice is
asked of the library), groups whose rows fill the exchange area and reach out of it, token counts that leave a CTA of the cluster few
rows or none."""
import ctypes as C

import numpy as np
import pytest
import torch

from paper_2503_09387_b200 import binding, synth
from tests.parity import Pair, errors, to_dev, to_f64

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


def _cluster_size(G, D, row_tiles, key_tiles):
    lib = binding.load_library()
    clusters = (C.c_int * 9)(0, 0, *(2 * lib._ZN2vs30prefill_attention_max_clustersEii(D, s) for s in range(2, 9)))
    return lib._ZN2vs15attention_splitEiiiiiiPKi(D, G, row_tiles, key_tiles, 0, torch.cuda.get_device_properties(0).multi_processor_count, clusters)


# streams of a call and its rows: 10, 32, 80, 128 and 160 row tiles, the last one of a stream often ragged
CALLS = ((1, 153), (2, 251), (5, 243), (8, 256), (10, 242))


@pytest.mark.parametrize("G,D,sizes", [(7, 128, [8, 4, 3, 2, 1]), (8, 128, [4, 4, 2, 2, 1]), (5, 128, [8, 6, 3, 2, 1]),
                                       (8, 64, [8, 4, 2, 2, 1]), (7, 64, [8, 4, 3, 2, 1])])
def test_the_cluster_sizes_in_use(G, D, sizes):
    S, d = 10, G * D
    w = synth.workload("deep", n_layers=2, d_model=d, n_q_heads=G, n_kv_heads=1, head_dim=D, tokens_per_frame=5, n_frames=0, bank_capacity=1,
                       prefix_len=3, question_len=0, decode_tokens=0, n_streams=S, frame_model="iid", seed=67)
    p = Pair(w, with_gain=True, max_prefix=1200, max_step_tokens=256)
    used, at = [], [0] * S
    for i, (n, T) in enumerate(CALLS):
        ids = list(range(n))
        tiles = max((at[s] + 63) // 64 for s in ids) + (T + 63) // 64
        used.append(_cluster_size(G, D, n * ((T + 15) // 16), tiles))
        p.text(ids, [synth.normal_bf16(w.seed, synth.TAG_QUESTION, (T, d), 1.0, offset=(i * S + s) * 256 * d) for s in ids], f"{n} x {T} rows")
        for s in ids:
            at[s] += T
    assert used == sizes
    p.check_bank(0)
    p.close()


# rows that no cluster shares (many streams), to the least aligned address that is taken; heads that leave softmax warps idle, several layers' residual.
# Every stream is compared: each is fed the rows of one of seven, in no regular order, so that an entry, row tile or head mixed up with another shows.
@pytest.mark.parametrize("G,D,L,out_dtype", [(7, 128, 2, 1), (8, 128, 1, 0), (1, 128, 2, 0), (3, 64, 2, 1), (8, 64, 1, 0)])
def test_rows_without_peers(G, D, L, out_dtype):
    # (chained layers: flipped roundings of the stored rows reach the next layer's scores, whose size grows with the width -- 7168 wide, one row of
    # the second layer was 5.1e-2 off at a relative RMS of 4.7e-3.  So no wider than 2688, and 2e-2 * sqrt(L), as the deep chain's test has it.)
    S, Hkv, kinds = 60, 3, 7
    d = G * Hkv * D
    w = synth.workload("deep", n_layers=L, d_model=d, n_q_heads=G * Hkv, n_kv_heads=Hkv, head_dim=D, tokens_per_frame=17, n_frames=0, bank_capacity=1,
                       prefix_len=3, question_len=0, decode_tokens=0, n_streams=S, frame_model="iid", seed=71)
    p = Pair(w, with_gain=True, max_prefix=160, max_step_tokens=128, out_dtype=out_dtype, n_oracles=kinds)
    kind = np.concatenate([np.arange(kinds), np.random.default_rng(5).integers(0, kinds, S - kinds)])
    at = 0
    for i, T in enumerate((2, 63, 64, 18)):                   # one to three tiles of keys, ragged row tiles
        assert _cluster_size(G, D, S * Hkv * ((T + 15) // 16), (at + 63) // 64 + (T + 63) // 64) == 1
        x = [synth.normal_bf16(w.seed, synth.TAG_QUESTION, (T, d), 1.0, offset=(i * S + s) * 128 * d) for s in range(kinds)]
        n = S * T * d
        big = torch.full((n + 64,), 7.0, dtype=p.gpu.out_torch_dtype, device="cuda")
        out = big[4:4 + n].view(S, T, d)                      # 16 bytes (fp32) or 8 (bf16) off
        p.gpu.decode_step(list(range(S)), to_dev(np.stack([x[k] for k in kind])), out=out)
        assert torch.all(big[:4] == 7.0) and torch.all(big[4 + n:] == 7.0)
        got = to_f64(out)
        want = [p.ora[s].text_step(synth.bf16_bits_to_f64(x[s])) for s in range(kinds)]
        # Beside the arithmetic's 2e-2 * sqrt(L): with few keys a row is nearly a V row, whose stored elements may have been rounded to the other
        # neighbour, a unit, at most 2^-7 of the largest |v|, apart (with n keys of like weight those average down as 1 / sqrt(n): from nine on a
        # third of a unit, within the arithmetic's).  And half a unit, at most 2^-8 of the element, for rounding to a bf16 output.
        few = (at + np.arange(T) < 8)[:, None]
        for s in range(S):
            ref = want[kind[s]]
            tol = 2e-2 * L ** 0.5 + np.where(few, 2.0 ** -7 * np.max(np.abs(ref)), 0.0) + (0.0 if out_dtype else 2.0 ** -8) * np.abs(ref)
            rel_rms = errors(got[s], ref)[1]
            worst = np.max(np.abs(got[s] - ref) / tol)
            assert worst <= 1.0 and rel_rms <= 1e-2, (T, s, worst, rel_rms)
        at += T
    p.close()
