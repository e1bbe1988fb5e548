"""The calls a program built on this package makes, as measured cases.

A streaming video assistant keeps one handle per backbone and makes four kinds of call on it: it feeds frames as they
arrive (one stream or many in a call), feeds a whole clip in chunks of frames, prefills a question, and generates the
answer token by token.  A batch job may also recompute the bank from its carriers alone.  The two backbones are the
Qwen2-7B shape the package is configured for throughout and a small generic one with 64-wide heads.  Handles come in the
two forms the package has: the attention path alone (stacked through a residual stream, fp32 rows) and full decoder
layers with the language-model head (query/key/value biases and norm gains as such checkpoints bring them, bf16 rows).

Every state is a stream in mid-flight: prompt prefix in place, the bank filled by earlier frames (full, for frame and
clip calls, so that every frame evicts), inputs drawn from the seed with the package's own recipe -- weights
N(0, 0.02^2), scaled down by depth where they write to the residual stream of a full decoder; frames a slowly drifting
scene vector plus N(0, 0.5^2) token noise; text rows N(0, 1).
"""
import math

import torch

from paper_2503_09387_b200 import binding

BACKBONES = {
    "qwen2_7b": dict(d=3584, hq=28, hkv=4, hd=128, dff=18944, vocab=152064),
    "small": dict(d=1024, hq=16, hkv=4, hd=64, dff=4096, vocab=32000),
}
ANSWER = 128            # tokens of one answer: the tail a token step walks through before the turn ends
FILL_TOKENS = 8         # visual tokens of the frames that fill the bank beforehand
SHAPE = dict(backbone="qwen2_7b", layers=1, full=False, streams=1, tokens=169, frames=1, text=0, bank=64, fill=64, prefix=64,
             policy=0)


def _case(name, kind, **kw):
    c = dict(SHAPE, name=name, kind=kind)
    c.update(kw)
    return c


def listed():
    return [
        # the package's headline workload: one attention layer at the Qwen2-7B shape, a live stream of 169-token frames
        _case("frame_1layer", "frame"),
        # ... and the answer tokens that follow; the smallest call there is, all latency and launches
        _case("token_1layer", "token"),
        # the same attention path through all 28 layers, a long bank: live frames, a question, answer tokens
        _case("frame_28layers", "frame", layers=28, bank=512, fill=512),
        _case("question_28layers", "text", layers=28, bank=512, fill=512, text=32),
        _case("token_28layers", "token", layers=28, bank=512, fill=512),
        # sixteen viewers served by one call: frames of 196 tokens, then their answers side by side
        _case("frame_16streams", "frame", streams=16, tokens=196, bank=1024, fill=1024),
        _case("token_16streams", "token", streams=16, tokens=196, bank=1024, fill=1024),
        # offline clip, eight frames to a call
        _case("clip_1layer", "clip", frames=8),
        # the whole model of the paper's serving numbers (28 decoder layers and the head): a live frame of 210 tokens,
        # an answer token with its logits, a clip
        _case("model_frame", "frame", layers=28, full=True, tokens=210, bank=128, fill=128),
        _case("model_token", "token", layers=28, full=True, bank=128, fill=128),
        _case("model_clip", "clip", layers=28, full=True, frames=16, bank=128, fill=128),
        # a small model, odd sizes: the bank's carriers re-run without their stored keys and values
        _case("small_carriers", "carriers", backbone="small", layers=6, full=True, tokens=75, bank=117, fill=101, prefix=19),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more call of the ranges above: 1 to 28 layers of either backbone and form, frames of 49 to 255 tokens, banks of
    16 to 1024 carriers, questions of 2 to 192 tokens, clips of 2 to 24 frames, 1 to 24 streams in a call."""
    largest = _cost(listed()[10])
    while True:
        kind = rng.choice(["frame", "frame", "token", "token", "text", "clip", "carriers"])
        full = rng.random() < 0.5
        bank = _log_int(rng, 16, 1024)
        c = dict(SHAPE, kind=kind, backbone="qwen2_7b" if rng.random() < 0.75 else "small", full=full,
                 layers=_log_int(rng, 1, 28), tokens=rng.randint(49, 255), bank=bank, prefix=rng.randint(8, 160),
                 policy=1 if rng.random() < 0.2 else 0)
        # a bank still filling up is met by the calls that leave it as it is
        c["fill"] = bank if kind in ("frame", "clip") else rng.randint(max(1, bank // 4), bank)
        if kind in ("frame", "token", "text") and rng.random() < 0.4:
            c["streams"] = _log_int(rng, 2, 24)
        if kind == "text":
            c["text"] = _log_int(rng, 2, 192)
        if kind == "clip":
            c["frames"] = _log_int(rng, 2, 24)
        if _cost(c) <= largest and _rows(c) <= 4096:
            return c


# ---- sizes ------------------------------------------------------------------------------------------------------------
def _rows(c):
    return {"frame": c["streams"] * (c["tokens"] + 1), "clip": c["frames"] * (c["tokens"] + 1), "text": c["streams"] * c["text"],
            "token": c["streams"], "carriers": c["fill"]}[c["kind"]]


def _keys(c):
    """Keys a row of the call attends to, on average."""
    n = {"frame": (c["tokens"] + 2) / 2, "clip": (c["tokens"] + 2) / 2, "text": (c["text"] + 1) / 2,
         "token": (ANSWER + 1) / 2, "carriers": (c["fill"] + 1) / 2}[c["kind"]]
    return c["prefix"] + n + (0 if c["kind"] == "carriers" else c["fill"])


def work(case):
    b = BACKBONES[case["backbone"]]
    d, q, kv = b["d"], b["hq"] * b["hd"], b["hkv"] * b["hd"]
    rows, keys, L = _rows(case), _keys(case), case["layers"]
    matrix = (q + 2 * kv) * d + ((d * q + 3 * d * b["dff"]) if case["full"] else 0)
    # stored keys and values: the prompt's and the bank's, and the answer so far of a token step
    stored = case["prefix"] + (0 if case["kind"] == "carriers" else case["fill"]) + (ANSWER / 2 if case["kind"] == "token" else 0)
    nbytes = L * (matrix * 2 + case["streams"] * stored * kv * 4) + rows * d * 2 + rows * q * (2 if case["full"] else 4)
    flops = L * (2 * rows * matrix + 4 * rows * keys * q)
    if case["full"] and case["kind"] == "token":
        nbytes += b["vocab"] * d * 2 + rows * b["vocab"] * 4
        flops += 2 * rows * d * b["vocab"]
    return {"bytes": nbytes, "flops": flops}


def _cost(c):
    w = work(c)
    return max(w["bytes"] / 6.5e12, w["flops"] / 1.4e15)


def tolerance(case):
    # bf16 operands and a bf16 residual stream.  One layer's attention rows agree to a few 1e-3 of their norm; in full
    # decoder layers the flipped roundings of the stored stream and activations add up like a random walk over the
    # layers (two summation orders of this package's own projections: 0.8e-2 after 6 layers, 1.6e-2 after 28)
    if case["full"]:
        return {"rel": min(2.5e-2, 5e-3 * math.sqrt(1 + case["layers"])), "max": 0.3}
    return {"rel": 5e-3 if case["layers"] == 1 else 1e-2, "max": 0.2}


# ---- a program's state and its calls --------------------------------------------------------------------------------------
class _Program:
    pass


def prepare(case, seed):
    c, b = case, BACKBONES[case["backbone"]]
    dev = torch.device("cuda", 0)
    g = torch.Generator(device=dev)
    g.manual_seed(seed)

    def normal(*shape, std=1.0, mean=0.0):
        return torch.empty(shape, dtype=torch.bfloat16, device=dev).normal_(mean, std, generator=g)

    L, S, N, d, q = c["layers"], c["streams"], c["tokens"], b["d"], b["hq"] * b["hd"]
    e_out = q + 2 * b["hkv"] * b["hd"]
    w = [normal(e_out, d, std=0.02) for _ in range(L)]
    bias = gain = block = lm = None
    if c["full"]:
        bias = [normal(e_out, std=0.1) for _ in range(L)]
        gain = [normal(d, std=0.1, mean=1.0) for _ in range(L)]
        res = 0.02 / math.sqrt(2 * L)          # matrices that write to the residual stream: scaled by depth, as such models are
        block = dict(w_o=[normal(d, q, std=res) for _ in range(L)], w_gate=[normal(b["dff"], d, std=0.02) for _ in range(L)],
                     w_up=[normal(b["dff"], d, std=0.02) for _ in range(L)], w_down=[normal(d, b["dff"], std=res) for _ in range(L)],
                     norm2_w=[normal(d, std=0.1, mean=1.0) for _ in range(L)])
        lm = (normal(b["vocab"], d, std=0.02), normal(d, std=0.1, mean=1.0))
    multi = L > 1 or c["full"]
    cfg = binding.make_config(L, d, b["hq"], b["hkv"], b["hd"], N, max_prefix=c["prefix"], max_text=max(ANSWER, c["text"]),
                              bank_capacity=c["bank"], n_streams=S, max_step_tokens=max(64, c["text"], c["prefix"]),
                              evict_policy=c["policy"], use_rmsnorm=int(multi), residual=int(multi), out_dtype=0 if c["full"] else 1,
                              max_chunk_frames=c["frames"], d_ff=b["dff"] if c["full"] else 0, vocab=b["vocab"] if c["full"] else 0)
    p = _Program()
    p.kind, p.full, p.ids, p.fill = c["kind"], c["full"], list(range(S)), c["fill"]
    p.batch = binding.StreamBatch(cfg, w, biases=bias, norm_weights=gain, block=block, lm=lm)
    # the prompt, then the frames seen so far
    p.batch.decode_step(p.ids, normal(S, c["prefix"], d))
    scene = normal(S, 1, d).float()
    noise = [normal(S, FILL_TOKENS, d, std=0.5) for _ in range(4)]

    def drift(scene):
        return 0.9 * scene + math.sqrt(1 - 0.81) * normal(S, 1, d).float()

    for t in range(c["fill"]):
        scene = drift(scene)
        p.batch.frame_prefill(p.ids, (scene + noise[t % 4]).bfloat16().contiguous(), want_out=False)
    # what comes next: some inputs to go round, so that no call sees the rows of the one before
    p.inputs, p.step, p.tail = [], 0, 0
    for _ in range(2 if c["kind"] == "clip" else 4):
        if c["kind"] == "frame":
            scene = drift(scene)
            p.inputs.append((scene + normal(S, N, d, std=0.5)).bfloat16().contiguous())
        elif c["kind"] == "clip":
            clip = []
            for _ in range(c["frames"]):
                scene = drift(scene)
                clip.append((scene[0] + normal(N, d, std=0.5)).bfloat16())
            p.inputs.append(torch.stack(clip).contiguous())
        elif c["kind"] == "text":
            p.inputs.append(normal(S, c["text"], d))
        elif c["kind"] == "token":
            p.inputs.append(normal(S, 1, d))
        else:
            p.inputs.append(None)
    return p


def run(p):
    x = p.inputs[p.step % len(p.inputs)]
    p.step += 1
    if p.kind == "frame":
        return p.batch.frame_prefill(p.ids, x)
    if p.kind == "clip":
        return p.batch.frame_prefill_chunk(0, x)
    if p.kind == "carriers":
        return p.batch.bank_forward(0, p.fill)
    if p.kind == "text":
        out = p.batch.decode_step(p.ids, x)
        p.batch.end_turn(p.ids)
        return out
    # an answer token; the turn ends after ANSWER of them
    if p.tail == ANSWER:
        p.batch.end_turn(p.ids)
        p.tail = 0
    out = p.batch.decode_step(p.ids, x)
    p.tail += 1
    if not p.full:
        return out
    # (the greedy token comes with the logits; it is theirs to decide, a near tie either way, so the logits stand for it)
    logits, _ = p.batch.lm_head(out.view(len(p.ids), -1))
    return out, logits
