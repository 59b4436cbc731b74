"""The work a user of this decoder has it do, as cases that can be timed: transcribing one utterance, batches of every
size, a stream through slots, scoring given transcripts step by step, feeding prompts, and the fp32 configuration.

A serving program creates one decoder per model when it starts, sized for its largest batch, and then sees one batch
after the other; so does this file (``_decoder``).  A case fixes the model, the options and the lengths of its
utterances (drawn from ``case["lengths"]``); the seed of ``prepare`` draws the encoder states and the order in which
the utterances arrive.  All sizes follow ``paper_2503_05931_b200.workloads``.
"""
from __future__ import annotations

import functools
import heapq
import math

import numpy as np
import torch

from paper_2503_05931_b200 import binding, streaming
from paper_2503_05931_b200 import workloads as wl

DEVICE = "cuda:0"
MAX_ENC, MAX_DEC = 500, 240               # 40 s of 80 ms frames; 40 s at 6 tokens a second
EOS_ID = 2
# largest batch and most encoder frames of one batch that the program sizes its decoder for
CAPACITY = {"canary24": (512, 150_000), "flash4": (512, 160_000), "tiny": (64, 4_000)}
# how strongly a token calls for its successor, see _weights
SURE = {"canary24": 0.95, "flash4": 0.45, "tiny": 0.0}


def _greedy(name, model, batch, law, lengths, dtype="bf16", cross_kv="dtype", eos=False):
    return {"name": name, "kind": "greedy", "model": model, "dtype": dtype, "batch": batch, "law": law, "lengths": lengths,
            "cross_kv": cross_kv, "eos": eos}


def listed():
    return [
        # a voice command of about two seconds, alone: the smallest call, where launches and latency are everything
        _greedy("command_flash4", "flash4", 1, "lognormal", 26),
        # one ordinary utterance through the deep decoder, as an interactive user sends it
        _greedy("one_canary24", "canary24", 1, "lognormal", 2),
        # a few callers at once, with an end-of-sequence id as a deployed model has one
        _greedy("callers_flash4", "flash4", 12, "lognormal", 3, eos=True),
        # offline transcription: the three bf16 batches of the repository's benchmark
        _greedy("batch64_canary24", "canary24", 64, "lognormal", 20250307),
        _greedy("batch128_flash4", "flash4", 128, "lognormal", 20250308),
        _greedy("batch512_canary24", "canary24", 512, "uniform", 20250309),
        # a large batch with the 8-bit cross-attention store
        _greedy("batch200_e4m3", "canary24", 200, "lognormal", 11, cross_kv="e4m3"),
        # a queue of utterances through continuously refilled slots
        {"name": "stream_flash4", "kind": "stream", "model": "flash4", "dtype": "bf16", "batch": 400, "slots": 96, "law": "lognormal",
         "lengths": 5, "cross_kv": "dtype", "eos": False},
        # scoring given transcripts: the caller feeds the tokens and reads every step's logits
        {"name": "score_canary24", "kind": "steps", "model": "canary24", "dtype": "bf16", "batch": 24, "steps": 12, "law": "lognormal",
         "lengths": 6, "cross_kv": "dtype", "eos": False},
        # a task and language prompt in front of a batch, then the first tokens of the transcripts
        {"name": "prompt_canary24", "kind": "prompt", "model": "canary24", "dtype": "bf16", "batch": 37, "prompt": 9, "steps": 3,
         "law": "lognormal", "lengths": 7, "cross_kv": "dtype", "eos": False},
        # time to the first token of a large batch of long recordings: nearly all cross-attention keys and values
        {"name": "first_token_flash4", "kind": "steps", "model": "flash4", "dtype": "bf16", "batch": 301, "steps": 1, "law": "uniform",
         "lengths": 8, "cross_kv": "dtype", "eos": False},
        # the fp32 configuration of the repository
        _greedy("tiny_fp32", "tiny", 4, "tiny", 20250306, dtype="fp32"),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["greedy", "greedy", "greedy", "stream", "steps", "prompt", "fp32"])
    lengths = rng.randrange(1 << 30)
    if kind == "fp32":
        return {"kind": "greedy", "model": "tiny", "dtype": "fp32", "batch": _log_int(rng, 1, 64), "law": "tiny", "lengths": lengths,
                "cross_kv": "dtype", "eos": False}
    case = {"kind": kind, "model": rng.choice(["canary24", "flash4"]), "dtype": "bf16", "law": "lognormal", "lengths": lengths,
            "cross_kv": "dtype", "eos": False}
    if kind == "greedy":
        case["batch"] = _log_int(rng, 1, 480)
        case["law"] = rng.choice(["lognormal", "lognormal", "uniform"])
        case["eos"] = rng.random() < 0.25
        if case["model"] == "canary24" and not case["eos"]:
            case["cross_kv"] = rng.choice(["dtype", "dtype", "e4m3"])
        if case["eos"]:
            case["model"] = "flash4"
    elif kind == "stream":
        case["model"] = "flash4"
        case["slots"] = _log_int(rng, 4, 256)
        case["batch"] = int(case["slots"] * rng.uniform(1.5, 4.0))
    elif kind == "steps":
        case["batch"] = _log_int(rng, 1, 400)
        case["steps"] = _log_int(rng, 1, 16)
        case["law"] = rng.choice(["lognormal", "uniform"])
    else:
        case["batch"] = _log_int(rng, 1, 96)
        case["prompt"] = _log_int(rng, 2, 24)
        case["steps"] = rng.randint(1, 4)
    return case


def _lengths(case):
    """Encoder frames and output tokens of the case's utterances."""
    _, enc_lens, dec_lens = wl.draw_lengths(np.random.default_rng(case["lengths"]), case["batch"], case["law"])
    return enc_lens, np.minimum(dec_lens, MAX_DEC).astype(np.int32)


class _DeviceNormals:
    """The one method of a numpy generator that ``draw_weights`` calls, with the numbers drawn on the GPU."""

    def __init__(self, seed):
        self.gen = torch.Generator(device=DEVICE).manual_seed(seed)

    def standard_normal(self, size, dtype):
        return torch.randn(size, generator=self.gen, device=DEVICE).cpu().numpy()


def _weights(model, dtype):
    """Random weights, with an output matrix that is sure of most tokens as a trained one is: all but the start token
    have a successor whose output row leans towards their embedding.  The first token, and about one in ten of the
    others, is decided by the audio and the history instead.  (With plain random rows nearly every choice of a token is
    a near-tie among thousands.)"""
    weights = wl.draw_weights(_DeviceNormals(20250305), wl.MODELS[model], dtype)
    tokens = np.random.default_rng(20250305).permutation(wl.MODELS[model]["vocab"])
    before, after = tokens[:-1], tokens[1:]
    after, before = after[before != 1], before[before != 1]
    rows = weights["w_out"]
    sure = np.float32(SURE[model])
    rows[after] = sure * weights["embed"][before] + np.sqrt(1 - sure * sure) * rows[after]
    weights["w_out"] = wl.round_to_bf16(rows) if dtype == "bf16" else rows
    return weights


@functools.lru_cache(maxsize=None)
def _decoder(model, dtype, cross_kv, eos):
    weights = _weights(model, dtype)
    max_batch, max_frames = CAPACITY[model]
    return binding.Decoder(wl.MODELS[model], weights, dtype, max_batch=max_batch, max_total_enc_frames=max_frames, max_enc_len=MAX_ENC,
                           max_dec_len=MAX_DEC, eos_id=EOS_ID if eos else -1, cross_kv_e4m3=cross_kv == "e4m3", device=DEVICE)


def prepare(case, seed):
    model = wl.MODELS[case["model"]]
    dec = _decoder(case["model"], case["dtype"], case["cross_kv"], case["eos"])
    rng = np.random.default_rng(seed)
    gen = torch.Generator(device=DEVICE).manual_seed(seed)
    enc_lens, dec_lens = _lengths(case)
    order = rng.permutation(case["batch"])
    enc_lens, dec_lens = enc_lens[order].copy(), dec_lens[order].copy()
    # the states of one recording have a component in common (its speaker, its subject) beside what changes from frame to frame
    enc = 0.8 * torch.randn((int(enc_lens.sum()), model["d_enc"]), generator=gen, device=DEVICE)
    common = 0.6 * torch.randn((case["batch"], model["d_enc"]), generator=gen, device=DEVICE)
    enc += common.repeat_interleave(torch.from_numpy(enc_lens).to(DEVICE), dim=0)
    enc = enc.to(dec.tdtype)
    state = {"case": case, "dec": dec, "enc": enc, "enc_lens": enc_lens, "dec_lens": dec_lens}
    tokens = lambda *shape: torch.randint(0, model["vocab"], shape, generator=gen, device=DEVICE, dtype=torch.int32)
    if case["kind"] in ("steps", "prompt"):
        batch, steps = case["batch"], case["steps"]
        state["tokens"] = tokens(steps, batch)
        state["logits"] = torch.empty((steps + 1, batch, model["vocab"]), dtype=torch.float32, device=DEVICE)
        state["next"] = torch.empty((steps + 1, batch), dtype=torch.int32, device=DEVICE)
        if case["kind"] == "prompt":
            state["prompt"] = tokens(batch, case["prompt"])
    elif case["kind"] == "stream":
        state["host_tokens"] = torch.empty((case["batch"], MAX_DEC), dtype=torch.int32).pin_memory()
        state["host_lens"] = torch.zeros(case["batch"], dtype=torch.int32).pin_memory()
    return state


def run(state):
    case, dec = state["case"], state["dec"]
    if case["kind"] == "stream":
        tokens, _ = streaming.decode_stream(dec, state["enc"], state["enc_lens"], state["dec_lens"], case["slots"],
                                            tokens_out=state["host_tokens"], out_lens=state["host_lens"])
        return {"tokens": np.concatenate(tokens), "lens": state["host_lens"]}
    dec.precompute_cross_kv(state["enc"], state["enc_lens"])
    if case["kind"] == "greedy":
        tokens, lens = dec.greedy_decode(state["dec_lens"])
        return {"tokens": tokens, "lens": lens}
    logits, chosen, steps = state["logits"], state["next"], case["steps"]
    first = 0
    if case["kind"] == "prompt":
        dec.prefill(state["prompt"], logits[steps], chosen[steps])
        first = 1
    for t in range(steps):
        dec.step(state["tokens"][t], None, logits[t], chosen[t])
    used = steps + first
    return {"logits": logits[:used], "next": chosen[:used]}


def _stream_steps(dec_lens, slots):
    """Steps of a stream whose utterances enter in order as slots become free."""
    ends = []
    for n in dec_lens:
        start = heapq.heappop(ends) if len(ends) == slots else 0
        heapq.heappush(ends, start + int(n))
    return max(ends)


def work(case):
    """Weights once per step that reads them, every row's keys and values once per step and layer, the encoder states
    in and the cross-attention keys and values out once, and the results."""
    m = wl.MODELS[case["model"]]
    e = 2 if case["dtype"] == "bf16" else 4
    ec = 1 if case["cross_kv"] == "e4m3" else e
    layers, d, f, v, d_enc = m["n_layers"], m["d_model"], m["d_ffn"], m["vocab"], m["d_enc"]
    enc_lens, dec_lens = (a.astype(np.int64) for a in _lengths(case))
    params = layers * (6 * d * d + 2 * d * f) + v * d
    frames = int(enc_lens.sum())
    total = e * (frames * d_enc + layers * 2 * d * d_enc) + ec * frames * layers * 2 * d
    flops = 4 * frames * d_enc * layers * d
    if case["kind"] in ("greedy", "stream"):
        rows = int(dec_lens.sum())
        passes = int(dec_lens.max()) if case["kind"] == "greedy" else _stream_steps(dec_lens, case["slots"])
        cross = int((dec_lens * enc_lens).sum())
        own = int((dec_lens * (dec_lens + 1) // 2).sum())
        total += 4 * rows
        heads = rows
    else:
        prompt = case.get("prompt", 0)
        length = prompt + case["steps"]
        rows, passes = case["batch"] * length, case["steps"] + (1 if prompt else 0)
        # a prompt pass reads an utterance's cross-attention keys and values once for all of its positions
        cross = passes * frames
        own = case["batch"] * (length * (length + 1) - prompt * (prompt + 1)) // 2 + case["batch"] * prompt
        heads = case["batch"] * passes
        total += 4 * heads * v
    total += passes * e * params + layers * 2 * d * (ec * cross + e * own)
    flops += 2 * rows * (params - v * d) + 2 * heads * v * d + 4 * d * layers * (cross + own)
    return {"bytes": int(total), "flops": int(flops)}


def tolerance(case):
    # tokens: greedy choices are the same but for near-ties, after which an utterance goes its own way
    return {"rel": 1e-5 if case["dtype"] == "fp32" else 1e-2, "differ": 0.01}
