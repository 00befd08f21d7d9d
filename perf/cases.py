"""The measured cases of this library: what a program that generates audio with it calls, over the range of sizes that
such programs use.  Shapes are those of `paper_1802_08435_b200/synth.py` (H = 896 dense, H = 2048 with 96 % of the blocks
of R, O1, O3 pruned, 64-value conditioning frames held for 120 samples, 24 kHz), with weights, frames and Philox key made
from the seed.  Every case goes through the ctypes binding's public calls."""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_1802_08435_b200 import binding as B
from paper_1802_08435_b200 import synth

HOP = synth.HOP
D = synth.COND_DIM

# parameters of a step (Eq. 2 and the two heads), multiply-adds per row and step
PARAMS_896 = 3 * 896 * 896 + 3 * 896 * 3 + 2 * 448 * 448 + 2 * 256 * 448
PARAMS_FUSED = 3 * 896 * 896 + 3 * 896 * 12 + 2 * 448 * 448 + 2 * 64 * 448
PARAMS_2048_PRUNED = (3 * 2048 * 2048 + 2 * 1024 * 1024) // 25 + 3 * 2048 * 3 + 2 * 256 * 1024
NET_PARAMS = 10 * (3 * 768 * 384 + 384 * 768) + 16 * 768 + 768 * 64


def listed():
    return [
        # live playback: one voice in 5 ms pieces (one conditioning frame each), the state carried from call to call
        dict(name="stream_5ms", kind="stream", dtype="bf16", chunk=120, chunks=8),
        # one second of one voice in one call: the library's headline use
        dict(name="voice_1s", kind="sample", dtype="bf16", batch=1, steps=24000),
        # the same model kept in fp32, a short prompt
        dict(name="voice_f32_50ms", kind="sample", dtype="f32", batch=1, steps=1200),
        # fp32 models, four voices in step
        dict(name="voices4_f32", kind="sample", dtype="f32", batch=4, steps=333),
        # pruned model, 4 x 4 blocks, a quarter of a second
        dict(name="sparse_4x4", kind="sparse", block_rows=4, block_cols=4, steps=6000),
        # an utterance folded into 16 interleaved rows, advanced together and unfolded
        dict(name="subscale_fold16", kind="fold", rows=16, total=24000),
        # a small server: four utterances from host buffers to host buffers
        dict(name="voices4_host", kind="host", dtype="bf16", batch=4, steps=6000),
        # a mid-sized and ragged batch of utterances
        dict(name="voices37", kind="sample", dtype="bf16", batch=37, steps=1501),
        # bulk synthesis: a full batch of utterances
        dict(name="voices256", kind="sample", dtype="bf16", batch=256, steps=2400),
        # two samples per step from one state (four 4-bit softmaxes per sample)
        dict(name="fused2x", kind="fused", steps=6002),
        # subscale generation, 16 dependent rows conditioned through the ten-layer network: four seconds of audio
        dict(name="subscale_net", kind="net", rows=16, positions=6000, chunk=128, lag=256),
        # scoring given audio: the samples fed back are supplied, gates, states and logits of every step are read
        dict(name="score8", kind="score", dtype="bf16", batch=8, steps=400),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["stream", "sample", "sample", "sample", "sample", "f32", "sparse", "fold", "host", "fused", "net", "score"])
    if kind == "stream":
        return dict(kind="stream", dtype="bf16", chunk=_log(rng, 60, 480), chunks=rng.randint(2, 12))
    if kind in ("sample", "host"):
        batch = _log(rng, 1, 256) if kind == "sample" else _log(rng, 1, 16)
        top = 24000 if batch == 1 else 6000 if batch <= 16 else 2400
        return dict(kind=kind, dtype="bf16", batch=batch, steps=_log(rng, 240, top))
    if kind == "f32":
        batch = rng.choice([1, 1, 2, 3, 4, 6, 8])
        return dict(kind="sample", dtype="f32", batch=batch, steps=_log(rng, 200, 3000 if batch == 1 else 500))
    if kind == "sparse":
        br, bc = rng.choice([(4, 4), (4, 4), (16, 1)])
        return dict(kind="sparse", block_rows=br, block_cols=bc, steps=_log(rng, 400, 6000))
    if kind == "fold":
        rows = rng.choice([2, 4, 8, 16])
        return dict(kind="fold", rows=rows, total=rows * _log(rng, 200, 3000))
    if kind == "fused":
        return dict(kind="fused", steps=_log(rng, 200, 12000))
    if kind == "net":
        rows = rng.choice([4, 8, 16])
        return dict(kind="net", rows=rows, positions=_log(rng, 400, 6000), chunk=128, lag=256)
    return dict(kind="score", dtype="bf16", batch=_log(rng, 1, 48), steps=_log(rng, 100, 400))


class _State:
    """What a program holds between calls; the library's handles are given back with it."""

    def __init__(self):
        self.model = self.net = None

    def __del__(self):
        if self.net is not None:
            B.wrnn_subscale_net_destroy(self.net)
        if self.model is not None:
            B.wrnn_destroy(self.model)


def _rows_steps(case):
    k = case["kind"]
    if k == "stream":
        return 1, case["chunk"] * case["chunks"]
    if k == "fold":
        return case["rows"], case["total"] // case["rows"]
    if k == "net":
        return case["rows"], case["positions"]
    return case.get("batch", 1), case["steps"]


def _frames(case):
    rows, steps = _rows_steps(case)
    return (rows * steps if case["kind"] in ("fold", "net") else steps) // HOP + 1


def prepare(case, seed):
    s = _State()
    s.case, k = case, case["kind"]
    s.key = (synth.SEED_SAMPLING + 7919 * seed) & (2 ** 63 - 1)
    rows, steps = _rows_steps(case)
    masks = None
    if k == "sparse":
        block = (case["block_rows"], case["block_cols"])
        w = synth.make_weights(2048, seed_w=seed, seed_b=seed + 1)
        masks = synth.make_block_masks(2048, 0.96, seed=seed + 2, block=block)
        w = synth.rescale_kept(w, masks)
        s.model = B.wrnn_create(w, "bf16", masks, max_batch=1, block=block)
    elif k == "fused":
        s.model = B.wrnn_create(synth.make_weights(896, n_inputs=12, n_logits=64, seed_w=seed, seed_b=seed + 1), "bf16", variant=1)
    else:
        s.model = B.wrnn_create(synth.make_weights(896, seed_w=seed, seed_b=seed + 1), case.get("dtype", "bf16"), max_batch=rows)
    cond = synth.make_cond(rows, _frames(case), seed=seed + 3)
    dev = torch.device("cuda")
    if k == "host":
        s.cond = torch.from_numpy(cond).pin_memory().numpy()
        s.out = torch.zeros((rows, steps), dtype=torch.int16).pin_memory().numpy()
        return s
    s.cond = torch.from_numpy(cond).to(dev)
    if k == "stream":
        s.out = torch.zeros((case["chunks"], 1, case["chunk"]), dtype=torch.int16, device=dev)
        s.h = torch.zeros((1, 896), device=dev)
        s.c = torch.zeros(1, dtype=torch.uint8, device=dev)
        s.f = torch.zeros(1, dtype=torch.uint8, device=dev)
    elif k == "fold":
        s.out = torch.zeros(case["total"], dtype=torch.int16, device=dev)
    elif k == "net":
        s.net = B.wrnn_subscale_net_create(synth.make_subscale_net(rows, seed=seed + 4))
        s.out = torch.zeros(rows * steps, dtype=torch.int16, device=dev)
    elif k == "fused":
        s.ab = torch.zeros((2, steps), dtype=torch.int16, device=dev)
        s.out = torch.zeros(2 * (steps - 2), dtype=torch.int16, device=dev)
    elif k == "score":
        r = np.random.default_rng(seed + 5)
        # audio of a voice: a few low tones with noise, as the bytes that are fed back
        t = np.arange(steps)[None, :] / 24000.0
        x = sum(np.sin(2 * np.pi * r.uniform(80, 900, (rows, 1)) * t + r.uniform(0, 6, (rows, 1))) for _ in range(4))
        x = np.clip((x * 6000 + r.standard_normal((rows, steps)) * 400), -32768, 32767).astype(np.int64) + 32768
        s.cf = torch.from_numpy((x >> 8).astype(np.uint8)).to(dev)
        s.ff = torch.from_numpy((x & 255).astype(np.uint8)).to(dev)
        s.co, s.fo = torch.zeros_like(s.cf), torch.zeros_like(s.ff)
        s.gates = torch.zeros((steps, rows, 3 * 896), device=dev)
        s.hs = torch.zeros((steps, rows, 896), device=dev)
        s.logits = torch.zeros((steps, rows, 2, 256), device=dev)
    else:
        s.out = torch.zeros((rows, steps), dtype=torch.int16, device=dev)
    return s


def run(s):
    case, k = s.case, s.case["kind"]
    rows, steps = _rows_steps(case)
    if k == "stream":
        s.h.zero_(), s.c.fill_(128), s.f.zero_()
        for i in range(case["chunks"]):
            B.wrnn_sample(s.model, s.cond, case["chunk"], 1, s.key, s.out[i], h=s.h, c_prev=s.c, f_prev=s.f, step0=i * case["chunk"])
        return s.out, s.h
    if k == "host":
        B.wrnn_sample_host(s.model, s.cond, steps, rows, s.key, s.out)
    elif k == "fold":
        B.wrnn_sample_subscale(s.model, s.cond, case["total"], rows, s.key, s.out)
    elif k == "net":
        B.wrnn_sample_subscale_net(s.model, s.net, s.cond, 128, case["chunk"], case["lag"], rows * steps, s.key, s.out)
    elif k == "fused":
        B.wrnn_fs2_sample(s.model, s.cond, steps, s.key, s.ab)
        B.wrnn_fs2_unfold(s.ab, steps, s.out)
    elif k == "score":
        B.wrnn_step_teacher_forced(s.model, s.cond, steps, rows, s.key, s.cf, s.ff, s.co, s.fo, dbg_gates=s.gates, dbg_h=s.hs,
                                   dbg_logits=s.logits)
        return s.co, s.fo, s.gates, s.hs, s.logits
    else:
        B.wrnn_sample(s.model, s.cond, steps, rows, s.key, s.out)
    return s.out


def work(case):
    """Weights, frames and what is fed back read once, samples (and, for scoring, the dumps) written once; two operations
    per weight, row and step."""
    k = case["kind"]
    rows, steps = _rows_steps(case)
    params = PARAMS_2048_PRUNED if k == "sparse" else PARAMS_FUSED if k == "fused" else PARAMS_896
    bytes_ = params * (4 if case.get("dtype") == "f32" else 2) + rows * _frames(case) * D * 4
    bytes_ += rows * steps * (4 if k == "fused" else 2)
    flops = 2.0 * params * rows * steps
    if k == "net":
        bytes_ += 2 * NET_PARAMS
        flops += 2.0 * NET_PARAMS * rows * steps
    if k == "score":
        bytes_ += rows * steps * 4 * (4 * 896 + 512)
    return {"bytes": bytes_, "flops": flops}


def tolerance(case):
    """Measured against the any-shape kernel (plain fp32 sums in another order) over three seeds of every case: states and
    gates within 7e-7 (2-norm), logits within 3.4e-6 (largest 2.2e-5), and 0 to 9e-5 of the drawn samples different.  A draw
    whose uniform lies within rounding of a CDF boundary goes the other way; the stream then falls back in step, because
    the state forgets one neighbouring symbol within a few steps.  Short calls: room for two such draws."""
    rows, steps = _rows_steps(case)
    return {"rel": 1.5e-5, "max": 1e-4, "differ": min(0.009, max(4e-4, 2.5 / (rows * steps)))}
