"""The work whose speed this repository is judged by: calls of the public entry points (dc_decode_chunk,
dc_decode_batch, dc_decode_batch_host, dc_decode_wavefront) over the networks of dc_workloads, as a
speech server or an offline renderer issues them.

A case names a network, an entry point, the number of streams of one call and the frames that each
stream presents; with "ragged" the streams of a call present different numbers of frames (a turn that
ends, a session that has just begun).  The model is loaded once per network and kept, with room for the
largest batch, as a serving process keeps it; streams come from a pool of open sessions and are reset
when a new session takes one over.  A streaming case starts behind the retained history, where a
session spends nearly all of its life.
"""
import math

import numpy as np
import torch

import dc_workloads as wl
import paper_2609_35115_b200 as dc

MAX_STREAMS = 32
ROUNDS = 4                      # distinct inputs that the passes over one state cycle through

NETS = {
    "conv": wl.CONFIGS["cfg1"],                     # causal conv stack, fp32
    "flow_small": wl.CONFIGS["cfg2"],               # small bf16 flow decoder
    "flow": wl.CONFIGS["cfg3"],                     # Token2Wav-sized bf16 flow decoder (cfg5 is the same network)
    "flow_guided": wl.EXTRA_CONFIGS["cfg3_guided"],  # ... with classifier-free guidance
    "flow_prompt": wl.EXTRA_CONFIGS["cfg3_paper"],  # ... with a kept prompt, a short window and look-ahead frames
    "vocoder": wl.CONFIGS["cfg4"],                  # fp32 vocoder tail with inverse STFT
    "token2wav": wl.EXTRA_CONFIGS["token2wav"],     # flow decoder and vocoder tail in one call
}


def listed():
    def case(name, net, call, streams=1, frames=None, ragged=False):
        return {"name": name, "net": net, "call": call, "streams": streams, "frames": frames or NETS[net].f_chunk, "ragged": ragged}

    return [
        # the smallest call: one session of the conv stack, latency and launches only
        case("conv_chunk", "conv", "chunk"),
        # one interactive session, a full chunk per call: the latency that a listener waits for
        case("flow_small_chunk", "flow_small", "chunk"),
        case("flow_chunk", "flow", "chunk"),
        # ... at the operating point with a voice prompt: 302 kept frames, 100 retained, 6 of look-ahead
        case("flow_prompt_chunk", "flow_prompt", "chunk", frames=56),
        # a lightly loaded server: a few sessions, each at a chunk boundary of its own
        case("flow_batch7_ragged", "flow", "batch", streams=7, ragged=True),
        # a server whose requests arrive in page-locked host memory
        case("flow_host16", "flow", "batch_host", streams=16),
        # a fully loaded server
        case("flow_batch32", "flow", "batch", streams=32),
        # offline rendering of 20 s of audio from one utterance whose features are all there
        case("flow_offline_20s", "flow", "wavefront", frames=1000),
        # the vocoder tail on its own: the last, odd piece of a turn; eight sessions
        case("vocoder_chunk", "vocoder", "chunk"),
        case("vocoder_batch8_ragged", "vocoder", "batch", streams=8, ragged=True),
        # the whole decoder, features in and PCM out: one listener, and a full server
        case("token2wav_chunk", "token2wav", "chunk"),
        case("token2wav_batch32", "token2wav", "batch", streams=32),
    ]


def draw(rng):
    net = rng.choice(["conv", "flow_small", "flow", "flow", "flow_guided", "flow_prompt", "vocoder", "vocoder", "token2wav", "token2wav"])
    cfg = NETS[net]
    call = rng.choice(["chunk", "batch", "batch", "batch_host"] + (["wavefront"] if net in ("flow_small", "flow") else []))
    streams = 1
    if call in ("batch", "batch_host"):
        most = 16 if net == "flow_guided" else MAX_STREAMS
        streams = int(round(math.exp(rng.uniform(math.log(2), math.log(most)))))
    if call == "wavefront":
        frames = int(round(math.exp(rng.uniform(math.log(50), math.log(1000)))))
    else:
        full = cfg.f_chunk + cfg.f_lookahead
        frames = full if streams > 1 and rng.random() < 0.5 else int(round(math.exp(rng.uniform(0.0, math.log(full)))))
    return {"net": net, "call": call, "streams": streams, "frames": frames, "ragged": streams > 1 and rng.random() < 0.5}


def frame_counts(case):
    """Frames presented by each stream of one call."""
    T, n = case["frames"], case["streams"]
    return [1 + int(T * ((0.98 + 0.618034 * i) % 1.0)) if case["ragged"] else T for i in range(n)]


def history_frames(cfg):
    """Frames a session has behind it: the prompt and the retained window are full."""
    if cfg.pipeline in ("flow", "token2wav"):
        return math.ceil((cfg.f_prompt + cfg.kv_cap) / cfg.f_chunk) * cfg.f_chunk
    return cfg.f_chunk


# ---- what a serving process keeps: one model per network, a pool of open sessions ----------------------------------------

_models = {}
_idle = {}


def model_of(net):
    if net not in _models:
        cfg = NETS[net]
        weights = wl.make_weights(cfg, np.random.default_rng(cfg.seed))
        _models[net] = dc.Model(cfg, weights, max_batch=MAX_STREAMS)
        _idle[net] = []
    return _models[net]


class State:
    """The sessions of one case and the inputs and outputs of their calls."""

    def __init__(self, case):
        self.net, self.call = case["net"], case["call"]
        self.model = model_of(self.net)
        idle = _idle[self.net]
        self.streams = [idle.pop() if idle else self.model.open_stream() for _ in range(case["streams"])]
        self.feats, self.outs, self.at = [], None, 0
        for s in self.streams:
            s.reset()

    def __del__(self):
        _idle[self.net].extend(self.streams)


def prepare(case, seed):
    cfg, n = NETS[case["net"]], case["streams"]
    st = State(case)
    gen = torch.Generator(device="cuda").manual_seed(seed)

    def noise(*shape):
        return torch.randn(*shape, generator=gen, device="cuda")

    counts = frame_counts(case)
    if case["call"] != "wavefront":
        past = torch.empty(n, cfg.f_chunk, cfg.out_per_frame, device="cuda")
        for _ in range(history_frames(cfg) // cfg.f_chunk):
            dc.decode_batch(st.model, st.streams, noise(n, cfg.f_chunk, cfg.in_dim), past)
    if case["call"] in ("chunk", "wavefront"):
        st.feats = [noise(counts[0], cfg.in_dim) for _ in range(ROUNDS)]
        return st
    committed = [min(T, cfg.f_chunk) for T in counts]
    host = case["call"] == "batch_host"

    def blank(*shape):
        return torch.zeros(*shape).pin_memory() if host else torch.zeros(*shape, device="cuda")

    for _ in range(ROUNDS):
        x = [noise(T, cfg.in_dim) for T in counts] if case["ragged"] else noise(n, counts[0], cfg.in_dim)
        if host:
            x = [t.cpu().pin_memory() for t in x] if case["ragged"] else x.cpu().pin_memory()
        st.feats.append(x)
    st.outs = [blank(T, cfg.out_per_frame) for T in committed] if case["ragged"] else blank(n, committed[0], cfg.out_per_frame)
    return st


def run(st):
    feats = st.feats[st.at % ROUNDS]
    st.at += 1
    if st.call == "chunk":
        return st.streams[0].decode_chunk(feats)
    if st.call == "wavefront":                      # a new utterance on an open session
        st.streams[0].reset()
        return st.streams[0].decode_wavefront(feats)
    if st.call == "batch_host":
        dc.decode_batch_host(st.model, st.streams, feats, st.outs)
    else:
        dc.decode_batch(st.model, st.streams, feats, st.outs)
    return st.outs


# ---- the least work of one pass ------------------------------------------------------------------------------------------

def _flow_work(cfg, chunks):
    """chunks: (frames presented, frames of history attended) of every chunk that the call decodes."""
    C, m, S = cfg.hidden, cfg.mel_dim, cfg.n_steps
    passes = 2 if cfg.cfg_scale else 1
    weights = 2 * m * C + len(cfg.dilations) * 3 * C * C + cfg.n_attn_layers * 4 * C * C + C * m
    flops = bytes_ = 0
    for T, carried in chunks:
        keys = carried + T
        flops += passes * S * (2 * T * weights + cfg.n_attn_layers * 4 * T * keys * C)
        bytes_ += passes * S * cfg.n_attn_layers * 2 * keys * C * 2              # keys and values: carried ones read, new ones written
        bytes_ += passes * S * len(cfg.dilations) * 2 * 2 * max(cfg.dilations) * C * 2   # conv left context, read and written
        bytes_ += 4 * T * (2 * m + m)
    return bytes_ + 2 * weights, flops


def _f32_work(cfg, counts):
    """Layers as (frames per chunk frame, multiply-adds per frame); the weights are read once for all the streams."""
    if cfg.pipeline == "conv":
        weights = len(cfg.dilations) * 3 * cfg.hidden ** 2
        per_frame = weights
    else:
        ch, rate = cfg.up_channels, 1
        weights = per_frame = 3 * cfg.mel_dim * ch[0]
        for q, s in enumerate(cfg.up_strides):
            weights += 2 * s * ch[q] * ch[q + 1] + len(cfg.res_dilations) * 3 * ch[q + 1] ** 2
            rate *= s
            per_frame += rate * (2 * ch[q] * ch[q + 1] + len(cfg.res_dilations) * 3 * ch[q + 1] ** 2)
        head = 3 * ch[-1] * (cfg.n_fft + 2)
        weights += head
        per_frame += rate * (head + cfg.n_fft * (cfg.n_fft + 2))
    T = sum(counts)
    return 4 * weights + 4 * T * (cfg.mel_dim if cfg.pipeline != "conv" else cfg.hidden) + 4 * T * cfg.out_per_frame, 2 * T * per_frame


def work(case):
    cfg, counts = NETS[case["net"]], frame_counts(case)
    if cfg.pipeline in ("conv", "vocoder"):
        b, f = _f32_work(cfg, counts)
        return {"bytes": b, "flops": f}
    if case["call"] == "wavefront":
        F = counts[0]
        chunks = [(min(cfg.f_chunk + cfg.f_lookahead, F - t), min(t, cfg.f_prompt + cfg.kv_cap)) for t in range(0, F, cfg.f_chunk)]
    else:
        chunks = [(T, cfg.f_prompt + cfg.kv_cap) for T in counts]
    if cfg.pipeline == "flow":
        b, f = _flow_work(cfg, chunks)
        return {"bytes": b, "flops": f}
    b, f = _flow_work(cfg.flow_part(), chunks)
    bv, fv = _f32_work(cfg.vocoder_part(), counts)
    return {"bytes": b + bv, "flops": f + fv}


def tolerance(case):
    pipeline = NETS[case["net"]].pipeline
    if pipeline == "conv":
        return {"rel": 1e-5}
    if pipeline == "vocoder":
        return {"rel": 2e-5}            # 32-bit sums through twelve layers and the exponential of the magnitudes
    if pipeline == "flow":
        return {"rel": 1e-2}            # bf16 activations
    return {"rel": 2e-2}                # the vocoder tail expands what the bf16 flow decoder leaves
