"""The decoder's performance cases: what users of this framework have it do, through its public entry points.

A case is one model shape, one batch shape and one way of calling:
  decode   frames on the GPU, one call of TwDecoder.decode for the batch
  host     frames in pinned host memory, one call of TwDecoder.decode_host, results back on the host
  stream   live sessions: open, chunks pushed as they arrive with the N best read after each, close
  stages   the separately callable stages, as a caller with a search of its own runs them for one pass of its loop
The model shapes are the ones of tw_synth/configs.py: weights N(0, 1/fan_in), embeddings and frames N(0, 1), LSTM
biases 0, output bias 0 except at blank.
"""
import math

import torch

from paper_2302_14357_b200.binding import MODE_BF16, MODE_F32, TwDecoder

# Model shapes: encoder width D, predictor (layers of width H, 0 layers: stateless embedding of width H), joiner width J,
# vocabulary V with blank = 0, bias of blank, joiner nonlinearity and output normalisation.
_TINY = dict(D=64, layers=0, H=64, J=64, V=32, blank_bias=3.0, act="tanh", norm="softmax")
_LIBRISPEECH = dict(D=512, layers=1, H=640, J=640, V=1024, blank_bias=4.0, act="tanh", norm="softmax")
_PAPER = dict(D=512, layers=3, H=512, J=512, V=501, blank_bias=4.0, act="relu", norm="softmax")
_HAT = dict(D=512, layers=1, H=640, J=640, V=1024, blank_bias=1.5, act="tanh", norm="hat")
_ASSISTANT = dict(D=1024, layers=2, H=1024, J=1024, V=4096, blank_bias=4.0, act="tanh", norm="softmax")


def _case(name, model, call, mode, B, T, T_min, N, S, chunk=0, tau=1.0):
    """T_min: utterance lengths are drawn from [T_min, T].  chunk: frames per push of a stream.  tau: blank threshold."""
    c = dict(model, call=call, mode=mode, B=B, T=T, T_min=T_min, N=N, S=S, chunk=chunk, tau=tau)
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # the accuracy path on a short command, the smallest thing a decoder is asked for
        _case("f32_one_short", _TINY, "decode", "f32", B=1, T=40, T_min=40, N=2, S=2),
        # one utterance as it comes in, on the large model: latency of a single offline request
        _case("one_utterance", _ASSISTANT, "decode", "bf16", B=1, T=600, T_min=600, N=10, S=3),
        # live captioning: 16 microphones, chunks of 20 frames that are no multiple of the segment, partial results shown
        _case("live_stream", _LIBRISPEECH, "stream", "bf16", B=16, T=100, T_min=85, N=5, S=3, chunk=20),
        # one pass of a caller's own search: project the new frames, step the predictor, expand (ragged segments)
        _case("stages", _ASSISTANT, "stages", "bf16", B=100, T=3, T_min=1, N=10, S=3),
        # a ragged batch of utterances of a public test set, small beam
        _case("librispeech_b32", _LIBRISPEECH, "decode", "bf16", B=32, T=400, T_min=200, N=5, S=3),
        # the same model, long segments: the right end of the sweep over S
        _case("librispeech_s20", _LIBRISPEECH, "decode", "bf16", B=64, T=400, T_min=400, N=10, S=20),
        # the paper's Librispeech model: ReLU joiner, three LSTM layers, a vocabulary that is a multiple of nothing
        _case("paper_v501", _PAPER, "decode", "bf16", B=32, T=300, T_min=150, N=5, S=5),
        # factorised output with blank thresholding
        _case("hat_threshold", _HAT, "decode", "bf16", B=64, T=400, T_min=400, N=10, S=3, tau=0.85),
        # the accuracy path on a batch
        _case("f32_batch", _LIBRISPEECH, "decode", "f32", B=32, T=400, T_min=200, N=5, S=3),
        # the headline workload, frames on the GPU
        _case("assistant_b128", _ASSISTANT, "decode", "bf16", B=128, T=600, T_min=600, N=10, S=3),
        # and from host memory to host memory, as a server calls it
        _case("assistant_host", _ASSISTANT, "host", "bf16", B=128, T=600, T_min=600, N=10, S=3),
        # throughput: a large ragged batch with long segments
        _case("assistant_b512", _ASSISTANT, "decode", "bf16", B=512, T=1000, T_min=500, N=10, S=10),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    while True:
        model = dict(rng.choice([_LIBRISPEECH, _LIBRISPEECH, _PAPER, _HAT, _ASSISTANT, _ASSISTANT]))
        call = rng.choice(["decode", "decode", "decode", "decode", "host", "stream", "stages"])
        mode = rng.choice(["bf16", "bf16", "bf16", "bf16", "f32"])
        if mode == "f32" and rng.random() < 0.5:
            model = dict(_TINY)
        if rng.random() < 0.5:                            # another vocabulary for the same network
            model["V"] = rng.randint(max(17, model["V"] // 2), model["V"])
        if rng.random() < 0.3:                            # another width
            model["J"] = 16 * rng.randint(model["J"] // 32, model["J"] // 16)
        S = rng.choice([1, 2, 2, 3, 3, 3, 4, 5, 5, 6, 8, 10, 10, 13, 20, 50])
        N = rng.choice([1, 2, 4, 5, 5, 8, 10, 10, 10, 16])
        T = S if call == "stages" else _log_int(rng, 40, 1000)
        T_min = rng.choice([T, max(1, T // 2)])
        B = _log_int(rng, 1, 512)
        if call == "stream":
            B, T = min(B, 64), min(T, 200)
            T_min = min(T_min, T)
        chunk = rng.randint(4, max(5, min(T, 64))) if call == "stream" else 0
        tau = rng.choice([1.0, 0.85, 0.6]) if model["norm"] == "hat" else 1.0
        c = _case(None, model, call, mode, B, T, T_min, N, S, chunk, tau)
        w = work(c)
        if w["flops"] > (1.5e12 if mode == "f32" else 1.0e14 if S in (1, 2, 3, 4, 5, 8, 10) else 1.5e13):
            continue                                      # no dearer than the largest listed case
        if B * S * N * model["V"] > 1 << 29:
            continue                                      # materialised logits of the staged path: at most 2 GiB
        return c


# ---------------------------------------------------------------------------------------------------------------------
def _weights(c, g, dt):
    def normal(shape, std):
        return (torch.randn(shape, device="cuda", generator=g) * std).to(dt)
    w = dict(W_e=normal((c["J"], c["D"]), c["D"] ** -0.5), W_p=normal((c["J"], c["H"]), c["H"] ** -0.5),
             W_out=normal((c["V"], c["J"]), c["J"] ** -0.5), emb=normal((c["V"], c["H"]), 1.0))
    b = torch.zeros(c["V"], device="cuda", dtype=dt)
    b[0] = c["blank_bias"]
    w["b_out"] = b
    if c["layers"]:
        H = c["H"]
        w["lstm_W_ih"] = [normal((4 * H, H), H ** -0.5) for _ in range(c["layers"])]
        w["lstm_W_hh"] = [normal((4 * H, H), H ** -0.5) for _ in range(c["layers"])]
        w["lstm_b"] = [torch.zeros(4 * H, device="cuda", dtype=dt) for _ in range(c["layers"])]
    return w


def prepare(case, seed):
    """A decoder that holds the model's weights, and the batch."""
    c = case
    g = torch.Generator(device="cuda").manual_seed(seed)
    f32 = c["mode"] == "f32"
    dt = torch.float32 if f32 else torch.bfloat16
    B, T, N, S = c["B"], c["T"], c["N"], c["S"]
    dec = TwDecoder(_weights(c, g, dt), N=N, S=S, mode=MODE_F32 if f32 else MODE_BF16, max_batch=B, max_T=T,
                    joiner_act=c["act"], joiner_norm=c["norm"], dtype="f32" if f32 else "bf16")
    if c["tau"] < 1.0:
        dec.set_blank_threshold(c["tau"])
    enc = torch.randn((B, T, c["D"]), device="cuda", generator=g).to(dt)
    lens = torch.randint(c["T_min"], T + 1, (B,), device="cuda", generator=g, dtype=torch.int32)
    s = dict(call=c["call"], dec=dec, enc=enc, lens=lens)
    if c["call"] == "host":
        s["enc"] = enc.cpu().pin_memory()
        s["lens"] = lens.cpu().numpy()
        s["out"] = tuple(torch.empty(shape, dtype=t).pin_memory().numpy() for shape, t in (
            ((B, N, dec.U_cap), torch.int32), ((B, N), torch.int32), ((B, N), torch.float64), ((B,), torch.int32)))
    elif c["call"] == "stream":
        s["B"] = B
        s["chunks"] = [(enc[:, t:t + c["chunk"]].contiguous(), (lens - t).clamp(0, min(c["chunk"], T - t)).to(torch.int32))
                       for t in range(0, T, c["chunk"])]
    elif c["call"] == "stages":
        R, L, H = B * N, c["layers"], c["H"]
        s["tokens"] = torch.randint(1, c["V"], (R,), device="cuda", generator=g, dtype=torch.int32)
        s["state"] = torch.tanh(torch.randn((R, L, 2, H), device="cuda", generator=g)) if L else None
        s["group"] = (torch.arange(R, device="cuda", dtype=torch.int32) // N).contiguous()
        s["ld_old"] = torch.randn((R, S), device="cuda", generator=g) - 2.0
        s["shape"] = (B, S, c["J"])
    return s


def run(state):
    s = state
    dec = s["dec"]
    if s["call"] == "decode":
        return dec.decode(s["enc"], s["lens"])[:4]
    if s["call"] == "host":
        return dec.decode_host(s["enc"], s["lens"], out=s["out"])[:4]
    if s["call"] == "stream":
        dec.stream_open(s["B"])
        for frames, valid in s["chunks"]:
            dec.stream_push(frames, valid)
            partial = dec.stream_nbest()
        return partial, dec.stream_close()[:4]
    E = dec.project_encoder(s["enc"])
    hc, Pp = dec.predictor_step(s["tokens"], s["state"])
    return E, hc, Pp, dec.joiner_expand(E.view(s["shape"]), Pp, s["group"], s["lens"], s["ld_old"])


def work(case):
    """Inputs read once, outputs written once; the contractions of the encoder projection, of the predictor for every new
    hypothesis and of the joiner for every (hypothesis, frame) pair of every pass.  The number of passes depends on the
    inputs; per frame the search joins about 1.4 + 0.58 S times with this kind of model (half of that with the factorised
    output's higher blank probability), for 0.95 N hypotheses on average, of which 0.7 are new."""
    c = case
    B, S, N, J, V, H, D, L = (c[k] for k in ("B", "S", "N", "J", "V", "H", "D", "layers"))
    el = 4 if c["mode"] == "f32" else 2
    pred = 16.0 * H * H * L + 2.0 * J * H                 # flops of one predictor step and its projection
    weights = el * (J * D + J * H + V * J + V + V * H + L * (8.0 * H * H + 4 * H))
    if c["call"] == "stages":
        R, t = B * N, (c["T"] + c["T_min"]) / 2
        flops = 2.0 * J * D * B * S + R * (pred + 2.0 * J * V * t)
        return {"bytes": weights + el * B * S * D + 4.0 * (B * S * J + R * (4 * L * H + J + V + 2 * S + 2)), "flops": flops}
    frames = B * (c["T"] + c["T_min"]) / 2
    joins = (1.4 + 0.58 * S) * (0.5 if c["norm"] == "hat" else 1.0)
    rows = frames * joins / S * 0.95 * N                  # hypothesis rows of all passes
    flops = 2.0 * J * D * frames + rows * (2.0 * J * V * S + 0.7 * (pred if L else 0.0))
    return {"bytes": weights + el * frames * D + B * N * (4.0 * 512 + 12), "flops": flops}


def tolerance(case):
    # whole values: token sequences, which may swap places in a list where two scores are a rounding apart
    if case["mode"] == "f32":
        return {"rel": 1e-5, "max": 1e-4, "differ": 2e-3}
    if case["call"] == "stages":
        return {"rel": 1e-2, "max": 4e-2}                 # bf16 operands: log-probabilities to 2e-2
    return {"rel": 1e-3, "max": 1e-2, "differ": 1e-2}     # scores add such errors of random sign up
