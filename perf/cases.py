"""The work that programs have this library do, as timed cases.

Five kinds of call, all through the public binding (`paper_2506_01380_b200.nfd`):

frame      one step of the interactive generation loop on one stream: `speculate(k)` under the current action,
           then `rollback(accept)` (k = 1: plain frame by frame; k > 1: speculative decoding, of which `accept`
           frames survive), with a full context window behind it.
streams    the same step for several independent streams, one batched call per frame (a server).
prompt     the start of a session: `reset`, the prompt's frames committed in chunks, the first denoising pass
           of the new frame (prefill and its first use).
dpmpp      one frame from the undistilled sampler (one model evaluation per solver step), then its rollback.
attention  the allocation-free attention call, for hosts that bring their own pages.

A case of the first four kinds names a configuration of `inputs.make_cfg` and what is changed in it.  fp32
contexts are the library's validation mode and are not timed; the attention call serves hosts in both types.
"""
import math

import numpy as np
import torch

from paper_2506_01380_b200 import inputs as I
from paper_2506_01380_b200 import nfd as N

DEV = "cuda:0"
N_NOISE = 4            # sets of noise a state holds and takes in turn
CHAIN = 256            # length of a state's action chain
L2_BYTES = 126e6       # what does not fit on the chip has to be read again in every forward pass


# ---------------------------------------------------------------------------------------------------------------
# cases
# ---------------------------------------------------------------------------------------------------------------
def _model(kind, model, act=0, ctx=16, latent_h=0, latent_w=0, k=1, accept=1, streams=1, **more):
    """A case on a model context; latent 0 x 0 = the configuration's own size."""
    return dict(kind=kind, model=model, act=act, ctx=ctx, latent_h=latent_h, latent_w=latent_w, k=k, accept=accept,
                streams=streams, **more)


def _attention(dtype, heads, head_dim, tokens, n_q, n_kv, window):
    return dict(kind="attention", dtype=dtype, heads=heads, head_dim=head_dim, tokens=tokens, n_q=n_q, n_kv=n_kv,
                window=window)


def listed():
    return [
        # a toy world model (2 layers, 64 tokens per frame): nothing but launches, latency and host work
        dict(name="frame_tiny", **_model("frame", "tiny_bf16", ctx=4)),
        # the headline: 310M-class model, 384 x 224 video, one player, frame by frame
        dict(name="frame_nfd310m", **_model("frame", "nfd310m")),
        # the same player with four-frame speculation, three frames accepted (repeat probability 0.8)
        dict(name="spec4_nfd310m", **_model("frame", "nfd310m", k=4, accept=3)),
        # a server: eight players on one GPU, long context
        dict(name="streams8_nfd310m", **_model("streams", "nfd310m", ctx=32, streams=8)),
        # another resolution (320 x 176 video: 220 tokens per frame, no multiple of a tile), short context
        dict(name="frame_nfd310m_220tok", **_model("frame", "nfd310m", ctx=9, latent_h=40, latent_w=22)),
        # the paper's three model sizes, gated MLP: the small one frame by frame,
        dict(name="frame_paper130m", **_model("frame", "paper130m", act=1)),
        # the middle one (MLP 2730, no multiple of anything) with two-frame speculation, one accepted,
        dict(name="spec2_paper310m", **_model("frame", "paper310m", act=1, k=2, accept=1)),
        # and the large one frame by frame
        dict(name="frame_paper774m", **_model("frame", "paper774m", act=1)),
        # a session opens: 16 prompt frames go into the cache, then the first pass of the first new frame
        dict(name="prompt_nfd310m", **_model("prompt", "nfd310m", frames=16)),
        # offline generation with the undistilled model: 18 evaluations per frame
        dict(name="dpmpp18_nfd310m", **_model("dpmpp", "nfd310m", evals=18)),
        # attention for a host with its own cache: one frame of the 310M-class model behind 16 frames
        dict(name="attention_bf16", **_attention("bf16", 16, 64, 336, 1, 17, 16)),
        # and a small fp32 model's two frames at an odd size
        dict(name="attention_fp32_odd", **_attention("fp32", 6, 32, 77, 2, 9, 5)),
    ]


def _log_int(rng, lo, hi):
    return min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    if rng.random() < 0.15:
        dtype = rng.choice(["bf16", "bf16", "fp32"])
        n_q = rng.randint(1, 4)
        n_kv = n_q + rng.randint(0, 20)
        heads, head_dim = rng.choice([(4, 32), (12, 64), (16, 64), (24, 64), (8, 128)])
        return _attention(dtype, heads, head_dim, _log_int(rng, 40, 400), n_q, n_kv, rng.randint(1, 20))
    kind = rng.choice(["frame"] * 6 + ["streams"] * 2 + ["prompt"] * 2 + ["dpmpp"])
    model, act = rng.choice([("tiny_bf16", 0), ("nfd310m", 0), ("nfd310m", 0), ("paper130m", 1), ("paper310m", 1),
                             ("paper310m", 0), ("paper774m", 1)])
    c = dict(act=act, ctx=_log_int(rng, 2, 32))
    if rng.random() < 0.4 and model != "tiny_bf16":         # another resolution than 384 x 224
        c.update(latent_h=2 * rng.randint(8, 26), latent_w=2 * rng.randint(6, 15))
    if kind == "frame":
        c["k"] = rng.randint(1, 4)
        c["accept"] = rng.randint(1, c["k"])
    elif kind == "streams":
        c["streams"] = rng.randint(2, 4 if model == "paper774m" else 7)
    elif kind == "prompt":
        c["frames"] = rng.randint(1, 24)
    else:
        c["evals"] = rng.randint(8, 20)
    return _model(kind, model, **c)


# ---------------------------------------------------------------------------------------------------------------
# state
# ---------------------------------------------------------------------------------------------------------------
def _cfg(case):
    over = dict(act=case["act"], ctx_frames=case["ctx"], n_streams=case["streams"])
    if case["latent_h"]:
        over.update(latent_h=case["latent_h"], latent_w=case["latent_w"])
    return I.make_cfg(case["model"], **over)


def _weights(cfg, gen):
    """Random weights with every residual branch at full strength, as in a trained model: matrices N(0, 1/fan_in),
    biases N(0, 0.1^2), gate biases of the modulation 1 (the distributions of inputs.make_weights(kind="stress"),
    drawn on the device)."""
    d, out = cfg["d_model"], {}
    for name, shape in I.weight_shapes(cfg).items():
        w = torch.randn(shape, generator=gen, device=DEV, dtype=torch.float32)
        if name == "a_emb":
            pass
        elif len(shape) == 2:
            w *= 1.0 / math.sqrt(shape[0])
        else:
            w *= 0.1
            if name.startswith("b_mod."):
                w[2 * d:3 * d] = 1.0
                w[5 * d:6 * d] = 1.0
        out[name] = w.to(torch.bfloat16)
    return out


class _State:
    """What a generating program keeps: the context, its noise and action sources and where it is in them."""

    def __init__(self, case, seed):
        self.case, self.cfg = case, _cfg(case)
        gen = torch.Generator(device=DEV)
        gen.manual_seed(seed)
        cfg, fs = self.cfg, I.frame_shape(self.cfg)
        self.nfd = N.NFD(cfg, _weights(cfg, gen), device=DEV)
        n, k = case["streams"], case["k"]

        def randn(*shape):
            return torch.randn(shape, generator=gen, device=DEV, dtype=torch.float32)

        self.chains = [I.make_action_chain(cfg, CHAIN, seed=seed + 1000 * s, p_repeat=0.8) for s in range(n)]
        self.i = 0
        self.streams = list(range(n))
        steps = cfg["n_steps"]
        lead = {"frame": (steps, k), "streams": (steps, n, k), "prompt": (1,), "dpmpp": (k,)}[case["kind"]]
        self.noise = [randn(*lead, *fs) for _ in range(N_NOISE)]
        self.ctx_noise = [randn(*((n, k) if case["kind"] == "streams" else (k,)), *fs) for _ in range(N_NOISE)]
        n_prompt = case["frames"] if case["kind"] == "prompt" else cfg["ctx_frames"]
        latents = cfg["sigma_d"] * randn(n, n_prompt, *fs)
        prompt_noise = randn(n, n_prompt, *fs)
        step = cfg["max_spec"]
        self.prompt = [(s, latents[s, a:a + step].contiguous(), self.chains[s][-n_prompt:][a:a + step],
                        prompt_noise[s, a:a + step].contiguous())
                       for s in self.streams for a in range(0, n_prompt, step)]
        # load time: the modulation of the sampler's (time, action) pairs
        self.nfd.warm_modulation()
        if case["kind"] != "prompt":
            self.fill()
            # the session is under way: the first frames (and with them the library's graphs) are behind it
            for _ in range(2):
                run(self)
        torch.cuda.synchronize()

    def fill(self):
        for s, x0, actions, noise in self.prompt:
            self.nfd.commit_frame(x0, actions, noise, stream=s)

    def next(self):
        i, self.i = self.i, self.i + 1
        return i % CHAIN, self.noise[i % N_NOISE], self.ctx_noise[i % N_NOISE]


class _Attention:
    def __init__(self, case, seed):
        gen = torch.Generator(device=DEV)
        gen.manual_seed(seed)
        self.case = case
        dt = torch.bfloat16 if case["dtype"] == "bf16" else torch.float32
        H, T, dh = case["heads"], case["tokens"], case["head_dim"]

        def randn(*shape):
            return torch.randn(shape, generator=gen, device=DEV, dtype=torch.float32).to(dt)

        self.q = randn(H, case["n_q"] * T, dh)
        self.k, self.v = randn(case["n_kv"], H, T, dh), randn(case["n_kv"], H, T, dh)
        self.out = torch.empty(case["n_q"] * T, H * dh, device=DEV, dtype=dt)


def prepare(case, seed):
    return (_Attention if case["kind"] == "attention" else _State)(case, seed)


# ---------------------------------------------------------------------------------------------------------------
# one pass
# ---------------------------------------------------------------------------------------------------------------
def run(st):
    c = st.case
    if c["kind"] == "attention":
        return N.attention_noalloc(st.q, st.k, st.v, c["n_q"], c["window"], st.out)
    nfd = st.nfd
    i, noise, ctx_noise = st.next()
    if c["kind"] == "frame":
        x0 = nfd.speculate(c["k"], st.chains[0][i], noise, ctx_noise)
        nfd.rollback(c["accept"])
        return x0
    if c["kind"] == "streams":
        x0 = nfd.speculate_batched(st.streams, c["k"], [chain[i] for chain in st.chains], noise, ctx_noise)
        for s in st.streams:
            nfd.rollback(c["accept"], stream=s)
        return x0
    if c["kind"] == "prompt":
        nfd.reset(0)
        st.fill()
        return nfd.denoise_step(noise, 1.0, st.chains[0][i])
    x0 = nfd.sample_dpmpp(c["k"], st.chains[0][i], noise, n_evals=c["evals"], ctx_noise=ctx_noise)
    nfd.rollback(c["accept"])
    return x0


# ---------------------------------------------------------------------------------------------------------------
# what a pass cannot do without, and how far two correct implementations may be apart
# ---------------------------------------------------------------------------------------------------------------
def work(case):
    if case["kind"] == "attention":
        size = 2 if case["dtype"] == "bf16" else 4
        H, T, dh, n_q, n_kv = (case[x] for x in ("heads", "tokens", "head_dim", "n_q", "n_kv"))
        firsts = [max(0, f - case["window"]) for f in range(n_kv - n_q, n_kv)]
        pairs = sum(f - a + 1 for f, a in zip(range(n_kv - n_q, n_kv), firsts))
        page = H * T * dh
        return {"bytes": size * page * (2 * n_q + 2 * (n_kv - firsts[0])), "flops": 4.0 * pairs * page * T}
    cfg = _cfg(case)
    L, d, T, W = cfg["n_layers"], cfg["d_model"], I.tokens_per_frame(cfg), cfg["ctx_frames"]
    n, k, fe = case["streams"], case["k"], int(np.prod(I.frame_shape(cfg)))
    params = L * (4 * d * d + (3 if case["act"] == 1 else 2) * d * cfg["d_mlp"]) + 2 * d * I.patch_len(cfg)

    def frame(context):                      # FLOPs of one frame of a pass that sees `context` frames
        return 2.0 * T * params + 4.0 * T * (context + 1) * T * d * L

    kv = 2.0 * 2 * L * T * d                 # bytes of one frame's K and V
    if case["kind"] == "prompt":
        m = case["frames"]
        return {"bytes": (-(-m // cfg["max_spec"]) + 1) * 2.0 * params + m * (2 * kv + 8 * fe) + 8 * fe,
                "flops": sum(frame(min(f, W)) for f in range(m + 1))}
    evals = case.get("evals", cfg["n_steps"])
    keep = 2.0 * params + n * W * kv         # weights and context, read in every evaluation unless the chip holds them
    flops = n * (evals * k + case["accept"]) * frame(W)
    byts = keep * (evals if keep > L2_BYTES else 1) + n * (k * kv + 4 * fe * (k * evals + 2 * k))
    if case["kind"] == "dpmpp":              # the solver's times are no schedule times: their modulation is computed
        byts += 2.0 * 6 * d * d * L
        flops += 2.0 * 6 * d * d * L * evals
    return {"bytes": byts, "flops": flops}


def tolerance(case):
    # Model passes: about four times what the same pass differs by when its LayerNorms run as kernels of their own
    # instead of folded into the projections, or when the K ranges of its sums are split in another way (measured
    # on one B200: rel up to 4.0e-3 and max up to 1.6e-2 with the GELU MLP, 5.6e-3 and 2.5e-2 with the gated one;
    # every activation of up to 24 layers x 5 passes is rounded to bf16).
    # Attention: bf16 outputs whose products may take probabilities rounded to bf16 (2.3e-3 against 64 bits for
    # normal data of these sizes); fp32 sums in any order.
    if case["kind"] == "attention":
        return {"rel": 1e-2, "max": 0.05} if case["dtype"] == "bf16" else {"rel": 1e-5, "max": 4e-4}
    return {"rel": 2.2e-2, "max": 0.1} if case["act"] == 1 else {"rel": 1.5e-2, "max": 0.07}
