"""The calls whose speed is measured, as a user's program makes them: the denoising loop over its batch sizes, storage
types and conditioning modes, the serving worker around it, the feature-handoff head, and the operators either side.

Shapes are those of ``synth`` (pi0- / pi0.5-shaped experts, the tiny fp32 expert, the feature-handoff head) and of the
benchmark; weights are random with the same distribution (N(0, 0.02)), prefix K / V, states and noise are N(0, 1)."""
import math

import torch

from paper_2608_03682_b200 import binding, frontend, synth

WEIGHT_STD = 0.02
FEAT_DIM = 2048          # width of the vision-language features of the feature-handoff head


# ------------------------------------------------------------------------------------------------------------------
# cases
# ------------------------------------------------------------------------------------------------------------------
def _loop(name, cond, dtype, batch, lo, hi, horizon=50, n_steps=10):
    return dict(name=name, kind="loop", cond=cond, dtype=dtype, batch=batch, lo=lo, hi=hi, horizon=horizon, n_steps=n_steps)


def listed():
    return [
        # one layer's suffix attention as an operator of its own: the smallest call, one robot's query rows
        dict(name="attention-b1", kind="attention", batch=1, lo=816, hi=816, suffix=51),
        # the adapter's steps around a call for eight robots: padded backbone K / V -> ragged cache, raw chunk -> actions
        dict(name="adapter-b8", kind="adapter", batch=8, lo=600, hi=968, p_max=968, out_dim=14),
        # the tiny fp32 expert: true fp32 arithmetic, launch-bound
        dict(name="tiny-f32", kind="tiny", batch=1, lo=64, hi=64, horizon=16, n_steps=4),
        # one robot, pi0 shape: latency of an action chunk
        _loop("pi0-b1", "pi0", "bf16", 1, 816, 816),
        # one robot, pi0.5 shape: adaptive norms, no state token
        _loop("pi05-b1", "pi05", "bf16", 1, 968, 968),
        # one robot, e4m3 weights
        _loop("pi0-e4m3-b1", "pi0", "w8e4m3", 1, 816, 816),
        # the data-parallel front-end's worker: 32 pending observations over eight GPUs = 4 requests per worker, from
        # host tensors to host arrays
        dict(name="worker-b4", kind="worker", cond="pi0", dtype="bf16", batch=4, lo=600, hi=968, horizon=50, n_steps=10),
        # a few robots share a GPU, e4m3 weights
        _loop("pi0-e4m3-b8", "pi0", "w8e4m3", 8, 816, 816),
        # a middling batch of the adaptive-norm expert, ragged prefixes
        _loop("pi05-b16", "pi05", "bf16", 16, 600, 968),
        # batched rollouts with ragged prefixes
        _loop("pi0-b64", "pi0", "bf16", 64, 600, 968),
        # the largest batch of the e4m3 sweep
        _loop("pi0-e4m3-b256", "pi0", "w8e4m3", 256, 816, 816),
        # one robot with a feature-handoff head: K / V projections of the features, then four steps on a 40 x 132 chunk
        dict(name="groot-b1", kind="groot", batch=1, lo=640, hi=640, n_steps=4),
    ]


def _log_int(rng, lo, hi):
    return min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def _lens(rng, lo, hi):
    """Bounds of the prefix lengths: fixed or ragged."""
    a, b = sorted((rng.randint(lo, hi), rng.randint(lo, hi)))
    return (a, b) if rng.random() < 0.6 else (b, b)


def draw(rng):
    kind = rng.choice(["loop"] * 7 + ["worker", "groot", "attention", "adapter", "tiny"])
    if kind == "attention":
        lo, hi = _lens(rng, 32, 968)
        return dict(kind=kind, batch=_log_int(rng, 1, 16), lo=lo, hi=hi, suffix=rng.randint(17, 64))
    if kind == "adapter":
        lo, hi = _lens(rng, 200, 968)
        return dict(kind=kind, batch=_log_int(rng, 1, 32), lo=lo, hi=hi, p_max=968, out_dim=rng.randint(7, 32))
    if kind == "tiny":
        lo, hi = _lens(rng, 8, 64)
        return dict(kind=kind, batch=_log_int(rng, 1, 8), lo=lo, hi=hi, horizon=rng.randint(8, 24), n_steps=rng.randint(2, 8))
    if kind == "groot":
        lo, hi = _lens(rng, 100, 640)
        return dict(kind=kind, batch=_log_int(rng, 1, 16), lo=lo, hi=hi, n_steps=4)
    lo, hi = _lens(rng, 300, 968)
    horizon, n_steps = rng.choice([10, 16, 32, 50, 50, 50]), rng.choice([5, 8, 10, 10, 10])
    cond = rng.choice(["pi0", "pi0", "pi05"])
    if kind == "worker":
        return dict(kind=kind, cond=cond, dtype="bf16", batch=_log_int(rng, 1, 8), lo=lo, hi=hi, horizon=horizon, n_steps=n_steps)
    # (not the W8A8 mode: its activation quantizer is a step function that carries rounding-level differences up to
    # several per cent of the actions, so two of its results cannot be told apart from two correct ones)
    dtype = rng.choice(["bf16", "bf16", "w8e4m3", "w4a16"])
    # (at most 192 requests: a drawn case costs no more than the largest listed one)
    return dict(kind=kind, cond=cond, dtype=dtype, batch=_log_int(rng, 1, 192), lo=lo, hi=hi, horizon=horizon, n_steps=n_steps)


# ------------------------------------------------------------------------------------------------------------------
# inputs
# ------------------------------------------------------------------------------------------------------------------
def _config(case):
    kind, B, hi = case["kind"], case["batch"], case["hi"]
    if kind == "tiny":
        return synth.tiny_config().with_(max_batch=B, max_prefix_len=hi, horizon=case["horizon"])
    if kind == "groot":
        return synth.groot_like_config(max_batch=B, max_prefix_len=hi)
    make = synth.pi0_config if case["cond"] == "pi0" else synth.pi05_config
    return make(max_batch=B, dtype=case["dtype"], max_prefix_len=hi).with_(horizon=case["horizon"])


def _lengths(case):
    """The requests' prefix lengths: spread evenly over lo..hi, in a fixed shuffled order."""
    B, lo, hi = case["batch"], case["lo"], case["hi"]
    return [lo + (hi - lo) * ((i * 37 + 11) % B) // max(1, B - 1) if B > 1 else hi for i in range(B)]


def _cu(lens, device="cuda"):
    return torch.tensor([0] + lens, dtype=torch.int64).cumsum(0).to(torch.int32).to(device)


def _normal(gen, shape, dtype, std=1.0):
    t = torch.empty(shape, dtype=torch.float32 if dtype == torch.float32 else torch.bfloat16, device="cuda")
    return t.normal_(0.0, std, generator=gen)


def _weights(cfg, gen):
    """The expert's weights in its storage format, on the device."""
    store = torch.float32 if cfg.dtype == "f32" else torch.bfloat16
    out = {}
    for name, shape in synth.weight_shapes(cfg):
        big = name.split(".")[0] in synth.BIG_MATS
        if big and cfg.dtype == "w8e4m3":
            out[name] = synth.quantize_e4m3_columns(_normal(gen, shape, torch.float32, WEIGHT_STD))
        elif big and cfg.dtype == "w4a16":
            out[name] = synth.quantize_int4_columns(_normal(gen, shape, torch.float32, WEIGHT_STD))
        else:
            out[name] = _normal(gen, shape, store, WEIGHT_STD)
    return out


def prepare(case, seed):
    gen = torch.Generator(device="cuda").manual_seed(seed)
    kind, B, lens = case["kind"], case["batch"], _lengths(case)
    if kind == "attention":
        Hq, Hkv, dh, S, L = 8, 1, 256, case["suffix"], 2
        pos = torch.arange(max(lens) + S, dtype=torch.float64, device="cuda")[:, None]
        ang = pos * 10000.0 ** (-2.0 * torch.arange(dh // 2, dtype=torch.float64, device="cuda") / dh)[None, :]
        return dict(kind=kind, desc=binding.attention_desc(Hq, Hkv, dh, S, n_layers=L, layer=1),
                    qkv=_normal(gen, (B * S, (Hq + 2 * Hkv) * dh), torch.float32),
                    kv=_normal(gen, (L, 2, sum(lens), Hkv, dh), torch.bfloat16), cu=_cu(lens),
                    rope=torch.stack([ang.cos(), ang.sin()], dim=-1).float().contiguous())
    if kind == "adapter":
        cfg = synth.pi0_config(max_batch=B)
        shape = (cfg.n_layers, B, case["p_max"], cfg.n_kv_heads, cfg.head_dim)
        q = _normal(gen, (2, cfg.action_dim), torch.float32).abs() + 0.1
        return dict(kind=kind, k=_normal(gen, shape, torch.bfloat16), v=_normal(gen, shape, torch.bfloat16),
                    lens=torch.tensor(lens, dtype=torch.int32, device="cuda"),
                    x=_normal(gen, (B, cfg.horizon, cfg.action_dim), torch.float32), q01=-q[0].contiguous(),
                    q99=q[1].contiguous(), out_dim=case["out_dim"])
    cfg = _config(case)
    state = dict(kind=kind, n=case["n_steps"], ex=binding.Expert(cfg, _weights(cfg, gen)), batch=B, lens=lens)
    kv_dtype = torch.float32 if cfg.dtype == "f32" else torch.bfloat16
    noise = _normal(gen, (B, cfg.horizon, cfg.action_dim), torch.float32)
    states = _normal(gen, (B, cfg.state_dim), torch.float32) if cfg.has_state_token else None
    kv_shape = (cfg.n_layers, 2, sum(lens), cfg.n_kv_heads, cfg.head_dim)
    if kind == "worker":
        # requests as they arrive at a rank: host tensors in ordinary memory
        state["worker"] = frontend.ExpertWorker(state["ex"], cfg, case["n_steps"])
        noise, states = noise.cpu(), None if states is None else states.cpu()
        state["requests"] = [dict(prefix_kv=_normal(gen, kv_shape[:2] + (p,) + kv_shape[3:], kv_dtype).cpu(),
                                  state=None if states is None else states[b].clone(), noise=noise[b].clone(),
                                  n_steps=case["n_steps"]) for b, p in enumerate(lens)]
        return state
    state.update(noise=noise, states=states, cu=_cu(lens), out=torch.empty_like(noise))
    if kind == "groot":
        std = FEAT_DIM ** -0.5
        wk, wv = ([_normal(gen, (FEAT_DIM, cfg.kv_dim), torch.bfloat16, std) for _ in range(cfg.n_layers)] for _ in range(2))
        state["proj"] = binding.KvProjector(wk, wv, cfg.n_kv_heads, cfg.head_dim, max_tokens=sum(lens))
        state["features"] = _normal(gen, (sum(lens), FEAT_DIM), torch.bfloat16)
        return state
    state["kv"] = _normal(gen, kv_shape, kv_dtype)
    return state


# ------------------------------------------------------------------------------------------------------------------
# one pass
# ------------------------------------------------------------------------------------------------------------------
def run(s):
    kind = s["kind"]
    if kind == "attention":
        return binding.suffix_attention(s["desc"], s["qkv"], s["kv"], s["cu"], s["rope"])
    if kind == "adapter":
        kv, cu, status = binding.pack_prefix_kv(s["k"], s["v"], s["lens"])
        return kv, cu, status, binding.postprocess_actions(s["x"], s["q01"], s["q99"], out_dim=s["out_dim"])
    if kind == "worker":
        return s["worker"](s["requests"])
    kv = s["proj"].run(s["features"]) if kind == "groot" else s["kv"]
    if s["batch"] == 1:
        s["ex"].denoise(kv, s["lens"][0], None if s["states"] is None else s["states"][0], s["noise"][0], s["n"], out=s["out"][0])
    else:
        s["ex"].denoise_batched(kv, s["cu"], s["states"], s["noise"], s["n"], out=s["out"])
    return (kv, s["out"]) if kind == "groot" else s["out"]


# ------------------------------------------------------------------------------------------------------------------
# what a pass cannot do without
# ------------------------------------------------------------------------------------------------------------------
def work(case):
    kind, lens = case["kind"], _lengths(case)
    B, T = case["batch"], sum(lens)
    if kind == "attention":
        Hq, Hkv, dh, S = 8, 1, 256, case["suffix"]
        return {"bytes": B * S * (Hq + 2 * Hkv) * dh * 4 + T * 2 * Hkv * dh * 2 + B * S * Hq * dh * 2 + (max(lens) + S) * dh * 4,
                "flops": sum(4 * S * (p + S) * Hq * dh for p in lens)}
    if kind == "adapter":
        cfg = synth.pi0_config()
        row = cfg.n_layers * 2 * cfg.kv_dim * 2     # the rows that exist are read, the whole cache (zero tail included) is written
        return {"bytes": row * (T + B * case["p_max"]) + B * cfg.horizon * (cfg.action_dim + case["out_dim"]) * 4, "flops": 0}
    cfg = _config(case)
    n, D, F, L, S = case["n_steps"], cfg.width, cfg.mlp_dim, cfg.n_layers, cfg.suffix_len
    wb = {"f32": 4.0, "bf16": 2.0, "w8e4m3": 1.0, "w4a16": 0.5}[cfg.dtype]
    eb = 4 if cfg.dtype == "f32" else 2
    layer = D * (cfg.q_dim + 2 * cfg.kv_dim) + cfg.q_dim * D + 3 * D * F
    # The steps depend on one another, so every step reads all weights and the whole prefix cache.
    nbytes = n * (L * layer * wb + (D * D * eb if cfg.cond == "pi0" else 0) + 2 * cfg.action_dim * D * eb + T * L * 2 * cfg.kv_dim * eb)
    flops = n * (2 * B * S * L * layer + (2 * B * cfg.horizon * D * D if cfg.cond == "pi0" else 0)
                 + 4 * B * cfg.horizon * cfg.action_dim * D + L * sum(4 * S * (p + S) * cfg.q_dim for p in lens))
    if kind == "groot":
        nbytes += L * FEAT_DIM * 2 * cfg.kv_dim * 2 + T * FEAT_DIM * 2 + T * L * 2 * cfg.kv_dim * 2
        flops += 2 * T * FEAT_DIM * 2 * cfg.kv_dim * L
    return {"bytes": nbytes + 2 * B * cfg.horizon * cfg.action_dim * 4, "flops": flops}


def tolerance(case):
    kind = case["kind"]
    if kind == "adapter":
        return {"rel": 1e-6}                       # moved bytes, and one fused multiply-add per action in fp32
    if kind == "tiny":
        return {"rel": 1e-5}                       # fp32 throughout
    return {"rel": 1e-2}                           # bf16 operands, fp32 accumulation
