"""The performance cases of the library: what its users have it do, through the public entry points.

A vision-language serving engine calls the library in two places.  Once per request batch, after (or layer by layer
during) the prefill, it compresses the cache: aircache_score, then aircache_budget and aircache_compact.  Then, for
every generated token, it runs one attention call over the compressed cache: aircache_decode_attn, or
aircache_decode_step when the call also appends the new token's K and V.  A host-side caller has both done by
aircache_pipeline_host.  The kinds of case:

  attn    one decode attention call over all layers and sequences
  steps   the decoding of `rounds` tokens of a request batch, each call appending a token
  score   the importance scores of all visual tokens, one call over all layers; alpha = 0 takes every window query
  layers  the same, one call per layer, as an engine does that scores a layer while its keys are hot
  keep    budgets, selection and compaction from given scores
  host    the whole path from and to host memory

The compression is measured in two kinds of case, each with its own inputs, because whole numbers follow from the
scores: two tokens whose scores differ by a rounding may change places in a kept list.
"""
import math

import torch

import paper_2503_23956_b200 as ac
from paper_2503_23956_b200.session import Session

_DEV = "cuda:0"

# layers, query heads, KV heads, head_dim: the tiny cache, the Qwen2-7B-shaped decoder and the Qwen2-72B-shaped stack
# of this repository's configurations, and two generic decoders (two KV heads; eight KV heads of 64 channels)
_MODELS = {
    "tiny": (4, 8, 2, 64),
    "7b": (28, 28, 4, 128),
    "72b": (80, 64, 8, 128),
    "two_kv": (24, 32, 2, 128),
    "small_heads": (24, 32, 8, 64),
}


def listed():
    return [
        # one token of the smallest cache: launch latency and host work, hardly any bytes
        dict(name="attn_tiny", kind="attn", model="tiny", batch=1, visual=576, text=64, ratio=0.10, heads=False),
        # interactive use: one high-resolution image, one user, 32 tokens generated
        dict(name="steps_image", kind="steps", model="7b", batch=1, visual=7290, text=128, ratio=0.10, heads=False,
             rounds=32),
        # one token of four video requests
        dict(name="attn_video", kind="attn", model="7b", batch=4, visual=6272, text=512, ratio=0.10, heads=False),
        # one token of a full serving batch
        dict(name="attn_batch", kind="attn", model="7b", batch=64, visual=2916, text=256, ratio=0.10, heads=False),
        # one token of a long-context request to a large model whose budgets differ by KV head
        dict(name="attn_heads", kind="attn", model="72b", batch=1, visual=7290, text=2048, ratio=0.05, heads=True),
        # scores for one high-resolution image (an odd number of tokens: 90 x 81)
        dict(name="score_image", kind="score", model="7b", batch=1, visual=7290, text=128, window=16, alpha=0.9,
             heads=False),
        # scores for a full serving batch
        dict(name="score_batch", kind="score", model="7b", batch=64, visual=2916, text=256, window=16, alpha=0.9,
             heads=False),
        # scores of four video requests, layer by layer during the prefill
        dict(name="layers_video", kind="layers", model="7b", batch=4, visual=6272, text=512, window=16, alpha=0.9,
             heads=False),
        # scores from the whole window (no elite selection): the dense contraction
        dict(name="score_window", kind="score", model="7b", batch=1, visual=7290, text=128, window=16, alpha=0.0,
             heads=False),
        # compaction for one image
        dict(name="keep_image", kind="keep", model="7b", batch=1, visual=7290, text=128, ratio=0.10, heads=False),
        # compaction for a full serving batch
        dict(name="keep_batch", kind="keep", model="7b", batch=64, visual=2916, text=256, ratio=0.10, heads=False),
        # a host-side caller: one image and the queries of 64 rounds come from pinned host memory, outputs go back
        dict(name="host_image", kind="host", model="7b", batch=1, visual=7290, text=128, window=16, alpha=0.9,
             ratio=0.10, heads=False, rounds=64),
    ]


# A drawn case stays below the largest listed ones: bytes and operations of a pass, and the full cache's K and V.
_MOST_BYTES = 4.0e9
_MOST_FLOPS = 4.5e10
_MOST_CACHE = 10.0e9


def draw(rng):
    def log_uniform(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(["attn", "attn", "steps", "score", "score", "layers", "keep", "keep", "host"])
    model = rng.choice(["tiny", "7b", "7b", "7b", "72b", "two_kv", "small_heads"])
    L, _, Hkv, d = _MODELS[model]
    case = dict(kind=kind, model=model, visual=log_uniform(400, 9000), text=log_uniform(24, 2048),
                heads=rng.random() < 0.2)
    if kind in ("attn", "steps", "keep", "host"):
        case["ratio"] = rng.choice([0.05, 0.10, 0.25, 0.50])
    if kind in ("score", "layers", "host"):
        case["window"] = min(rng.choice([16, 16, 16, 32, 64]), case["text"])
        case["alpha"] = 0.0 if kind == "score" and rng.random() < 0.25 else rng.choice([0.9, 0.9, 0.5])
    if kind in ("steps", "host"):
        case["rounds"] = log_uniform(8, 64)
    batch = log_uniform(1, 64)
    if kind == "host":
        batch = min(batch, 2)
    # the library takes at most 1792 regions (cells, with budgets per KV head)
    batch = min(batch, 1792 // (L * (Hkv if case["heads"] else 1)))
    case["batch"] = batch
    while True:
        need = work(case)
        full = 4 * L * case["batch"] * (case["visual"] + case["text"]) * Hkv * d
        if need["bytes"] <= _MOST_BYTES and need["flops"] <= _MOST_FLOPS and full <= _MOST_CACHE:
            return case
        if case["batch"] > 1:
            case["batch"] = case["batch"] * 3 // 4
        elif case.get("rounds", 1) > 1:
            case["rounds"] = case["rounds"] * 3 // 4
        else:
            case["visual"] = case["visual"] * 3 // 4


# ---------------------------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------------------------
def _shape(case):
    L, Hq, Hkv, d = _MODELS[case["model"]]
    slack = case["rounds"] if case["kind"] == "steps" else 0
    return ac.shape(L, case["batch"], Hq, Hkv, d, case["visual"], case["text"], case.get("window", 16), slack,
                    per_kv_head=int(case["heads"]))


def _normal(shape, gen):
    return torch.empty(shape, dtype=torch.bfloat16, device=_DEV).normal_(generator=gen)


def _keys_and_window(sh, gen):
    """Token-major keys [L, B, N, Hkv, d] and window queries [L, B, W, Hq, d]: standard normal, with a twentieth of
    the visual keys moved along a direction that the window's queries share, by an amount that differs by layer."""
    L, B, Hq, Hkv, d, W = sh.n_layers, sh.batch, sh.n_q_heads, sh.n_kv_heads, sh.head_dim, sh.window
    k = _normal((L, B, sh.n_visual + sh.n_text, Hkv, d), gen)
    qw = _normal((L, B, W, Hq, d), gen)
    u = torch.randn((L, B, Hkv, d), generator=gen, device=_DEV)
    u /= u.norm(dim=-1, keepdim=True)
    amp = 0.5 + 3.5 * torch.rand((L, B, 1, 1), generator=gen, device=_DEV)
    planted = torch.rand((L, B, sh.n_visual, 1, 1), generator=gen, device=_DEV) < 0.05
    for l in range(L):
        k[l, :, :sh.n_visual] += (planted[l] * (amp[l] * u[l])[:, None]).to(torch.bfloat16)
    qw += (math.sqrt(d) * u).repeat_interleave(Hq // Hkv, dim=2)[:, :, None].to(torch.bfloat16)
    return k, qw


def _heads_first(t):
    return t.permute(0, 1, 3, 2, 4)   # the logical order of the entry points, [L, B, Hkv, N, d]


def _compressed_cache(s, gen):
    """A filled ragged cache: the budgets of a sequence's cells differ and sum to the sequence's total."""
    sh = s.sh
    cells = sh.n_kv_heads if sh.per_kv_head else 1
    total = ac.aircache_kept_per_sequence(sh, s.ratio)
    share = 0.5 + torch.rand((sh.batch, sh.n_layers * cells), generator=gen, device=_DEV, dtype=torch.float64)
    ends = (share.cumsum(1) / share.sum(1, keepdim=True) * total).round().to(torch.int64)
    kept = torch.diff(ends, dim=1, prepend=torch.zeros_like(ends[:, :1]))
    kept = kept.view(sh.batch, sh.n_layers, cells).transpose(0, 1).reshape(-1)
    s.lens.copy_(kept + sh.n_text)
    s.offsets[1:] = (kept + sh.n_text + sh.slack).cumsum(0)
    s.k_c.normal_(generator=gen)
    s.v_c.normal_(generator=gen)


def _prepare_attn(case, gen):
    s = Session(_shape(case), case["ratio"], device=_DEV)
    _compressed_cache(s, gen)
    return dict(s=s, q=_normal(tuple(s.out.shape), gen))


def _prepare_steps(case, gen):
    s = Session(_shape(case), case["ratio"], device=_DEV)
    _compressed_cache(s, gen)
    L, B, Hq, d = s.out.shape
    new = (case["rounds"], L, B, s.sh.n_kv_heads, d)
    return dict(s=s, lens=s.lens.clone(), q=_normal((case["rounds"], L, B, Hq, d), gen), k=_normal(new, gen),
                v=_normal(new, gen), out=torch.empty((case["rounds"], L, B, Hq, d), device=_DEV))


def _prepare_score(case, gen):
    s = Session(_shape(case), 0.1, case["alpha"], device=_DEV)
    k, qw = _keys_and_window(s.sh, gen)
    s.set_full(_heads_first(k), _heads_first(k))   # scoring reads no values
    return dict(s=s, qw=qw)


def _prepare_keep(case, gen):
    s = Session(_shape(case), case["ratio"], device=_DEV)
    sh = s.sh
    k = _normal((sh.n_layers, sh.batch, sh.n_visual + sh.n_text, sh.n_kv_heads, sh.head_dim), gen)
    v = _normal(tuple(k.shape), gen)
    s.set_full(_heads_first(k), _heads_first(v))
    # importance as softmax mass: log-normal, wider in some cells than in others, most of the mass on visual tokens
    x = torch.randn(tuple(s.scores.shape), generator=gen, device=_DEV)
    width = 0.3 + 0.9 * torch.rand(tuple(s.scores.shape[:-1]) + (1,), generator=gen, device=_DEV)
    mass = 0.8 + 0.2 * torch.rand(tuple(width.shape), generator=gen, device=_DEV)
    s.scores.copy_(torch.softmax(width * x, dim=-1) * mass)
    return dict(s=s)


def _pinned(t):
    h = torch.empty(t.shape, dtype=t.dtype, pin_memory=True)
    h.copy_(t)
    return h


def _prepare_host(case, gen):
    s = Session(_shape(case), case["ratio"], case["alpha"], device=_DEV)
    L, B, Hq, d = s.out.shape
    k, qw = _keys_and_window(s.sh, gen)
    v = _normal(tuple(k.shape), gen)
    q = _normal((case["rounds"], L, B, Hq, d), gen)
    out = torch.empty((case["rounds"], L, B, Hq, d), device=_DEV)
    return dict(s=s, h_k=_pinned(k), h_v=_pinned(v), h_qw=_pinned(qw), h_q=_pinned(q), d_k=k, d_v=v, d_qw=qw, d_q=q,
                d_out=out, h_out=torch.empty(out.shape, pin_memory=True),
                h_budgets=torch.empty(s.budgets.shape, dtype=torch.int32, pin_memory=True))


_PREPARE = dict(attn=_prepare_attn, steps=_prepare_steps, score=_prepare_score, layers=_prepare_score,
                keep=_prepare_keep, host=_prepare_host)


def prepare(case, seed):
    gen = torch.Generator(device=_DEV)
    gen.manual_seed(seed)
    state = _PREPARE[case["kind"]](case, gen)
    state["case"] = case
    return state


# ---------------------------------------------------------------------------------------------
# one pass
# ---------------------------------------------------------------------------------------------
def _run_attn(st):
    st["s"].decode(st["q"])
    return st["s"].out


def _run_steps(st):
    s = st["s"]
    s.lens.copy_(st["lens"])   # the request starts again behind its compressed prompt
    for i in range(st["case"]["rounds"]):
        ac.aircache_decode_step(s.sh, s.cache, st["q"][i], st["k"][i], st["v"][i], i, st["out"][i], s.ws)
    return st["out"], s.k_c, s.v_c, s.lens


def _run_score(st):
    st["s"].score(st["qw"])
    return st["s"].scores, st["s"].mask


def _run_layers(st):
    s = st["s"]
    for l in range(s.sh.n_layers):
        ac.aircache_score_layers(s.sh, s.full, st["qw"], s.alpha, l, 1, s.scores, s.mask, s.ws)
    return s.scores, s.mask


def _run_keep(st):
    s = st["s"]
    s.budget()
    s.compact()
    return s.budgets, s.strength, s.skew, s.offsets, s.lens, s.kept[:s.kept_n], s.k_c, s.v_c


def _run_host(st):
    s, case = st["s"], st["case"]
    h_full = ac.full_view(_heads_first(st["h_k"]), _heads_first(st["h_v"]))
    ac.aircache_pipeline_host(s.sh, h_full, st["h_k"].numel(), st["d_k"], st["d_v"], st["h_qw"], st["d_qw"],
                              st["h_q"], st["d_q"], case["rounds"], s.alpha, s.ratio, 0, s.scores, s.budgets, s.cache,
                              st["d_out"], st["h_out"], st["h_budgets"], s.ws)
    return st["h_out"], st["h_budgets"]


_RUN = dict(attn=_run_attn, steps=_run_steps, score=_run_score, layers=_run_layers, keep=_run_keep, host=_run_host)


def run(state):
    return _RUN[state["case"]["kind"]](state)


# ---------------------------------------------------------------------------------------------
# what a pass cannot do without
# ---------------------------------------------------------------------------------------------
def work(case):
    kind = case["kind"]
    L, Hq, Hkv, d = _MODELS[case["model"]]
    LB = L * case["batch"]
    row = 2 * Hkv * d   # bytes of a token's keys (or values) in one layer
    rounds = case.get("rounds", 1)
    bytes_, flops = 0.0, 0.0
    if kind in ("score", "layers", "host"):
        W = case["window"]
        queries = W if case["alpha"] == 0 else 1   # elite queries per head: all of them, or the best one at least
        bytes_ += LB * (case["visual"] * row + W * row + W * Hq * d * 2)
        flops += 2.0 * LB * case["visual"] * Hq * d * queries
        if kind != "host":
            bytes_ += 4.0 * LB * case["visual"] * (Hkv if case["heads"] else 1)
    if "ratio" in case:
        # rows (of all KV heads) of the compressed cache
        rows = case["batch"] * math.floor(case["ratio"] * case["visual"] * L + 0.5) + LB * case["text"]
        if kind == "keep":
            bytes_ += 4.0 * LB * case["visual"] * (Hkv if case["heads"] else 1) + 2 * 2 * row * rows
        if kind == "host":
            bytes_ += 2 * 2 * row * rows
        if kind in ("attn", "steps", "host"):
            bytes_ += rounds * (2.0 * row * rows + 6.0 * Hq * d * LB)
            flops += rounds * 4.0 * Hq * d * rows
        if kind == "steps":
            grown = LB * (rounds - 1) * rounds / 2   # the tokens appended in earlier rounds are read again
            bytes_ += 2.0 * row * grown + rounds * 2 * 2.0 * row * LB
            flops += 4.0 * Hq * d * grown
    return {"bytes": bytes_, "flops": flops}


def tolerance(case):
    # Measured against the same path in 64 bits (relative error of the whole, largest error of one value), and stated
    # about four times as large.
    if case["kind"] == "keep":
        # whole numbers and copied rows; the moments are sums of up to 9000 terms in 64 bits (6e-16; another order of
        # such a sum differs by up to 1e-14)
        return {"rel": 1e-13, "max": 1e-12}
    if case["kind"] == "host":
        # Rounding of the scores (2e-7) can let two tokens with nearly equal scores change places at a layer's
        # budget; one token of some 800 then differs in that layer, which is 5e-2 of its attention output and, over
        # 28 layers, 1e-2 of the whole.
        return {"rel": 1e-2, "max": 0.5}
    if case["kind"] in ("attn", "steps"):
        # 32-bit sums of exact products, probabilities of 16 bits or more (2.2e-6, 1.1e-5)
        return {"rel": 1e-5, "max": 5e-5}
    # 32-bit logits and softmax sums (2.3e-7, 6.7e-7 with a few elite rows; larger logits round more coarsely)
    return {"rel": 2e-6, "max": 1e-5}
