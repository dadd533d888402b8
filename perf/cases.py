"""The work that users of this library have it do, as cases that can be timed and compared.

Each case is one pass through the torch layer (``api.Evictor.run`` over a prefill cache, or the
decode steps of ``api.DecodeEvictor`` that end in an eviction), with the plan and the buffers that
a serving program keeps from pass to pass made beforehand. ``kind`` is "prefill" or "decode"; the
other fields are the cache's shape and the pass's options:

  layers, hq, hkv     layers and query / KV heads (Llama-3-8B and Mistral-7B 32 / 8, Qwen3-14B 40 / 8,
                      Nemotron-7B 28 / 4, multi-head 8 / 8)
  seqlens             the requests' cached tokens, as a text of numbers and spaces (prefill)
  window, budget      window queries, tokens kept per request and KV head
  dtype, sinks        "bf16" or "f32"; attention-sink tokens at the start of each request
  tau, option         softmax temperature; "" (the method's defaults), "full_covariance", "linear" or
                      "out_directions" (u = W v instead of the proxy u = v)
  requests, interval  decode: requests that fill together, decode steps from one eviction to the next

The pass over a cache in host memory (``api.HostEvictor``) runs the same kernels behind the host
link, whose rate is all of its time, so it has no case of its own.
"""

import math

import torch

from paper_2609_08131_gb300 import jacap_params
from paper_2609_08131_gb300.api import Cache, DecodeEvictor, Evictor
from paper_2609_08131_gb300.workloads import Workload, generate

D = 128


def _prefill(name, layers, hq, hkv, seqlens, budget, window=32, dtype="bf16", sinks=0, tau=10.0, option=""):
    c = {"kind": "prefill", "layers": layers, "hq": hq, "hkv": hkv, "seqlens": " ".join(str(n) for n in seqlens),
         "budget": budget, "window": window, "dtype": dtype, "sinks": sinks, "tau": tau, "option": option}
    return {"name": name, **c} if name else c


def _decode(name, layers, hq, hkv, requests, budget, interval):
    c = {"kind": "decode", "layers": layers, "hq": hq, "hkv": hkv, "requests": requests, "budget": budget,
         "interval": interval, "window": 32, "tau": 10.0}
    return {"name": name, **c} if name else c


# sixteen prompts between 2K and 64K tokens that a batch packs together
_RAGGED = (6231, 41987, 2304, 58113, 17020, 33391, 9600, 64502, 25111, 4097, 51200, 13873, 37449, 2999, 46026, 20533)


def listed():
    return [
        # one float32 layer of multi-head attention, as a model that is evaluated in float32 keeps it
        _prefill("f32_layer_4k", 1, 8, 8, (4096,), 256, dtype="f32"),
        # one layer right after its own prefill, a short prompt of an odd length: the smallest call a
        # serving program makes (it evicts layer by layer, so that no more than one layer is ever held whole)
        _prefill("layer_4k", 1, 32, 8, (4099,), 512),
        # four prompts of a chat service, the whole model, lengths as they come
        _prefill("chat_4_prompts", 32, 32, 8, (1500, 731, 3072, 2177), 256),
        # Llama-3-8B's cache after a prompt of 32K tokens: the headline workload
        _prefill("llama_32k", 32, 32, 8, (32768,), 512),
        # Mistral-7B, half the prompt, a wider window, attention sinks and a tenth of the tokens kept
        _prefill("mistral_16k", 32, 32, 8, (16384,), 1638, window=64, sinks=4),
        # a document of 128K tokens, under 1 % kept: the largest single request
        _prefill("llama_128k", 32, 32, 8, (131072,), 1024),
        # a packed batch of very different prompts, evicted a group of eight layers at a time
        _prefill("ragged_16_prompts", 8, 32, 8, _RAGGED, 512),
        # five query heads per KV head (Qwen3-14B) and seven (Nemotron-7B), odd lengths
        _prefill("qwen3_14b_9k", 40, 40, 8, (9001,), 900),
        _prefill("nemotron_7b_20k", 28, 28, 4, (20011,), 2048),
        # the method's variants: the window's full covariance, and the true output directions
        _prefill("full_covariance_16k", 16, 32, 8, (16384,), 512, option="full_covariance"),
        _prefill("out_directions_16k", 16, 32, 8, (16384,), 512, option="out_directions"),
        # decoding with a fixed number of reserved tokens: every step appends one token to each of four
        # requests, and every fourth step evicts them back to the budget
        _decode("decode_4_requests", 28, 28, 4, 4, 2048, 4),
    ]


def _between(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(("one", "one", "batch", "batch", "f32", "option", "decode"))
    heads = rng.choice(((32, 8), (32, 8), (40, 8), (28, 4), (8, 8), (16, 8), (48, 8), (64, 8)))
    if kind == "f32":
        hq, hkv = rng.choice(((8, 8), (32, 8), (28, 4)))
        n = _between(rng, 300, 16384)
        return _prefill("", rng.randint(1, 4), hq, hkv, (n,), _between(rng, 32, max(33, n // 4)), dtype="f32",
                        window=rng.choice((16, 32, 64)))
    if kind == "decode":
        hq, hkv = rng.choice(((28, 4), (32, 8)))
        requests = rng.choice((1, 1, 2, 4, 8))
        return _decode("", 28 if hkv == 4 else 32, hq, hkv, requests, _between(rng, 256, 8192 // requests),
                       rng.randint(1, 6))
    if kind == "batch":
        seqs = rng.randint(2, 24)
        total = _between(rng, 200 * seqs, 200000)
        weights = [rng.uniform(0.05, 1.0) for _ in range(seqs)]
        lens = tuple(max(40, int(total * w / sum(weights))) for w in weights)
        return _prefill("", rng.randint(1, 8), *heads, lens, _between(rng, 32, 1024), window=rng.choice((16, 32, 64)))
    n = _between(rng, 500, 120000)
    layers = rng.choice((1, 2, 4, 8, 16, 32))
    while layers > 1 and layers * heads[1] * n > 16_000_000:
        layers //= 2
    budget = _between(rng, 64, max(65, min(4096, n // 2)))
    if kind == "option":
        option = rng.choice(("full_covariance", "out_directions", "linear"))
        window = rng.choice((16, 32)) if option == "full_covariance" else 32
        return _prefill("", layers, *heads, (n,), budget, window=window, option=option)
    return _prefill("", layers, *heads, (n,), budget, window=rng.choice((16, 32, 64)), sinks=rng.choice((0, 0, 4)),
                    tau=rng.choice((10.0, 10.0, 5.0, 20.0)))


def _seqlens(case):
    return [int(n) for n in case["seqlens"].split()]


def _params(case):
    option = case.get("option", "")
    return jacap_params(tau=case["tau"], full_covariance=int(option == "full_covariance"),
                        linear_weighting=int(option == "linear"))


def _cache(case, seed):
    """The prefill cache (per-channel scales, window queries that share a latent with the keys)."""
    f32 = case["dtype"] == "f32"
    return generate(Workload("case", case["layers"], case["hq"], case["hkv"], tuple(_seqlens(case)), case["window"],
                             case["budget"], dtype=case["dtype"], dist="outlier" if f32 else "latent", seed=seed,
                             outlier_channels=4 if f32 else 0, outlier_scale=8.0, sink_tokens=case["sinks"],
                             sink_scale=4.0), "cuda")


def _out_factor(case, seed):
    """F with F^T F = W^T W for a map W of 512 x 128 per layer and KV head (four heads' output slices)."""
    g = torch.Generator(device="cuda").manual_seed(seed + 77)
    w = torch.randn(case["layers"], case["hkv"], 512, D, generator=g, device="cuda", dtype=torch.float64) / math.sqrt(D)
    return torch.linalg.cholesky(w.mT @ w).mT.float().contiguous()


def _decode_tokens(case, seed):
    """The prefilled slots, the window queries and the tokens of the decode steps up to the eviction."""
    S, L, Hq, Hkv = case["requests"], case["layers"], case["hq"], case["hkv"]
    B, steps, G = case["budget"], case["interval"], case["hq"] // case["hkv"]
    g = torch.Generator(device="cuda").manual_seed(seed)

    def randn(*shape):
        return torch.randn(*shape, generator=g, device="cuda")

    sk, sv = torch.exp(0.5 * randn(1, L, Hkv, 1, D)), torch.exp(0.5 * randn(1, L, Hkv, 1, D))
    z = randn(S, L, Hkv, B + steps, D)  # the latent that a position's key and queries share
    k = (sk * (math.sqrt(0.3) * z + math.sqrt(0.7) * randn(S, L, Hkv, B + steps, D))).bfloat16()
    v = (sv * randn(S, L, Hkv, B + steps, D)).bfloat16()
    w = case["window"] + steps
    zq = z[:, :, :, -w:].repeat_interleave(G, dim=2)
    q = (math.sqrt(0.3) * zq + math.sqrt(0.7) * randn(S, L, Hq, w, D)).bfloat16()
    return k, v, q


def prepare(case, seed):
    if case["kind"] == "decode":
        B, w = case["budget"], case["window"]
        k, v, q = _decode_tokens(case, seed)
        dec = DecodeEvictor(case["requests"], case["layers"], case["hq"], case["hkv"], B, case["interval"],
                            params=_params(case))
        dec.start(k[:, :, :, :B], v[:, :, :, :B], q[:, :, :, :w], [B] * case["requests"])
        steps = [(k[:, :, :, B + j].contiguous(), v[:, :, :, B + j].contiguous(), q[:, :, :, w + j].contiguous())
                 for j in range(case["interval"])]
        return {"dec": dec, "steps": steps}
    t = _cache(case, seed)
    out = _out_factor(case, seed) if case["option"] == "out_directions" else None
    cache = Cache(t.q_win, t.k, t.v, t.cu_seqlens, t.seqlens, case["hq"])
    return {"ev": Evictor(cache, case["budget"], _params(case), out_factor=out)}


def _bits(x):
    """Copied rows are compared as the whole numbers that their bytes are."""
    return x.view(torch.int16 if x.dtype == torch.bfloat16 else torch.int32)


def run(state):
    if "dec" in state:
        dec = state["dec"]
        for k, v, q in state["steps"]:
            dec.step(k, v, q)
        return {"scores": dec.scores, "idx": dec.idx, "pos": dec.pos, "k": _bits(dec.k), "v": _bits(dec.v),
                "stats": dec.stats, "counts": dec.counts}
    ev = state["ev"]
    ev.run()
    return {"scores": ev.scores, "idx": ev.idx, "kept": ev.kept, "k_out": _bits(ev.k_out), "v_out": _bits(ev.v_out)}


def work(case):
    """Q window, K and V read once; scores, positions and the retained rows written once (decode: the new tokens
    written, and the rows that fill the evicted ones' places moved). Operations of a token and KV head: the logits
    and kappa of its G query heads, one triangle of the weighted Gram, and the triangular quadratic form; of a
    unit: its Cholesky factor."""
    L, Hkv, G = case["layers"], case["hkv"], case["hq"] // case["hkv"]
    if case["kind"] == "decode":
        S, B, T = case["requests"], case["budget"], case["interval"]
        tokens, units, es = S * (B + T), S * L * Hkv, 2
        moved = T * S * L * (2 * Hkv * D * es + case["hq"] * D * es)     # the steps' tokens, read ...
        moved += T * S * L * Hkv * 2 * D * es + 4 * T * S * L * Hkv      # ... and written, with their tags
        moved += 2 * 2 * T * S * L * Hkv * 2 * D * es                    # the rows that move, read and written
        moved += 2 * T * S * L * case["hq"] * 2 * D * 4                  # the running statistics
        nbytes = tokens * L * Hkv * (2 * D * es + 4) + 4 * units * B + moved
    else:
        lens, B = _seqlens(case), case["budget"]
        tokens, units = sum(lens), len(lens) * L * Hkv
        es = 4 if case["dtype"] == "f32" else 2
        nbytes = len(lens) * L * case["hq"] * case["window"] * D * es + tokens * L * Hkv * (2 * D * es + 4)
        nbytes += units * B * (4 + 2 * D * es)
    per_token = 2 * G * D * (2 if case.get("option") != "full_covariance" else 1 + case["window"]) + 2 * D * (D + 1)
    if case.get("option") == "out_directions":
        per_token += D * (D - 1)  # a full matrix instead of a triangular one
        nbytes += L * Hkv * D * D * 4
    return {"bytes": nbytes, "flops": tokens * L * Hkv * per_token + units * (2 * D ** 3 // 3)}


def tolerance(case):
    """Scores carry float32 sums and the splits of float32 values into two bf16 parts (2^-17 relative per product,
    averaged out over a score's many); against ``exact`` they measure 2e-7 (float32 caches) to 1.0e-6. Positions and
    copied rows may differ for near ties at the budget: one such tie shifts a unit's rows by a place up to the other."""
    return {"rel": 4e-6, "max": 2e-4, "differ": 0.01}


def _unit_scores(q, k, v, tau, mu=None, lam=None, full=False, linear=False, F=None):
    """Algorithm 1 up to the scores for one unit in float64: q [G, w, D], k and v [n, D]."""
    k, v = k.double(), v.double()
    if mu is None:
        q = q.double()
        mu = q.mean(1)
        dev = q - mu[:, None]
        lam = dev.square().mean(1)
    if full:
        kappa = torch.stack([(k @ d.T).square().mean(1) for d in dev])
    else:
        kappa = lam @ k.square().T
    a = torch.softmax(mu @ k.T / (tau * math.sqrt(D)), dim=1)
    rho = torch.ones_like(a) if linear else a * (1 - a)
    w = (rho.square() * kappa).sum(0) / D
    u = v if F is None else v @ F.double().T
    A = torch.eye(D, dtype=torch.float64, device=k.device) + u.T @ (w[:, None] * u)
    y = torch.linalg.solve_triangular(torch.linalg.cholesky(A), u.T, upper=False)
    return w * y.square().sum(0)


def exact(case, seed):
    L, Hkv, G = case["layers"], case["hkv"], case["hq"] // case["hkv"]
    if case["kind"] == "decode":
        S, cap = case["requests"], case["budget"] + case["interval"]
        k, v, q = _decode_tokens(case, seed)
        qd = q.double()
        mean = qd.mean(3)
        m2 = (qd - mean[:, :, :, None]).square().sum(3)
        scores = torch.empty((L, Hkv, S * cap), dtype=torch.float64, device="cuda")
        for s in range(S):
            for l in range(L):
                for g in range(Hkv):
                    h = slice(g * G, (g + 1) * G)
                    scores[l, g, s * cap:(s + 1) * cap] = _unit_scores(
                        None, k[s, l, g], v[s, l, g], case["tau"], mean[s, l, h], m2[s, l, h] / qd.shape[3])
        return {"scores": scores, "idx": None, "pos": None, "k": None, "v": None,
                "stats": torch.stack([mean, m2], dim=3), "counts": None}
    t = _cache(case, seed)
    F = _out_factor(case, seed) if case["option"] == "out_directions" else None
    scores = torch.empty((L, Hkv, t.k.shape[2]), dtype=torch.float64, device="cuda")
    at = 0
    for s, n in enumerate(t.seqlens):
        for l in range(L):
            for g in range(Hkv):
                scores[l, g, at:at + n] = _unit_scores(
                    t.q_win[s, l, g * G:(g + 1) * G], t.k[l, g, at:at + n], t.v[l, g, at:at + n], case["tau"],
                    full=case["option"] == "full_covariance", linear=case["option"] == "linear",
                    F=None if F is None else F[l, g])
        at += n
    return {"scores": scores, "idx": None, "kept": None, "k_out": None, "v_out": None}
