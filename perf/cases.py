"""The workloads this library is measured on, through its public entry points.

Two families of model shapes, the ones the benchmark and the tests use: Pythia-160M (12 layers of 12
query heads, head_dim 64, one to four KV heads per owner layer) and Llama-2-7B (32 layers of 32
heads, head_dim 128, 8 KV heads), with the layer-to-owner maps of MLKV, GQA and MQA.  A case is one
of five kinds of call:

  step      one mlkv_decode_step: every layer of one decode step, all queries at hand
  host      the same with the step's tensors in page-locked host memory (mlkv_decode_step_host),
            the outputs awaited on the host: the call as a client of the library sees it
  layers    the step layer by layer (mlkv_append_decode_attention for owner layers,
            mlkv_decode_attention for the others), as a model runs it whose layer n queries come
            from layer n - 1
  prefill   the prompt of every sequence through an owner layer and the readers of its cache
  merge     the conversion of an MHA projection's weights to MLKV (mlkv_merge_kv_weights)

Inputs are bf16 normals (the Llama keys at half the scale, as a trained model's logits are less
spread than random ones); lengths are one for all sequences or uniform in [1, L].
"""
import math
import random

import torch

import paper_2406_09297_gb300 as mlkv

MODELS = {"pythia": {"l": 12, "h": 12, "d": 64, "sigma_k": 1.0},
          "llama": {"l": 32, "h": 32, "d": 128, "sigma_k": 0.5}}


def _step(name, kind, model, m, g, b, L, ragged=False):
    return {"name": name, "kind": kind, "model": model, "layers": MODELS[model]["l"], "m": m, "g": g,
            "b": b, "L": L, "ragged": ragged}


def _prefill(name, model, readers, g, b, L, ragged=False):
    return {"name": name, "kind": "prefill", "model": model, "layers": 1 + readers, "m": 1, "g": g,
            "b": b, "L": L, "ragged": ragged}


def listed():
    return [
        # one user, a short chat turn: nothing but latency
        _step("step-pythia-mlkv6-b1-L128", "step", "pythia", 6, 1, 1, 128),
        # a serving batch in the middle of its generation: the benchmark's own workload
        _step("step-pythia-mlkv2-b64-L2048", "step", "pythia", 2, 1, 64, 2048),
        # continuous batching: every sequence at a length of its own, KV heads shared both ways
        _step("step-pythia-mlkv4-gqa4-b128-ragged4096", "step", "pythia", 4, 4, 128, 4096, True),
        # the large model under load: streaming the cache is all there is
        _step("step-llama-mlkv8-gqa4-b32-L4096", "step", "llama", 8, 8, 32, 4096),
        # one very long document
        _step("step-pythia-mlkv2-b1-L131072", "step", "pythia", 2, 1, 1, 131072),
        # the serving batch as a client calls it, host memory to host memory
        _step("host-pythia-mlkv2-b64-L2048", "host", "pythia", 2, 1, 64, 2048),
        # a model's own forward pass, layer after layer: the serving batch, and a ragged small one
        _step("layers-pythia-mlkv2-b64-L2048", "layers", "pythia", 2, 1, 64, 2048),
        _step("layers-llama-mlkv8-gqa4-b8-ragged3000", "layers", "llama", 8, 8, 8, 3000, True),
        # prompts: one batch of full-length ones for each head_dim, and many short uneven ones
        _prefill("prefill-pythia-mlkv2-b8-S2048", "pythia", 1, 1, 8, 2048),
        _prefill("prefill-pythia-gqa4-b32-ragged777", "pythia", 1, 4, 32, 777, True),
        _prefill("prefill-llama-gqa4-b4-S2048", "llama", 1, 8, 4, 2048),
        # uptraining starts from a merged checkpoint: one projection of the large model
        {"name": "merge-llama-mlkv8-gqa4", "kind": "merge", "model": "llama", "layers": 32, "m": 8,
         "g": 8, "d_model": 4096},
    ]


def draw(rng):
    kind = rng.choice(["step", "step", "host", "layers", "layers", "prefill", "prefill", "merge"])
    model = rng.choice(["pythia", "pythia", "llama"])
    s = MODELS[model]
    if kind == "merge":
        m = rng.choice([1, 2, 3, 4, 6, 12] if model == "pythia" else [4, 8, 16, 32])
        g = rng.choice([1, 3, 4, 6] if model == "pythia" else [8, 16])
        return {"kind": kind, "model": model, "layers": s["l"], "m": m, "g": g,
                "d_model": 8 * rng.randint(32, 96 if model == "pythia" else 512)}
    ragged = rng.random() < 0.5
    g = rng.choice([1, 3, 4, 12] if model == "pythia" else [2, 4, 8])
    top = {"step": 131072, "host": 16384, "layers": 16384, "prefill": 4096}[kind]
    L = max(1, min(top, round(math.exp(rng.uniform(math.log(16), math.log(top * 1.05))))))
    b = max(1, round(math.exp(rng.uniform(0.0, math.log(256)))))
    if kind == "prefill":
        c = dict(_prefill("", model, rng.choice([0, 1, 2]), g, b, L, ragged))
        limit = 4e11
    else:
        m = rng.choice([1, 2, 3, 4, 6, 12] if model == "pythia" else [4, 8, 16])
        c = dict(_step("", kind, model, m, g, b, L, ragged))
        limit = 4e9
    del c["name"]
    size = (lambda: work(c)["flops"]) if kind == "prefill" else (
        lambda: 4.0 * c["m"] * c["b"] * c["g"] * c["L"] * s["d"])
    while size() > limit:   # no more than the largest listed one
        if c["b"] > 1:
            c["b"] = max(1, c["b"] * 2 // 3)
        else:
            c["L"] = max(1, c["L"] * 2 // 3)
    return c


# ------------------------------------------------------------------------------------------------
# inputs
# ------------------------------------------------------------------------------------------------


def _lens(case):
    """The sequences' lengths: part of the case, not of its inputs."""
    if not case["ragged"]:
        return [case["L"]] * case["b"]
    r = random.Random("%(model)s %(b)d %(L)d" % case)
    return [r.randint(1, case["L"]) for _ in range(case["b"])]


def _normal(seed, what, shape, sigma=1.0):
    gen = torch.Generator(device="cuda").manual_seed((seed * 1000003 + what) % (1 << 62))
    return torch.empty(shape, dtype=torch.bfloat16, device="cuda").normal_(0.0, sigma, generator=gen)


def _q(case, seed, layer):
    s = MODELS[case["model"]]
    rows = (case["b"], case["L"]) if case["kind"] == "prefill" else (case["b"],)
    return _normal(seed, 1000 + layer, rows + (s["h"], s["d"]))


def _kv(case, seed, slot):
    """One owner's keys and values at positions [0, L)."""
    s = MODELS[case["model"]]
    shape = (case["b"], case["g"], case["L"], s["d"])
    return _normal(seed, 2000 + slot, shape, s["sigma_k"]), _normal(seed, 3000 + slot, shape)


def _new(case, seed, slot):
    """One owner's new token."""
    s = MODELS[case["model"]]
    shape = (case["b"], case["g"], s["d"])
    return _normal(seed, 4000 + slot, shape, s["sigma_k"]), _normal(seed, 5000 + slot, shape)


def _weights(case, seed):
    s = MODELS[case["model"]]
    return _normal(seed, 6000, (s["l"], s["h"], s["d"] * case["d_model"]), 0.02)


def _owners(case):
    per = case["layers"] // case["m"]
    return [n - n % per for n in range(case["layers"])]


class _DeviceMemory:
    """A view of cache memory for torch; it keeps the cache alive as long as a tensor uses it."""

    def __init__(self, cache, ptr, shape, strides):
        self.cache = cache
        self.__cuda_array_interface__ = {"data": (ptr, False), "shape": shape, "typestr": "<i2",
                                         "strides": tuple(2 * x for x in strides), "version": 3}


def _stored(cache, case, lens):
    """What a step or a prefill stores, where it lies in the cache: the new token's position (one
    length for all), every position (uneven lengths), or the prompt."""
    views = []
    for slot in range(case["m"]):
        k, v, st = cache.kv_ptr(slot)
        for ptr in (k, v):
            t = torch.as_tensor(_DeviceMemory(cache, ptr, (cache.b, cache.g, cache.max_seq, cache.d),
                                              st), device="cuda").view(torch.bfloat16)
            views.append(t if case["ragged"] or case["kind"] == "prefill" else t[:, :, lens[0] - 1])
    return views[:16]


def prepare(case, seed):
    s = MODELS[case["model"]]
    if case["kind"] == "merge":
        return {"case": case, "owner": _owners(case), "W": _weights(case, seed),
                "out": torch.zeros((case["m"], case["g"], s["d"] * case["d_model"]),
                                   dtype=torch.bfloat16, device="cuda")}
    lens = _lens(case)
    cache = mlkv.MLKVCache(case["layers"], s["h"], s["d"], _owners(case), case["g"], case["b"],
                           case["L"])
    state = {"case": case, "cache": cache, "lens": mlkv.as_seq_lens(lens), "owner": _owners(case)}
    q = [_q(case, seed, n) for n in range(case["layers"])]
    if case["kind"] == "prefill":
        state["K"], state["V"] = _kv(case, seed, 0)
        state["Q"], state["out"] = q, [torch.zeros_like(x) for x in q]
        state["stored"] = _stored(cache, case, lens)
        return state
    per = case["layers"] // case["m"]
    for slot in range(case["m"]):
        k, v = _kv(case, seed, slot)
        cache.load_prefix(slot * per, k, v, case["L"])
    new = [_new(case, seed, slot) for slot in range(case["m"])]
    Q, K, V = torch.stack(q), torch.stack([k for k, _ in new]), torch.stack([v for _, v in new])
    out = torch.zeros_like(Q)
    state["stored"] = _stored(cache, case, lens)
    if case["kind"] == "host":
        Q, K, V, out = [x.cpu().pin_memory() for x in (Q, K, V, out)]
    if case["kind"] == "layers":
        Q, out = list(Q), list(out)
        K = {slot * per: k for slot, k in enumerate(K)}
        V = {slot * per: v for slot, v in enumerate(V)}
    state.update(Q=Q, K=K, V=V, out=out)
    torch.cuda.synchronize()   # the cache copies its prefix from tensors that end here
    return state


def run(state):
    kind = state["case"]["kind"]
    if kind == "merge":
        case = state["case"]
        mlkv.mlkv_merge_kv_weights(state["owner"], MODELS[case["model"]]["h"], case["g"],
                                   state["W"], state["out"])
        return state["out"]
    cache, lens, Q, K, V, out = (state[k] for k in ("cache", "lens", "Q", "K", "V", "out"))
    if kind == "step":
        cache.decode_step(Q, K, V, out, lens)
    elif kind == "host":
        cache.decode_step_host(Q, K, V, out, lens)
        torch.cuda.current_stream().synchronize()   # the client reads the outputs
    elif kind == "layers":
        for n, o in enumerate(state["owner"]):
            if n == o:
                cache.append_decode_attention(n, K[n], V[n], Q[n], out[n], lens)
            else:
                cache.decode_attention(n, Q[n], out[n], lens)
    else:
        for n, o in enumerate(state["owner"]):
            cache.prefill(n, Q[n], K if n == o else None, V if n == o else None, out[n], lens)
    return {"out": out, "stored": state["stored"]}


# ------------------------------------------------------------------------------------------------
# what a pass cannot do without, and how far correct results may lie apart
# ------------------------------------------------------------------------------------------------


def work(case):
    s = MODELS[case["model"]]
    if case["kind"] == "merge":
        row = s["d"] * case["d_model"]
        return {"bytes": 2.0 * row * (s["l"] * s["h"] + case["m"] * case["g"]),
                "flops": 1.0 * row * s["l"] * s["h"]}
    lens, l, h, d, m, g = _lens(case), case["layers"], s["h"], s["d"], case["m"], case["g"]
    total = float(sum(lens))
    if case["kind"] == "prefill":
        # queries in, outputs out, the prompt's K/V in and (all s_max positions) into the cache
        return {"bytes": l * total * h * d * 2 * 2 + 2 * 2 * (total + case["b"] * case["L"]) * g * d,
                "flops": 4.0 * l * h * d * sum(n * (n + 1) / 2 for n in lens)}
    # every owner's visible K/V once, queries and outputs, the new tokens in and into the cache
    return {"bytes": 4.0 * m * g * d * total + 4.0 * l * case["b"] * h * d + 8.0 * m * case["b"] * g * d,
            "flops": 4.0 * l * h * d * total}


def tolerance(case):
    if case["kind"] == "merge":
        return {"rel": 1e-3, "max": 8e-3}   # bf16 from the exact mean: at most a neighbour now and then
    # bf16 weights and bf16 outputs around fp32 sums
    return {"rel": 8e-3, "max": 6e-2}


# ------------------------------------------------------------------------------------------------
# the same in 64 bits
# ------------------------------------------------------------------------------------------------


def _attend(q, k, v, lens, causal):
    """softmax(q k^T / sqrt(d)) v for q [b][h][d] (one token) or [b][s][h][d] (a causal prompt)."""
    b, g, L, d = k.shape
    out = torch.zeros(q.shape, dtype=torch.float64, device="cuda")
    pos = torch.arange(L, device="cuda")
    for i in range(b):
        n = lens[i]
        kk, vv = k[i, :, :n].double(), v[i, :, :n].double()
        if causal:
            qq = q[i, :n].double().view(n, g, -1, d).permute(1, 2, 0, 3)   # [g][G][n][d]
            sc = torch.matmul(qq, kk.transpose(1, 2).unsqueeze(1)) / math.sqrt(d)
            sc = sc.masked_fill(pos[:n].view(1, 1, 1, n) > pos[:n].view(1, 1, n, 1), -math.inf)
            o = torch.matmul(torch.softmax(sc, -1), vv.unsqueeze(1))
            out[i, :n] = o.permute(2, 0, 1, 3).reshape(n, -1, d)
        else:
            sc = torch.matmul(q[i].double().view(g, -1, d), kk.transpose(1, 2)) / math.sqrt(d)
            out[i] = torch.matmul(torch.softmax(sc, -1), vv).reshape(-1, d)
    return out


def exact(case, seed):
    s = MODELS[case["model"]]
    if case["kind"] == "merge":
        W = _weights(case, seed).view(case["m"], s["l"] // case["m"], case["g"], s["h"] // case["g"], -1)
        return torch.stack([w.double().mean(dim=(0, 2)) for w in W])
    lens, per, outs, stored = _lens(case), case["layers"] // case["m"], [], []
    for slot in range(case["m"]):
        k, v = _kv(case, seed, slot)
        if case["kind"] != "prefill":
            kn, vn = _new(case, seed, slot)
            at = torch.tensor(lens, device="cuda") - 1
            rows = torch.arange(case["b"], device="cuda")
            k[rows, :, at], v[rows, :, at] = kn, vn
            stored += [None, None] if case["ragged"] else [kn.double(), vn.double()]
        else:
            stored += [k.double(), v.double()]
        for n in range(slot * per, (slot + 1) * per):
            outs.append(_attend(_q(case, seed, n), k, v, lens, case["kind"] == "prefill"))
    out = outs if case["kind"] in ("layers", "prefill") else torch.stack(outs)
    return {"out": out.cpu() if case["kind"] == "host" else out, "stored": stored[:16]}
