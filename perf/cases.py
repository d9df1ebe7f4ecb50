"""The serving steps whose speed is looked after: what a program that serves models with this library has it do.

A case is one serving step of one context: the requests of every placed model are submitted, the step is launched,
and the answers of earlier steps are collected while it runs, the way a serving loop keeps the device busy.  The
families are the workload configurations of this repository: small MLPs, ViT encoders, Llama-style decoders
(decode, whole prompts, prompt chunks beside decode requests) and the co-resident mix of all three.

Sizes are those of paper_2511_00603_b200/configs.py.  Weights are random with biases and gains that carry signal.
Two things are set the way trained models have them and random ones do not, so that a tie does not decide the answer
of a request: a classifier prefers a class by several standard deviations of its logits (head bias), and a decoder's
LM head is its embedding (scaled), which makes the next token decisive.
"""
from __future__ import annotations

import collections
import ctypes as C
import math

import numpy as np
import torch

from paper_2511_00603_b200 import configs
from paper_2511_00603_b200 import epara as E
from paper_2511_00603_b200 import synth
from paper_2511_00603_b200.server import Server

MLP_STD = 0.06          # keeps the activations of a 512-wide layer near unit variance
PERTURB = 0.05          # gains 1 + N(0, 0.05), biases N(0, 0.05)
VITS = {"vit_s": configs.VIT_S, "vit_b": configs.VIT_B}
DECODERS = {"dec_1b": configs.DEC_1B, "dec_8b": configs.DEC_8B}
CACHE_PIECE = 1 << 30   # elements; a large cache is returned in pieces of whole layers


def listed():
    return [
        # the two-model step of small MLPs (8 latency-sensitive and 32 frequency-sensitive requests): a step of a
        # handful of kernels, where the calls and the launches are the time
        {"name": "mlp_two_models", "family": "mlp", "ls": 8, "fs": 32},
        # one image through ViT-B/16: the latency of a single classification request
        {"name": "vit_b_1", "family": "vit", "model": "vit_b", "batch": 1, "capacity": 1, "mf": 0},
        # the large ViT-B/16 batch of the vision configuration
        {"name": "vit_b_64", "family": "vit", "model": "vit_b", "batch": 64, "capacity": 64, "mf": 0},
        # video: 29 streams of ViT-S/16, seven frames from each, grouped by the multi-frame rule; an odd batch
        {"name": "vit_s_203_frames", "family": "vit", "model": "vit_s", "batch": 203, "capacity": 203, "mf": 7},
        # a single chat: one token of the 1B decoder
        {"name": "decode_1b_1", "family": "decoder", "model": "dec_1b", "decode": 1, "capacity": 1, "kv_lo": 128, "kv_hi": 4096,
         "prompts": 0, "prompt_len": 0, "prefix": 0},
        # a moderately loaded decoder: 27 requests on an instance placed for 32
        {"name": "decode_1b_27_of_32", "family": "decoder", "model": "dec_1b", "decode": 27, "capacity": 32, "kv_lo": 128, "kv_hi": 4096,
         "prompts": 0, "prompt_len": 0, "prefix": 0},
        # the full decode batch of the LLM configuration
        {"name": "decode_1b_128", "family": "decoder", "model": "dec_1b", "decode": 128, "capacity": 128, "kv_lo": 128, "kv_hi": 4096,
         "prompts": 0, "prompt_len": 0, "prefix": 0},
        # the 8B decoder (head size 128) with long caches
        {"name": "decode_8b_64", "family": "decoder", "model": "dec_8b", "decode": 64, "capacity": 64, "kv_lo": 512, "kv_hi": 4096,
         "prompts": 0, "prompt_len": 0, "prefix": 0},
        # time to first token of one short prompt of odd length
        {"name": "prompt_1b_509", "family": "decoder", "model": "dec_1b", "decode": 0, "capacity": 512, "kv_lo": 128, "kv_hi": 4096,
         "prompts": 1, "prompt_len": 509, "prefix": 0},
        # whole prompts in one step: the compute-bound end of serving a decoder
        {"name": "prompts_1b_4x2048", "family": "decoder", "model": "dec_1b", "decode": 0, "capacity": 8192, "kv_lo": 128, "kv_hi": 4096,
         "prompts": 4, "prompt_len": 2048, "prefix": 0},
        # chunked prefill: a 512-token chunk on a cached prefix shares its step with 24 decode requests
        {"name": "chunk_1b_512_and_24", "family": "decoder", "model": "dec_1b", "decode": 24, "capacity": 536, "kv_lo": 128, "kv_hi": 4096,
         "prompts": 1, "prompt_len": 512, "prefix": 1500},
        # the co-resident mix, saturated: 3 MLPs, 3 ViT-S/16 and 2 decoders, 4 latency-sensitive requests on the first
        # instance of a family and 256 frequency-sensitive ones on the others
        {"name": "mixed_saturated", "family": "mixed", "ls": 4, "fs": 256, "capacity": 256, "kv_lo": 128, "kv_hi": 4096},
    ]


def _log_int(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi + 1)) - 1e-9)))))


def draw(rng):
    """One more step of the same families: batches and lengths over the whole range, instances placed for what they
    carry or for more."""
    family = rng.choice(["mlp", "vit", "vit", "decode", "decode", "decode", "prompts", "prompts", "chunk", "mixed"])
    if family == "mlp":
        return {"family": "mlp", "ls": rng.randint(1, 8), "fs": _log_int(rng, 1, 256)}
    if family == "vit":
        model = rng.choice(["vit_s", "vit_b"])
        hi = 256 if model == "vit_s" else 64
        mf = rng.choice([0, 0, rng.randint(2, 8)])
        batch = _log_int(rng, 1, hi)
        if mf:
            batch = max(1, batch // mf) * mf if batch >= mf else batch
            mf = mf if batch >= mf else 0
        return {"family": "vit", "model": model, "batch": batch, "capacity": rng.choice([batch, min(hi, batch + rng.randint(0, batch))]), "mf": mf}
    if family == "decode":
        model = rng.choice(["dec_1b", "dec_1b", "dec_8b"])
        hi = 128 if model == "dec_1b" else 64
        n = _log_int(rng, 1, hi)
        return {"family": "decoder", "model": model, "decode": n, "capacity": rng.choice([n, min(hi, n + rng.randint(0, n))]),
                "kv_lo": rng.choice([128, 512]), "kv_hi": rng.randint(600, 4096), "prompts": 0, "prompt_len": 0, "prefix": 0}
    if family == "prompts":
        model = rng.choice(["dec_1b", "dec_1b", "dec_8b"])
        n = rng.randint(1, 4)
        length = _log_int(rng, 32, 2048 if model == "dec_1b" else 768)
        length = min(length, 2048 if model == "dec_1b" else 1024 // n)
        return {"family": "decoder", "model": model, "decode": 0, "capacity": n * length + rng.choice([0, rng.randint(0, 64)]), "kv_lo": 128,
                "kv_hi": 4096, "prompts": n, "prompt_len": length, "prefix": 0}
    if family == "chunk":
        n, length = rng.randint(1, 64), _log_int(rng, 16, 1024)
        return {"family": "decoder", "model": "dec_1b", "decode": n, "capacity": n + length + rng.randint(0, 64), "kv_lo": 128,
                "kv_hi": rng.randint(600, 4096), "prompts": 1, "prompt_len": length, "prefix": rng.randint(1, 3000)}
    fs = _log_int(rng, 4, 255)
    return {"family": "mixed", "ls": rng.randint(1, 4), "fs": fs, "capacity": rng.choice([fs, 256]), "kv_lo": 128, "kv_hi": rng.randint(600, 4096)}


# ------------------------------------------------------------------ what a program has in hand before the step
def _mlp(dims, seed, device):
    p = synth.make_mlp(dims, seed=seed, device=device, std=MLP_STD, perturb=PERTURB)
    p["b"][-1][seed % dims[-1]] += 8.0
    return p


def _vit(model, seed, device):
    p = synth.make_vit(seed=seed, device=device, perturb=PERTURB, **VITS[model])
    p["bhead"][seed % p["n_cls"]] += 4.0
    return p


def _decoder(model, seed, device):
    p = synth.make_decoder(seed=seed, device=device, perturb=PERTURB, **DECODERS[model])
    p["packed_layers"] = [synth.pack_decoder_layer(layer) for layer in p["layers"]]
    p["layers"] = None                               # the packed layout is all the library reads
    # (embedding of unit variance at 16 layers; more for deeper models, whose layers add up to a larger residual stream)
    p["Emb"] = (p["Wlm"].float() * 50.0 * (p["n_layers"] / 16.0) ** 2).to(torch.bfloat16)
    return p


def _workspace(specs, **cfg):
    """Bytes of workspace the models need; specs: (params, capacity, max_kv_len)."""
    config = E.Config(0, 256, 1 << 40, cfg.get("cap_ls", 0), cfg.get("cap_fs", 0), cfg.get("mf_max", 0), E.GEMM_TCGEN05, 0, 0)
    need = 64 << 20
    for p, capacity, max_kv_len in specs:
        pool = None
        if p["kind"] == "decoder":
            pool = torch.empty((p["n_layers"], 1, 2, p["n_kv_heads"], synth.PAGE, p["head_dim"]), dtype=torch.bfloat16, device="cuda")
        desc, _keep = E.make_model_desc(p, kv_pool=pool, max_kv_len=max_kv_len, max_batch=capacity)
        need += E.lib.epara_model_workspace_bytes(C.byref(config), C.byref(desc))
    return need


class _Requests:
    """The requests of one placed model: descriptors ready for epara_submit_many, inputs and outputs."""

    def __init__(self, mid, category, n, n_out, device):
        self.mid, self.category, self.n = mid, category, n
        self.logits = torch.zeros((n, n_out), dtype=torch.bfloat16, device=device)
        self.argmax = torch.full((n,), -1, dtype=torch.int32, device=device)
        self.inputs = (E.Inputs * n)()
        for i in range(n):
            self.inputs[i].out_logits = self.logits.data_ptr() + i * n_out * 2
            self.inputs[i].out_argmax = self.argmax.data_ptr() + i * 4
        self.keep = []
        self.cache = []

    def results(self):
        return [self.logits, self.argmax] + self.cache


def _add_dense(srv, p, category, n, capacity, seed, mf=0):
    if p["kind"] == "mlp":
        x, n_out = synth.make_mlp_inputs(n, p["dims"][0], seed, device=srv.device), p["dims"][-1]
    else:
        x, n_out = synth.make_images(n, seed, device=srv.device, img=p["img"]), p["n_cls"]
    q = _Requests(srv.add_model(p, max_batch=capacity), category, n, n_out, srv.device)
    q.keep.append(x)
    step = x[0].numel() * 2
    for i in range(n):
        q.inputs[i].input = x.data_ptr() + i * step
        q.inputs[i].stream = i // mf if mf else 0
    return q


def _cached(case, i):
    """Cached tokens of the i-th shortest decode request."""
    return case["kv_lo"] + int((case["kv_hi"] - case["kv_lo"]) * (int(i) + 0.5) / case["decode"])


def _add_decoder(srv, p, category, case, seed):
    """`decode` requests with cached lengths evenly spread over [kv_lo, kv_hi], in an order of the seed, and `prompts`
    chunks of prompt_len tokens on `prefix` cached ones; every sequence has pages of its own, spread over the pool."""
    n_dec, n_pre, length, prefix = case["decode"], case["prompts"], case["prompt_len"], case["prefix"]
    rng = np.random.default_rng(seed)
    lens = [_cached(case, i) for i in rng.permutation(n_dec)] + [prefix] * n_pre
    new = [1] * n_dec + [length] * n_pre
    pages = [-(-(a + b) // synth.PAGE) for a, b in zip(lens, new)]
    order = rng.permutation(sum(pages)).astype(np.int32)
    pool = synth.make_kv_pool(p["n_layers"], sum(pages), p["n_kv_heads"], p["head_dim"], seed + 1, device=srv.device)
    tables = torch.as_tensor(order, device=srv.device)
    mid = srv.add_model(p, kv_pool=pool, max_kv_len=max(case["kv_hi"], prefix + length), max_batch=case["capacity"])
    q = _Requests(mid, category, n_dec + n_pre, p["vocab"], srv.device)
    at = 0
    for i in range(n_dec + n_pre):
        toks = rng.integers(0, p["vocab"], new[i])
        inp = q.inputs[i]
        inp.token, inp.kv_len = int(toks[0]), lens[i]
        inp.block_table, inp.n_blocks = tables.data_ptr() + 4 * at, pages[i]
        if new[i] > 1:
            arr = (C.c_int32 * new[i])(*[int(t) for t in toks])
            inp.tokens, inp.n_tokens = arr, new[i]
            q.keep.append(arr)
        at += pages[i]
    q.keep += [tables, pool]
    per = max(1, CACHE_PIECE // pool[0].numel())
    q.cache = list(pool.split(per))
    return q


def prepare(case, seed):
    dev = torch.device("cuda", torch.cuda.current_device())
    family = case["family"]
    if family == "mlp":
        a, b = _mlp(configs.MLP_A, seed * 10, dev), _mlp(configs.MLP_B, seed * 10 + 1, dev)
        cfg = {"cap_ls": 8}
        srv = Server(device=dev.index, workspace_bytes=_workspace([(a, case["ls"], 0), (b, case["fs"], 0)], **cfg), **cfg)
        reqs = [_add_dense(srv, a, E.CAT_LS, case["ls"], case["ls"], seed * 10 + 2),
                _add_dense(srv, b, E.CAT_FS, case["fs"], case["fs"], seed * 10 + 3)]
    elif family == "vit":
        p = _vit(case["model"], seed * 10, dev)
        cfg = {"mf_max": case["mf"], "cap_fs": max(case["capacity"], case["batch"])}
        srv = Server(device=dev.index, workspace_bytes=_workspace([(p, case["capacity"], 0)], **cfg), **cfg)
        reqs = [_add_dense(srv, p, E.CAT_FS, case["batch"], case["capacity"], seed * 10 + 1, mf=case["mf"])]
    elif family == "decoder":
        p = _decoder(case["model"], seed * 10, dev)
        longest = max(case["kv_hi"], case["prefix"] + case["prompt_len"])
        srv = Server(device=dev.index, workspace_bytes=_workspace([(p, case["capacity"], longest)]))
        reqs = [_add_decoder(srv, p, E.CAT_FS, case, seed * 10 + 1)]
    else:
        specs, reqs = [], []
        for k, kind in enumerate(["mlp"] * 3 + ["vit"] * 3 + ["dec"] * 2):
            first = k in (0, 3, 6)
            p = (_mlp(configs.MLP_A, seed * 100 + k, dev) if kind == "mlp" else
                 _vit("vit_s", seed * 100 + k, dev) if kind == "vit" else _decoder("dec_1b", seed * 100 + k, dev))
            specs.append((p, case["ls"] if first else case["capacity"], case["kv_hi"] if kind == "dec" else 0))
        srv = Server(device=dev.index, workspace_bytes=_workspace(specs))
        for k, (p, capacity, _kv) in enumerate(specs):
            first = k in (0, 3, 6)
            n, cat = (case["ls"], E.CAT_LS) if first else (case["fs"], E.CAT_FS)
            if p["kind"] == "decoder":
                one = {"decode": n, "prompts": 0, "prompt_len": 0, "prefix": 0, "kv_lo": case["kv_lo"], "kv_hi": case["kv_hi"], "capacity": capacity}
                reqs.append(_add_decoder(srv, p, cat, one, seed * 100 + 20 + k))
            else:
                reqs.append(_add_dense(srv, p, cat, n, capacity, seed * 100 + 20 + k))
    return {"srv": srv, "requests": reqs, "in_flight": collections.deque()}


def run(state):
    """One pass of a serving loop: submit, step, and collect what earlier steps have finished by now."""
    srv, flying = state["srv"], state["in_flight"]
    tickets = [srv.ctx.epara_submit_many(q.mid, q.category, q.inputs, q.n) for q in state["requests"]]
    srv.step()
    while flying:
        status = srv.ctx.epara_collect(flying[0][0][0])[0]
        if status == E.PENDING:
            break
        first = True
        for tks in flying.popleft():
            for t in tks:
                if not first:
                    status = srv.ctx.epara_collect(t)[0]
                first = False
                if status != E.OK:
                    raise RuntimeError("request answered %s" % E.lib.epara_strerror(status).decode())
    flying.append(tickets)
    return [q.results() for q in state["requests"]]


# ------------------------------------------------------------------ the least work of one pass
def _dense_work(dims, n):
    w = sum(a * b for a, b in zip(dims, dims[1:]))
    return {"bytes": 2.0 * (w + sum(dims[1:]) + n * (dims[0] + dims[-1])) + 4.0 * n, "flops": 2.0 * w * n}


def _vit_work(model, n):
    c = VITS[model]
    d, layers, ffn, cls = c["d"], c["n_layers"], c["mlp"], c["n_cls"]
    tokens, per_layer = 197, 4 * c["d"] ** 2 + 2 * c["d"] * c["mlp"]
    w = layers * per_layer + d * 768 + tokens * d + cls * d
    flops = n * (2.0 * tokens * layers * per_layer + 4.0 * tokens * tokens * d * layers + 2.0 * 196 * 768 * d + 2.0 * cls * d)
    return {"bytes": 2.0 * (w + layers * (9 * d + ffn) + n * (3 * 224 * 224 + cls)) + 4.0 * n, "flops": flops}


def _decoder_work(model, case):
    c = DECODERS[model]
    d, layers, hd, hq, hkv = c["d"], c["n_layers"], c["head_dim"], c["n_q_heads"], c["n_kv_heads"]
    per_layer = d * (hq + 2 * hkv) * hd + d * hq * hd + 3 * d * c["ffn"]
    n_dec, n_pre, length, prefix = case["decode"], case["prompts"], case["prompt_len"], case["prefix"]
    rows, answers = n_dec + n_pre * length, n_dec + n_pre
    lens = sum(_cached(case, i) for i in range(n_dec))
    cached = lens + n_pre * prefix
    seen = lens + n_dec + n_pre * (length * prefix + length * (length + 1) / 2.0)
    kv_token = 2 * hkv * hd * layers
    w = layers * (per_layer + 2 * d) + d + c["vocab"] * d
    return {"bytes": 2.0 * (w + rows * d + (cached + rows) * kv_token + answers * c["vocab"]) + 4.0 * answers,
            "flops": 2.0 * rows * layers * per_layer + 2.0 * answers * c["vocab"] * d + 4.0 * hq * hd * layers * seen}


def work(case):
    family = case["family"]
    if family == "mlp":
        parts = [_dense_work(configs.MLP_A, case["ls"]), _dense_work(configs.MLP_B, case["fs"])]
    elif family == "vit":
        parts = [_vit_work(case["model"], case["batch"])]
    elif family == "decoder":
        parts = [_decoder_work(case["model"], case)]
    else:
        parts = []
        for n, times in ((case["ls"], 1), (case["fs"], 2)):
            parts += [_dense_work(configs.MLP_A, n), _vit_work("vit_s", n)] * times
        for n in (case["ls"], case["fs"]):
            parts.append(_decoder_work("dec_1b", {"decode": n, "prompts": 0, "prompt_len": 0, "prefix": 0, "kv_lo": case["kv_lo"], "kv_hi": case["kv_hi"]}))
    return {k: sum(p[k] for p in parts) for k in ("bytes", "flops")}


def tolerance(case):
    """About four times the difference between this path and itself with every sum in another order (plain CUDA-core
    kernels): 1.3e-4 / 6e-3 (relative 2-norm / largest element) for the MLPs, whose preferred class carries most of the
    norm, 4.6e-3 / 2.0e-2 for the encoders, 8.8e-3 / 5.0e-2 for the 16-layer decoders, in which one bf16 rounding that
    falls the other way is carried on by every later layer."""
    if case["family"] == "mlp":
        return {"rel": 0.002, "max": 0.025}
    if case["family"] == "vit":
        return {"rel": 0.018, "max": 0.08}
    return {"rel": 0.03, "max": 0.2}
