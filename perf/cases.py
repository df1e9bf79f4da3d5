"""The calls that users of the library make, as cases that can be timed and compared.

A case is a dict of plain values.  `kind` says which entry points it goes through:

  step        gram_step, Single-step: a whole training step with the Adam / Noam update
  window      gram_step, Multi-step: the K steps of one window, the last of which runs the encoder
  task        gram_task: the task module's forward and backward on given encodings
  encode      gram_encode_unique without saved activations (filling a cache, serving encodings)
  pass        gram_encode_unique with saved activations, then gram_encoder_backward
  dedup       gram_dedup
  accumulate  gram_accumulate: sums of gradient rows over the occurrences of an item
  gather      gram_gather: encodings copied to their occurrences

`prepare` draws everything from the seed on the GPU; `run` is one pass; `exact` is the same computation in 64-bit
torch, written from the model's definition (post-LayerNorm transformer encoder, causal or additive-attention task
module) without the library.
"""
import math

import numpy as np
import torch

from paper_2204_04179_b200 import binding, synth

LN_EPS = 1e-5


# --------------------------------------------------------------------------- the cases

def _case(kind, name=None, config="kt", **over):
    """A plain dict: the fields of a named workload of the package that matter for `kind`, with changes."""
    s = synth.config(config)
    keep = ["dtype", "n_items", "l_t", "vocab", "zipf_s", "d", "n_heads", "d_ff", "n_layers", "pooling", "task",
            "task_layers", "task_heads", "task_d_ff", "task_attn_only", "d_a", "n_cand", "B", "L"]
    c = {"kind": kind}
    c.update({k: getattr(s, k) for k in keep})
    c.update(K=1, micro=0, items=0, shortest=0)
    c.update(over)
    if name is not None:
        c["name"] = name
    return c


def _index_case(kind, P, n_items, zipf_s, d=0, dtype="f32", name=None):
    c = {"kind": kind, "P": P, "n_items": n_items, "zipf_s": zipf_s}
    if d:
        c.update(d=d, dtype=dtype)
    if name is not None:
        c["name"] = name
    return c


def listed():
    return [
        # the smallest whole call: the fp32 check-sized model, launches and host waits count
        _case("step", "tiny_step", config="tiny"),
        # an ordinary training step of the knowledge-tracing workload: 12 layers, 32 histories of 100 exercises
        _case("step", "kt_step", config="kt", B=32, micro=2048),
        # the news workload as configured: 64 users, 50 clicks + 5 candidates, titles of 32 tokens, 10^5 items
        _case("step", "nr_step", config="nr", micro=2048),
        # Multi-step training with the 6-layer encoder: three light steps, then the encoder over the touched items
        _case("window", "kt_window", config="kt_6l", B=64, K=4, micro=1024),
        # the task module at the knowledge-tracing batch: what a Multi-step light step consists of
        _case("task", "kt_task", config="kt", B=256),
        # encodings for a cache: texts of 4 to 64 tokens, mean pooling, two layers
        _case("encode", "encode_ragged", config="kt", n_layers=2, pooling="mean", items=2048, shortest=4),
        # the encoder's training pass, exercises of 64 tokens
        _case("pass", "pass_kt", config="kt", n_layers=2, items=1024),
        # the encoder's training pass on long texts (two attention tiles; one of the paper's datasets has 147 tokens
        # per item)
        _case("pass", "pass_long", config="kt", n_layers=2, l_t=147, pooling="mean", items=371),
        # the index of one knowledge-tracing batch
        _index_case("dedup", 25_600, 10_000, 1.0, name="dedup_step"),
        # the index at the far end of the kernel sweep
        _index_case("dedup", 10_000_000, 1_000_000, 1.1, name="dedup_large"),
        # the benchmark's cell for the two row movers: 10^6 positions of 768 columns over 10^5 items
        _index_case("accumulate", 1_000_000, 100_000, 1.1, 768, name="accumulate_large"),
        _index_case("gather", 1_000_000, 100_000, 1.1, 768, "bf16", name="gather_large"),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["tiny", "step", "step", "window", "task", "task", "encode", "pass", "pass", "dedup", "dedup",
                       "accumulate", "gather"])
    if kind == "tiny":           # fp32 models of the check's size and somewhat larger
        d = rng.choice([32, 64, 128])
        return _case("step", config="tiny", n_items=_log(rng, 50, 2000), l_t=rng.randint(4, 40), d=d, d_ff=4 * d,
                     n_layers=rng.randint(1, 3), task_layers=rng.randint(1, 2), task_attn_only=rng.random() < 0.5,
                     task_d_ff=4 * d, B=rng.randint(2, 24), L=rng.randint(5, 50),
                     pooling=rng.choice(["mean", "cls"]))
    if kind == "step":
        if rng.random() < 0.4:
            n = rng.randint(10, 60)
            return _case("step", config=rng.choice(["nr", "nr_mhsa", "nr_additive"]), n_layers=rng.randint(1, 6),
                         l_t=rng.randint(8, 48), B=_log(rng, 8, 64), L=n + 5, n_items=_log(rng, 3000, 100_000),
                         micro=2048)
        return _case("step", config="kt", n_layers=rng.randint(1, 6), l_t=rng.randint(12, 96), B=_log(rng, 4, 32),
                     L=rng.randint(20, 128), n_items=_log(rng, 500, 10_000), zipf_s=rng.choice([0.8, 1.0, 1.1]),
                     pooling=rng.choice(["cls", "cls", "mean"]), micro=1024)
    if kind == "window":
        return _case("window", config="kt", n_layers=rng.randint(1, 4), l_t=rng.randint(12, 64), B=_log(rng, 8, 64),
                     L=rng.randint(20, 100), n_items=_log(rng, 500, 4000), K=rng.choice([2, 4, 8]), micro=1024)
    if kind == "task":
        if rng.random() < 0.4:
            return _case("task", config=rng.choice(["nr", "nr_mhsa"]), B=_log(rng, 16, 512),
                         L=rng.randint(10, 60) + 5)
        return _case("task", config="kt", B=_log(rng, 8, 256), L=rng.randint(16, 100), task_layers=rng.randint(1, 2),
                     task_attn_only=rng.random() < 0.3)
    if kind in ("encode", "pass"):
        l_t = _log(rng, 5, 256)
        d = rng.choice([256, 512, 768, 768])
        return _case(kind, config="kt", n_layers=rng.randint(1, 2), l_t=l_t, d=d, n_heads=d // 64, d_ff=4 * d,
                     d_a=256, pooling=rng.choice(["mean", "cls", "additive" if l_t <= 128 else "mean"]),
                     items=max(4, min(4096, _log(rng, 1500, 65_536) // l_t)),
                     shortest=rng.choice([0, 0, max(1, l_t // 10)]))
    if kind == "dedup":
        return _index_case("dedup", _log(rng, 1000, 10_000_000), _log(rng, 100, 1_000_000),
                           rng.choice([0.8, 1.0, 1.1, 1.5]))
    d = rng.choice([64, 128, 200, 256, 768, 1024])
    P = min(_log(rng, 3000, 3_000_000), 768_000_000 // d)
    n = max(100, min(_log(rng, 100, 1_000_000), 400_000_000 // d))
    return _index_case(kind, P, n, rng.choice([0.8, 1.0, 1.1, 1.5]), d,
                       rng.choice(["bf16", "f32"]) if kind == "gather" else "f32")


# --------------------------------------------------------------------------- inputs

def _generator(seed, stream):
    return torch.Generator(device="cuda").manual_seed(int(seed) * 16 + stream)


def _zipf(seed, n_items, s, size, stream):
    """IDs: rank r with probability ~ (r+1)^-s, ranks scattered over the IDs."""
    g = _generator(seed, 1)
    perm = torch.randperm(n_items, generator=g, device="cuda")
    cdf = torch.cumsum(torch.arange(1, n_items + 1, device="cuda", dtype=torch.float64).pow(-float(s)), 0)
    u = torch.rand(size, generator=_generator(seed, stream), device="cuda", dtype=torch.float64) * cdf[-1]
    return perm[torch.searchsorted(cdf, u, right=True).clamp_(max=n_items - 1)].to(torch.int32)


def _layer_spec(pre, d, d_ff, attn_only):
    spec = [(pre + "wqkv", (3 * d, d)), (pre + "bqkv", (3 * d,)), (pre + "wo", (d, d)), (pre + "bo", (d,))]
    if not attn_only:
        spec += [(pre + "ln1_g", (d,)), (pre + "ln1_b", (d,)), (pre + "w1", (d_ff, d)), (pre + "b1", (d_ff,)),
                 (pre + "w2", (d, d_ff)), (pre + "b2", (d,)), (pre + "ln2_g", (d,)), (pre + "ln2_b", (d,))]
    return spec


def _ce_spec(c):
    d = c["d"]
    spec = [("tok_emb", (c["vocab"], d)), ("pos_emb", (c["l_t"], d)), ("emb_ln_g", (d,)), ("emb_ln_b", (d,))]
    for l in range(c["n_layers"]):
        spec += _layer_spec("l%d." % l, d, c["d_ff"], False)
    if c["pooling"] == "additive":
        spec += [("pool_wa", (c["d_a"], d)), ("pool_ba", (c["d_a"],)), ("pool_qa", (c["d_a"],))]
    return spec


def _task_spec(c):
    d = c["d"]
    spec = [("pos", (c["L"], d)), ("resp", (3, d))] if c["task"] == "kt" else []
    for l in range(c["task_layers"]):
        spec += _layer_spec("t%d." % l, d, c["task_d_ff"], c["task_attn_only"])
    return spec + ([("head_w", (d,)), ("head_b", (1,))] if c["task"] == "kt" else
                   [("wa", (c["d_a"], d)), ("ba", (c["d_a"],)), ("qa", (c["d_a"],))])


def _size(spec):
    return sum(math.prod(s) for _, s in spec)


def _split(flat, spec):
    out, o = {}, 0
    for name, shape in spec:
        n = math.prod(shape)
        out[name] = flat[o:o + n].view(shape)
        o += n
    return out


def _params(spec, seed, stream):
    """Weights as training has them: about N(0, 0.02^2), LayerNorm gains near 1."""
    flat = torch.randn(_size(spec), generator=_generator(seed, stream), device="cuda") * 0.02
    for name, v in _split(flat, spec).items():
        if name.endswith("_g"):
            v.add_(1.0)
    return flat


def _item_texts(c, seed):
    tokens = torch.randint(0, c["vocab"], (c["n_items"], c["l_t"]), generator=_generator(seed, 4), device="cuda",
                           dtype=torch.int32)
    if not c["shortest"]:
        return tokens, None
    n = torch.randint(c["shortest"], c["l_t"] + 1, (c["n_items"],), generator=_generator(seed, 5), device="cuda",
                      dtype=torch.int32)
    return tokens, n


def _batch(c, seed, step):
    ids = _zipf(seed, c["n_items"], c["zipf_s"], c["B"] * c["L"], 6 + 2 * step).view(c["B"], c["L"])
    lab = torch.rand(c["B"], c["L"], generator=_generator(seed, 1000 + step), device="cuda") < 0.65
    return ids, lab.to(torch.int32)


def _encodings(c, seed):
    """Encodings as a LayerNorm leaves them."""
    return torch.randn(c["B"], c["L"], c["d"], generator=_generator(seed, 7), device="cuda")


def _items(c, seed):
    return torch.randperm(c["n_items"], generator=_generator(seed, 8), device="cuda")[:c["items"]].sort()[0].to(torch.int32)


def _cotangent(c, seed):
    """Accumulated gradients of a mean loss over some thousands of predictions."""
    return torch.randn(c["items"], c["d"], generator=_generator(seed, 9), device="cuda") * 1e-4


def _index_inputs(c, seed):
    ids = _zipf(seed, c["n_items"], c["zipf_s"], c["P"], 6)
    if c["kind"] == "dedup":
        return ids
    if c["kind"] == "gather":
        src = torch.randn(c["n_items"], c["d"], generator=_generator(seed, 7), device="cuda")
        return ids, src.to(torch.bfloat16 if c["dtype"] == "bf16" else torch.float32)
    perm = torch.sort(ids, stable=True)[1].to(torch.int32)
    n = torch.unique(ids, return_counts=True)[1]
    seg = torch.zeros(n.numel() + 1, dtype=torch.int32, device="cuda")
    seg[1:] = n.cumsum(0)
    dE = torch.rand(c["P"], c["d"], generator=_generator(seed, 7), device="cuda") * 2 - 1
    return dE, perm, seg


class _GradView:
    """A module's gradient buffer as a tensor over the same memory; keeps the context alive."""

    def __init__(self, g, module):
        self.owner = g
        p, n = g.grads_device(module)
        self.__cuda_array_interface__ = {"shape": (n,), "typestr": "<f4", "data": (p, False), "version": 3}


def _grad_views(g, module, spec, whole_layers):
    """Views of a gradient buffer: one per parameter, or one per layer for the deep encoders."""
    flat = torch.as_tensor(_GradView(g, module), device="cuda")
    return _grouped(flat, spec) if whole_layers else _split(flat, spec)


def _grouped(flat, spec):
    groups = []
    for name, shape in spec:
        key = name.split(".")[0]
        if "." not in name or not groups or groups[-1][0] != key:
            groups.append([key, 0])
        groups[-1][1] += math.prod(shape)
    out, o = {}, 0
    for key, n in groups:
        out[key] = flat[o:o + n]
        o += n
    return out


def _context(c, **over):
    cfg = binding.GramConfig()
    cfg.dtype = binding.GRAM_BF16 if c["dtype"] == "bf16" else binding.GRAM_F32
    for k in ("n_items", "l_t", "vocab", "d", "n_heads", "d_ff", "n_layers", "task_layers", "task_heads", "task_d_ff",
              "d_a", "n_cand", "L", "K"):
        setattr(cfg, k, int(c[k]))
    cfg.pooling = {"mean": binding.GRAM_POOL_MEAN, "cls": binding.GRAM_POOL_CLS,
                   "additive": binding.GRAM_POOL_ADDITIVE}[c["pooling"]]
    cfg.task = {"kt": binding.GRAM_TASK_KT, "nr": binding.GRAM_TASK_NR}[c["task"]]
    cfg.task_attn_only = int(c["task_attn_only"])
    cfg.B_max = int(c["B"])
    cfg.ce_micro_batch = int(c["micro"])
    for k, v in over.items():
        setattr(cfg, k, v)
    return binding.Gram(cfg)


def prepare(case, seed):
    c, k = case, case["kind"]
    if k in ("dedup", "accumulate", "gather"):
        cfg = binding.GramConfig()
        cfg.dtype, cfg.n_items, cfg.K = binding.GRAM_F32, c["n_items"], 1
        cfg.d = cfg.d_max = c.get("d", 4)
        cfg.B_max = cfg.L = 1
        cfg.P_max = c["P"]
        g = binding.Gram(cfg)
        st = {"case": c, "g": g}
        if k == "dedup":
            U = min(c["P"], c["n_items"])
            st["ids"] = _index_inputs(c, seed)
            for name, n in (("unique", U), ("inverse", c["P"]), ("perm", c["P"]), ("seg_off", U + 1), ("n", 1)):
                st[name] = torch.zeros(n, dtype=torch.int32, device="cuda")
        elif k == "accumulate":
            st["dE"], st["perm"], st["seg"] = _index_inputs(c, seed)
            st["U"] = st["seg"].numel() - 1
            st["G"] = torch.zeros(min(c["P"], c["n_items"]), c["d"], device="cuda")       # as many rows as there can be
        else:
            st["ids"], st["src"] = _index_inputs(c, seed)
            st["E"] = torch.empty(c["P"], c["d"], dtype=st["src"].dtype, device="cuda")
        return st
    if k in ("step", "window"):
        # early in the warm-up, so that the weights stay near where they were drawn over many passes: Adam's first
        # updates move every weight the same way, and at 1e-4 three of them already show in the loss
        g = _context(c, lr_task=1e-6, lr_ce=1e-6, optimizer=binding.GRAM_OPT_ADAM, noam_warmup=4000)
    elif k == "task":
        g = _context(c, n_layers=0, n_items=1, l_t=1, vocab=1, ce_micro_batch=1)
    else:
        g = _context(c, B_max=1, L=1, task=binding.GRAM_TASK_NONE, task_layers=0, P_max=c["items"],
                     ce_micro_batch=c["items"])
    st = {"case": c, "g": g}
    if k != "task":
        g.set_params(binding.GRAM_MODULE_CE, _params(_ce_spec(c), seed, 2).cpu().numpy())
        tokens, lengths = _item_texts(c, seed)
        g.set_item_tokens(tokens.cpu().numpy())
        if lengths is not None:
            g.set_item_lengths(lengths.cpu().numpy())
        st["ce"] = _grad_views(g, binding.GRAM_MODULE_CE, _ce_spec(c), k in ("step", "window") and c["dtype"] == "bf16")
    if k in ("step", "window", "task"):
        g.set_params(binding.GRAM_MODULE_TASK, _params(_task_spec(c), seed, 3).cpu().numpy())
        st["cf"] = _grad_views(g, binding.GRAM_MODULE_TASK, _task_spec(c), False)
    if k in ("step", "window"):
        st["batches"] = [_batch(c, seed, i) for i in range(c["K"])]
        if k == "window":
            g.cache_fill()
    elif k == "task":
        st["E"], st["labels"] = _encodings(c, seed), _batch(c, seed, 0)[1]
        if c["task"] == "nr":
            st["labels"].clamp_(min=0)
        st["dE"] = torch.empty(c["B"] * c["L"], c["d"], device="cuda")
        st["loss"] = torch.empty(1, device="cuda")
    else:
        st["items"] = _items(c, seed)
        st["H"] = torch.empty(c["items"], c["d"], device="cuda")
        if k == "pass":
            st["G"] = _cotangent(c, seed)
    torch.cuda.synchronize()
    return st


# --------------------------------------------------------------------------- one pass

def run(st):
    c, g = st["case"], st["g"]
    k = c["kind"]
    if k == "dedup":
        g.dedup(st["ids"], c["n_items"], st["unique"], st["inverse"], st["perm"], st["seg_off"], st["n"])
        return {n: st[n] for n in ("unique", "inverse", "perm", "seg_off", "n")}
    if k == "accumulate":
        g.accumulate(st["dE"], st["perm"], st["seg"], st["U"], st["G"])
        return st["G"]
    if k == "gather":
        g.gather(st["src"], st["ids"], st["E"])
        return st["E"]
    if k in ("step", "window"):
        loss, unique = [], []
        for ids, lab in st["batches"]:
            rep = g.step(ids, lab, c["B"])
            loss.append(float(rep.loss))
            unique.append(int(rep.n_unique))
        return {"loss": loss, "unique": unique, "ce": st["ce"], "cf": st["cf"]}
    if k == "task":
        g.task(st["E"], st["labels"], c["B"], st["dE"], st["loss"])
        return {"loss": st["loss"], "dE": st["dE"], "cf": st["cf"]}
    if k == "encode":
        g.encode_unique(None, st["items"], c["items"], st["H"])
        return st["H"]
    g.encode_unique(None, st["items"], c["items"], st["H"], save_activations=True)
    g.zero_grads(binding.GRAM_MODULE_CE)
    g.encoder_backward(st["G"], st["items"], c["items"])
    return {"H": st["H"], "ce": st["ce"]}


# --------------------------------------------------------------------------- what a pass cannot do without

def _expected_unique(n_items, s, P):
    p = np.arange(1, n_items + 1, dtype=np.float64) ** -float(s)
    return float(-np.expm1(P * np.log1p(-np.minimum(p / p.sum(), 1 - 1e-12))).sum())


def _mean_length(c):
    return c["l_t"] if not c["shortest"] else (c["shortest"] + c["l_t"]) / 2


def _layer_flops(d, d_ff, S, attn_only):
    """Forward, per row: the projections, the two attention products, the feed-forward."""
    return 2 * 4 * d * d + 4 * S * d + (0 if attn_only else 4 * d * d_ff)


def _encoder_flops(c, items):
    d, S = c["d"], _mean_length(c)
    f = items * S * c["n_layers"] * _layer_flops(d, c["d_ff"], S, False)
    if c["pooling"] == "cls" and c["n_layers"]:      # the last layer: keys and values of every token, one query row
        f += items * (S * 4 * d * d + _layer_flops(d, c["d_ff"], S, False) - 4 * d * d
                      - S * _layer_flops(d, c["d_ff"], S, False))
    if c["pooling"] == "additive":
        f += items * S * 2 * d * c["d_a"]
    return f


def _task_flops(c):
    rows = c["B"] * (c["L"] if c["task"] == "kt" else c["L"] - c["n_cand"])
    S = c["L"] / 2 if c["task"] == "kt" else c["L"] - c["n_cand"]
    f = rows * c["task_layers"] * _layer_flops(c["d"], c["task_d_ff"], S, c["task_attn_only"])
    return f + (0 if c["task"] == "kt" else rows * 2 * c["d"] * c["d_a"])


def work(case):
    c, k = case, case["kind"]
    if k in ("dedup", "accumulate", "gather"):
        U = _expected_unique(c["n_items"], c["zipf_s"], c["P"])
        if k == "dedup":
            return {"bytes": 12.0 * c["P"] + 8.0 * U, "flops": 0}
        e = 2 if c["dtype"] == "bf16" else 4
        return {"bytes": c["P"] * (4.0 + e * c["d"]) + U * e * c["d"], "flops": float(c["P"] * c["d"]) if k == "accumulate" else 0}
    w = 2 if c["dtype"] == "bf16" else 4              # parameters as the products read them
    ce, cf = _size(_ce_spec(c)), _size(_task_spec(c))
    if k == "task":
        return {"bytes": 8.0 * c["B"] * c["L"] * c["d"] + (w + 4.0) * cf, "flops": 3.0 * _task_flops(c)}
    if k in ("step", "window"):
        U = _expected_unique(c["n_items"], c["zipf_s"], c["B"] * c["L"] * c["K"])
        adam = 28 + (w if w == 2 else 0)              # parameter, two moments read and written, gradient
        return {"bytes": (w + 4.0 + adam) * (ce + c["K"] * cf) + U * c["l_t"] * 4.0 + 8.0 * c["K"] * c["B"] * c["L"],
                "flops": 3.0 * (_encoder_flops(c, U) + c["K"] * _task_flops(c))}
    n = c["items"]
    f, b = _encoder_flops(c, n), n * _mean_length(c) * 4.0 + n * c["d"] * 4.0 + w * float(ce - c["vocab"] * c["d"])
    return {"bytes": b, "flops": f} if k == "encode" else {"bytes": b + n * c["d"] * 4.0 + 4.0 * ce, "flops": 3.0 * f}


def tolerance(case):
    k = case["kind"]
    if k in ("dedup", "gather"):
        return "exact"
    if k == "accumulate":
        return {"rel": 1e-6}              # fp32 sums; 1.6e-7 measured against 64 bits
    if case["dtype"] == "f32":
        return {"rel": 1e-5}              # up to 2e-6 measured on the worst parameter tensor
    # bf16 operands, fp32 sums; against 64 bits: encodings 0.1 to 0.25 % off, the worst parameter tensor's gradient
    # 0.4 % (one encoder pass), 0.8 % (the news task, whole steps)
    return {"rel": {"encode": 0.01, "pass": 0.02}.get(k, 0.03)}


# --------------------------------------------------------------------------- the same in 64 bits

def _ln(x, g, b):
    return torch.nn.functional.layer_norm(x, x.shape[-1:], g, b, LN_EPS)


def _layer(x, th, pre, heads, mask, attn_only):
    """x [n, S, d]; mask [.., S, S] additive (0 or -inf) or None."""
    n, S, d = x.shape
    q, k, v = (x @ th[pre + "wqkv"].T + th[pre + "bqkv"]).view(n, S, 3, heads, d // heads).permute(2, 0, 3, 1, 4)
    s = q @ k.transpose(-1, -2) / math.sqrt(d // heads)
    if mask is not None:
        s = s + mask
    a = (torch.softmax(s, -1) @ v).transpose(1, 2).reshape(n, S, d) @ th[pre + "wo"].T + th[pre + "bo"]
    if attn_only:
        return x + a
    h = _ln(x + a, th[pre + "ln1_g"], th[pre + "ln1_b"])
    f = torch.nn.functional.gelu(h @ th[pre + "w1"].T + th[pre + "b1"]) @ th[pre + "w2"].T + th[pre + "b2"]
    return _ln(h + f, th[pre + "ln2_g"], th[pre + "ln2_b"])


def _ce(c, th, tokens, lengths):
    """Encodings [n, d] of texts [n, l_t] of which the first `lengths` tokens count."""
    x = _ln(th["tok_emb"][tokens.long()] + th["pos_emb"], th["emb_ln_g"], th["emb_ln_b"])
    mask = there = None
    if lengths is not None:
        there = torch.arange(c["l_t"], device=x.device)[None] < lengths[:, None]
        mask = torch.zeros(there.shape, dtype=x.dtype, device=x.device).masked_fill_(~there, -math.inf)[:, None, None]
    for l in range(c["n_layers"]):
        x = _layer(x, th, "l%d." % l, c["n_heads"], mask, False)
    if c["pooling"] == "cls":
        return x[:, 0]
    if c["pooling"] == "mean":
        return x.mean(1) if there is None else (x * there[..., None]).sum(1) / lengths[:, None]
    a = torch.tanh(x @ th["pool_wa"].T + th["pool_ba"]) @ th["pool_qa"]
    if there is not None:
        a = a.masked_fill(~there, -math.inf)
    return (torch.softmax(a, -1)[..., None] * x).sum(1)


def _cf_loss(c, th, E, lab):
    B, L, _ = E.shape
    if c["task"] == "kt":
        prev = torch.cat([torch.full((B, 1), 2, device=E.device), lab[:, :-1].long()], 1)
        x = E + th["pos"] + th["resp"][prev]
        mask = torch.full((L, L), -math.inf, dtype=E.dtype, device=E.device).triu_(1)
        for l in range(c["task_layers"]):
            x = _layer(x, th, "t%d." % l, c["task_heads"], mask, c["task_attn_only"])
        z = x @ th["head_w"] + th["head_b"]
        return torch.nn.functional.binary_cross_entropy_with_logits(z, lab.to(E.dtype))
    n = L - c["n_cand"]
    x, cand = E[:, :n], E[:, n:]
    for l in range(c["task_layers"]):
        x = _layer(x, th, "t%d." % l, c["task_heads"], None, c["task_attn_only"])
    a = torch.softmax(torch.tanh(x @ th["wa"].T + th["ba"]) @ th["qa"], -1)
    s = torch.einsum("bn,bnd,bcd->bc", a, x, cand)
    return -torch.log_softmax(s, -1)[:, 0].mean()


def _leaf(spec, seed, stream):
    flat = _params(spec, seed, stream).double()
    grad = torch.zeros_like(flat)
    th = _split(flat, spec)
    for name, g in _split(grad, spec).items():
        th[name] = th[name].detach().requires_grad_(True)
        th[name].grad = g
    return th, grad


def _chunks(c, n):
    """Items at a time, so that the saved 64-bit activations stay near 20 GB."""
    per = c["l_t"] * 8.0 * (c["n_layers"] + 1) * (14 * c["d"] + 3 * c["d_ff"] + 3 * c["n_heads"] * c["l_t"])
    step = max(1, int(20e9 / per))
    return [slice(i, min(n, i + step)) for i in range(0, n, step)]


def _exact_encode(c, th, texts, items):
    tokens, lengths = texts
    with torch.no_grad():
        return torch.cat([_ce(c, th, tokens[items[s].long()], None if lengths is None else lengths[items[s].long()])
                          for s in _chunks(c, items.numel())])


def _exact_ce_backward(c, th, texts, items, G):
    tokens, lengths = texts
    for s in _chunks(c, items.numel()):
        i = items[s].long()
        _ce(c, th, tokens[i], None if lengths is None else lengths[i]).backward(G[s])


def exact(case, seed):
    c, k = case, case["kind"]
    if k in ("dedup", "gather"):
        return None                       # whole numbers and copies: compared bit for bit
    if k == "accumulate":
        dE, perm, seg = _index_inputs(c, seed)
        G = torch.zeros(min(c["P"], c["n_items"]), c["d"], dtype=torch.float64, device="cuda")
        where = torch.repeat_interleave(torch.arange(seg.numel() - 1, device="cuda"), (seg[1:] - seg[:-1]).long())
        for o in range(0, c["P"], 250_000):
            G.index_add_(0, where[o:o + 250_000], dE[perm[o:o + 250_000].long()].double())
        return G
    if k == "task":
        cf, gcf = _leaf(_task_spec(c), seed, 3)
        E = _encodings(c, seed).double()
        dE = torch.empty_like(E)
        lab, total = _batch(c, seed, 0)[1], 0.0
        for o in range(0, c["B"], 32):    # the loss is a mean over histories of equal length
            e = E[o:o + 32].clone().requires_grad_(True)
            loss = _cf_loss(c, cf, e, lab[o:o + 32]) * (e.shape[0] / c["B"])
            loss.backward()
            dE[o:o + 32], total = e.grad, total + loss.detach()
        return {"loss": total.reshape(1), "dE": dE.view(-1, c["d"]), "cf": _split(gcf, _task_spec(c))}
    th, grad = _leaf(_ce_spec(c), seed, 2)
    texts = _item_texts(c, seed)
    if k in ("encode", "pass"):
        items = _items(c, seed)
        H = _exact_encode(c, th, texts, items)
        if k == "encode":
            return H
        _exact_ce_backward(c, th, texts, items, _cotangent(c, seed).double())
        return {"H": H, "ce": _split(grad, _ce_spec(c))}
    batches = [_batch(c, seed, i) for i in range(c["K"])]
    items = torch.unique(torch.cat([ids.reshape(-1) for ids, _ in batches]))
    H = _exact_encode(c, th, texts, items)
    G, losses, unique = torch.zeros_like(H), [], []
    cf, gcf = _leaf(_task_spec(c), seed, 3)
    for ids, lab in batches:              # task gradients are those of the last step; the updates between the steps
        gcf.zero_()                       # (1e-6 / 4000 each) are far below what 16-bit operands show
        u, inv = torch.unique(ids, return_inverse=True)
        at = torch.searchsorted(items, u)
        E = H[at][inv].requires_grad_(True)
        loss = _cf_loss(c, cf, E, lab)
        loss.backward()
        G.index_add_(0, at[inv].reshape(-1), E.grad.reshape(-1, c["d"]))
        losses.append(float(loss.detach()))
        unique.append(None)
    _exact_ce_backward(c, th, texts, items, G)
    deep = _grouped if c["dtype"] == "bf16" else _split
    return {"loss": losses, "unique": unique, "ce": deep(grad, _ce_spec(c)), "cf": _split(gcf, _task_spec(c))}
