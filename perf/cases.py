"""The calls that users of this package make, as cases to be timed and compared.

A case is one call (or the three stage calls) of the compression path at the
end of a prefill: shapes of the package's own workloads (GQA 32/8, 28/4 and
64/8 heads, head_dim 128, W = 32 / 64, pooling width 7), the same families at
other lengths, and the options that are used in earnest: both 16-bit types,
ragged batches, given log-sum-exps, per-layer selection, head-level budgets,
max pooling, the call without a workspace and the separate stages.

SRH masks, lengths and layer budgets are a model's and a request's
configuration: they follow from the case alone.  Queries, keys and values
are drawn from the seed: keys and values N(0, 1); the window queries of one
head share a direction (they ask about the same thing) and give scaled
logits of standard deviation 1.5 on ordinary keys, 4 attention sinks at about
+5 and 16 needles per KV group at about +6, so scores span the decades that
attention scores span.
"""
import math

import numpy as np
import torch

import paper_2606_24467_gb300 as ckv

D = 128  # head_dim
SHAPES = {"llama8b": (32, 8), "qwen7b": (28, 4), "llama70b": (64, 8)}


def _case(name, call, shape, layers, batch, lo, hi, window=32, pool=7, srh=(1, 2), budget=256.0,
          dtype="bf16", scores=False, config=1):
    """`lo`..`hi`: prompt lengths (equal: every prompt has that length);
    `budget`: mean kept tokens per layer, or a share of the length below 1;
    `config`: seed of lengths, SRH masks and layer budgets; `scores`: the
    caller asks for the raw and pooled scores as well."""
    return {"name": name, "call": call, "shape": shape, "layers": layers, "batch": batch, "lo": lo,
            "hi": hi, "window": window, "pool": pool, "srh_lo": srh[0], "srh_hi": srh[1],
            "budget": budget, "dtype": dtype, "scores": scores, "config": config}


def listed():
    return [
        # a short prompt's layer inside an engine that owns all device memory
        _case("short_layer_noalloc", "noalloc", "llama8b", 1, 1, 777, 777, budget=128.0),
        # one layer of a 4K prompt, compressed inside its forward pass; the
        # caller keeps the scores (for statistics or its own budgets)
        _case("layer_4k_f16", "layers", "llama8b", 1, 1, 4096, 4096, srh=(1, 1), budget=128.0,
              dtype="f16", scores=True),
        # the three stages called one by one (a caller that edits scores or
        # indices in between), an odd length
        _case("stages_16k", "stages", "qwen7b", 1, 1, 16001, 16001, srh=(2, 2), budget=512.0,
              scores=True),
        # a serving batch of short prompts, all layers of the model
        _case("short_batch_32layers", "layers", "llama8b", 32, 8, 300, 4000, budget=256.0),
        # one long prompt, all layers: the package's benchmark
        _case("llama8b_32k", "layers", "llama8b", 32, 1, 32768, 32768),
        # ... and at the longest context
        _case("llama8b_128k", "layers", "llama8b", 32, 1, 131072, 131072, budget=917.0),
        # a ragged batch of long prompts, seven query heads per group
        _case("qwen7b_ragged", "layers", "qwen7b", 28, 8, 8192, 65536, srh=(2, 2), budget=0.03),
        # the largest: a 70B-shaped model, four prompts, 64-192 query rows
        _case("llama70b_32k_x4", "layers", "llama70b", 80, 4, 32768, 32768, window=64, srh=(1, 3),
              budget=328.0),
        # the prefill attention kernel hands over its log-sum-exps
        _case("lse_32k", "lse", "llama8b", 32, 1, 32768, 32768, scores=True),
        # one selection per layer shared by all KV groups, four layers a call
        _case("shared_selection_32k", "shared", "llama8b", 4, 1, 32768, 32768, scores=True),
        # budgets per KV group (head-level allocation), one layer
        _case("head_budgets_32k", "head_budgets", "llama8b", 1, 1, 32768, 32768, budget=512.0),
        # max pooling of each SRH head, one layer
        _case("maxpool_24k", "maxpool", "qwen7b", 1, 1, 24000, 24000, srh=(2, 2), budget=512.0),
    ]


def draw(rng):
    call = rng.choice(["layers", "layers", "layers", "layers", "lse", "lse", "noalloc", "stages",
                       "shared", "head_budgets", "maxpool"])
    shape = rng.choice(["llama8b", "llama8b", "qwen7b", "llama70b"])
    heads = SHAPES[shape][1]
    window = rng.choice([16, 32, 32, 32, 64])
    hi = int(round(math.exp(rng.uniform(math.log(400), math.log(131072)))))
    if call == "noalloc":
        hi = int(round(math.exp(rng.uniform(math.log(300), math.log(1800)))))
    lo = hi if rng.random() < 0.5 else max(window + 1, int(hi * rng.uniform(0.1, 0.9)))
    batch = 1 if call == "noalloc" else rng.choice([1, 1, 2, 4, 8])
    if call == "shared":
        layers = rng.choice([1, 4])
    elif call in ("layers", "lse"):
        layers = rng.choice([1, 4, 16, 32, 48])
    else:
        layers = 1
    # no more (layer, prompt, group, token)s than 32 layers of a 128K prompt,
    # and a batch within what one call takes
    room = 32 * 8 * 131072
    while layers * batch * heads * hi > room:
        if batch > 1:
            batch //= 2
        elif layers > 1:
            layers //= 2
        else:
            hi //= 2
            lo = min(lo, hi)
    srh_hi = rng.randint(1, 3)
    budget = rng.choice([0.01, 0.03, 0.1, 128.0, 256.0, 917.0])
    return {"call": call, "shape": shape, "layers": layers, "batch": batch, "lo": lo, "hi": hi,
            "window": window, "pool": rng.choice([5, 7, 7, 13]), "srh_lo": rng.randint(1, srh_hi),
            "srh_hi": srh_hi, "budget": budget, "dtype": rng.choice(["bf16", "bf16", "f16"]),
            "scores": call == "stages" or rng.random() < 0.3, "config": rng.randint(1, 1 << 20)}


# ------------------------------------------------------------- configuration
class _Config:
    """What follows from the case alone: lengths, masks, budgets, offsets."""

    def __init__(self, c):
        rng = np.random.default_rng(c["config"])
        self.hq, self.hkv = SHAPES[c["shape"]]
        self.group = self.hq // self.hkv
        nl, b, w = c["layers"], c["batch"], c["window"]
        lens = rng.integers(c["lo"], c["hi"] + 1, size=b)
        self.lens = np.tile(lens, nl).astype(np.int64)  # [layers * batch]
        self.cu = np.concatenate([[0], np.cumsum(self.lens)]).astype(np.int32)
        self.masks = np.zeros((nl, self.hq), bool)
        for l in range(nl):
            for g in range(self.hkv):
                k = int(rng.integers(c["srh_lo"], c["srh_hi"] + 1))
                self.masks[l, g * self.group + rng.choice(self.group, k, replace=False)] = True
        # layer budgets: Dirichlet shares of the mean, at least W + 16
        share = rng.dirichlet([2.0] * nl) * nl
        mean = c["budget"] * lens if c["budget"] < 1 else np.full(b, c["budget"])
        floor = w + 16
        bud = floor + share[:, None] * np.maximum(mean[None, :] - floor, 0)
        self.budgets = np.minimum(bud.astype(np.int64), np.maximum(self.lens.reshape(nl, b), w))
        self.budgets = np.maximum(self.budgets, w).reshape(-1).astype(np.int32)
        # head-level budgets: the layer's budget spread unevenly over the groups
        hb = floor + rng.dirichlet([2.0] * self.hkv, size=nl * b) * self.hkv * np.maximum(
            self.budgets[:, None] - floor, 0)
        self.group_budgets = np.clip(hb.astype(np.int64), w, np.maximum(self.lens, w)[:, None])
        self.group_budgets = self.group_budgets.astype(np.int32)

    def units(self):
        """(sequence, group, offset, length, SRH heads) of every unit."""
        per = len(self.lens) // len(self.masks)
        for s, n in enumerate(self.lens):
            m = self.masks[s // per]
            for g in range(self.hkv):
                h = [h for h in range(g * self.group, (g + 1) * self.group) if m[h]]
                yield s, g, int(self.cu[s]), int(n), h


def _inputs(c, cfg, seed):
    dev = torch.device("cuda")
    dt = torch.bfloat16 if c["dtype"] == "bf16" else torch.float16
    gen = torch.Generator(device=dev)
    gen.manual_seed(int(seed))
    ns, w, t = len(cfg.lens), c["window"], int(cfg.cu[-1])
    k = torch.empty((t, cfg.hkv, D), dtype=dt, device=dev).normal_(generator=gen)
    v = torch.empty((t, cfg.hkv, D), dtype=dt, device=dev).normal_(generator=gen)
    common = torch.randn((ns, cfg.hq, 1, D), generator=gen, device=dev)
    q = 1.5 * (0.8 * common + 0.6 * torch.randn((ns, cfg.hq, w, D), generator=gen, device=dev))
    # the direction the SRH heads of a group look for, and its keys
    per = ns // len(cfg.masks)
    mask = torch.from_numpy(np.repeat(cfg.masks, per, axis=0)).to(dev)
    aim = (common[:, :, 0] * mask[:, :, None]).view(ns, cfg.hkv, cfg.group, D).sum(2)
    aim = aim / aim.norm(dim=-1, keepdim=True)
    away = torch.randn((ns, 16, cfg.hkv, D), generator=gen, device=dev)
    place = torch.rand((ns, 16), generator=gen, device=dev) * 0.99
    step = torch.arange(16, device=dev)
    for s in range(ns):
        n = int(cfg.lens[s])
        if n > w + 64:
            row = int(cfg.cu[s])
            # one needle per sixteenth of the prefix: never two in one place
            at = row + 4 + ((step + place[s]) * ((n - w - 4) / 16)).long()
            k[at] = (4.8 * aim[s][None] + 0.9 * away[s]).to(dt)
            k[row:row + 4] = (4.0 * aim[s][None].expand(4, -1, -1)).to(dt)
    return q.to(dt), k, v


def _lse(c, cfg, q, k):
    """The window queries' log-sum-exps, as a prefill attention returns them."""
    w = c["window"]
    out = torch.empty((len(cfg.lens), cfg.hq, w), dtype=torch.float32, device=q.device)
    for s, g, row, n, _ in cfg.units():
        h0 = g * cfg.group
        z = q[s, h0:h0 + cfg.group].float().reshape(-1, D) @ k[row:row + n, g].float().T
        z = z.view(cfg.group, w, n) / math.sqrt(D)
        later = torch.arange(n, device=q.device) > n - w + torch.arange(w, device=q.device)[:, None]
        out[s, h0:h0 + cfg.group] = z.masked_fill_(later, -math.inf).logsumexp(-1)
    return out


# ------------------------------------------------------------------ the calls
def prepare(case, seed):
    c, cfg = case, _Config(case)
    q, k, v = _inputs(c, cfg, seed)
    call = c["call"]
    prob = ckv.Problem(q, k, cfg.cu, c["window"], c["pool"],
                       selection="layer" if call == "shared" else "group",
                       pool="max" if call == "maxpool" else "avg")
    st = {"call": call, "cfg": cfg, "prob": prob, "q": q, "k": k, "v": v,
          "masks": cfg.masks.astype(np.uint8)}
    n_pre = int(np.maximum(cfg.lens - c["window"], 0).sum())
    if call == "head_budgets":
        _, rows = ckv.head_budget_layout(prob, cfg.group_budgets)
        shape = (rows, D)
        st["indices"] = torch.empty((rows,), dtype=torch.int32, device=k.device)
    else:
        rows = int(np.minimum(cfg.budgets, cfg.lens).sum())
        shape = (rows, cfg.hkv, D)
        st["indices"] = torch.empty((cfg.hkv, rows), dtype=torch.int32, device=k.device)
    st["k_out"] = torch.empty(shape, dtype=k.dtype, device=k.device)
    st["v_out"] = torch.empty(shape, dtype=k.dtype, device=k.device)
    if c["scores"]:
        st["raw"] = torch.empty((cfg.hkv, n_pre), dtype=torch.float32, device=k.device)
        if call != "shared":
            st["pooled"] = torch.empty_like(st["raw"])
    if call != "noalloc":
        st["ws"] = ckv.workspace(prob)
    if call == "lse":
        st["lse"] = _lse(c, cfg, q, k)
    return st


def run(st):
    cfg, prob, call = st["cfg"], st["prob"], st["call"]
    q, k, v, ind, ko, vo = st["q"], st["k"], st["v"], st["indices"], st["k_out"], st["v_out"]
    raw, pooled = st.get("raw"), st.get("pooled")
    if call == "stages":
        ckv.score(prob, q, k, st["masks"][0], raw, st["ws"])
        cu_out = ckv.select(prob, raw, cfg.budgets, ind, st["ws"], pooled=pooled)
        ckv.gather(prob, ind, cu_out, k, v, ko, vo, ws=st["ws"])
    elif call == "noalloc":
        ckv.compress_layer_noalloc(prob, q, k, v, st["masks"][0], cfg.budgets, ind, ko, vo,
                                   raw=raw, pooled=pooled)
    elif call == "lse":
        ckv.compress_layers_lse(prob, len(st["masks"]), q, k, v, st["lse"], st["masks"],
                                cfg.budgets, ind, ko, vo, st["ws"], raw=raw, pooled=pooled)
    elif call == "head_budgets":
        ckv.compress_layer_head_budgets(prob, q, k, v, st["masks"][0], cfg.group_budgets, ind, ko,
                                        vo, st["ws"], raw=raw, pooled=pooled)
    elif len(st["masks"]) == 1:
        ckv.compress_layer(prob, q, k, v, st["masks"][0], cfg.budgets, ind, ko, vo, st["ws"],
                           raw=raw, pooled=pooled)
    else:
        ckv.compress_layers(prob, len(st["masks"]), q, k, v, st["masks"], cfg.budgets, ind, ko, vo,
                            st["ws"], raw=raw, pooled=pooled)
    # the compressed cache holds copies: compared as the 16-bit words they are
    out = {"indices": ind, "k_out": ko.view(torch.int16), "v_out": vo.view(torch.int16)}
    if raw is not None:
        out["raw"] = raw
    if pooled is not None:
        out["pooled"] = pooled
    return out


def work(case):
    """Bytes: every key, the SRH window queries and the kept value rows read
    once, the compressed cache, its indices and the scores asked for written
    once.  Operations: one product of the SRH window queries and the keys."""
    cfg, w = _Config(case), case["window"]
    bytes_, flops = 0, 0
    for s, g, _, n, h in cfg.units():
        if n <= w:
            continue
        kept = cfg.group_budgets[s, g] if case["call"] == "head_budgets" else cfg.budgets[s]
        rows = len(h) * w
        bytes_ += 2 * D * n + 2 * D * rows + int(min(kept, n)) * (3 * 2 * D + 4)
        bytes_ += (4 if case["call"] == "shared" else 8) * (n - w) if case["scores"] else 0
        bytes_ += 4 * rows if case["call"] == "lse" else 0
        flops += 2 * D * rows * n
    return {"bytes": int(bytes_), "flops": int(flops)}


def tolerance(case):
    """Scores are fp32 sums of fp32 exponentials of fp32 logits (against 64
    bits: about 1e-6 of the norm); per-layer selection, head-level budgets and
    other calls outside the persistent kernel may keep their exponentials in
    16 bits (2^-11 a term, 2e-5 over a sum).  A rounding in the last place can
    swap two tokens whose pooled scores are neighbours at the budget's edge,
    and shift the rows between them."""
    wide = case["call"] in ("shared", "head_budgets")
    return {"rel": 1e-4 if wide else 1e-5, "max": 2e-3 if wide else 1e-4, "differ": 0.01}


def exact(case, seed):
    """Raw and pooled scores in 64 bits; None where the caller asks for none
    (the rest is a choice by these scores and copies)."""
    if not case["scores"]:
        return None
    c, cfg = case, _Config(case)
    q, k, _ = _inputs(c, cfg, seed)
    w, half = c["window"], (c["pool"] - 1) // 2
    pre = np.concatenate([[0], np.cumsum(np.maximum(cfg.lens - w, 0))])
    raw = torch.zeros((cfg.hkv, int(pre[-1])), dtype=torch.float64, device=k.device)
    pooled = torch.zeros_like(raw)
    for s, g, row, n, heads in cfg.units():
        if n <= w:
            continue
        key = k[row:row + n, g].double()
        later = torch.arange(n, device=k.device) > n - w + torch.arange(w, device=k.device)[:, None]
        each = torch.zeros((len(heads), n - w), dtype=torch.float64, device=k.device)
        for i, h in enumerate(heads):
            z = (q[s, h].double() @ key.T) / math.sqrt(D)
            p = z.masked_fill_(later, -math.inf).softmax(-1)
            each[i] = p[:, :n - w].sum(0)
        a, b = int(pre[s]), int(pre[s + 1])
        raw[g, a:b] = each.sum(0)
        if c["call"] == "maxpool":
            pooled[g, a:b] = torch.nn.functional.max_pool1d(each[None], c["pool"], 1, half)[0].sum(0)
        else:
            pooled[g, a:b] = torch.nn.functional.avg_pool1d(
                each.sum(0)[None], c["pool"], 1, half, count_include_pad=True)[0]
    out = {"indices": None, "k_out": None, "v_out": None, "raw": raw}
    if c["call"] != "shared":
        out["pooled"] = pooled
    return out
