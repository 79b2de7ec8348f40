"""The work that programs have this library do, as measured cases.

A diffusion-LLM server calls one decoding step per iteration over the active
windows of its sequences (`ebd_step`, or `ebd_step_host` where the backbone's
results arrive in host memory); programs that drive the stages themselves call
`ebd_attention`, `ebd_lm_stats` and `ebd_decide`.  The sizes are the
repository's own: the tiny step, the LLaDA-8B and Dream-7B shapes of
`synth/configs.py`, the batch x prefix x window sweep, and the full-sequence
setting; `draw` spreads over the same ranges and adds generic backbones (any
width and vocabulary, 64- and 128-wide heads, grouped K/V heads).

Values follow `synth/gen.py`: hidden rows N(0,1) times a per-row scale
log-uniform in [0.5, 8], W_lm ~ N(0, 1/64) (0.02 at the tiny width), W_e, q, K
and V ~ N(0, 1); router weights are imported as a trained blob would be, drawn
U(+-1/sqrt(fan_in)).  Everything is drawn on the GPU from the seed alone.

A pass of a step starts from the window's decode state as the program holds
it: one device copy puts tokens, mask and block state in place, then the call
updates them.  A pass of the host-buffer step ends when its results are in the
caller's buffers, which is when such a program can read them.
"""
from __future__ import annotations

import math

import torch

from paper_2609_16450_gb300 import _ebd as E
from paper_2609_16450_gb300 import runtime as rt

GEN_LEN, G_MAX, L_MIN, L_B = 512, 5, 8, 32
TAU, TAU_PSI = 0.9, 0.89
MASK_TOKEN = -1

# d_model, vocab, query heads, K/V heads, head width
TINY = (256, 4096, 4, 4, 64)
LLADA_8B = (4096, 126464, 32, 32, 128)
DREAM_7B = (3584, 152064, 28, 4, 128)


def _case(entry, model, batch, prefix, window, *, ragged=False, block=False, suffix=0,
          append=False, packed=True, mask=0.75, mode=0, name=None):
    d, v, hq, hkv, hd = model
    c = dict(entry=entry, d_model=d, vocab=v, heads_q=hq, heads_kv=hkv, head_dim=hd, batch=batch,
             prefix=prefix, window=window, ragged=ragged, block=block, suffix=suffix,
             append=append, packed=packed, mask=mask, mode=mode)
    return dict(c, name=name) if name else c


def listed():
    return [
        # one small step: kernel latency, launches and the host's enqueue
        _case("step", TINY, 1, 128, 32, name="tiny_step"),
        # the interactive step of one user, a block to be selected (both routers run)
        _case("step", LLADA_8B, 1, 512, 32, name="llada_step"),
        # the step that most iterations are: inside a block, dual cache, cache append
        _case("step", LLADA_8B, 1, 512, 32, block=True, suffix=448, append=True,
              name="llada_step_block_dual"),
        # the same step for a program whose backbone's results are in pinned host memory
        _case("host_step", LLADA_8B, 1, 512, 64, name="llada_host_step"),
        # a small batch with grouped heads and ragged windows
        _case("step", DREAM_7B, 8, 1024, 64, ragged=True, name="dream_step_b8"),
        # batched serving: short windows over a long cache, and the largest step
        _case("step", LLADA_8B, 64, 1024, 32, mask=0.6, name="llada_step_b64_w32"),
        _case("step", LLADA_8B, 64, 256, 64, mask=0.6, name="llada_step_b64_w64"),
        # every position of a 512-token response is a row (no K/V cache)
        _case("step", LLADA_8B, 1, 0, 512, name="llada_full_sequence"),
        # the stages by themselves: attention over a long ragged cache, and of many short windows
        _case("attention", DREAM_7B, 16, 4096, 32, ragged=True, name="dream_attention_b16"),
        _case("attention", LLADA_8B, 64, 256, 16, name="llada_attention_b64"),
        # statistics of an odd number of rows on the checkpoint's own row-major weight
        _case("lm_stats", LLADA_8B, 3, 0, 51, packed=False, name="llada_lm_stats_153"),
        # the decision of a batch on statistics that another LM head made
        _case("decide", LLADA_8B, 16, 0, 64, ragged=True, name="llada_decide_b16"),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _generic(rng):
    hd = rng.choice((64, 128))
    hkv = rng.choice((1, 2, 4, 8))
    return (8 * _log_int(rng, 32, 512), _log_int(rng, 2000, 130000), hkv * rng.choice((1, 2, 4, 7)),
            hkv, hd)


def draw(rng):
    model = rng.choice((TINY, LLADA_8B, LLADA_8B, DREAM_7B, _generic(rng), _generic(rng)))
    entry = rng.choice(("step", "step", "step", "host_step", "full", "attention", "attention",
                        "lm_stats", "decide", "decide"))
    mask = rng.choice((0.5, 0.6, 0.75, 1.0))
    ragged = rng.random() < 0.5
    packed = rng.random() < 0.75
    block = rng.random() < 0.4
    if entry == "full":
        return _case("step", model, _log_int(rng, 1, 4), 0, rng.randint(65, 512), ragged=ragged,
                     block=block, packed=packed, mask=mask)
    batch = _log_int(rng, 1, 64)
    window = _log_int(rng, 4, 64)
    prefix = _log_int(rng, 64, min(4096, 64 * 1024 // batch))
    if entry == "lm_stats":
        return _case(entry, model, batch, 0, window, packed=packed, ragged=ragged)
    if entry == "decide":
        if rng.random() < 0.25:
            batch, window = _log_int(rng, 1, 8), rng.randint(65, 512)
        return _case(entry, model, batch, 0, window, ragged=ragged, block=block, mask=mask,
                     mode=rng.choice((0, 0, 0, 1, 2)))
    suffix = rng.choice((0, 0, _log_int(rng, 8, 512)))
    if entry == "attention":
        return _case(entry, model, batch, prefix, window, ragged=ragged, suffix=suffix)
    return _case(entry, model, batch, prefix, window, ragged=ragged, block=block, suffix=suffix,
                 append=rng.random() < 0.3, packed=packed, mask=mask)


# ------------------------------------------------------------------ inputs
def _gen(seed, what, device="cuda"):
    return torch.Generator(device=device).manual_seed((seed * 1000003 + what * 7919 + 17) % (1 << 62))


def _normal(seed, what, shape, std=1.0):
    x = torch.empty(shape, dtype=torch.bfloat16, device="cuda")
    return x.normal_(0.0, std, generator=_gen(seed, what))


def _std_w(case):
    return 0.02 if case["d_model"] <= 256 else 1.0 / 64.0


def _lens(case):
    """Window rows and cached prefix of every sequence (host lists); a ragged
    case's are part of the case, so that its outputs keep their shapes."""
    b, w, p = case["batch"], case["window"], case["prefix"]
    if not case["ragged"]:
        return [w] * b, [p] * b
    g = _gen(b * 8191 + w * 131 + p, 1, "cpu")
    ws = torch.randint(max(1, w // 4), w + 1, (b,), generator=g).tolist()
    ps = torch.randint(p // 2, p + 1, (b,), generator=g).tolist()
    return ws, ps


def _router(seed, d_base):
    """Router weights in the blob's order (bf16, host): name -> tensor."""
    g = _gen(seed, 2, "cpu")
    out = {}

    def lin(name, n_out, n_in):
        a = n_in ** -0.5
        out[name + ".w"] = (torch.rand((n_out, n_in), generator=g) * 2 - 1) * a
        out[name + ".b"] = (torch.rand((n_out,), generator=g) * 2 - 1) * a

    def ln(name, n):
        out[name + ".g"] = 1 + 0.1 * torch.randn((n,), generator=g)
        out[name + ".b"] = 0.1 * torch.randn((n,), generator=g)

    lin("ent1", 64, 1), lin("ent2", 64, 64), ln("ent_ln", 64)
    lin("tok", 64, d_base), lin("comb", 128, 128)
    out["pos"] = 0.02 * torch.randn((GEN_LEN, 128), generator=g)
    for i in range(2):
        lin(f"s{i}.qkv", 384, 128), lin(f"s{i}.out", 128, 128), ln(f"s{i}.ln1", 128)
        lin(f"s{i}.ff1", 256, 128), lin(f"s{i}.ff2", 128, 256), ln(f"s{i}.ln2", 128)
    lin("shead", 1, 128)
    lin("in", 32, 5), ln("in_ln", 32)
    for i in range(2):
        ln(f"p{i}.ln1", 32), lin(f"p{i}.qkv", 96, 32), lin(f"p{i}.out", 32, 32)
        ln(f"p{i}.ln2", 32), lin(f"p{i}.ff1", 64, 32), lin(f"p{i}.ff2", 32, 64)
    lin("phead", 1, 32)
    return {k: v.to(torch.bfloat16) for k, v in out.items()}


def _inputs(case, seed):
    """The step's tensors on the GPU, by name."""
    d, hq, hkv, hd = (case[k] for k in ("d_model", "heads_q", "heads_kv", "head_dim"))
    ws, ps = _lens(case)
    n, b, entry = sum(ws), case["batch"], case["entry"]
    x = {}
    cu = [0]
    for w in ws:
        cu.append(cu[-1] + w)
    dev = dict(device="cuda")
    i32 = dict(dtype=torch.int32, **dev)
    x["cu_rows"] = torch.tensor(cu, **i32)
    x["prefix_len"] = torch.tensor(ps, **i32)
    x["row_pos"] = torch.tensor([p + i for w, p in zip(ws, ps) for i in range(w)], **i32)
    if entry in ("step", "host_step", "lm_stats"):
        u = torch.empty((n, 1), dtype=torch.float32, **dev).uniform_(generator=_gen(seed, 3))
        x["hidden"] = (_normal(seed, 4, (n, d)).float() * torch.exp(math.log(0.5) + u * math.log(16.0))).bfloat16()
        x["w_lm"] = _normal(seed, 5, (case["vocab"], d), _std_w(case))
    if entry in ("step", "host_step", "attention") and case["window"] <= 64:
        cap = case["prefix"] + (case["window"] + case["suffix"] if case["suffix"] or case["append"] else 0)
        x["q"] = _normal(seed, 6, (n, hq, hd))
        x["k_win"], x["v_win"] = _normal(seed, 7, (n, hkv, hd)), _normal(seed, 8, (n, hkv, hd))
        x["k_cache"], x["v_cache"] = _normal(seed, 9, (b, cap, hkv, hd)), _normal(seed, 10, (b, cap, hkv, hd))
        if case["suffix"]:
            x["suffix"] = torch.tensor([[p + w, case["suffix"]] for w, p in zip(ws, ps)], **i32)
    if entry in ("step", "host_step", "decide"):
        x["w_emb"] = _normal(seed, 11, (case["vocab"], d))
        g = _gen(seed, 12, "cpu")
        mask, in_block, meta = [], [], []
        for i, w in enumerate(ws):
            m = torch.zeros(w, dtype=torch.uint8)
            m[torch.randperm(w, generator=g)[: max(1, round(case["mask"] * w))]] = 1
            inside = torch.zeros(w, dtype=torch.uint8)
            k = min(20, w)
            if case["block"] and int(m[:k].sum()):
                inside[:k] = 1
            mask.append(m), in_block.append(inside)
            meta.append([ps[i], k] if int(inside.sum()) else [0, 0])
        tok = torch.randint(0, case["vocab"], (n,), generator=g, dtype=torch.int32)
        mask = torch.cat(mask)
        tok[mask == 1] = MASK_TOKEN
        x["tokens"], x["mask"], x["in_block"] = tok, mask, torch.cat(in_block)
        x["blk_meta"] = torch.tensor(meta, dtype=torch.int32)
    if entry == "decide":
        u = torch.rand((3, n), generator=_gen(seed, 13, "cpu"))
        conf = u[0] ** 0.5 * 0.98 + 0.01
        x["conf"] = conf.cuda()
        x["ent_norm"] = ((1 - conf) * (0.2 + 0.8 * u[1])).cuda()
        x["gap"] = (conf * (0.3 + 0.7 * u[2])).cuda()
        x["argmax"] = torch.randint(0, case["vocab"], (n,), generator=_gen(seed, 14, "cpu"), dtype=torch.int32).cuda()
    return x


STATE = ("tokens", "blk_meta", "mask", "in_block")


class _Step:
    """The handle, buffers and arguments that a program keeps between calls."""


def _state_blob(x, make):
    """The decode state's arrays as views of one buffer, so that one copy sets them all."""
    at, size = {}, 0
    for k in STATE:
        at[k] = size
        size += (x[k].numel() * x[k].element_size() + 63) // 64 * 64
    blob = make(size)
    views = {k: blob[at[k]: at[k] + x[k].numel() * x[k].element_size()].view(x[k].dtype).view(x[k].shape)
             for k in STATE}
    for k in STATE:
        views[k].copy_(x[k])
    return blob, views


def prepare(case, seed):
    x = _inputs(case, seed)
    s = _Step()
    s.x, s.entry = x, case["entry"]
    n, b = x["row_pos"].numel(), case["batch"]
    cap = x["k_cache"].shape[1] if "k_cache" in x else case["prefix"]
    cfg = E.ebd_config(d_model=case["d_model"], vocab=case["vocab"], n_heads_q=case["heads_q"],
                       n_heads_kv=case["heads_kv"], head_dim=case["head_dim"],
                       d_base=case["d_model"], max_batch=b, max_window=case["window"],
                       max_rows=b * case["window"], max_prefix=cap, gen_len=GEN_LEN, g_max=G_MAX,
                       l_min=L_MIN, l_b=L_B, eos_id=case["vocab"] - 1, lps_enabled=1, tau=TAU,
                       tau_psi=TAU_PSI, seed=seed & 0xFFFF, debug_flags=0,
                       decode_mode=case["mode"], top_m=4)
    s.handle = rt.Handle(cfg)
    h = s.handle.h
    if "w_emb" in x:
        blob = torch.cat([t.reshape(-1) for t in _router(seed, case["d_model"]).values()])
        E.check(E.ebd_import_weights(h, blob.view(torch.int16).numpy().view("uint16")), h)
        s.handle.bind(x["w_emb"])
    if "w_lm" in x and case["packed"]:
        x["w_lm"] = rt.pack_weights(s.handle, rt.DeviceWeights(w_lm=x["w_lm"], w_emb=None)).w_lm
    host = s.entry == "host_step"
    if host:  # per-step tensors in pinned host memory; weights and cache stay on the GPU
        for k in ("cu_rows", "prefix_len", "row_pos", "hidden", "q", "k_win", "v_win", "suffix"):
            if k in x:
                x[k] = x[k].cpu().pin_memory()

    def out(*shape, dtype=torch.float32):
        # positions that a call leaves alone hold zero
        return torch.zeros(shape, dtype=dtype, pin_memory=True) if host else torch.zeros(shape, dtype=dtype, device="cuda")

    s.out = {}
    if "tokens" in x:
        make = (lambda k: torch.zeros(k, dtype=torch.uint8, pin_memory=True)) if host else (
            lambda k: torch.zeros(k, dtype=torch.uint8, device="cuda"))
        s.state, views = _state_blob(x, make)
        s.start = s.state.clone()
        x.update(views)
        s.out.update(views)
        s.out.update(lbs_logit=out(n), lps_prob=out(n), accepted=out(n, dtype=torch.uint8))
    if "w_lm" in x:
        s.out.update(conf=out(n), entropy=out(n), ent_norm=out(n), gap=out(n), argmax=out(n, dtype=torch.int32))
    if "q" in x:
        s.out["attn_out"] = out(n, case["heads_q"], case["head_dim"])
    if case["append"] and "q" in x:
        s.out.update(k_cache=x["k_cache"], v_cache=x["v_cache"])
    a = E.ebd_step_args()
    a.batch, a.rows = b, n
    for k, t in {**x, **s.out}.items():
        if k not in ("w_emb",):
            setattr(a, k, t.data_ptr())
    a.w_lm_layout = int(case["packed"])
    a.kv_append = int(bool(case["append"]) and "q" in x)
    s.args = a
    s.call = {"step": E.ebd_step, "host_step": E.ebd_step_host, "decide": E.ebd_decide,
              "lm_stats": E.ebd_lm_stats, "attention": E.ebd_attention}[s.entry]
    torch.cuda.synchronize()
    return s


def run(s):
    h = s.handle.h
    stream = rt.stream_handle(None)
    if s.entry not in ("attention", "lm_stats"):
        s.state.copy_(s.start)
    E.check(s.call(h, s.args, stream), h)
    if s.entry == "host_step":  # the results are in the caller's buffers from here on
        E.check(E.ebd_sync_status(h, stream), h)
    return s.out


# ------------------------------------------------------------------ what a pass cannot do without
def work(case):
    d, v, hq, hkv, hd = (case[k] for k in ("d_model", "vocab", "heads_q", "heads_kv", "head_dim"))
    ws, ps = _lens(case)
    n = sum(ws)
    entry = case["entry"]
    nbytes = flops = 0.0
    if entry in ("step", "host_step", "lm_stats"):
        nbytes += 2.0 * v * d + 2.0 * n * d + 20.0 * n
        flops += 2.0 * n * v * d
    if entry in ("step", "host_step", "attention") and case["window"] <= 64:
        nbytes += 6.0 * n * hq * hd
        for w, p in zip(ws, ps):
            keys = p + w + case["suffix"]
            nbytes += 4.0 * keys * hkv * hd
            flops += 4.0 * w * keys * hq * hd
        if case["append"]:  # the rows that a step commits, about a quarter of the masked ones
            nbytes += 8.0 * n * hkv * hd * case["mask"] * 0.25
    if entry in ("step", "host_step", "decide"):
        nbytes += 45.0 * n + 2.0 * 17000
        if not case["block"] and case["mode"] == 0:
            nbytes += 2.0 * 290000
            for w in ws:
                m = case["mask"] * w
                nbytes += 256.0 * m
                flops += 2.0 * m * (4096 + 16384 + 2 * (49152 + 16384 + 65536 + 256 * m))
        flops += 2.0 * n * 17000
    return {"bytes": nbytes, "flops": flops}


def tolerance(case):
    # About four times what fp32 accumulation shows against 64 bits: attention
    # 2e-6..4.5e-6, statistics up to 2.2e-5 (the gap of peaked rows; logits of
    # some tens make 1 ulp there 4e-6 of a probability), the routers 5e-6.
    # `differ`: a top-2 tie of a row among thousands.
    rel = {"attention": 2e-5, "decide": 4e-5}.get(case["entry"], 1e-4)
    return {"rel": rel, "max": 40 * rel, "differ": 0.002}


# ------------------------------------------------------------------ the same in 64 bits
def _exact_stats(x, v):
    hid = x["hidden"].double()
    w = x["w_lm"]
    logits = torch.cat([hid @ w[i: i + 16384].double().T for i in range(0, v, 16384)], dim=1)
    top = torch.topk(logits, 2, dim=1)
    m = top.values[:, :1]
    z = torch.exp(logits - m).sum(1)
    logits.sub_(m)
    t = (torch.exp(logits) * logits).sum(1)
    ent = torch.log(z) - t / z
    return dict(conf=1 / z, entropy=ent, ent_norm=ent / math.log(v),
                gap=(1 - torch.exp(top.values[:, 1] - m[:, 0])) / z, argmax=None)


def _exact_attention(case, x):
    ws, ps = _lens(case)
    rep = case["heads_q"] // case["heads_kv"]
    outs, r = [], 0
    for i, (w, p) in enumerate(zip(ws, ps)):
        k = [x["k_cache"][i, :p], x["k_win"][r: r + w]]
        v = [x["v_cache"][i, :p], x["v_win"][r: r + w]]
        if case["suffix"]:
            k.append(x["k_cache"][i, p + w: p + w + case["suffix"]])
            v.append(x["v_cache"][i, p + w: p + w + case["suffix"]])
        k = torch.cat(k).double().repeat_interleave(rep, 1).transpose(0, 1)
        v = torch.cat(v).double().repeat_interleave(rep, 1).transpose(0, 1)
        q = x["q"][r: r + w].double().transpose(0, 1)
        a = torch.softmax(q @ k.transpose(1, 2) / math.sqrt(case["head_dim"]), dim=-1)
        outs.append((a @ v).transpose(0, 1))
        r += w
    return torch.cat(outs)


def _lin(z, w, name):
    return z @ w[name + ".w"].T + w[name + ".b"]


def _ln(z, w, name):
    mu = z.mean(-1, keepdim=True)
    var = ((z - mu) ** 2).mean(-1, keepdim=True)
    return (z - mu) / torch.sqrt(var + 1e-5) * w[name + ".g"] + w[name + ".b"]


def _gelu(z):
    return 0.5 * z * (1 + torch.erf(z / math.sqrt(2.0)))


def _mha(z, w, name, heads=4):
    n, d = z.shape
    q, k, v = _lin(z, w, name + ".qkv").view(n, 3, heads, d // heads).permute(1, 2, 0, 3)
    a = torch.softmax(q @ k.transpose(1, 2) / math.sqrt(d // heads), dim=-1) @ v
    return _lin(a.transpose(0, 1).reshape(n, d), w, name + ".out")


def _lbs(ent, tok, w, w_emb):
    e = _ln(_lin(_gelu(_lin(ent[:, None], w, "ent1")), w, "ent2"), w, "ent_ln")
    z = _lin(torch.cat([e, _lin(w_emb[tok].double(), w, "tok")], 1), w, "comb") + w["pos"][: len(ent)]
    for i in range(2):
        z = _ln(z + _mha(z, w, f"s{i}"), w, f"s{i}.ln1")
        z = _ln(z + _lin(_gelu(_lin(z, w, f"s{i}.ff1")), w, f"s{i}.ff2"), w, f"s{i}.ln2")
    return _lin(z, w, "shead")[:, 0]


def _lps(f, w):
    z = _gelu(_ln(_lin(f, w, "in"), w, "in_ln"))
    for i in range(2):
        z = z + _mha(_ln(z, w, f"p{i}.ln1"), w, f"p{i}")
        z = z + _lin(_gelu(_lin(_ln(z, w, f"p{i}.ln2"), w, f"p{i}.ff1")), w, f"p{i}.ff2")
    return torch.sigmoid(_lin(z, w, "phead")[:, 0])


def _select(pos, logit, tok, eos):
    """Indexes, among the masked rows, of the block that the router's logits give."""
    n = len(pos)
    if n <= L_MIN:
        return list(range(n))
    got = []
    for j in range(n):
        if logit[j] > 0 and tok[j] != eos:
            if got and pos[j] - pos[got[-1]] > G_MAX:
                break
            got.append(j)
    return got if len(got) >= L_MIN else list(range(min(L_B, n)))


def _exact_decide(case, seed, x):
    w = {k: t.cuda().double() for k, t in _router(seed, case["d_model"]).items()}
    nan = float("nan")
    n = x["row_pos"].numel()
    lbs, lps = torch.full((n,), nan, dtype=torch.float64), torch.full((n,), nan, dtype=torch.float64)
    pos, tok = x["row_pos"].tolist(), x["argmax"].tolist()
    mask, inside, meta = x["mask"].tolist(), x["in_block"].tolist(), x["blk_meta"].tolist()
    r = 0
    for i, wn in enumerate(_lens(case)[0]):
        rows = [r + j for j in range(wn) if mask[r + j]]
        b0, size = meta[i]
        blk = [j for j in rows if inside[j]]
        if size == 0:
            at, logit = torch.tensor(rows), [0.0] * len(rows)
            if len(rows) > L_MIN:
                o = _lbs(x["ent_norm"][at.cuda()].double(), x["argmax"][at.cuda()].long(), w, x["w_emb"])
                lbs[at], logit = o.cpu(), o.tolist()
            blk = [rows[j] for j in _select([pos[j] for j in rows], logit, [tok[j] for j in rows], case["vocab"] - 1)]
            b0, size = pos[blk[0]], len(blk)
        if blk:
            at = torch.tensor(blk).cuda()
            f = torch.stack([x["conf"][at].double(), x["ent_norm"][at].double(), x["gap"][at].double(),
                             torch.full((len(blk),), len(blk) / size, dtype=torch.float64, device="cuda"),
                             (x["row_pos"][at].double() - b0) / size], 1)
            lps[at.cpu()] = _lps(f, w).cpu()
        r += wn
    return dict(lbs_logit=lbs, lps_prob=lps)


def exact(case, seed):
    x = _inputs(case, seed)
    out = {}
    if "w_lm" in x:
        out.update(_exact_stats(x, case["vocab"]))
    if "q" in x:
        out["attn_out"] = _exact_attention(case, x)
    if case["entry"] == "decide" and case["mode"] == 0:
        out.update(_exact_decide(case, seed, x))
    return out or None
