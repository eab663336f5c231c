"""The work that users of the library have it do, as measurable cases.

Every case goes through the package's public calls (fb_draft, fb_refine, fb_block_forward,
fb_op_attention, fb_op_gemm and their Model methods) on seeded random-init weights and
inputs of the shapes that the repository's configurations, tests and benchmark use:

  kind "draft"      a candidate pool through (part of) the schedule, with skips, proxies,
                    guidance and SDE noise where the case asks for them
  kind "refine"     one latent through a full-computation schedule
  kind "block"      one transformer block on a residual stream (layer studies, proxies
                    calibrated block by block)
  kind "attention"  one attention layer (self- or cross-attention) on projected q, k, v
  kind "gemm"       one linear layer with its epilogue

exact() is the same arithmetic in plain torch float64.
"""
import math

import numpy as np
import torch

from paper_2607_04461_gb300 import flashbon, synth

MODELS = {"tiny": synth.TINY, "small": synth.SMALL, "wan13": synth.WAN13, "wan14": synth.WAN14}
# exact() in float64 runs at about 1 TFLOP/s; past this many operations it is left out
EXACT_FLOPS = 1.3e13


# ---- the cases ------------------------------------------------------------------------

def listed():
    return [
        # The smallest whole call: the tiny model's draft pool, 4 steps, one skip, one
        # proxy. Latency and launches: a smoke test, a CI job, a tutorial.
        _draft("tiny_draft", "tiny", n=4, steps=4, of=4, plan="tiny"),
        # One linear layer alone: the FFN down-projection of one refined candidate, with
        # bias, gate and fp32 residual.
        dict(name="gemm_ffn_down_n1", kind="gemm", M=1560, N=1536, K=8960, epi=2),
        # One self-attention layer of a small pool at 480 x 832 (1560 tokens: a ragged
        # last query and key tile).
        dict(name="attn_self_1560", kind="attention", batch=4, heads=12, Lq=1560, Lkv=1560,
             shared=False),
        # One cross-attention layer at 1024 x 1024 against the shared 512 text tokens.
        dict(name="attn_cross_4096", kind="attention", batch=4, heads=12, Lq=4096, Lkv=512,
             shared=True),
        # One block for one candidate: what the refinement of a selected draft repeats.
        _block("block_wan13_n1", "wan13", n=1),
        # The ordinary block of a draft pool: 16 candidates.
        _block("block_wan13_n16", "wan13", n=16),
        # One candidate at 1024 x 1024: 4096 tokens.
        _block("block_1k_n1", "wan13", n=1, lat_h=128, lat_w=128),
        # The wide model's block for its draft pool of 8.
        _block("block_wan14_n8", "wan14", n=8),
        # A few full steps on one candidate, all 30 blocks, the prompt encoded in the call.
        dict(name="refine_wan13", kind="refine", model="wan13", lat_h=60, lat_w=104, text=512,
             steps=2, of=50, first=10),
        # An instant draft pool: 8 candidates, the first 10 of 50 steps, a third of the
        # blocks skipped, half of the rest proxied on odd steps.
        _draft("draft_pool_wan13", "wan13", n=8, steps=10, of=50, plan="random", skip=1 / 3,
               proxy=0.5),
        # The paper's searched plan for two candidates: 49 of 50 steps, full steps every
        # fifth, second-order forecasts between, blocks 22-23 skipped from step 3.
        _draft("draft_phi_star", "wan13", n=2, steps=49, of=50, plan="phi"),
        # Guidance (two prompts, two rows per candidate) with SDE noise, as exploration
        # of one seed does.
        _draft("draft_guided_sde", "wan13", n=1, steps=2, of=50, plan="random", skip=0.25,
               proxy=0.5, order=1, guided=True, sde=0.7),
    ]


def draw(rng):
    """One more case of the listed ones' ranges."""
    while True:
        case = _draw_any(rng)
        if work(case)["flops"] <= 1.8e14 and work(case)["bytes"] <= 6e10:
            return case


def _draw_any(rng):
    pick = rng.random()
    if pick < 0.12:  # the small models' whole calls
        c = synth.TINY if rng.random() < 0.5 else synth.SMALL
        name = "tiny" if c is synth.TINY else "small"
        steps = rng.randint(1, 6)
        return _draft(None, name, n=rng.randint(1, c.max_n), steps=steps,
                      of=steps + rng.randint(0, 4), plan="random", skip=rng.choice([0, 0.34, 0.5]),
                      proxy=rng.choice([0, 0.5]), order=rng.randint(0, 2),
                      lat_h=2 * rng.randint(2, 12), lat_w=2 * rng.randint(2, 16))
    if pick < 0.32:
        D, F = rng.choice([(256, 1024), (1536, 8960), (5120, 13824)])
        N, K = rng.choice([(3 * D, D), (D, D), (F, D), (D, F), (2 * D, D)])
        return dict(kind="gemm", M=_log_int(rng, 1, 25000), N=N, K=K, epi=rng.randint(0, 3))
    if pick < 0.55:
        shared = rng.random() < 0.4
        Lq = _log_int(rng, 1, 4096)
        return dict(kind="attention", batch=_log_int(rng, 1, 16), heads=rng.choice([2, 12, 40]),
                    Lq=Lq, Lkv=rng.choice([8, 40, 77, 226, 512]) if shared else Lq, shared=shared)
    lat_h, lat_w = 2 * _log_int(rng, 8, 64), 2 * _log_int(rng, 8, 64)
    text = rng.choice([77, 226, 512])
    if pick < 0.8:
        model = rng.choice(["wan13", "wan13", "wan14"])
        return _block(None, model, n=_log_int(rng, 1, 16), lat_h=lat_h, lat_w=lat_w, text=text,
                      t=round(rng.uniform(0.02, 1.0), 3))
    if pick < 0.88:
        of = rng.choice([10, 25, 50])
        steps = rng.randint(1, 5)
        return dict(kind="refine", model="wan13", lat_h=lat_h, lat_w=lat_w, text=text,
                    steps=steps, of=of, first=rng.randint(0, of - steps))
    steps = rng.randint(2, 10)
    guided = rng.random() < 0.3
    return _draft(None, "wan13", n=_log_int(rng, 1, 4 if guided else 8), steps=steps,
                  of=rng.choice([10, 25, 50]), plan="random", skip=rng.choice([0, 0.25, 1 / 3, 0.5]),
                  proxy=rng.choice([0, 0.5]), order=rng.randint(0, 2), guided=guided,
                  sde=rng.choice([0.0, 0.7]), lat_h=lat_h, lat_w=lat_w, text=text)


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _draft(name, model, n, steps, of, plan, skip=0.0, proxy=0.0, order=0, guided=False, sde=0.0,
           lat_h=None, lat_w=None, text=None):
    c = MODELS[model]
    case = dict(kind="draft", model=model, n=n, steps=steps, of=of, plan=plan, skip=skip,
                proxy=proxy, order=order, guided=guided, sde=sde, lat_h=lat_h or c.latent_h,
                lat_w=lat_w or c.latent_w, text=text or c.text_len)
    if name:
        case["name"] = name
    return case


def _block(name, model, n, lat_h=60, lat_w=104, text=512, t=0.7):
    case = dict(kind="block", model=model, n=n, lat_h=lat_h, lat_w=lat_w, text=text, t=t)
    if name:
        case["name"] = name
    return case


def _cfg(case):
    rows = {"draft": case.get("n", 1) * (2 if case.get("guided") else 1),
            "block": case.get("n", 1), "refine": 1}[case["kind"]]
    c = MODELS[case["model"]].with_(latent_h=case["lat_h"], latent_w=case["lat_w"],
                                    text_len=case["text"], max_n=rows)
    return c.with_(depth=1) if case["kind"] == "block" else c


def _schedule(case):
    first = case.get("first", 0)
    return synth.make_schedule(case["of"])[first: first + case["steps"] + 1]


def _plan(case):
    depth = MODELS[case["model"]].depth
    if case["plan"] == "tiny":
        return synth.tiny_plan()
    if case["plan"] == "phi":
        return flashbon.fb_plan_from_phi(case["of"], case["steps"], 3, 22, 23, 5, 2, depth)
    return synth.random_plan(case["steps"], depth, case["skip"], case["proxy"],
                             order=case["order"])


# ---- inputs ---------------------------------------------------------------------------

def _gen(seed, stream):
    return torch.Generator(device="cuda").manual_seed(int(seed) * 1009 + stream)


def _randn(shape, seed, stream, dtype=torch.float32, scale=1.0):
    x = torch.randn(shape, generator=_gen(seed, stream), device="cuda", dtype=torch.float32)
    return (x * scale if scale != 1.0 else x).to(dtype)


def _weights(cfg, seed):
    """Packed random-init weights (fp32 values that are exact in bf16) and named views."""
    specs = synth.weight_specs(cfg)
    sizes = [math.prod(shape) for _, shape, _ in specs]
    buf = torch.randn(sum(sizes), generator=_gen(seed, 0), device="cuda", dtype=torch.float32)
    buf.mul_(0.02)
    views, off = {}, 0
    for (name, shape, kind), size in zip(specs, sizes):
        views[name] = buf[off: off + size].view(shape)
        if kind == "norm":
            views[name].add_(1.0)
        views[name].copy_(views[name].bfloat16())
        off += size
    return buf, views


def _sampler_inputs(case, cfg, seed):
    n = case.get("n", 1)
    shape = (n, cfg.latent_c, cfg.latent_h, cfg.latent_w)
    z = _randn(shape, seed, 1)
    text = _randn((cfg.text_len, cfg.text_dim), seed, 2)
    uncond = _randn((cfg.text_len, cfg.text_dim), seed, 3) if case.get("guided") else None
    noise = _randn((case["steps"],) + shape, seed, 4) if case.get("sde") else None
    return z, text, uncond, noise


def _attention_inputs(case, seed):
    """q and k of unit variance (they leave an RMSNorm), v of a projection's; q, k and v
    interleaved by row as the QKV projection writes them (self), k and v as the text
    projection does (cross)."""
    D = case["heads"] * 128
    rows = case["batch"] * case["Lq"]
    if case["shared"]:
        q = _randn((rows, D), seed, 1, torch.bfloat16)
        kv = _randn((case["Lkv"], 2 * D), seed, 2, torch.bfloat16)
        return q, kv[:, :D], kv[:, D:]
    qkv = _randn((rows, 3 * D), seed, 1, torch.bfloat16)
    return qkv[:, :D], qkv[:, D: 2 * D], qkv[:, 2 * D:]


def _gemm_inputs(case, seed):
    M, N, K, epi = case["M"], case["N"], case["K"], case["epi"]
    f32 = torch.float32
    return dict(A=_randn((M, K), seed, 1, torch.bfloat16),
                W=_randn((N, K), seed, 2, torch.bfloat16, 0.02), bias=_randn((N,), seed, 3, f32, 0.02),
                resid=_randn((M, N), seed, 4) if epi >= 2 else None,
                gate=_randn((N,), seed, 5) if epi >= 2 else None,
                base=_randn((M, N), seed, 6) if epi == 3 else None)


class _State:
    """What a user's program keeps: the model and its buffers."""

    def __init__(self, case):
        self.case = case
        self.model = None

    def __del__(self):
        if self.model is not None:
            self.model.close()


def prepare(case, seed):
    s = _State(case)
    kind = case["kind"]
    if kind in ("attention", "gemm"):
        # the single-layer calls run on any model's stream: a tiny one carries them
        s.model = flashbon.Model(synth.TINY, synth.make_weights(synth.TINY))
        if kind == "gemm":
            s.io = _gemm_inputs(case, seed)
            wide = torch.float32 if case["epi"] >= 2 else torch.bfloat16
            s.out = torch.empty((case["M"], case["N"]), dtype=wide, device="cuda")
            s.delta = (torch.empty((case["M"], case["N"]), dtype=torch.bfloat16, device="cuda")
                       if case["epi"] == 3 else None)
        else:
            s.q, s.k, s.v = _attention_inputs(case, seed)
            s.out = torch.empty((s.q.shape[0], case["heads"] * 128), dtype=torch.bfloat16,
                                device="cuda")
        return s
    cfg = _cfg(case)
    packed, _ = _weights(cfg, seed)
    torch.cuda.synchronize()
    s.model = flashbon.Model(cfg, packed)
    del packed, _
    if kind == "block":
        s.h0 = _randn((case["n"] * cfg.tokens, cfg.dim), seed, 1)
        s.h = torch.empty_like(s.h0)
        s.model.encode_text(_randn((cfg.text_len, cfg.text_dim), seed, 2))
        return s
    s.z0, s.text, s.uncond, s.noise = _sampler_inputs(case, cfg, seed)
    s.z = torch.empty_like(s.z0)
    s.schedule = _schedule(case)
    s.opts = None
    if kind == "draft":
        s.skip, s.proxy = _plan(case)
        if case["guided"] or case["sde"]:
            s.opts = flashbon.make_opts(guidance=5.0 if case["guided"] else 1.0,
                                        text_uncond=s.uncond, sde_a=case["sde"], noise=s.noise)
    return s


def run(s):
    case, kind = s.case, s.case["kind"]
    if kind == "gemm":
        i = s.io
        flashbon.fb_op_gemm(s.model.handle, case["M"], case["N"], case["K"], i["A"], i["W"],
                            i["bias"], case["epi"], s.out, i["resid"], i["gate"], i["base"], s.delta)
        return s.out if s.delta is None else (s.out, s.delta)
    if kind == "attention":
        # column slices of the projections' outputs: passed by address, with row strides
        flashbon.fb_op_attention(s.model.handle, s.q.data_ptr(), s.q.stride(0), s.k.data_ptr(),
                                 s.k.stride(0), s.v.data_ptr(), s.v.stride(0), s.out,
                                 s.out.stride(0), case["batch"], case["Lq"], case["Lkv"],
                                 0 if case["shared"] else case["Lkv"], case["heads"], 128)
        return s.out
    if kind == "block":
        s.h.copy_(s.h0)  # the block updates the residual stream in place
        s.model.block_forward(0, s.h, case["n"], case["t"])
        return s.h
    s.z.copy_(s.z0)      # the sampler updates the latents in place
    if kind == "refine":
        s.model.refine(s.z, s.text, s.schedule)
    else:
        s.model.draft(s.z, s.text, s.schedule, s.skip, s.proxy, opts=s.opts)
    return s.z


# ---- work -----------------------------------------------------------------------------

def _block_work(cfg, rows, batches, kv_sets):
    """Operations and bytes of one block: weights and the text K/V read once, the residual
    stream read and written once."""
    D, F, P, T = cfg.dim, cfg.ffn, cfg.tokens, cfg.text_len
    mats = 6 * D * D + 2 * D * F
    flops = 2.0 * rows * mats + 4.0 * batches * P * D * (P + T)
    return flops, 2.0 * mats + 2.0 * kv_sets * T * 2 * D + 8.0 * rows * D


def work(case):
    kind = case["kind"]
    if kind == "gemm":
        M, N, K = case["M"], case["N"], case["K"]
        out = {0: 2, 1: 2, 2: 8, 3: 14}[case["epi"]]
        return {"bytes": 2.0 * (M * K + N * K) + float(out) * M * N, "flops": 2.0 * M * N * K}
    if kind == "attention":
        D, B, Lq, Lkv = case["heads"] * 128, case["batch"], case["Lq"], case["Lkv"]
        return {"bytes": 2.0 * D * (2 * B * Lq + 2 * (1 if case["shared"] else B) * Lkv),
                "flops": 4.0 * B * D * Lq * Lkv}
    cfg = _cfg(case)
    D, P, T = cfg.dim, cfg.tokens, cfg.text_len
    cond = 2.0 * D * (cfg.freq_dim + D + 6 * D)  # operations (= bytes) of a step's conditioning
    if kind == "block":
        f, b = _block_work(cfg, case["n"] * P, case["n"], 1)
        return {"bytes": b + cond, "flops": f + cond}
    n, sets = case.get("n", 1), 2 if case.get("guided") else 1
    rows = n * sets * P
    # the prompt once per call
    flops = sets * 2.0 * T * (cfg.text_dim * D + D * D + cfg.depth * 2 * D * D)
    bytes_ = 2.0 * (cfg.text_dim * D + D * D + cfg.depth * 2 * D * D) + sets * 4.0 * T * cfg.text_dim
    skip, proxy = _plan(case) if kind == "draft" else synth.empty_plan(case["steps"], cfg.depth)
    fb, bb = _block_work(cfg, rows, n * sets, sets)
    computed = int(((skip == 0) & (proxy == synth.COMPUTE)).sum())
    terms = sum(1 + (int(c) >> 16) for c in proxy[proxy != synth.COMPUTE].tolist())
    flops += computed * fb + terms * 2.0 * rows * D
    bytes_ += computed * bb + terms * 2.0 * rows * D
    lat = 4.0 * n * cfg.latent_c * cfg.latent_h * cfg.latent_w
    # conditioning, patch embedding, head and update of every step
    flops += case["steps"] * (cond + 4.0 * rows * D * cfg.patch_dim)
    bytes_ += case["steps"] * (cond + 4.0 * rows * D + 2 * lat + (lat if case.get("sde") else 0))
    return {"bytes": bytes_, "flops": flops}


# ---- the same in float64 --------------------------------------------------------------

def _norm(x, eps):
    x = x - x.mean(-1, keepdim=True)
    return x * torch.rsqrt((x * x).mean(-1, keepdim=True) + eps)


def _rms(x, w, eps):
    return x * torch.rsqrt((x * x).mean(-1, keepdim=True) + eps) * w


def _gelu(x):
    return 0.5 * x * (1 + torch.tanh(math.sqrt(2 / math.pi) * (x + 0.044715 * x ** 3)))


def _lin(x, w, b):
    return x @ w.double().t() + b.double()


def _attend(q, k, v):
    """q [Lq, H, d], k and v [Lkv, H, d] -> [Lq, H * d]."""
    q, k, v = (x.transpose(0, 1) for x in (q, k, v))
    p = torch.softmax(q @ k.transpose(1, 2) / math.sqrt(q.shape[-1]), -1)
    return (p @ v).transpose(0, 1).reshape(q.shape[1], -1)


class _Exact:
    def __init__(self, cfg, w):
        self.c, self.w = cfg, w
        half = cfg.head_dim // 2
        tok = torch.arange(cfg.tokens, device="cuda")
        j = torch.arange(half, device="cuda")
        pos = torch.where((j < half // 2)[None], (tok // cfg.grid_w)[:, None],
                          (tok % cfg.grid_w)[:, None]).double()
        ang = pos * torch.pow(torch.tensor(float(cfg.rope_theta), dtype=torch.float64, device="cuda"),
                              -2.0 * (j % (half // 2)).double() / half)
        self.cos, self.sin = torch.cos(ang)[:, None], torch.sin(ang)[:, None]

    def time(self, t):
        c, w = self.c, self.w
        half = c.freq_dim // 2
        f = torch.exp(-math.log(10000.0) * torch.arange(half, device="cuda").double() / half)
        arg = 1000.0 * float(np.float32(t)) * f
        emb = torch.cat([torch.cos(arg), torch.sin(arg)])
        x = torch.nn.functional.silu(_lin(emb, w["time.w1"], w["time.b1"]))
        temb = _lin(x, w["time.w2"], w["time.b2"])
        mod = _lin(torch.nn.functional.silu(temb), w["mod.w"], w["mod.b"])
        return temb, mod.view(6, c.dim)

    def text(self, ctx):
        w = self.w
        x = _lin(_gelu(_lin(ctx.double(), w["text.w1"], w["text.b1"])), w["text.w2"], w["text.b2"])
        out = []
        for l in range(self.c.depth):
            p = f"blocks.{l}.cross."
            k, v = _lin(x, w[p + "wkv"], w[p + "bkv"]).chunk(2, -1)
            out.append((_rms(k, w[p + "norm_k"].double(), self.c.eps_rms), v))
        return out

    def rope(self, x):
        a, b = x[..., 0::2], x[..., 1::2]
        return torch.stack([a * self.cos - b * self.sin, a * self.sin + b * self.cos], -1).flatten(-2)

    def block(self, l, h, mod, kv):
        """One candidate's rows h [tokens, dim]."""
        c, w, p = self.c, self.w, f"blocks.{l}."
        s1, c1, g1, s2, c2, g2 = mod + w[p + "table"].double()
        H, d = c.heads, c.head_dim
        q, k, v = _lin(_norm(h, c.eps_ln) * (1 + c1) + s1, w[p + "attn.wqkv"],
                       w[p + "attn.bqkv"]).chunk(3, -1)
        q = self.rope(_rms(q, w[p + "attn.norm_q"].double(), c.eps_rms).view(-1, H, d))
        k = self.rope(_rms(k, w[p + "attn.norm_k"].double(), c.eps_rms).view(-1, H, d))
        h = h + g1 * _lin(_attend(q, k, v.reshape(-1, H, d)), w[p + "attn.wo"], w[p + "attn.bo"])
        x = _norm(h, c.eps_ln) * w[p + "norm3.w"].double() + w[p + "norm3.b"].double()
        q = _rms(_lin(x, w[p + "cross.wq"], w[p + "cross.bq"]), w[p + "cross.norm_q"].double(),
                 c.eps_rms)
        k, v = kv[l]
        o = _attend(q.view(-1, H, d), k.reshape(-1, H, d), v.reshape(-1, H, d))
        h = h + _lin(o, w[p + "cross.wo"], w[p + "cross.bo"])
        x = _norm(h, c.eps_ln) * (1 + c2) + s2
        x = _gelu(_lin(x, w[p + "ffn.w1"], w[p + "ffn.b1"]))
        return h + g2 * _lin(x, w[p + "ffn.w2"], w[p + "ffn.b2"])

    def velocity(self, z, t, step, kv, skip, proxy, sched, cache):
        """One candidate's velocity; cache[l] holds (step, contribution), newest last."""
        c, w = self.c, self.w
        temb, mod = self.time(t)
        gh, gw, pp = c.grid_h, c.grid_w, c.patch
        x = z.view(c.latent_c, gh, pp, gw, pp).permute(1, 3, 0, 2, 4).reshape(gh * gw, -1)
        h = _lin(x, w["patch.w"], w["patch.b"])
        for l in range(c.depth):
            if skip[step, l]:
                continue
            code = int(proxy[step, l])
            if code == synth.COMPUTE:
                new = self.block(l, h, mod, kv)
                cache[l].append((step, new - h))
                h = new
                continue
            src, order = code & 0xFFFF, code >> 16
            past = [e for e in reversed(cache[l]) if e[0] <= src][: order + 1]
            d = past[0][1]
            if len(past) > 1:
                tau = [float(sched[e[0]]) for e in past]
                a = (float(t) - tau[0]) / (tau[0] - tau[1])
                d = d + a * (past[0][1] - past[1][1])
                if len(past) > 2:
                    d = d + 0.5 * a * a * (past[0][1] - 2 * past[1][1] + past[2][1])
            h = h + d
        shift, scale = w["head.table"].double() + temb
        v = _lin(_norm(h, c.eps_ln) * (1 + scale) + shift, w["head.w"], w["head.b"])
        v = v.view(gh, gw, c.latent_c, pp, pp).permute(2, 0, 3, 1, 4)
        return v.reshape(c.latent_c, c.latent_h, c.latent_w)

    def sample(self, z0, text, uncond, noise, sched, skip, proxy, w=1.0, sde=0.0):
        kv = self.text(text)
        kv_u = None if uncond is None else self.text(uncond)
        out = []
        for i in range(z0.shape[0]):
            z = z0[i].double()
            caches = [[[] for _ in range(self.c.depth)] for _ in range(2)]
            for k in range(len(sched) - 1):
                t, t1 = float(sched[k]), float(sched[k + 1])
                v = self.velocity(z, sched[k], k, kv, skip, proxy, sched, caches[0])
                if kv_u is not None:
                    vu = self.velocity(z, sched[k], k, kv_u, skip, proxy, sched, caches[1])
                    v = vu + w * (v - vu)
                dt = t1 - t
                if sde:
                    te = t1 if t >= 1.0 else t
                    sig = sde * math.sqrt(te / (1 - te))
                    z = z + (v + sig * sig / (2 * t) * (z + (1 - t) * v)) * dt \
                        + sig * math.sqrt(abs(dt)) * noise[k, i].double()
                else:
                    z = z + dt * v
            out.append(z)
        return torch.stack(out)


def exact(case, seed):
    if work(case)["flops"] > EXACT_FLOPS:
        return None
    kind = case["kind"]
    with torch.no_grad():
        if kind == "gemm":
            i = _gemm_inputs(case, seed)
            y = _lin(i["A"].double(), i["W"], i["bias"])
            if case["epi"] < 2:
                return _gelu(y) if case["epi"] == 1 else y
            y = i["resid"].double() + i["gate"].double() * y
            return y if case["epi"] == 2 else (y, y - i["base"].double())
        if kind == "attention":
            q, k, v = _attention_inputs(case, seed)
            B, H, Lkv = case["batch"], case["heads"], case["Lkv"]
            q = q.reshape(B, case["Lq"], H, 128)
            k, v = (x.reshape(-1, Lkv, H, 128) for x in (k, v))
            out = [torch.cat([_attend(q[b, :, h: h + 1].double(),
                                      k[0 if case["shared"] else b][:, h: h + 1].double(),
                                      v[0 if case["shared"] else b][:, h: h + 1].double())
                              for h in range(H)], -1) for b in range(B)]
            return torch.cat(out)
        cfg = _cfg(case)
        _, w = _weights(cfg, seed)
        e = _Exact(cfg, w)
        if kind == "block":
            h = _randn((case["n"] * cfg.tokens, cfg.dim), seed, 1)
            kv = e.text(_randn((cfg.text_len, cfg.text_dim), seed, 2))
            mod = e.time(case["t"])[1]
            return torch.cat([e.block(0, x.double(), mod, kv) for x in h.split(cfg.tokens)])
        z, text, uncond, noise = _sampler_inputs(case, cfg, seed)
        skip, proxy = _plan(case) if kind == "draft" else synth.empty_plan(case["steps"], cfg.depth)
        return e.sample(z, text, uncond, noise, _schedule(case), skip, proxy,
                        w=5.0 if case.get("guided") else 1.0, sde=case.get("sde", 0.0))


# ---- tolerances -----------------------------------------------------------------------
# About four times the error against exact() (relative 2-norm), measured on the listed and
# on drawn cases; bf16 operands, fp32 sums:
#   gemm       fp32 outputs 4e-6, bf16 outputs 1.7e-3 to 2.2e-3 (one bf16 rounding)
#   attention  2.1e-3 to 2.3e-3
#   block      3.7e-4 (dim 1536), 1.5e-3 (dim 5120): the residual stream dominates
#   sampler    6e-5 for a schedule that spans 0.04, 7e-4 for one that spans 0.8; with
#              guidance w = 5 (5 v - 4 v_u) 4e-4 for a span of 0.04. Where exact() is left
#              out: against the same call with the sums of the cut GEMM tiles in another
#              order (another number of SMs), 1.4e-4 for the pool of 8 and 5e-4 for the
#              searched plan.

def tolerance(case):
    kind = case["kind"]
    if kind == "gemm":
        return {"rel": 2e-5} if case["epi"] == 2 else {"rel": 8e-3}
    if kind == "attention":
        return {"rel": 9e-3}
    if kind == "block":
        return {"rel": 6e-3 if case["model"] == "wan14" else 1.5e-3}
    sched = _schedule(case)
    span = float(sched[0] - sched[-1])
    return {"rel": (2e-4 + 3e-3 * span) * (6 if case.get("guided") else 1)}
