"""What this framework is timed on: one pass of its public entry points, over the range of sizes
that a program which denoises with it uses.

A "model" case is a trajectory of ``binding.Denoiser`` (sgd_set_schedule, sgd_step, the sampler
update between two steps) at the real widths of the five synthetic architectures; all but two keep a
few blocks only, so that a case is a block with its stem and head.  The other cases are single
kernels of a step through the C ABI (``sgd_kernel_*``), for programs that call a layer by itself.
Weights are products of Gaussian factors with power-law singular values, as the paper's spectra
have, and every input comes from the seed.

``exact`` computes the same in float64 with torch alone.
"""
import math

import torch

from paper_2609_29505_gb300 import binding, synth

# stem, block, norm, mlp and head of the architectures, and what goes with them
ARCH = {
    "tiny": dict(stem="time_add", block="prenorm", norm="rms", mlp="swiglu", head="linear"),
    "dit": dict(stem="patch", block="adaln", norm="ln_plain", mlp="gelu_tanh", head="adaln_linear",
                channels=16, d_out=32, n_classes=1001, t_freq=256),
    "uvit": dict(stem="patch_tokens", block="prenorm", norm="ln", mlp="gelu_erf", head="linear",
                 channels=16, d_out=16, n_classes=1001, n_prefix=2),
    "sdxl": dict(stem="identity", block="xattn", norm="ln", mlp="geglu", head="identity",
                 ctx_len=77, d_ctx=2048),
    "llada": dict(stem="embed", block="prenorm", norm="rms", mlp="swiglu", head="logits", rope=True),
}
EPS = 1e-6
THETA = 10000.0


def _model(name, arch, n_blocks, n_heads, d_head, d_ff, batch, n_tokens, T, budget, vocab=0, host=False):
    c = dict(kind="model", arch=arch, n_blocks=n_blocks, n_heads=n_heads, d_head=d_head, d_ff=d_ff,
             batch=batch, n_tokens=n_tokens, T=T, budget=budget, vocab=vocab, host=host)
    return dict(c, name=name) if name else c


def _gemm(name, epi, M, N, K, act=0, cache=False, gate_rows=0, d_head=0):
    c = dict(kind="gemm", epi=epi, M=M, N=N, K=K, act=act, cache=cache, gate_rows=gate_rows, d_head=d_head)
    return dict(c, name=name) if name else c


def _attention(name, batch, n_heads, d_head, n_q, n_kv):
    c = dict(kind="attention", batch=batch, n_heads=n_heads, d_head=d_head, n_q=n_q, n_kv=n_kv)
    return dict(c, name=name) if name else c


def listed():
    return [
        # the smallest model: a whole 10-step trajectory where launches and latency are everything
        _model("tiny trajectory", "tiny", 4, 4, 64, 688, 1, 64, 10, 0.5),
        # class-conditional image model at full depth, a short trajectory at half the layer steps
        _model("dit trajectory", "dit", 28, 16, 72, 4608, 8, 256, 4, 0.5),
        # U-shaped image transformer: long skips, a ragged 258 tokens, buffers on the host
        _model("uvit host", "uvit", 5, 16, 64, 4096, 16, 258, 3, 0.5, host=True),
        # text-to-image transformer blocks: self- and cross-attention, context projected at step 1
        _model("sdxl blocks", "sdxl", 2, 20, 64, 5120, 2, 1024, 3, 0.5),
        # language model at the batch it is served with: blocks at full width and the whole vocabulary
        _model("llada blocks", "llada", 2, 32, 128, 12288, 4, 1024, 2, 0.5, vocab=126464),
        # the same for one short prompt of an odd length
        _model("llada prompt", "llada", 2, 32, 128, 12288, 1, 333, 2, 0.5, vocab=126464),
        # one large projection with its gated activation
        _gemm("gated projection", "gated", 4096, 12288, 4096),
        # a residual projection of a mid-size model, odd rows, the update stored for later steps
        _gemm("residual projection", "delta", 1003, 1280, 5120, cache=True),
        # self-attention over a long context
        _attention("attention 4k", 1, 32, 128, 4096, 4096),
        # cross-attention: many queries, 77 keys
        _attention("cross attention", 2, 20, 64, 1024, 77),
        # the norm ahead of every branch of the language model
        dict(name="norm", kind="norm", norm="rms", rows=4096, d=4096, mod_rows=0),
        # the cached updates of nine frozen units added to the stream
        dict(name="frozen run", kind="frozen", rows=4128, d=1024, caches=9),
    ]


# ---------------------------------------------------------------------------
# drawn cases: the same ranges
# ---------------------------------------------------------------------------

def _log(rng, lo, hi, step=1):
    v = math.exp(rng.uniform(math.log(lo), math.log(hi)))
    return max(step, min(hi, int(round(v / step)) * step))


def draw(rng):
    kind = rng.choice(["model"] * 6 + ["gemm"] * 3 + ["attention"] * 2 + ["norm", "frozen"])
    if kind == "model":
        arch = rng.choice(["tiny", "dit", "uvit", "sdxl", "llada"])
        budget = rng.choice([1.0, 0.5, 0.5, 0.33])
        host = rng.random() < 0.2
        if arch == "tiny":
            return _model(None, arch, rng.randint(1, 4), rng.randint(1, 4), rng.choice([64, 128]),
                          _log(rng, 128, 1376, 8), rng.randint(1, 2), _log(rng, 8, 192), rng.randint(4, 10),
                          budget, host=host)
        if arch == "dit":
            heads, dh = rng.choice([(4, 72), (16, 72), (16, 72), (12, 64)])
            return _model(None, arch, _log(rng, 1, 28), heads, dh, 4 * heads * dh, _log(rng, 1, 8),
                          _log(rng, 64, 256), rng.randint(2, 4), budget, host=host)
        if arch == "uvit":
            heads = rng.choice([4, 8, 16, 16])
            return _model(None, arch, 2 * rng.randint(1, 4) + 1, heads, 64, 256 * heads, _log(rng, 1, 16),
                          _log(rng, 64, 256) + 2, rng.randint(2, 4), budget, host=host)
        if arch == "sdxl":
            heads = rng.choice([5, 10, 20, 20])
            return _model(None, arch, rng.randint(1, 4), heads, 64, rng.choice([128, 256]) * heads,
                          rng.randint(1, 2), _log(rng, 196, 2048), rng.randint(2, 4), budget, host=host)
        heads = rng.choice([4, 16, 32, 32])
        batch = rng.randint(1, 4)
        return _model(None, arch, rng.randint(1, 2), heads, 128, rng.choice([344, 384]) * heads, batch,
                      _log(rng, 17, 4096 // batch), 2, budget, vocab=rng.choice([1000, 32000, 126464]))
    if kind == "gemm":
        epi = rng.choice(["f16", "f32", "delta", "delta", "gated", "gelu", "rope"])
        M = _log(rng, 1, 8192)
        dh = rng.choice([64, 128]) if epi == "rope" else 0
        N = 3 * dh * _log(rng, 2, 32) if dh else _log(rng, 64, 12288, 8)
        K = _log(rng, 64, 12288, 8)
        while 2.0 * M * N * K * (2 if epi == "gated" else 1) > 2e12:
            M = (M + 1) // 2
        return _gemm(None, epi, M, N, K, act=rng.randint(0, 1), cache=epi == "delta" and rng.random() < 0.5,
                     gate_rows=rng.choice([0, 0, _log(rng, 16, 1024)]) if epi == "delta" else 0, d_head=dh)
    if kind == "attention":
        dh = rng.choice([64, 64, 72, 128, 128])
        n = _log(rng, 16, 4096)
        heads = _log(rng, 1, 32)
        batch = max(1, min(_log(rng, 1, 16), 16384 // n))
        return _attention(None, batch, heads, dh, n, 77 if rng.random() < 0.25 else n)
    if kind == "norm":
        return dict(kind="norm", norm=rng.choice(["rms", "ln", "ln_plain"]), rows=_log(rng, 1, 16384),
                    d=_log(rng, 64, 4096, 8), mod_rows=rng.choice([0, 256]))
    return dict(kind="frozen", rows=_log(rng, 1, 8192), d=_log(rng, 64, 4096, 8), caches=_log(rng, 1, 64))


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------

def _generator(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed))


def _randn(g, *shape):
    return torch.randn(*shape, generator=g, device="cuda")


def _matrix(g, m, n):
    """bf16 [m, n] with power-law singular values and Frobenius norm about sqrt(min(m, n))."""
    r = min(m, n)
    s = torch.arange(1, r + 1, device="cuda").float().pow(-(0.3 + 1.2 * torch.rand((), generator=g, device="cuda")))
    s = s * (math.sqrt(r) / torch.linalg.vector_norm(s))
    u, v = _randn(g, m, r) / math.sqrt(m), _randn(g, n, r) / math.sqrt(n)
    return ((u * s) @ v.T).bfloat16()


def _dims(c):
    a = ARCH[c["arch"]]
    d = c["n_heads"] * c["d_head"]
    ch = a.get("channels", d)
    return d, c["d_ff"], a, ch


def _weights(c, g):
    d, f, a, ch = _dims(c)
    skips = (c["n_blocks"] - 1) // 2 if c["arch"] == "uvit" else 0
    w = {}

    def gain(name):
        w[name + "_w"] = (1 + 0.1 * _randn(g, d)).bfloat16()
        if a["norm"] == "ln":
            w[name + "_b"] = (0.1 * _randn(g, d)).bfloat16()

    for b in range(c["n_blocks"]):
        p = "blocks.%d." % b
        if a["norm"] != "ln_plain":
            gain(p + "norm1")
            gain(p + "norm2")
        w[p + "w_qkv"], w[p + "w_o"] = _matrix(g, 3 * d, d), _matrix(g, d, d)
        if a["block"] == "xattn":
            gain(p + "normx")
            w[p + "wx_q"], w[p + "wx_kv"] = _matrix(g, d, d), _matrix(g, 2 * d, a["d_ctx"])
            w[p + "wx_o"] = _matrix(g, d, d)
        w[p + "w_1"] = _matrix(g, 2 * f if a["mlp"] in ("swiglu", "geglu") else f, d)
        w[p + "w_2"] = _matrix(g, d, f)
        if a["block"] == "adaln":
            w[p + "w_mod"] = _matrix(g, 6 * d, d)
    if a["stem"].startswith("patch"):
        w["w_stem"], w["pos_emb"] = _matrix(g, d, ch), (0.1 * _randn(g, c["n_tokens"], d)).bfloat16()
        w["class_emb"] = _randn(g, a["n_classes"], d).bfloat16()
    if a["block"] == "adaln":
        w["w_t1"], w["w_t2"] = _matrix(g, d, a["t_freq"]), _matrix(g, d, d)
        w["w_modf"] = _matrix(g, 2 * d, d)
    for j in range(skips):
        w["skips.%d.w" % j] = _matrix(g, d, 2 * d)
    if a["head"] in ("linear", "logits"):
        gain("normf")
    if a["head"] != "identity":
        w["w_head"] = _matrix(g, c["vocab"] or a.get("d_out", d), d)
    if a["stem"] == "embed":
        w["embed"] = _randn(g, c["vocab"], d).bfloat16()
    return w


def _lifetimes(c):
    """Lifetimes per block: a ramp over the horizon whose mean is the budget, in scattered order."""
    n, T = c["n_blocks"], c["T"]
    if c["budget"] >= 1.0:
        return [T] * n
    life = [T] * n
    for i, b in enumerate(sorted(range(n), key=lambda b: (b * 0.6180339887) % 1.0)):
        life[b] = min(T, max(1, round(2 * c["budget"] * T * (i + 0.5) / n)))
    return life


def _timestep(c, s):
    return 1000.0 * (c["T"] - s + 1) / c["T"]


def _model_inputs(c, g):
    """State (or the ids of every step), class ids and context."""
    d, _, a, ch = _dims(c)
    B, n = c["batch"], c["n_tokens"] - a.get("n_prefix", 0)
    x = {}
    if a["stem"] == "embed":  # a growing share of each row is revealed, the rest is the mask id
        target = torch.randint(0, c["vocab"] - 1, (B, n), generator=g, device="cuda", dtype=torch.int32)
        rank = torch.rand(B, n, generator=g, device="cuda").argsort(dim=1)
        x["ids"] = [torch.where(rank < (s * n) // c["T"], target, torch.full_like(target, c["vocab"] - 1))
                    for s in range(c["T"])]
    else:
        x["z0"] = _randn(g, B, n, ch).bfloat16().float()
    if "n_classes" in a:
        x["class_ids"] = torch.randint(0, a["n_classes"] - 1, (B,), generator=g, device="cuda", dtype=torch.int32)
    if "ctx_len" in a:
        x["ctx"] = _randn(g, B, a["ctx_len"], a["d_ctx"]).bfloat16()
    return x


def _layer_inputs(c, g):
    """Inputs of the single-kernel cases."""
    x = {}
    if c["kind"] == "gemm":
        M, N, K = c["M"], c["N"], c["K"]
        x["A"] = _randn(g, M, K).half()
        x["B"] = (_randn(g, 2 * N if c["epi"] == "gated" else N, K) / math.sqrt(K)).half()
        if c["epi"] == "delta":
            x["h"] = _randn(g, M, N)
        if c["gate_rows"]:
            x["gate"] = 0.3 * _randn(g, -(-M // c["gate_rows"]), N)
        if c["epi"] == "rope":
            half = c["d_head"] // 2
            freq = THETA ** (-torch.arange(half, device="cuda", dtype=torch.float64) / half)
            angle = torch.arange(1024, device="cuda", dtype=torch.float64)[:, None] * freq
            x["cos"], x["sin"] = angle.cos().float(), angle.sin().float()
    elif c["kind"] == "attention":
        B, H, dh = c["batch"], c["n_heads"], c["d_head"]
        hs = 80 if dh == 72 else dh  # heads of 72 columns lie 80 apart, zeros between them
        for name, n in (("q", c["n_q"]), ("k", c["n_kv"]), ("v", c["n_kv"])):
            t = torch.zeros(B, n, H, hs, device="cuda", dtype=torch.float16)
            t[..., :dh] = _randn(g, B, n, H, dh) * (1.0 if name == "v" else 1.5)
            x[name] = t
    elif c["kind"] == "norm":
        x["h"] = 2.0 * _randn(g, c["rows"], c["d"]) + 0.3
        if c["norm"] != "ln_plain":
            x["g"] = (1 + 0.1 * _randn(g, c["d"])).bfloat16()
        if c["norm"] == "ln":
            x["b"] = (0.1 * _randn(g, c["d"])).bfloat16()
        if c["mod_rows"]:  # shift and scale of every sample, side by side
            x["mod"] = 0.3 * _randn(g, -(-c["rows"] // c["mod_rows"]), 2 * c["d"])
            x["shift"], x["scale"] = x["mod"].split(c["d"], 1)
    else:
        x["h"] = _randn(g, c["rows"], c["d"])
        x["caches"] = [_randn(g, c["rows"], c["d"]).half() for _ in range(c["caches"])]
    return x


# ---------------------------------------------------------------------------
# the calls
# ---------------------------------------------------------------------------

def _prepare_model(c, g):
    d, f, a, ch = _dims(c)
    w = _weights(c, g)
    x = _model_inputs(c, g)
    keys = ("stem", "block", "norm", "mlp", "head")
    cfg = synth.ModelConfig(
        name=c["arch"], **{k: a[k] for k in keys}, n_blocks=c["n_blocks"], d=d, n_heads=c["n_heads"],
        d_head=c["d_head"], d_ff=f, batch=c["batch"], n_tokens=c["n_tokens"], d_in=0 if c["vocab"] else ch,
        d_out=0 if a["head"] == "identity" else c["vocab"] or a.get("d_out", d), out_channels=c["vocab"] or ch,
        T=c["T"], rope=a.get("rope", False), rope_theta=THETA, eps=EPS, n_prefix=a.get("n_prefix", 0),
        n_skips=(c["n_blocks"] - 1) // 2 if c["arch"] == "uvit" else 0, ctx_len=a.get("ctx_len", 0),
        d_ctx=a.get("d_ctx", 0), vocab=c["vocab"], n_classes=a.get("n_classes", 0), t_freq=a.get("t_freq", 0))
    life = _lifetimes(c)
    groups = synth.block_groups(cfg)
    model = binding.Denoiser(cfg, w)
    model.set_schedule(c["T"], [life[b] for b in groups], groups)
    where = dict(device="cpu", pin_memory=True) if c["host"] else dict(device="cuda")
    shape = (c["batch"], cfg.n_out_tokens, cfg.out_channels)
    outs = [torch.empty(shape, dtype=torch.float16 if c["vocab"] else torch.float32, **where) for _ in range(c["T"])]
    if c["host"]:
        x = {k: [t.cpu().pin_memory() for t in v] if isinstance(v, list) else v.cpu().pin_memory()
             for k, v in x.items()}
    z = None if c["vocab"] else torch.empty_like(x["z0"])
    return dict(case=c, model=model, x=x, outs=outs, z=z)


def _run_model(s):
    c, x, model, T = s["case"], s["x"], s["model"], s["case"]["T"]
    cls, ctx = x.get("class_ids"), x.get("ctx")
    if c["host"]:  # every step on the noisy state, results in the caller's buffers after the wait
        for k in range(1, T + 1):
            state = x["ids"][k - 1] if c["vocab"] else x["z0"]
            model.step_host_async(state, s["outs"][k - 1], _timestep(c, k), k, class_ids_host=cls, ctx_host=ctx)
        model.host_wait()
        return s["outs"]
    if c["vocab"]:
        for k in range(1, T + 1):
            model.step(x["ids"][k - 1], s["outs"][k - 1], _timestep(c, k), k)
        return s["outs"]
    z = s["z"]
    z.copy_(x["z0"])
    for k in range(1, T + 1):
        model.step(z, s["outs"][k - 1], _timestep(c, k), k, class_ids=cls, ctx=ctx)
        binding.sgd_sampler_update(z, s["outs"][k - 1], 1.0, 1.0 / T)
    return s["outs"] + [z]


EPI = {"f16": binding.EPI_F16, "f32": binding.EPI_F32, "delta": binding.EPI_DELTA, "gated": binding.EPI_GATED,
       "gelu": binding.EPI_GELU, "rope": binding.EPI_ROPE}
NORM = {"rms": 0, "ln": 1, "ln_plain": 2}


def prepare(case, seed):
    g = _generator(seed)
    if case["kind"] == "model":
        return _prepare_model(case, g)
    c, x = case, _layer_inputs(case, g)
    s = dict(case=c, x=x)
    if c["kind"] == "gemm":
        M, N = c["M"], c["N"]
        e = binding.sgd_epilogue_args(kind=EPI[c["epi"]], alpha=1.0, act=c["act"])
        if c["epi"] == "delta":
            e.h, e.ldh = x["h"].data_ptr(), N
            if c["cache"]:
                s["cache"] = torch.empty(M, N, device="cuda", dtype=torch.float16)
                e.cache, e.ld_cache = s["cache"].data_ptr(), N
            if c["gate_rows"]:
                e.gate, e.ld_gate, e.rows_per_batch = x["gate"].data_ptr(), N, c["gate_rows"]
        else:
            s["out"] = torch.empty(M, N, device="cuda", dtype=torch.float32 if c["epi"] == "f32" else torch.float16)
            e.out, e.ldo = s["out"].data_ptr(), N
        if c["epi"] == "rope":  # queries and keys are rotated, values are not
            e.rope_cos, e.rope_sin, e.rope_tokens = x["cos"].data_ptr(), x["sin"].data_ptr(), 1024
            e.d_head, e.rope_cols = c["d_head"], 2 * N // 3
        s["epi"] = e
    elif c["kind"] == "attention":
        s["out"] = torch.empty(c["batch"], c["n_q"], c["n_heads"], c["d_head"], device="cuda", dtype=torch.float16)
    elif c["kind"] == "norm":
        s["out"] = torch.empty(c["rows"], c["d"], device="cuda", dtype=torch.float16)
    return s


def run(s):
    c = s["case"]
    if c["kind"] == "model":
        return _run_model(s)
    x = s["x"]
    if c["kind"] == "gemm":
        binding.sgd_kernel_gemm(x["A"], x["B"], c["M"], c["N"], c["K"], s["epi"])
        if c["epi"] != "delta":
            return s["out"]
        return [x["h"], s["cache"]] if c["cache"] else x["h"]
    if c["kind"] == "attention":
        H, dh, hs = c["n_heads"], c["d_head"], x["q"].shape[-1]
        binding.sgd_kernel_attention_hs(x["q"], H * hs, x["k"], x["v"], H * hs, hs, s["out"], H * dh, c["batch"],
                                        c["n_q"], c["n_kv"], H, dh)
        return s["out"]
    if c["kind"] == "norm":
        binding.sgd_kernel_norm(x["h"], s["out"], c["rows"], c["d"], NORM[c["norm"]], g=x.get("g"), b=x.get("b"),
                                shift=x.get("shift"), scale=x.get("scale"), ld_mod=2 * c["d"],
                                rows_per_batch=c["mod_rows"] or 1, eps=EPS)
        return s["out"]
    binding.sgd_kernel_frozen_run(x["h"], x["caches"])
    return x["h"]


# ---------------------------------------------------------------------------
# work, tolerance
# ---------------------------------------------------------------------------

def _model_work(c):
    d, f, a, ch = _dims(c)
    B, n = c["batch"], c["n_tokens"]
    M, out = B * n, c["vocab"] or ch
    up = 2 * f if a["mlp"] in ("swiglu", "geglu") else f
    par = 4 * d * d + up * d + f * d            # weights of one block
    flops = 2.0 * M * par + 4.0 * M * n * d     # and its self-attention
    if a["block"] == "xattn":
        par += 3 * d * d
        flops += 6.0 * M * d * d - 2.0 * M * d * d + 4.0 * M * a["ctx_len"] * d
    if a["block"] == "adaln":
        par += 6 * d * d
        flops += 12.0 * B * d * d
    n_skips = (c["n_blocks"] - 1) // 2 if c["arch"] == "uvit" else 0
    head = 0 if a["head"] == "identity" else out * d
    total_b = total_f = 0.0
    for s in range(1, c["T"] + 1):
        active = sum(L >= s for L in _lifetimes(c))
        total_f += active * flops + 2.0 * M * head + n_skips * 4.0 * M * d * d
        # weights of the active blocks, the cached updates of the frozen ones, input and output
        total_b += 2.0 * (active * par + head + n_skips * 2 * d * d)
        total_b += 2.0 * M * d * len([1 for L in _lifetimes(c) if L < s])
        total_b += M * 4.0 if c["vocab"] else M * ch * 4.0
        total_b += (2.0 if c["vocab"] else 4.0) * M * out
    if a["block"] == "xattn":
        kv = c["n_blocks"] * 2 * d * a["d_ctx"]
        total_f += 2.0 * B * a["ctx_len"] * kv
        total_b += 2.0 * kv + 2.0 * B * a["ctx_len"] * a["d_ctx"]
    return dict(bytes=total_b, flops=total_f)


def work(c):
    if c["kind"] == "model":
        return _model_work(c)
    if c["kind"] == "gemm":
        M, N, K = c["M"], c["N"], c["K"]
        rows = 2 * N if c["epi"] == "gated" else N
        out = {"f32": 4.0, "delta": 10.0 if c["cache"] else 8.0}.get(c["epi"], 2.0)
        return dict(bytes=2.0 * M * K + 2.0 * rows * K + out * M * N, flops=2.0 * M * rows * K)
    if c["kind"] == "attention":
        d = c["n_heads"] * c["d_head"]
        return dict(bytes=4.0 * c["batch"] * (c["n_q"] + c["n_kv"]) * d, flops=4.0 * c["batch"] * c["n_q"] * c["n_kv"] * d)
    if c["kind"] == "norm":
        return dict(bytes=6.0 * c["rows"] * c["d"], flops=8.0 * c["rows"] * c["d"])
    return dict(bytes=c["rows"] * c["d"] * (8.0 + 2.0 * c["caches"]), flops=1.0 * c["rows"] * c["d"] * c["caches"])


def tolerance(c):
    """About four times the error against float64 that was measured.  Models 2e-4 to 6.5e-4 at every
    step (fp16 operands; the residual stream is fp32, so depth and the closed loop add little), fp16
    results 2.1e-4 to 3e-4.  An fp32 result or residual of a projection holds the tensor cores'
    accumulation error, which grows with K: 4.3e-6 at 5120 for a residual as large as its update.
    A frozen run 3.5e-8 with nine updates."""
    if c["kind"] == "model":
        return {"rel": 2.5e-3}
    if c["kind"] == "gemm":
        return {"rel": 4e-5} if c["epi"] in ("f32", "delta") and not c["cache"] else {"rel": 1e-3}
    if c["kind"] == "frozen":
        return {"rel": 5e-7}
    return {"rel": 1.2e-3 if c["kind"] == "attention" else 8e-4}


# ---------------------------------------------------------------------------
# the same in float64
# ---------------------------------------------------------------------------

def _gelu_tanh(x):
    return torch.nn.functional.gelu(x, approximate="tanh")


def _norm64(kind, x, g=None, b=None):
    if kind == "rms":
        y = x * torch.rsqrt((x * x).mean(-1, keepdim=True) + EPS)
    else:
        x = x - x.mean(-1, keepdim=True)
        y = x * torch.rsqrt((x * x).mean(-1, keepdim=True) + EPS)
    y = y if g is None else y * g.double()
    return y if b is None else y + b.double()


def _rotate64(x, dh):
    """Rotary embedding of x [..., n, dh] at positions 0 .. n - 1."""
    half = dh // 2
    freq = THETA ** (-torch.arange(half, device="cuda", dtype=torch.float64) / half)
    a = torch.arange(x.shape[-2], device="cuda", dtype=torch.float64)[:, None] * freq
    cos, sin, p, q = a.cos(), a.sin(), x[..., :half], x[..., half:]
    return torch.cat([p * cos - q * sin, q * cos + p * sin], -1)


def _attention64(q, k, v, n_heads, rope=False):
    """q [B, Nq, d], k and v [B, Nk, d]; one sample at a time."""
    B, nq, d = q.shape
    dh = d // n_heads
    out = torch.empty_like(q)
    for b in range(B):
        x, y, w = (t[b].view(-1, n_heads, dh).transpose(0, 1) for t in (q, k, v))
        if rope:
            x, y = _rotate64(x, dh), _rotate64(y, dh)
        p = torch.softmax(x @ y.transpose(1, 2) / math.sqrt(dh), -1)
        out[b] = (p @ w).transpose(0, 1).reshape(nq, d)
    return out


def _sinusoid64(t, dim):
    half = dim // 2
    a = t * torch.exp(-math.log(10000.0) * torch.arange(half, device="cuda", dtype=torch.float64) / half)
    return torch.cat([a.cos(), a.sin()])


class _Exact:
    def __init__(self, c, seed):
        g = _generator(seed)
        self.c, self.w, self.x = c, _weights(c, g), _model_inputs(c, g)
        self.d, self.f, self.a, _ = _dims(c)
        self.cache = {}

    def lin(self, x, name, rows=slice(None)):
        w = self.w[name][rows]
        if w.shape[0] > 32768:  # a vocabulary, in parts
            return torch.cat([x @ p.double().T for p in w.split(16384)], -1)
        return x @ w.double().T

    def norm(self, x, name):
        return _norm64(self.a["norm"], x, self.w.get(name + "_w"), self.w.get(name + "_b"))

    def stem(self, state, t):
        a, w = self.a, self.w
        if a["stem"] == "embed":
            return w["embed"][state.long()].double()
        z = state.double()
        if a["stem"] == "identity":
            return z
        if a["stem"] == "time_add":
            return z + _sinusoid64(t, self.d)
        h = self.lin(z, "w_stem")
        if a["stem"] == "patch_tokens":
            first = _sinusoid64(t, self.d).expand(z.shape[0], 1, -1)
            h = torch.cat([first, w["class_emb"][self.x["class_ids"].long()].double()[:, None], h], 1)
        return h + w["pos_emb"].double()

    def branch(self, b, kind, h, cond):
        p, a, d, H = "blocks.%d." % b, self.a, self.d, self.c["n_heads"]
        mod = None
        if cond is not None:
            k = 0 if kind == "attn" else 3
            mod = [m[:, None] for m in self.lin(cond, p + "w_mod").split(d, -1)[k:k + 3]]
        if kind == "xattn":
            q = self.lin(self.norm(h, p + "normx"), p + "wx_q")
            kv = self.lin(self.x["ctx"].double(), p + "wx_kv")
            return self.lin(_attention64(q, kv[..., :d], kv[..., d:], H), p + "wx_o")
        x = self.norm(h, p + ("norm1" if kind == "attn" else "norm2"))
        if mod is not None:
            x = x * (1 + mod[1]) + mod[0]
        if kind == "attn":
            q, k, v = self.lin(x, p + "w_qkv").split(d, -1)
            y = self.lin(_attention64(q, k, v, H, a.get("rope", False)), p + "w_o")
        else:
            u, f = self.lin(x, p + "w_1"), self.f
            if a["mlp"] == "swiglu":
                u = torch.nn.functional.silu(u[..., :f]) * u[..., f:]
            elif a["mlp"] == "geglu":
                u = u[..., :f] * torch.nn.functional.gelu(u[..., f:])
            else:
                u = _gelu_tanh(u) if a["mlp"] == "gelu_tanh" else torch.nn.functional.gelu(u)
            y = self.lin(u, p + "w_2")
        return y if mod is None else y * mod[2]

    def step(self, state, s, with_head):
        c, a, life, t = self.c, self.a, _lifetimes(self.c), _timestep(self.c, s)
        h, cond, skips = self.stem(state, t), None, []
        if a["block"] == "adaln":
            e = torch.nn.functional.silu(self.lin(_sinusoid64(t, a["t_freq"])[None], "w_t1"))
            e = self.lin(e, "w_t2") + self.w["class_emb"][self.x["class_ids"].long()].double()
            cond = torch.nn.functional.silu(e)
        n_skips = (c["n_blocks"] - 1) // 2 if c["arch"] == "uvit" else 0
        kinds = ("attn", "xattn", "mlp") if a["block"] == "xattn" else ("attn", "mlp")
        for b in range(c["n_blocks"]):
            if n_skips and b > n_skips:
                h = self.lin(torch.cat([h, skips.pop()], -1), "skips.%d.w" % (b - n_skips - 1))
            for kind in kinds:
                if s <= life[b]:
                    self.cache[b, kind] = self.branch(b, kind, h, cond)
                h = h + self.cache[b, kind]
            if n_skips and b < n_skips:
                skips.append(h)
        if not with_head or a["head"] == "identity":
            return h if with_head else None
        if a["head"] == "adaln_linear":
            shift, scale = (m[:, None] for m in self.lin(cond, "w_modf").split(self.d, -1))
            return self.lin(_norm64("ln", h) * (1 + scale) + shift, "w_head")[..., :a["channels"]]
        return self.lin(self.norm(h, "normf")[:, a.get("n_prefix", 0):], "w_head")

    def trajectory(self):
        c, outs = self.c, []
        if c["vocab"]:  # the logits of the last step stand for all: the head is most of the work
            return [self.step(self.x["ids"][s - 1], s, s == c["T"]) for s in range(1, c["T"] + 1)]
        z = self.x["z0"].double()
        for s in range(1, c["T"] + 1):
            outs.append(self.step(z, s, True))
            z = z if c["host"] else z - outs[-1] / c["T"]
        return outs if c["host"] else outs + [z]


def exact(c, seed):
    if c["kind"] == "model":
        if _model_work(c)["flops"] > 1.6e13:
            return None
        return _Exact(c, seed).trajectory()
    x = _layer_inputs(c, _generator(seed))
    if c["kind"] == "gemm":
        y = x["A"].double() @ x["B"].double().T
        N = c["N"]
        if c["epi"] == "gated":
            p, q = y[:, :N], y[:, N:]
            return p * torch.nn.functional.gelu(q) if c["act"] else torch.nn.functional.silu(p) * q
        if c["epi"] == "gelu":
            return torch.nn.functional.gelu(y) if c["act"] else _gelu_tanh(y)
        if c["epi"] == "rope":
            dh, half = c["d_head"], c["d_head"] // 2
            row = torch.arange(c["M"], device="cuda") % 1024
            cos, sin = x["cos"][row].double()[:, None], x["sin"][row].double()[:, None]
            r = y[:, :2 * N // 3].reshape(c["M"], -1, dh)
            p, q = r[..., :half], r[..., half:]
            r = torch.cat([p * cos - q * sin, q * cos + p * sin], -1).reshape(c["M"], -1)
            return torch.cat([r, y[:, 2 * N // 3:]], 1)
        if c["epi"] == "delta":
            if c["gate_rows"]:
                y = y * x["gate"].double()[torch.arange(c["M"], device="cuda") // c["gate_rows"]]
            h = x["h"].double() + y
            return [h, y] if c["cache"] else h
        return y
    if c["kind"] == "attention":
        B, H, dh = c["batch"], c["n_heads"], c["d_head"]
        q, k, v = (x[n][..., :dh].double().reshape(B, -1, H * dh) for n in ("q", "k", "v"))
        return _attention64(q, k, v, H).view(B, -1, H, dh)
    if c["kind"] == "norm":
        y = _norm64(c["norm"], x["h"].double(), x.get("g"), x.get("b"))
        if c["mod_rows"]:
            m = x["mod"].double()[torch.arange(c["rows"], device="cuda") // c["mod_rows"]]
            y = y * (1 + m[:, c["d"]:]) + m[:, :c["d"]]
        return y
    h = x["h"].double()
    for t in x["caches"]:
        h = h + t.double()
    return h
