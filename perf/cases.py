"""The work that a diffusion-GRPO trainer gives this library, as measurable cases.

A trainer's loop over one group of G samples is: sample T steps (a forward that keeps
nothing, then one sampler step), score the window's transitions (step signals with the
aggregation), run the endpoint rows forward with their activations kept and take the joint
VJP with the two cotangents (Algorithm 1), and accumulate / compare gradients.  Four kinds
of case stand for it, each through the entry points of include/jagg.h:

  train    dit_forward_save (activations kept) and dit_joint_vjp over `rows` endpoint rows
           with given cotangents: velocities and the whole flat gradient.  A model of one
           block is a layer case: the block between its embeddings and final layer.
  sample   dit_forward_save without an arena and jagg_rollout_step: one step of the rollout.
  signals  grpo_step_signals with the fused aggregation over one window.
  reduce   grad_reduce: acc += alpha a and <a,b>, |a|^2, |b|^2.

The cotangents of a train case are given and not computed by a signals call before it: the
likelihood ratio exp(logp - logp_old) of Eq. grpo_loss amplifies the rounding of a 16-bit
velocity by orders of magnitude, so a chained pass has no value to compare.
"""
import math

import torch
import torch.nn.functional as F

import paper_2607_17572_gb300 as jagg

DEV = "cuda"

# Widths, depths, token counts and group sizes of the repository's workloads.
_DIT_B = dict(arch="dit", dtype="bf16", hidden=768, heads=12, depth=12, double=0, channels=16, patch=2, txt_dim=768)
_FLUX = dict(arch="mmdit", dtype="bf16", hidden=3072, heads=24, channels=16, patch=2, txt_dim=4096)
_QWEN = dict(_FLUX, txt_dim=3072)
_TINY = dict(arch="dit", dtype="f32", hidden=64, heads=4, depth=2, double=0, channels=4, patch=1, txt_dim=64)


def listed():
    return [
        # the smallest configuration (f32, 24 tokens): bound by launches and by latency
        dict(name="tiny_f32_train", op="train", rows=8, h=4, w=4, txt=8, **_TINY),
        # DiT-B, the paper's group of 8: one rollout step
        dict(name="dit_b_sample", op="sample", rows=8, h=32, w=32, txt=77, **_DIT_B),
        # DiT-B: the joint VJP of one window (2 G = 16 endpoint rows)
        dict(name="dit_b_train", op="train", rows=16, h=32, w=32, txt=77, **_DIT_B),
        # a non-square latent, an odd group, few rows: ragged tiles everywhere
        dict(name="dit_b_odd_train", op="train", rows=5, h=30, w=26, txt=50, **_DIT_B),
        # one dual-stream block at Flux width and 512^2
        dict(name="flux512_double_train", op="train", rows=4, h=64, w=64, txt=512, depth=0, double=1, **_FLUX),
        # one dual-stream block at Qwen-Image width; its prompts have any length, so the text
        # stream ends inside a 128-token tile, and the latent is not square
        dict(name="qwen_odd_double_train", op="train", rows=3, h=60, w=52, txt=211, depth=0, double=1, **_QWEN),
        # one Flux-style single block at 1024^2: long sequences, attention-heavy
        dict(name="flux1024_single_train", op="train", rows=2, h=128, w=128, txt=512, depth=1, double=0, **_FLUX),
        # the whole Flux-width model at 1024^2: one rollout step of a group of 4
        dict(name="flux1024_sample", op="sample", rows=4, h=128, w=128, txt=512, depth=8, double=4, **_FLUX),
        # the largest: one JAGG window of that group (8 endpoint rows), forward and joint VJP
        dict(name="flux1024_train", op="train", rows=8, h=128, w=128, txt=512, depth=8, double=4, **_FLUX),
        # step signals at DiT-B's latents (a group of 8) and at 1024^2 latents
        dict(name="dit_b_signals", op="signals", group=8, window=4, dim=16 * 32 * 32, dtype="bf16"),
        dict(name="flux1024_signals", op="signals", group=4, window=4, dim=16 * 128 * 128, dtype="bf16"),
        # accumulating a window's gradient of DiT-B and its cosine against another gradient
        dict(name="dit_b_reduce", op="reduce", params=_param_count(dict(_DIT_B, h=32, w=32, txt=77))),
    ]


_LARGEST_FLOPS = 100e12  # a drawn model case stays well below the largest listed one


def _log_int(rng, lo, hi):
    return min(hi, int(math.exp(rng.uniform(math.log(lo), math.log(hi + 1)))))


def draw(rng):
    kind = rng.choice(["train", "train", "train", "sample", "sample", "signals", "signals", "reduce"])
    if kind == "signals":
        # any latent (16 channels, even sides), any group and window of the paper's ranges
        return dict(op="signals", group=rng.randint(2, 16), window=rng.randint(2, 8),
                    dim=16 * 4 * _log_int(rng, 4, 64) * _log_int(rng, 4, 64), dtype=rng.choice(["bf16", "bf16", "f32"]))
    if kind == "reduce":
        return dict(op="reduce", params=_log_int(rng, 10_000, 400_000_000))
    while True:
        family = rng.choice(["dit", "dit", "mmdit", "mmdit", "f32"])
        if family == "dit":
            d = rng.choice([512, 768, 1024])
            c = dict(arch="dit", dtype="bf16", hidden=d, heads=d // 64, depth=_log_int(rng, 1, 12), double=0,
                     channels=16, patch=2, txt_dim=768, rows=_log_int(rng, 1, 64), h=2 * rng.randint(6, 24),
                     w=2 * rng.randint(6, 24), txt=_log_int(rng, 8, 160))
        elif family == "mmdit":
            d = rng.choice([1024, 2048, 3072])
            c = dict(arch="mmdit", dtype="bf16", hidden=d, heads=d // 128, depth=rng.randint(0, 2),
                     double=rng.randint(0, 2), channels=16, patch=2, txt_dim=rng.choice([3072, 4096]),
                     rows=_log_int(rng, 1, 8), h=2 * _log_int(rng, 12, 64), w=2 * _log_int(rng, 12, 64),
                     txt=rng.choice([128, 256, 512, rng.randint(20, 512)]))
        else:
            arch = rng.choice(["dit", "mmdit"])
            d = rng.choice([64, 128, 256])
            c = dict(arch=arch, dtype="f32", hidden=d, heads=d // rng.choice([16, 32, 64]), depth=rng.randint(1, 2),
                     double=rng.randint(0, 2) if arch == "mmdit" else 0, channels=4, patch=1, txt_dim=64,
                     rows=_log_int(rng, 1, 16), h=rng.randint(3, 12), w=rng.randint(3, 12), txt=rng.randint(3, 40))
        c = dict(op=kind, **c)
        if c["depth"] + c["double"] > 0 and work(c)["flops"] <= _LARGEST_FLOPS:
            return c


# ------------------------------------------------------------------ sizes
def _layout(c):
    """(name, offset, rows, cols) of every parameter tensor and the flat length, as
    jagg_param_info describes them: tensors in this order, each on a multiple of 64 elements."""
    d, dm, pd = c["hidden"], 4 * c["hidden"], c["channels"] * c["patch"] ** 2
    dh = d // c["heads"]
    t = [("x_embed.w", d, pd), ("x_embed.b", d, 1), ("txt_embed.w", d, c["txt_dim"]), ("txt_embed.b", d, 1),
         ("t_embed.w1", d, 256), ("t_embed.b1", d, 1), ("t_embed.w2", d, d), ("t_embed.b2", d, 1)]
    if c["arch"] == "dit":
        mods = [("blocks.%d.mod" % i, 6 * d) for i in range(c["depth"])]
    else:
        mods = [("double.%d.%s.mod" % (i, s), 6 * d) for i in range(c["double"]) for s in ("txt", "img")]
        mods += [("single.%d.mod" % i, 3 * d) for i in range(c["depth"])]
    mods.append(("final.mod", 2 * d))
    t += [(n + ".w", r, d) for n, r in mods] + [(n + ".b", r, 1) for n, r in mods]

    def mlp(p):
        return [(p + "proj.w", d, d), (p + "proj.b", d, 1), (p + "fc1.w", dm, d), (p + "fc1.b", dm, 1),
                (p + "fc2.w", d, dm), (p + "fc2.b", d, 1)]

    def qkv(p):
        return [(p + "qkv.w", 3 * d, d), (p + "qkv.b", 3 * d, 1)]

    if c["arch"] == "dit":
        for i in range(c["depth"]):
            t += qkv("blocks.%d." % i) + mlp("blocks.%d." % i)
    else:
        for i in range(c["double"]):
            for s in ("txt", "img"):
                p = "double.%d.%s." % (i, s)
                t += qkv(p) + [(p + "q_norm", dh, 1), (p + "k_norm", dh, 1)] + mlp(p)
        for i in range(c["depth"]):
            p = "single.%d." % i
            t += [(p + "lin1.w", 3 * d + dm, d), (p + "lin1.b", 3 * d + dm, 1), (p + "q_norm", dh, 1),
                  (p + "k_norm", dh, 1), (p + "lin2.w", d, d + dm), (p + "lin2.b", d, 1)]
    t += [("final.out.w", pd, d), ("final.out.b", pd, 1)]
    out, off = [], 0
    for n, r, k in t:
        off = (off + 63) // 64 * 64
        out.append((n, off, r, k))
        off += r * k
    return out, (off + 63) // 64 * 64


def _param_count(c):
    return _layout(c)[1]


def _tokens(c):
    return (c["h"] // c["patch"]) * (c["w"] // c["patch"]), c["txt"]


def _latent(c):
    return (c["channels"], c["h"], c["w"])


def work(c):
    if c["op"] == "signals":
        G, W, D = c["group"], c["window"], c["dim"]
        return {"bytes": D * (G * W * (2 if c["dtype"] == "bf16" else 4) + 4 * G * (W + 1) + 8 * G), "flops": 0}
    if c["op"] == "reduce":
        return {"bytes": 16 * c["params"], "flops": 0}
    d, dm, B = c["hidden"], 4 * c["hidden"], c["rows"]
    ni, nt = _tokens(c)
    n, pd, D = ni + nt, c["channels"] * c["patch"] ** 2, math.prod(_latent(c))
    lmod = (6 * c["depth"] if c["arch"] == "dit" else 12 * c["double"] + 3 * c["depth"]) * d + 2 * d
    blocks = c["depth"] + c["double"]
    embed = 2 * (ni * pd * d + nt * c["txt_dim"] * d + 256 * d)
    rest = 2 * (d * d + lmod * d) + blocks * (2 * n * (4 * d * d + 2 * d * dm) + 4 * n * n * d) + 2 * ni * d * pd
    e = 2 if c["dtype"] == "bf16" else 4
    P = _param_count(c)
    move = P * e + B * (D * e * 2 + nt * c["txt_dim"] * e)
    if c["op"] == "sample":
        return {"bytes": move + B * D * (4 + 4 + 4 + e), "flops": B * (embed + rest)}
    # the gradient: weights read once more, gradient written in f32, cotangents read
    return {"bytes": move + P * e + P * 4 + B * D * 4, "flops": B * (2 * embed + 3 * rest)}


# ------------------------------------------------------------------ inputs
def _gen(seed):
    return torch.Generator(device=DEV).manual_seed(seed)


def _weights(c, seed):
    """Xavier-uniform matrices, small biases, RMSNorm scales near 1, in the storage type."""
    g = _gen(seed)
    tensors, total = _layout(c)
    flat = torch.zeros(total, dtype=torch.bfloat16 if c["dtype"] == "bf16" else torch.float32, device=DEV)
    for name, off, r, k in tensors:
        v = flat[off:off + r * k]
        if k > 1:
            b = math.sqrt(6.0 / (r + k))
            v.uniform_(-b, b, generator=g)
        elif name.endswith("_norm"):
            v.uniform_(0.9, 1.1, generator=g)
        else:
            v.uniform_(-0.02, 0.02, generator=g)
    return flat


def _times(seed, rows):
    """Network-input times of the rows: points of a shifted 16-step grid."""
    k = torch.randint(0, 15, (rows,), generator=_gen(seed + 1), device=DEV).double() / 16
    t = 1.0 - k
    return (3.0 * t / (1.0 + 2.0 * t)).float()


def _model_inputs(c, seed):
    dt = torch.bfloat16 if c["dtype"] == "bf16" else torch.float32
    g = _gen(seed + 2)
    z = torch.randn(c["rows"], *_latent(c), generator=g, device=DEV).to(dt)
    prompt = torch.randn(c["txt"], c["txt_dim"], generator=g, device=DEV).to(dt)
    txt = prompt.expand(c["rows"], -1, -1).contiguous()  # one prompt for the group
    return z, _times(seed, c["rows"]), txt


def _cotangents(c, seed):
    return torch.randn(c["rows"], *_latent(c), generator=_gen(seed + 3), device=DEV) * 0.01


def _sampler(c, seed):
    """The f32 state the forward's input was rounded from, the step's noise, its times."""
    g = _gen(seed + 4)
    z0 = _model_inputs(c, seed)[0].float()
    xi = torch.randn(z0.shape, generator=g, device=DEV)
    return z0, xi, (0.9, 0.85, 0.7 * math.sqrt(0.05))


def _window(c, seed):
    """A window of trajectories drawn by the sampler from given velocities, with rollout
    log-probs that put half of the ratios inside the clip range and half well outside."""
    G, W, D = c["group"], c["window"], c["dim"]
    g = _gen(seed)
    dt = torch.bfloat16 if c["dtype"] == "bf16" else torch.float32
    v = torch.randn(G, W, D, generator=g, device=DEV).to(dt)
    k = torch.arange(W + 1, device=DEV, dtype=torch.float64) / 16
    t = 3.0 * (1 - k) / (1.0 + 2.0 * (1 - k))
    sigma = 0.7 * (t[1:] - t[:-1]).abs().sqrt()
    z = torch.empty(G, W + 1, D, device=DEV)
    z[:, 0] = torch.randn(D, generator=g, device=DEV)  # shared initial noise
    logp = torch.empty(G, W, dtype=torch.float64, device=DEV)
    for j in range(W):
        mu = z[:, j].double() + v[:, j].double() * (t[j + 1] - t[j])
        z[:, j + 1] = (mu + sigma[j] * torch.randn(G, D, generator=g, device=DEV)).float()
        r = z[:, j + 1].double() - mu
        logp[:, j] = -(r * r).sum(1) / (2 * sigma[j] ** 2) - D * torch.log(math.sqrt(2 * math.pi) * sigma[j])
    eps = 0.1
    u = torch.rand(G, W, 3, generator=g, device=DEV, dtype=torch.float64)
    delta = torch.where(u[..., 0] < 0.5, 0.3 * eps * (2 * u[..., 1] - 1),
                        (2 + u[..., 1]) * eps * torch.where(u[..., 2] < 0.5, -1.0, 1.0))
    rewards = torch.randn(G, generator=g, device=DEV)
    return v, z, t, sigma, logp + delta, rewards


def _reduce_inputs(c, seed):
    g = _gen(seed)
    return [1e-3 * torch.randn(c["params"], generator=g, device=DEV) for _ in range(3)]


def prepare(c, seed):
    if c["op"] == "signals":
        G, W, D = c["group"], c["window"], c["dim"]
        v, z, t, sigma, logp_old, rewards = _window(c, seed)
        f64 = dict(dtype=torch.float64, device=DEV)
        out = dict(logp_new=torch.empty(G, W, **f64), ratio=torch.empty(G, W, **f64),
                   clipped=torch.empty(G, W, dtype=torch.uint8, device=DEV), adv_out=torch.empty(G, **f64),
                   cot_out=torch.empty(2 * G, D, device=DEV))
        return dict(c=c, args=(v, z, t, sigma, logp_old, rewards, 0.1, 5.0, 1e-8, 1.0 / (16 * G)), out=out,
                    ws=jagg.alloc_bytes(jagg.signals_workspace_bytes(G, W, D)))
    if c["op"] == "reduce":
        a, b, acc = _reduce_inputs(c, seed)
        return dict(c=c, a=a, b=b, acc=acc, out3=torch.empty(3, dtype=torch.float64, device=DEV),
                    ws=jagg.alloc_bytes(jagg.grad_reduce_workspace_bytes(a.numel())))
    cfg = jagg.Config(arch=jagg.ARCH_DIT if c["arch"] == "dit" else jagg.ARCH_MMDIT,
                      dtype=jagg.DTYPE_BF16 if c["dtype"] == "bf16" else jagg.DTYPE_F32, hidden=c["hidden"],
                      heads=c["heads"], mlp=4 * c["hidden"], depth=c["depth"], depth_double=c["double"],
                      in_channels=c["channels"], latent_h=c["h"], latent_w=c["w"], patch=c["patch"],
                      txt_len=c["txt"], txt_dim=c["txt_dim"], freq_dim=256)
    weights = _weights(c, seed)
    assert jagg.param_count(cfg) == weights.numel()
    model = jagg.Model(cfg, weights)
    z, t, txt = _model_inputs(c, seed)
    s = dict(c=c, model=model, z=z, t=t, txt=txt, v=torch.empty_like(z),
             ws=jagg.alloc_bytes(model.workspace_bytes(c["rows"])))
    if c["op"] == "train":
        s.update(saved=jagg.alloc_bytes(model.saved_bytes(c["rows"])), cot=_cotangents(c, seed),
                 grad=torch.empty(weights.numel(), device=DEV))
    else:
        z0, xi, times = _sampler(c, seed)
        G = c["rows"]
        traj = torch.zeros(G, 2, *_latent(c), device=DEV)
        traj[:, 0] = z0
        s.update(traj=traj, xi=xi, times=times, z_model=torch.empty_like(z),
                 logp=torch.empty(G, 1, dtype=torch.float64, device=DEV),
                 step_ws=jagg.alloc_bytes(jagg.rollout_workspace_bytes(G, z0[0].numel())))
    return s


def run(s):
    op = s["c"]["op"]
    if op == "signals":
        jagg.grpo_step_signals(*s["args"], ws=s["ws"], **s["out"])
        return s["out"]
    if op == "reduce":
        jagg.grad_reduce(s["a"], s["b"], alpha=0.5, acc=s["acc"], out3=s["out3"], ws=s["ws"])
        return {"acc": s["acc"], "out3": s["out3"]}
    if op == "sample":
        jagg.dit_forward_save(s["model"], s["z"], s["t"], s["txt"], s["v"], ws=s["ws"])
        t0, t1, sigma = s["times"]
        jagg.jagg_rollout_step(s["v"], s["traj"], 0, s["xi"], t0, t1, sigma, s["logp"], s["step_ws"],
                               z_model=s["z_model"])
        return {"v": s["v"], "z": s["traj"], "logp": s["logp"], "z_model": s["z_model"]}
    jagg.dit_forward_save(s["model"], s["z"], s["t"], s["txt"], s["v"], saved=s["saved"], ws=s["ws"])
    s["grad"].zero_()
    jagg.dit_joint_vjp(s["model"], s["saved"], s["c"]["rows"], s["cot"], s["grad"], s["ws"])
    return {"v": s["v"], "grad": s["grad"]}


def tolerance(c):
    """About four times the error measured against `exact` (or between two passes, whose f32
    sums meet in another order): signals 4.6e-5 (the ratio exponentiates f32 residuals' sum),
    reduce 2.7e-8, f32 models 4.4e-7 to 1e-6, bf16 models 2.0e-3 to 2.8e-3 with single entries
    off by 0.13 of the root mean square between two passes of the largest case."""
    if c["op"] == "signals":
        return {"rel": 2e-4, "max": 1e-3, "differ": 0.0}
    if c["op"] == "reduce":
        return {"rel": 2e-7, "max": 2e-6}
    if c["dtype"] == "f32":
        return {"rel": 4e-6, "max": 2e-4}
    return {"rel": 1e-2, "max": 0.5}


# ------------------------------------------------------------------ the same values in 64 bits
def _backbone(c, P, z, t, txt):
    """The velocity network in plain torch: patch and text embeddings, adaLN blocks with
    joint [txt; img] attention, the modulated final layer."""
    d, heads, p, B = c["hidden"], c["heads"], c["patch"], z.shape[0]
    gh, gw, dh, nt, ck = c["h"] // p, c["w"] // p, c["hidden"] // c["heads"], c["txt"], dict(dtype=z.dtype, device=DEV)
    rows, cols = torch.arange(gh, **ck).repeat_interleave(gw), torch.arange(gw, **ck).repeat(gh)

    def lin(x, n):
        return F.linear(x, P[n + ".w"], P[n + ".b"])

    xi = lin(z.reshape(B, -1, gh, p, gw, p).permute(0, 2, 4, 1, 3, 5).reshape(B, gh * gw, -1), "x_embed")
    xt = lin(txt, "txt_embed")
    if c["arch"] == "dit":
        w = 10000.0 ** (-torch.arange(d // 4, **ck) / (d // 4))
        ar, ac = rows[:, None] * w, cols[:, None] * w
        xi = xi + torch.cat([ar.sin(), ar.cos(), ac.sin(), ac.cos()], 1)
    arg = 1000.0 * t.to(z.dtype)[:, None] * 10000.0 ** (-torch.arange(128, **ck) / 128)
    emb = F.silu(F.linear(torch.cat([arg.cos(), arg.sin()], 1), P["t_embed.w1"], P["t_embed.b1"]))
    cond = F.silu(F.linear(emb, P["t_embed.w2"], P["t_embed.b2"]))
    zero = torch.zeros(nt, **ck)
    th = 10000.0 ** (-4.0 * torch.arange(dh // 4, **ck) / dh)
    ang = torch.cat([torch.cat([zero, rows])[:, None] * th, torch.cat([zero, cols])[:, None] * th], 1)[:, None]

    def rope(x):
        a, b = x[..., 0::2], x[..., 1::2]
        return torch.stack([a * ang.cos() - b * ang.sin(), a * ang.sin() + b * ang.cos()], -1).flatten(-2)

    def rms(x, scale):
        return x / (x.square().mean(-1, keepdim=True) + 1e-6).sqrt() * scale

    def norm(x, shift, scale):
        return F.layer_norm(x, (d,), eps=1e-6) * (1 + scale[:, None]) + shift[:, None]

    def attend(q, k, v):
        return torch.cat([F.scaled_dot_product_attention(*(x[b:b + 1].transpose(1, 2) for x in (q, k, v)))
                          .transpose(1, 2).reshape(1, -1, d) for b in range(B)])

    def heads_of(x):
        return [y.reshape(B, -1, heads, dh) for y in x.split(d, -1)]

    def mlp(x, m, pre):
        return x + m[5][:, None] * lin(F.gelu(lin(norm(x, m[3], m[4]), pre + "fc1"), approximate="tanh"), pre + "fc2")

    if c["arch"] == "dit":
        x = torch.cat([xt, xi], 1)
        for i in range(c["depth"]):
            pre = "blocks.%d." % i
            m = lin(cond, pre + "mod").chunk(6, 1)
            x = x + m[2][:, None] * lin(attend(*heads_of(lin(norm(x, m[0], m[1]), pre + "qkv"))), pre + "proj")
            x = mlp(x, m, pre)
    else:
        for i in range(c["double"]):
            pre = ["double.%d.%s." % (i, s) for s in ("txt", "img")]
            m = [lin(cond, q + "mod").chunk(6, 1) for q in pre]
            s = [heads_of(lin(norm(x, a[0], a[1]), q + "qkv")) for x, a, q in zip((xt, xi), m, pre)]
            q, k = (rope(torch.cat([rms(s[u][e], P[pre[u] + n]) for u in (0, 1)], 1))
                    for e, n in ((0, "q_norm"), (1, "k_norm")))
            o = attend(q, k, torch.cat([s[0][2], s[1][2]], 1)).split([nt, gh * gw], 1)
            xt, xi = (mlp(x + a[2][:, None] * lin(y, r + "proj"), a, r) for x, a, y, r in zip((xt, xi), m, o, pre))
        x = torch.cat([xt, xi], 1)
        for i in range(c["depth"]):
            pre = "single.%d." % i
            m = lin(cond, pre + "mod").chunk(3, 1)
            y = lin(norm(x, m[0], m[1]), pre + "lin1")
            q, k, v = heads_of(y[..., :3 * d])
            o = attend(rope(rms(q, P[pre + "q_norm"])), rope(rms(k, P[pre + "k_norm"])), v)
            x = x + m[2][:, None] * lin(torch.cat([o, F.gelu(y[..., 3 * d:], approximate="tanh")], -1), pre + "lin2")
    m = lin(cond, "final.mod").chunk(2, 1)
    y = lin(norm(x[:, nt:], m[0], m[1]), "final.out")
    return y.reshape(B, gh, gw, -1, p, p).permute(0, 3, 1, 4, 2, 5).reshape(B, *_latent(c))


_EXACT_FLOPS = 9e12  # what plain 64-bit products do in the time allowed for it


def exact(c, seed):
    if c["op"] == "signals":
        v, z, t, sigma, logp_old, rewards = _window(c, seed)
        G, W, D = c["group"], c["window"], c["dim"]
        z, v = z.double(), v.double()
        dt = (t[1:] - t[:-1])[None, :]
        r = z[:, 1:] - z[:, :-1] - v * dt[..., None]
        logp = -r.square().sum(2) / (2 * sigma ** 2) - D * torch.log(math.sqrt(2 * math.pi) * sigma)
        ratio = torch.exp(logp - logp_old)
        rw = rewards.double()
        adv = ((rw - rw.mean()) / (rw.std() + 1e-8)).clamp(-5, 5)[:, None]
        clipped = ((adv > 0) & (ratio > 1.1)) | ((adv < 0) & (ratio < 0.9))
        coef = torch.where(clipped, 0.0, -adv * ratio * dt / sigma ** 2 / (16 * G))
        s = coef[..., None] * r
        al = ((t[0] - t[:W]) / (t[0] - t[W - 1]))[None, :, None]
        return dict(logp_new=logp, ratio=ratio, clipped=clipped.to(torch.uint8), adv_out=adv[:, 0],
                    cot_out=torch.cat([((1 - al) * s).sum(1), (al * s).sum(1)]))
    if c["op"] == "reduce":
        a, b, acc = (x.double() for x in _reduce_inputs(c, seed))
        return {"acc": acc + 0.5 * a, "out3": torch.stack([a @ b, a @ a, b @ b])}
    if work(c)["flops"] > _EXACT_FLOPS:
        return None
    flat = _weights(c, seed).double().requires_grad_(c["op"] == "train")
    P = {n: flat[o:o + r * k].view(r, k) if k > 1 else flat[o:o + r] for n, o, r, k in _layout(c)[0]}
    z, t, txt = _model_inputs(c, seed)
    with torch.set_grad_enabled(c["op"] == "train"):
        v = _backbone(c, P, z.double(), t, txt.double())
    if c["op"] == "train":
        # the rows' cotangents enter the network in its storage type
        cot = _cotangents(c, seed).to(z.dtype).double()
        return {"v": v.detach(), "grad": torch.autograd.grad(v, flat, cot)[0]}
    z0, xi, (t0, t1, sigma) = _sampler(c, seed)
    z0, xi = z0.double(), xi.double()
    z1 = z0 + v * (t1 - t0) + sigma * xi
    logp = -xi.flatten(1).square().sum(1) / 2 - z0[0].numel() * math.log(math.sqrt(2 * math.pi) * sigma)
    return {"v": v, "z": torch.stack([z0, z1], 1), "logp": logp[:, None], "z_model": z1}
