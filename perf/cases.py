"""Timed cases of the optimizer step: what a training program has this library do, once per step.

A case is one parameter set of a decoder-only language model together with the options a run would set.  One pass is one
`adapm_step` over every block of that set, in the middle of a training run.  The sets are the ones `workloads` lists (3 M
to 1.5 B parameters, and layers of the 8 B shapes); drawn cases are models of other depths, widths, vocabularies and
feed-forward sizes between them, with the same options.
"""
import math

import torch

import paper_2510_09103_b200 as A
import workloads as WL

INNER_PASSES = 4                   # Algorithm 2 with K = 5: the last step size of the cosine schedule is zero
MAX_PARAMS = {"bf16": 1.6e9, "f32": 1.3e8}     # of a drawn case


def _case(**kw):
    """style, layers, d, heads, kv_heads (0: as many as heads), ffn, vocab, ctx: the model.  grad: dtype of the
    gradients; recipe: their distribution (see workloads.gen).  v: second moment per element, or one scalar per row or
    head.  rank: 0, or the rank of every low-rank block; else rank_pct percent of the full rank.  clip: threshold of the
    global gradient-norm clipping, 0 = off.  period: steps between two refits of the left factor (0: every step).
    shadow: the step also writes the bf16 weights of the next forward pass.  finite: NaN / Inf check of the gradients."""
    case = dict(style="gpt2", layers=12, d=768, heads=12, kv_heads=0, ffn=3072, vocab=50257, ctx=1024, grad="bf16",
                recipe="normal", beta2=0.95, v="blockmean", rank=0, rank_pct=5, clip=0.0, period=0, shadow=False,
                finite=False)
    case.update(kw)
    return case


def _tiny(**kw):
    return _case(layers=2, d=256, heads=4, ffn=1024, vocab=4096, ctx=2048, **kw)


def _llama350m(**kw):
    return _case(style="llama", layers=24, d=1024, heads=16, ffn=2736, vocab=32000, recipe="heavyrows", **kw)


def _gpt2_1p5b(**kw):
    return _case(layers=48, d=1600, heads=25, ffn=6400, **kw)


def listed():
    return [
        # the smallest set: a two-layer model in plain fp32, as one runs to debug a training loop; launches count
        _tiny(name="tiny f32", grad="f32", v="element", beta2=0.999),
        # the same model under mixed precision
        _tiny(name="tiny bf16"),
        # pre-training of a 60M model, gradients of very different row scales
        _case(name="llama60m", style="llama", layers=8, d=512, heads=8, ffn=1376, vocab=32000, recipe="rowscale"),
        # GPT-2 124M, heavy-tailed gradients, clipped to norm 1 as the paper's runs are
        _case(name="gpt2_124m", recipe="student_t3", clip=1.0),
        # the same model trained in fp32
        _case(name="gpt2_124m f32", recipe="student_t3", grad="f32"),
        # a feed-forward width of 8/3 d, not rounded to anything: the down projection's rows are not 16-byte aligned
        _case(name="llama ffn 2730", style="llama", layers=8, d=1024, heads=16, ffn=2730, vocab=32000),
        # the ends of the rank sweep on the 350M set; the second one with the plain per-element second moment
        _llama350m(name="llama350m r8", rank=8),
        _llama350m(name="llama350m r128", rank=128, v="element", clip=1.0),
        # the 1.5B set with block-wise second moments: the most compressed optimizer state
        _gpt2_1p5b(name="gpt2_1p5b"),
        # the same set with a per-element second moment, in a mixed-precision loop that clips and wants bf16 weights back
        _gpt2_1p5b(name="gpt2_1p5b element", v="element", clip=1.0, shadow=True),
        # and with the update period of 100 the paper sets: 99 of 100 steps hold the left factor
        _gpt2_1p5b(name="gpt2_1p5b period 100", period=100, clip=1.0),
        # fine-tuning of the 8B shapes (eight of its layers): rank 204, grouped-query attention, all the guards on
        _case(name="llama3_8b 8 layers", style="llama", layers=8, d=4096, heads=32, kv_heads=8, ffn=14336, vocab=128256,
              clip=1.0, shadow=True, finite=True),
    ]


def draw(rng):
    def log(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    grad = "f32" if rng.random() < 0.2 else "bf16"
    style = rng.choice(["gpt2", "llama"])
    while True:
        head_dim = rng.choice([32, 48, 64, 64, 80, 96, 100, 128])
        heads = max(2, log(256, 2048) // head_dim)
        d = heads * head_dim
        ffn = 4 * d if style == "gpt2" else log(2 * d, 4 * d)
        if style == "llama" and rng.random() < 0.6:
            ffn = (ffn + 15) // 16 * 16
        layers, vocab, ctx = log(2, 48), log(2000, 130000), log(512, 4096)
        mlp = 2 if style == "gpt2" else 3
        embed = vocab * d * (1 if style == "gpt2" else 2)
        if 2e6 <= layers * (4 * d * d + mlp * d * ffn) + embed <= MAX_PARAMS[grad]:
            break
    rank = rng.choice([8, 32, 128]) if rng.random() < 0.3 else 0
    return _case(style=style, layers=layers, d=d, heads=heads, ffn=ffn, vocab=vocab, ctx=ctx, grad=grad,
                 recipe=rng.choice(["normal", "rowscale", "student_t3", "heavyrows"]),
                 v=rng.choice(["blockmean", "blockmean", "element"]), rank=rank, rank_pct=rng.choice([2, 5, 5, 10]),
                 clip=rng.choice([0.0, 1.0]), period=rng.choice([0, 0, 0, 100]),
                 shadow=grad == "bf16" and rng.random() < 0.4)


def _tensors(case):
    d, ffn, vocab, heads = case["d"], case["ffn"], case["vocab"], case["heads"]

    def vec(n, init="ones"):
        return WL.Tensor("vector", WL.ROLE_VECTOR, 1, n, init=init)

    if case["style"] == "gpt2":
        out = [WL.Tensor("wte", WL.ROLE_EMBED, vocab, d), WL.Tensor("wpe", WL.ROLE_EMBED, case["ctx"], d)]
        for _ in range(case["layers"]):
            out += [vec(d), vec(d, "zeros"), WL.Tensor("qkv", WL.ROLE_QKV_FUSED, 3 * d, d, heads=heads), vec(3 * d, "zeros"),
                    WL.Tensor("attn_out", WL.ROLE_ATTN_OUT, d, d), vec(d, "zeros"), vec(d), vec(d, "zeros"),
                    WL.Tensor("fc", WL.ROLE_MLP, ffn, d), vec(ffn, "zeros"), WL.Tensor("proj", WL.ROLE_MLP, d, ffn),
                    vec(d, "zeros")]
        return out + [vec(d), vec(d, "zeros")]
    kv_heads = case["kv_heads"] or heads
    kv = kv_heads * (d // heads)
    out = [WL.Tensor("embed", WL.ROLE_EMBED, vocab, d)]
    for _ in range(case["layers"]):
        out += [vec(d), WL.Tensor("q", WL.ROLE_Q, d, d, heads=heads), WL.Tensor("k", WL.ROLE_K, kv, d, heads=kv_heads),
                WL.Tensor("v", WL.ROLE_V, kv, d), WL.Tensor("attn_out", WL.ROLE_ATTN_OUT, d, d), vec(d),
                WL.Tensor("gate", WL.ROLE_MLP, ffn, d), WL.Tensor("up", WL.ROLE_MLP, ffn, d),
                WL.Tensor("down", WL.ROLE_MLP, d, ffn)]
    return out + [vec(d), WL.Tensor("head", WL.ROLE_LM_HEAD, vocab, d)]


def _plan(case):
    """(tensors, blocks, elements of the flat buffers)."""
    tensors = _tensors(case)
    blocks, total = A.adapm_plan_default(tensors, case["rank_pct"], case["rank"],
                                         A.V_BLOCKMEAN if case["v"] == "blockmean" else A.V_ELEMENT, 0.1)
    return tensors, blocks, total


def _offsets(tensors):
    at, out = 0, []
    for t in tensors:
        at = (at + 7) // 8 * 8
        out.append(at)
        at += t.rows * t.cols
    return out


def _fill_gradients(grads, tensors, recipe, gen, row_gen):
    """The gradients of one step, standard deviation 1e-3, with the recipe's row scales or tail."""
    grads.normal_(0.0, 1e-3, generator=gen)
    if recipe == "student_t3":      # normal / sqrt(chi2_3 / 3)
        for i in range(0, grads.numel(), 1 << 26):
            part = grads[i:i + (1 << 26)]
            chi2 = torch.zeros(part.numel(), device=part.device)
            for _ in range(3):
                chi2.addcmul_(*[torch.randn(part.numel(), generator=gen, device=part.device)] * 2)
            part.copy_(part.float() * torch.rsqrt(chi2 / 3))
    elif recipe in ("rowscale", "heavyrows"):
        for t, at in zip(tensors, _offsets(tensors)):
            if t.role == WL.ROLE_VECTOR:
                continue
            u = torch.rand(t.rows, 1, generator=row_gen, device=grads.device)
            scale = torch.exp((2 * u - 1) * math.log(10.0)) if recipe == "rowscale" else torch.where(u < 0.05, 100.0, 1.0)
            grads[at:at + t.rows * t.cols].view(t.rows, t.cols).mul_(scale.to(grads.dtype))


def prepare(case, seed):
    """A training program two steps into its run: parameters, optimizer state, and the third step's gradients."""
    dev = torch.device("cuda")
    tensors, blocks, total = _plan(case)
    gen = torch.Generator(device=dev).manual_seed(seed)
    params = torch.empty(total, device=dev).normal_(0.0, 0.02, generator=gen)
    for t, at in zip(tensors, _offsets(tensors)):
        if t.init != "normal":
            params[at:at + t.rows * t.cols] = 1.0 if t.init == "ones" else 0.0
    hp = A.hparams(lr=1e-3, beta1=0.9, beta2=case["beta2"], grad_dtype=A.GRAD_F32 if case["grad"] == "f32" else A.GRAD_BF16,
                   seed=seed, max_grad_norm=case["clip"], refresh_period=case["period"],
                   flags=A.FLAG_CHECK_FINITE if case["finite"] else 0)
    ctx = A.adapm_create(blocks, hp)
    state = torch.empty(ctx.adapm_state_bytes() // 4, device=dev)
    work = torch.empty(max(ctx.adapm_workspace_bytes() // 4, 1), device=dev)
    ctx.adapm_set_workspace(work)
    ctx.adapm_state_init(state)
    shadow = None
    if case["shadow"]:
        shadow = params.to(torch.bfloat16)
        ctx.adapm_set_shadow_params(shadow)
    grads = torch.empty(total, dtype=torch.float32 if case["grad"] == "f32" else torch.bfloat16, device=dev)
    for t in (1, 2, 3):
        _fill_gradients(grads, tensors, case["recipe"], gen, torch.Generator(device=dev).manual_seed(seed + 1))
        if t < 3:
            ctx.adapm_step(params, grads, state, t)
    # what a checkpoint of the run would hold: the factors, the momentum of the full blocks, the second moments
    first = {A.STATE_M: state.numel(), A.STATE_V: state.numel()}
    for which in first:
        for i in range(len(blocks)):
            at, n = ctx.adapm_state_layout(i, which)
            if n > 0:
                first[which] = min(first[which], at)
    first[A.STATE_M] = min(first[A.STATE_M], first[A.STATE_V])
    out = {"params": params, "factors": state[:first[A.STATE_M]], "momentum": state[first[A.STATE_M]:first[A.STATE_V]],
           "second_moment": state[first[A.STATE_V]:]}
    if shadow is not None:
        out["shadow"] = shadow
    return {"ctx": ctx, "params": params, "grads": grads, "state": state, "work": work, "t": 2, "out": out}


def run(s):
    s["t"] += 1
    s["ctx"].adapm_step(s["params"], s["grads"], s["state"], s["t"])
    return s["out"]


def work(case):
    """Every gradient read once; parameters, momenta, factors and second moments read and written once; the bf16 weights
    written once.  Flops: the contractions of the low-rank blocks (two products with g per inner pass, the Gram matrices,
    the products with them, and the two products of the corrected momentum)."""
    _, blocks, _ = _plan(case)
    g = 4 if case["grad"] == "f32" else 2
    held = case["period"] > 1
    nbytes = flops = 0
    for b in blocks:
        m, n, r = b.rows, b.cols, b.rank
        nbytes += m * n * (g + 8 + (2 if case["shadow"] else 0))
        if b.v_mode == A.V_ELEMENT:
            nbytes += 8 * m * n
        else:
            nbytes += 8 * (m // b.v_group_rows if b.v_group_rows else 1)
        if b.mom_mode == A.MOM_FULL:
            nbytes += 8 * m * n
        elif b.mom_mode == A.MOM_LOWRANK:
            sides = 1 if held else 2
            nbytes += 8 * r * n + (4 if held else 8) * r * m
            flops += INNER_PASSES * (2 * sides * m * n * r) + 4 * m * n * r
            flops += INNER_PASSES * 4 * r * r * (n + m) if not held else 4 * r * r * m + INNER_PASSES * 4 * r * r * n
    return {"bytes": nbytes, "flops": flops}


def tolerance(case):
    """Sums of 32-bit values; the bf16 path carries its factors as two bf16 parts (2^-17).  A bf16 weight may round to
    either neighbour where the fp32 weight differs in its last bits."""
    if case["shadow"]:
        return {"rel": 1e-4, "max": 1e-2}
    return {"rel": 1e-5 if case["grad"] == "f32" else 2e-5, "max": 1e-3}
