"""What a user of this package has it do, as cases that can be timed and compared.

A case is one call, or the few calls that belong together, of a block-wise denoising run's first
layer, through the public entry points (``Context``, ``QkvProducer``).  ``op`` says which:

  step      one denoising step: the block's fresh q/k/v in, the normalised output of every position
            out.  The call made most often by far (16 to 64 times per block).
  enter     entering a block: the build of its cache, then the block's first step.
  advance   several blocks with the incremental rebuild: the build, then per block its last step and
            the advance to the next one, then a step of the block reached.
  full      every row over every key without a cache: the vanilla step the method replaces.
  tokens    a step fed with the block's token ids (embedding, norm and projection in front).
  enter_tokens  entering a block from token ids: all tokens projected, the build, the first step.
  sample    the sampling stage on the block's rows of the logits.

The host-buffer calls move the same work over PCIe and the tile-granular cache is a variant kept for
comparison: neither is timed here.  A context runs with its defaults (plain stream order) apart from
what the case names.  Values are those the path meets: prompt and decoded tokens drawn per head with
the spread of the workloads in ``paper_2607_16339_b200.workloads``, identical [MASK] rows from the
current block on, token tables with a few large channels, logits of spread 3.
"""
import torch

from paper_2607_16339_b200.binding import (DTYPE_BF16, DTYPE_FP32, OUT_BF16, OUT_FP32, PRECISION_FP16,
                                           PRECISION_PLAIN, PRECISION_SPLIT, Context, QkvProducer)

PRECISION = {"plain": PRECISION_PLAIN, "split": PRECISION_SPLIT, "fp16": PRECISION_FP16}
RAGGED8 = "500,256,798,584,526,932,396,371"


def _case(name, op, prompts, gen, block, heads, kv_heads, dim=128, dtype="bf16", precision="split", out="fp32",
          scale="small", theta=5.0e5, **more):
    return dict(name=name, op=op, prompts=prompts, gen=gen, block=block, heads=heads, kv_heads=kv_heads, dim=dim,
                dtype=dtype, precision=precision, out=out, scale=scale, theta=theta, **more)


def listed():
    # 64 few-shot prompts of 600 to 1000 tokens: the large-batch setting, a quarter of its batch
    batch64 = ",".join(str(600 + (i * 397 + 113) % 401) for i in range(64))
    return [
        # the smallest call there is: the tiny fp32 model, where the launches and the host count
        _case("step_tiny_fp32", "step", "48", 64, 16, 4, 4, dim=64, dtype="fp32", theta=1.0e4),
        # LLaDA-8B, one request, the binding's default operands and output
        _case("step_llada_p512", "step", "512", 256, 32, 32, 32, scale="head"),
        # LLaDA-8B, eight requests of different prompt lengths
        _case("step_llada_ragged8", "step", RAGGED8, 256, 32, 32, 32, precision="fp16", scale="head"),
        # Dream-7B (grouped heads, 64-row blocks), long prompt and generation, bf16 output
        _case("step_dream_p4096", "step", "4096", 1024, 64, 28, 4, precision="plain", out="bf16", theta=1.0e6),
        # a serving batch: the step bound by the cache it streams
        _case("step_gqa_batch64", "step", batch64, 320, 32, 28, 4, precision="fp16", theta=1.0e6),
        # entering a block: fp32 model of ordinary size (the engine without tensor cores)
        _case("enter_small_fp32", "enter", "200,171", 128, 32, 8, 8, dtype="fp32", theta=1.0e4),
        # LLaDA-8B, keys with outliers, which want the split operands
        _case("enter_llada_p1024", "enter", "1024", 512, 32, 32, 32, scale="head", outliers=True),
        # Dream-7B, the build bound by the tensor cores
        _case("enter_dream_p4096", "enter", "4096", 1024, 64, 28, 4, precision="fp16", theta=1.0e6),
        # the same generation walked block by block with the incremental rebuild
        _case("advance_dream_p4096", "advance", "4096", 1024, 64, 28, 4, precision="fp16", theta=1.0e6, blocks=5),
        # LLaDA-8B fed with token ids: the projection bound by one read of its weight
        _case("tokens_llada_p512", "tokens", "512", 256, 32, 32, 32, precision="fp16", scale="head", d_model=4096),
        # ... and the projection of every token of eight requests, bound by the tensor cores
        _case("enter_tokens_ragged8", "enter_tokens", RAGGED8, 256, 32, 32, 32, precision="fp16", scale="head",
              d_model=4096),
        # the sampling stage of eight requests over LLaDA-8B's vocabulary
        _case("sample_llada_ragged8", "sample", RAGGED8, 256, 32, 32, 32, precision="fp16", vocab=126464),
    ]


def _log(rng, lo, hi):
    return int(round(lo * (hi / lo) ** rng.random()))


def draw(rng):
    """Sizes between the tiny model's and the largest listed case's."""
    while True:
        op = rng.choice(["step"] * 5 + ["enter"] * 3 + ["advance", "full", "tokens", "enter_tokens", "sample"])
        fp32 = op in ("step", "enter", "full") and rng.random() < 0.2
        if fp32:      # models of the engine without tensor cores: fp32, or heads of 64 features
            dim = rng.choice([64, 128])
            dtype = "bf16" if dim == 64 and rng.random() < 0.3 else "fp32"
            heads, kv = rng.choice([(4, 4), (8, 8), (8, 2), (12, 12)])
            batch, longest, gen_hi = rng.randint(1, 3), 400, 256
        else:
            dim, dtype = 128, "bf16"
            heads, kv = rng.choice([(32, 32), (32, 32), (28, 4), (28, 4), (32, 8), (16, 16), (12, 2)])
            batch = _log(rng, 1, 32 if op == "step" else 8)
            longest, gen_hi = (4096, 1024) if batch <= 2 else (1100, 512)
        block = rng.choice([16, 32, 32, 32, 64] if fp32 else [16, 32, 32, 32, 48, 64])
        gen = block * max(2, _log(rng, 64, gen_hi) // block)
        top = _log(rng, 33, longest)
        prompts = [top] + [rng.randint(max(1, top // 2), top) for _ in range(batch - 1)]
        lens = [p + gen for p in prompts]
        case = _case(None, op, ",".join(map(str, prompts)), gen, block, heads, kv, dim, dtype,
                     rng.choice(["split", "fp16", "fp16", "plain"]), rng.choice(["fp32", "fp32", "bf16"]))
        del case["name"]
        if not fp32 and case["precision"] != "plain" and rng.random() < 0.6:
            case["scale"] = "head"
        if op == "advance":
            case["blocks"] = min(rng.randint(2, 4), gen // block)
        if op in ("tokens", "enter_tokens"):
            case["d_model"] = rng.choice([2048, 3584, 4096]) if heads > 16 else 2048
        if op == "sample":
            case["vocab"] = _log(rng, 32000, 152064)
            if sum(lens) * case["vocab"] > 8e8:
                continue
        # no dearer than the listed ones
        if sum(n * n for n in lens) * heads > (1.0e8 if fp32 else 7.3e8) or sum(lens) * heads > 7.0e5:
            continue
        if op == "advance" and sum(n * n for n in lens) * heads > 4e8:
            continue
        return case


# ---------------------------------------------------------------------------------------------------
class State:
    pass


def _lens(case):
    return [int(p) for p in case["prompts"].split(",")]


def _blocks(case):
    """(first block, blocks in all): the middle of the generation."""
    n = case["gen"] // case["block"]
    used = case.get("blocks", 1)
    return min(n // 2, n - used), n


def _spread(case, H, group, gen, dev):
    if case["scale"] == "small":
        return torch.full((H,), case["dim"] ** -0.5, device=dev)
    c = torch.rand(H, generator=gen, device=dev) * 1.5 + 0.5
    return c if group == 1 else c.view(-1, group)[:, :1].expand(-1, group).reshape(-1)


def prepare(case, seed):
    dev = torch.device("cuda")
    gen = torch.Generator(device=dev).manual_seed(seed)
    op, d, H, Hkv = case["op"], case["dim"], case["heads"], case["kv_heads"]
    prompts, G, L = _lens(case), case["gen"], case["block"]
    tdt = torch.bfloat16 if case["dtype"] == "bf16" else torch.float32
    s = State()
    s.case, s.block = case, _blocks(case)[0]
    s.ctx = Context(DTYPE_BF16 if case["dtype"] == "bf16" else DTYPE_FP32, H, Hkv, d, case["theta"], prompts, G, L,
                    out_dtype=OUT_BF16 if case["out"] == "bf16" else OUT_FP32,
                    precision_mode=PRECISION[case["precision"]])
    starts = [0]
    for p in prompts:
        starts.append(starts[-1] + p + G)
    T, n = starts[-1], len(prompts) * L

    cq = _spread(case, H, H // Hkv, gen, dev)
    ckv = cq[::H // Hkv]

    def rows(count, scales):
        x = torch.randn(count, len(scales), d, generator=gen, device=dev)
        return x.mul_(scales[None, :, None])

    if op in ("step", "enter", "advance", "full", "sample"):
        full = [rows(T, c) for c in (cq, ckv, ckv)]
        if case.get("outliers"):
            for start, p in zip(starts, prompts):
                at = torch.randperm(p, generator=gen, device=dev)[:max(1, p // 100)] + start
                full[1][at] *= 4.0
        mask = [rows(1, c) for c in (cq, ckv, ckv)]
        for start, p in zip(starts, prompts):
            lo, hi = start + p + s.block * L, start + p + G
            for x, m in zip(full, mask):
                x[lo:hi] = m
        s.full = [x.to(tdt) for x in full]
        del full
        s.blk = [[rows(n, c).to(tdt) for c in (cq, ckv, ckv)] for _ in range(case.get("blocks", 1))]
    else:
        dm, vocab, width = case["d_model"], 8192, (H + 2 * Hkv) * d
        embed = torch.randn(vocab, dm, generator=gen, device=dev)
        embed[:, torch.randperm(dm, generator=gen, device=dev)[:max(1, dm // 1024)]] *= 20.0
        norm = torch.rand(dm, generator=gen, device=dev) + 0.5
        w = torch.randn(width, dm, generator=gen, device=dev)
        w *= torch.cat([cq, ckv, ckv]).repeat_interleave(d)[:, None] * dm ** -0.5
        s.producer = QkvProducer(embed.bfloat16(), norm.bfloat16(), w.bfloat16(), H, Hkv, d, 1e-5, T)
        del embed, w
        ids = torch.randint(0, vocab - 1, (T,), generator=gen, device=dev, dtype=torch.int32)
        for start, p in zip(starts, prompts):
            ids[start + p + s.block * L:start + p + G] = vocab - 1
        s.ids = ids
        s.blk_ids = torch.randint(0, vocab - 1, (n,), generator=gen, device=dev, dtype=torch.int32)
        s.blk_ids[torch.rand(n, generator=gen, device=dev) < 0.5] = vocab - 1   # half of the block decoded

    if op in ("step", "sample"):
        s.ctx.build(s.block, *s.full)
        del s.full
    elif op == "tokens":
        s.ctx.build_tokens(s.producer, s.block, token_ids=s.ids)
    if op == "sample":
        s.logits = torch.randn(T, case["vocab"], generator=gen, device=dev, dtype=torch.bfloat16).mul_(3.0)
        s.conf = torch.empty(n, device=dev)
        s.token = torch.empty(n, device=dev, dtype=torch.int32)
        s.lse = torch.empty(n, device=dev)
    else:
        odt = torch.bfloat16 if case["out"] == "bf16" else torch.float32
        s.out = [torch.empty(T, H, d, device=dev, dtype=odt) for _ in range(case.get("blocks", 1))]
        s.lse = [torch.empty(T, H, device=dev) for _ in range(case.get("blocks", 1))]
    return s


def run(s):
    op, ctx = s.case["op"], s.ctx
    if op == "sample":
        ctx.sample_block(s.logits, s.conf, s.token, s.lse)
        return [s.conf, s.token, s.lse]
    if op == "step":
        ctx.step(*s.blk[0], s.out[0], s.lse[0])
    elif op == "enter":
        ctx.build(s.block, *s.full)
        ctx.step(*s.blk[0], s.out[0], s.lse[0])
    elif op == "advance":
        ctx.build_incremental(s.block, *s.full)
        ctx.step(*s.blk[0], s.out[0], s.lse[0])
        for j in range(1, len(s.blk)):
            ctx.build_advance(*s.blk[j - 1])
            ctx.step(*s.blk[j], s.out[j], s.lse[j])
    elif op == "full":
        ctx.full_recompute(*s.full, s.out[0], s.lse[0])
    elif op == "tokens":
        ctx.step_tokens(s.producer, s.out[0], s.lse[0], blk_token_ids=s.blk_ids)
    elif op == "enter_tokens":
        ctx.build_tokens(s.producer, s.block, token_ids=s.ids)
        ctx.step_tokens(s.producer, s.out[0], s.lse[0], blk_token_ids=s.blk_ids)
    return [s.out, s.lse]


def work(case):
    """What a pass cannot do without.  Rotated q/k/v are counted at the input's width and the cached
    state at fp32, whatever the operand mode stores."""
    d, H, Hkv, L, op = case["dim"], case["heads"], case["kv_heads"], case["block"], case["op"]
    es = 2 if case["dtype"] == "bf16" else 4
    lens = [p + case["gen"] for p in _lens(case)]
    T, n = sum(lens), len(lens) * L
    if op == "sample":
        return {"bytes": n * case["vocab"] * 2.0 + 12 * n, "flops": 4.0 * n * case["vocab"]}
    out = T * H * d * (2 if case["out"] == "bf16" else 4) + 4 * T * H
    fixed = (T - n) * H * (es * d + 4 * d + 8)                  # rotated queries and state of the fixed rows
    step = {"bytes": fixed + 2 * T * Hkv * d * es + n * (H + 2 * Hkv) * d * es + out,
            "flops": 4.0 * d * H * sum((m - L) * L + L * m for m in lens)}
    inputs = T * (H + 2 * Hkv) * d * es
    build = {"bytes": 2 * inputs + (T - n) * H * (4 * d + 8), "flops": 4.0 * d * H * sum((m - L) ** 2 for m in lens)}

    def project(tokens):
        width = (H + 2 * Hkv) * d
        return {"bytes": 2.0 * (width * case["d_model"] + tokens * (case["d_model"] + width)),
                "flops": 2.0 * tokens * width * case["d_model"]}

    def total(*parts):
        return {k: float(sum(p[k] for p in parts)) for k in ("bytes", "flops")}

    if op == "step":
        return total(step)
    if op == "enter":
        return total(build, step)
    if op == "full":
        return {"bytes": float(inputs + out), "flops": 4.0 * d * H * sum(m * m for m in lens)}
    if op == "tokens":
        return total(project(n), step)
    if op == "enter_tokens":
        return total(project(T), build, project(n), step)
    parts = [build, step]
    b0, n_blocks = _blocks(case)
    for j in range(1, case["blocks"]):
        # the finished block's keys onto every row's prefix state, the keys after the next block onto the
        # cached state; the finished block's own rows over everything before the next block
        after = case["gen"] - (b0 + j + 1) * L
        parts.append({"bytes": (T - n) * H * (es * d + 2 * (4 * d + 8)) + 2 * T * Hkv * d * es,
                      "flops": 4.0 * d * H * sum((m - 2 * L) * L + (m - L) * after + L * (m - after - L) for m in lens)})
        parts.append(step)
    return total(*parts)


def tolerance(case):
    if case["op"] == "sample":
        return {"rel": 1e-5, "max": 1e-4}      # fp32 sums over the vocabulary; the token ids are exact
    if case["dtype"] == "fp32" or case["dim"] == 64:
        # fp32 throughout; a bf16 output adds its rounding
        return {"rel": 1e-5, "max": 1e-4} if case["out"] == "fp32" else {"rel": 3e-3, "max": 1e-2}
    # tensor-core path: 16-bit probabilities and operands, fp32 sums
    if case["op"] in ("tokens", "enter_tokens"):
        return {"rel": 5e-3, "max": 0.1}       # ... and projections rounded to bf16 in front
    return {"rel": 1e-3, "max": 0.02} if case["out"] == "fp32" else {"rel": 4e-3, "max": 0.03}
