"""A context prepares the kernels that it may launch and no other.  What a kernel was prepared for stays with the
process, so each order of first contexts runs in a process of its own: build, steps, full recompute and the incremental
rebuild of every context agree with its own full recompute."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

SCRIPT = """
import sys
import torch
from paper_2607_16339_b200 import binding as b

def outputs(T):
    return torch.empty(T, 4, 128, device="cuda"), torch.empty(T, 4, device="cuda")

def run(mode, block, heads_kv):
    fp32 = mode == "fp32"
    kw = {} if fp32 else dict(precision_mode={"plain": b.PRECISION_PLAIN, "split": b.PRECISION_SPLIT, "fp16": b.PRECISION_FP16}[mode])
    ctx = b.Context(b.DTYPE_FP32 if fp32 else b.DTYPE_BF16, 4, heads_kv, 128, 1e4, [70, 33], 2 * block, block, **kw)
    assert ctx.engine == (b.ENGINE_SIMT if fp32 else b.ENGINE_TCGEN05)
    T, n = ctx.total_tokens, 2 * block
    g = torch.Generator(device="cuda").manual_seed(7)
    x = [(torch.randn(T, h, 128, generator=g, device="cuda") * 128 ** -0.5).to(torch.float32 if fp32 else torch.bfloat16)
         for h in (4, heads_kv, heads_kv)]
    starts = [70, 70 + 2 * block + 33]
    for build in ([ctx.build] if fp32 else [ctx.build, ctx.build_incremental]):
        build(0, *x)
        for blk in range(1 if fp32 or build == ctx.build else 2):
            rows = torch.cat([torch.arange(s + blk * block, s + (blk + 1) * block, device="cuda") for s in starts])
            if blk:
                prev = rows - block
                ctx.build_advance(*[t[prev].contiguous() for t in x])
            out, lse = outputs(T)
            ctx.step(*[t[rows].contiguous() for t in x], out, lse)
            ref, rlse = outputs(T)
            ctx.full_recompute(*x, ref, rlse)
            torch.cuda.synchronize()
            assert ctx.poll_status()[0] == 0, ctx.poll_status()
            assert (out - ref).abs().max().item() <= 1e-3 and (lse - rlse).abs().max().item() <= 1e-3, (mode, block, blk)
    return ctx

kept = [run(m, block, hkv) for m in sys.argv[1].split(",") for block, hkv in ((32, 4), (16, 2), (64, 4), (48, 2))]
"""


@pytest.mark.parametrize("order", ["plain", "split", "fp32", "fp32,fp16,split", "split,fp32,plain"])
def test_each_order_of_first_contexts(order):
    r = subprocess.run([sys.executable, "-c", SCRIPT, order], cwd=ROOT, capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stderr[-2000:]
