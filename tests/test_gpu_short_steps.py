"""Short steps with one-plane operands let the kernels behind them be scheduled early: steps and builds whose inputs
are written on the stream just before, and whose outputs are read just after, give bit for bit what synchronised calls
give, on both sides of the rule's limit (fixed-row tiles per CTA)."""
import pytest
import torch

from paper_2607_16339_b200 import binding
from paper_2607_16339_b200.workloads import SyntheticSchedule, small_workload

from lacache_testlib import advance_to_block, make_ctx, new_outputs, to_dev
from test_gpu_parity import _run_points

pytestmark = pytest.mark.gpu
MODES = {"plain": binding.PRECISION_PLAIN, "fp16": binding.PRECISION_FP16}


@pytest.mark.parametrize("prompts,block,hq,hkv,mode", [
    ((40,), 32, 4, 4, "fp16"),             # one tile a CTA, most SMs idle
    ((500,), 32, 32, 32, "fp16"),          # pairs of CTAs
    ((1100,), 16, 28, 4, "plain"),         # packed heads, three or four tiles a CTA
    ((1280, 57), 32, 32, 32, "plain"),     # about the limit
    ((1500, 700), 32, 32, 32, "fp16"),     # above it
])
def test_steps_and_builds_in_stream_order(prompts, block, hq, hkv, mode):
    wl = small_workload(name="short-%d-%d" % (sum(prompts), hq), prompt_lens=prompts, gen_len=2 * block, block_len=block,
                        steps=3, hq=hq, hkv=hkv)
    sch = SyntheticSchedule(wl, seed=5)
    full = [tuple(to_dev(a, wl) for a in sch.begin_block(0))]
    steps = [tuple(to_dev(a, wl) for a in sch.draw_step(0, s)) for s in (1, 2, 3)]
    full.append(tuple(t.flip(0).contiguous() for t in full[0]))
    ctx = make_ctx(wl, precision_mode=MODES[mode])
    bufs = [torch.empty_like(t) for t in full[0]]
    sbuf = [torch.empty_like(t) for t in steps[0]]
    out, lse = new_outputs(wl)

    def run(sync):
        res = []
        for f in full:
            for d, s in zip(bufs, f):
                d.copy_(s)
            ctx.build(0, *bufs)
            for st in steps:
                for d, s in zip(sbuf, st):
                    d.copy_(s)
                ctx.step(*sbuf, out, lse)
                if sync:
                    torch.cuda.synchronize()
                res.append((out.clone(), lse.clone()))
        torch.cuda.synchronize()
        assert ctx.poll_status()[0] == 0
        return res

    ref = run(True)
    for _ in range(4):
        for i, ((o0, l0), (o1, l1)) in enumerate(zip(ref, run(False))):
            assert torch.equal(o0, o1) and torch.equal(l0, l1), "call %d" % i
    ctx.destroy()


@pytest.mark.parametrize("block", [16, 32])
def test_two_key_chunks_as_a_pair_of_ctas_with_split_planes(block, monkeypatch):
    """The paired step with split planes, whose operand tiles leave the partner's state just room enough: against the
    oracle, and against the same step with the pairing switched off."""
    wl = small_workload(name="pair-split-%d" % block, prompt_lens=(100, 131, 90), gen_len=2 * block, block_len=block,
                        steps=2, hq=4, hkv=4)
    monkeypatch.setenv("LACACHE_STREAM_CTAS", str(wl.batch * 2 * wl.n_q_heads))   # (read when a context is created)
    outs = []
    for pair in (True, False):
        if not pair:
            monkeypatch.setenv("LACACHE_NO_PAIR", "1")
        _run_points(wl, "tc", seed=12, sc_tiles_per_chunk=1)
        sch = SyntheticSchedule(wl, seed=12)
        ctx = make_ctx(wl, sc_tiles_per_chunk=1)
        q, k, v = (to_dev(a, wl) for a in advance_to_block(sch, 1))
        ctx.build(1, q, k, v)
        out, lse = new_outputs(wl)
        ctx.step(*(to_dev(a, wl) for a in sch.draw_step(1, 1)), out, lse)
        torch.cuda.synchronize()
        assert ctx.poll_status()[0] == 0
        outs.append((out.clone(), lse.clone()))
        ctx.destroy()
    assert (outs[0][0] - outs[1][0]).abs().max().item() <= 1e-5
    assert (outs[0][1] - outs[1][1]).abs().max().item() <= 1e-5
