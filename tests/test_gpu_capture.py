"""Calls captured into a CUDA graph behind the things a captured stream has in it -- copies, another stream joined by an
event, ordinary kernels -- where their programmatically dependent launches follow no kernel, or more than one operation:
the replay gives what the same calls give when they are enqueued one by one."""
import pytest
import torch

from paper_2607_16339_b200 import binding
from paper_2607_16339_b200.workloads import SyntheticSchedule, small_workload

from lacache_testlib import make_ctx, new_outputs, to_dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype,hq,hkv,mode", [("bf16", 32, 32, binding.PRECISION_FP16), ("bf16", 4, 2, binding.PRECISION_SPLIT),
                                               ("fp32", 4, 4, None)])
def test_replay_matches_eager_calls(dtype, hq, hkv, mode):
    wl = small_workload(name="capture", dtype=dtype, prompt_lens=(300, 41), gen_len=64, block_len=32, steps=2, hq=hq, hkv=hkv)
    kw = {} if mode is None else dict(precision_mode=mode)
    sch = SyntheticSchedule(wl, seed=8)
    full = [to_dev(a, wl) for a in sch.begin_block(0)]
    steps = [[to_dev(a, wl) for a in sch.draw_step(0, i)] for i in (1, 2)]
    host = [t.cpu().pin_memory() for t in steps[1]]
    g = torch.Generator(device="cuda").manual_seed(1)
    logits = torch.randn(wl.total_tokens, 4099, generator=g, device="cuda")
    n = wl.batch * wl.block_len
    ctx = make_ctx(wl, **kw)
    bufs = [torch.empty_like(t) for t in full]
    sbuf = [torch.empty_like(t) for t in steps[0]]
    lbuf = torch.empty_like(logits)
    side = torch.cuda.Stream()
    outs = [new_outputs(wl) for _ in range(3)]
    samp = (torch.empty(n, device="cuda"), torch.empty(n, device="cuda", dtype=torch.int32), torch.empty(n, device="cuda"))

    def calls():
        for d, s in zip(bufs, full):
            d.copy_(s)                                   # kernels or copies on this stream
        ctx.build(0, *bufs)
        for d, s in zip(sbuf, steps[0]):
            d.copy_(s)
        ctx.step(*sbuf, *outs[0])
        side.wait_stream(torch.cuda.current_stream())
        with torch.cuda.stream(side):                    # the next step's inputs from another stream ...
            for d, s in zip(sbuf, host):
                d.copy_(s, non_blocking=True)
            lbuf.copy_(logits)
        torch.cuda.current_stream().wait_stream(side)    # ... joined right before the call
        ctx.step(*sbuf, *outs[1])
        ctx.sample_block(lbuf, samp[0], samp[1], samp[2])
        ctx.full_recompute(*bufs, *outs[2])

    calls()                                              # (first use allocates)
    torch.cuda.synchronize()
    want = [t.clone() for o in outs for t in o] + [t.clone() for t in samp]
    for t in [t for o in outs for t in o] + list(samp):
        t.zero_()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        calls()
    for _ in range(3):
        graph.replay()
    torch.cuda.synchronize()
    assert ctx.poll_status()[0] == 0
    for a, b in zip(want, [t for o in outs for t in o] + list(samp)):
        assert torch.equal(a, b)
    del graph
    ctx.destroy()
