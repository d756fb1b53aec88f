"""GPU parity of the row-tile kernel (builds, full recomputes and key windows) at the edges of
its tiles: sequences that end one row before, at and after a 128-row tile and a 256-row item, a second tile with a single
row or with whole warps of missing rows, blocks that straddle key tiles, and few CTAs that walk many items each."""
import pytest
import torch

from paper_2607_16339_b200 import binding
from paper_2607_16339_b200.workloads import SyntheticSchedule, small_workload

from lacache_testlib import make_ctx, new_outputs, to_dev
from test_gpu_incremental import _run as _run_generation
from test_gpu_parity import _run_points

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prompts,block,ctas", [
    ((95, 96, 97), 16, 0),          # 127, 128, 129 tokens
    ((223, 224, 225), 16, 2),       # 255, 256, 257
    ((0, 110, 353), 32, 3),         # 64, 174, 417
    ((640, 5), 64, 3),
])
# (split planes: another ring -- one stage of keys in four pieces -- and another way of storing rows)
@pytest.mark.parametrize("mode", [binding.PRECISION_PLAIN, binding.PRECISION_FP16, binding.PRECISION_SPLIT])
def test_tile_edges(prompts, block, ctas, mode, monkeypatch):
    if ctas:
        monkeypatch.setenv("LACACHE_MAX_CTAS", str(ctas))     # (experiment knobs are read when a context is created)
    wl = small_workload(name="rows", prompt_lens=prompts, gen_len=2 * block, block_len=block, steps=1, hq=4, hkv=2,
                        scale_mode="inv_sqrt_d" if mode == binding.PRECISION_PLAIN else "per_head_u(0.5,2)")
    _run_points(wl, "tc", seed=41, precision_mode=mode)
    _run_generation(wl, seed=42, precision_mode=mode)


@pytest.mark.parametrize("mode", [binding.PRECISION_FP16, binding.PRECISION_SPLIT])
@pytest.mark.parametrize("out_dtype", [binding.OUT_FP32, binding.OUT_BF16])
def test_rows_stored_in_either_output_type(mode, out_dtype):
    """A full recompute writes its rows itself: tiles with one row, a warp's worth and all but one, in both output types,
    against the same rows in fp32 (a bf16 output is that value rounded once)."""
    prompts, block = (0, 97, 223), 32          # 64, 161 (128 + 33), 287 (256 + 31) tokens
    wl = small_workload(name="rows-out", prompt_lens=prompts, gen_len=2 * block, block_len=block, steps=1, hq=4, hkv=2)
    sch = SyntheticSchedule(wl, seed=3)
    q, k, v = (to_dev(a, wl) for a in sch.begin_block(0))
    res = []
    for odt in (binding.OUT_FP32, out_dtype):
        ctx = make_ctx(wl, precision_mode=mode, out_dtype=odt)
        out, lse = new_outputs(wl)
        if odt == binding.OUT_BF16:
            out = out.bfloat16()
        ctx.full_recompute(q, k, v, out, lse)
        torch.cuda.synchronize()
        assert ctx.poll_status()[0] == 0
        res.append((out, lse))
        ctx.destroy()
    assert torch.isfinite(res[0][0]).all()
    assert torch.equal(res[1][0], res[0][0] if out_dtype == binding.OUT_FP32 else res[0][0].bfloat16())
    assert torch.equal(res[0][1], res[1][1])
