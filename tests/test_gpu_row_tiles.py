"""GPU parity of the row-tile kernel (builds, full recomputes and key windows with one plane per operand) at the edges of
its tiles: sequences that end one row before, at and after a 128-row tile and a 256-row item, a second tile with a single
row or with whole warps of missing rows, blocks that straddle key tiles, and few CTAs that walk many items each."""
import pytest

from paper_2607_16339_b200 import binding
from paper_2607_16339_b200.workloads import small_workload

from test_gpu_incremental import _run as _run_generation
from test_gpu_parity import _run_points

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prompts,block,ctas", [
    ((95, 96, 97), 16, 0),          # 127, 128, 129 tokens
    ((223, 224, 225), 16, 2),       # 255, 256, 257
    ((0, 110, 353), 32, 3),         # 64, 174, 417
    ((640, 5), 64, 3),
])
@pytest.mark.parametrize("mode", [binding.PRECISION_PLAIN, binding.PRECISION_FP16])
def test_tile_edges(prompts, block, ctas, mode, monkeypatch):
    if ctas:
        monkeypatch.setenv("LACACHE_MAX_CTAS", str(ctas))     # (experiment knobs are read when a context is created)
    wl = small_workload(name="rows", prompt_lens=prompts, gen_len=2 * block, block_len=block, steps=1, hq=4, hkv=2,
                        scale_mode="inv_sqrt_d" if mode == binding.PRECISION_PLAIN else "per_head_u(0.5,2)")
    _run_points(wl, "tc", seed=41, precision_mode=mode)
    _run_generation(wl, seed=42, precision_mode=mode)
