"""GPU parity of the fp32 engine where its units are cut over the CTAs of a cluster: every number of parts a
key range of 32-key tiles can give (a single tile up to more tiles than a cluster takes), row tiles with one
valid row or one row group missing, block rows that share their key tile with fixed rows, both head widths,
and bf16 inputs through the same kernel."""
import pytest

from paper_2607_16339_b200.workloads import small_workload

from test_gpu_parity import _run_points

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prompts,gen,block", [
    ((0,), 16, 16),             # one key tile, nothing fixed
    ((17,), 16, 16),            # two tiles, a row tile of 17
    ((33, 1), 64, 32),          # ragged: more parts than the short sequence has tiles
    ((65,), 48, 48),            # two row tiles of block rows, the second half full
    ((129, 95), 64, 64),        # whole block tiles that start inside a key tile
    ((410,), 96, 32),           # sixteen tiles: the largest cluster, two tiles a part
    ((700, 333, 61), 192, 64),  # more CTAs than SMs
])
@pytest.mark.parametrize("dtype,d", [("fp32", 64), ("fp32", 128), ("bf16", 64)])
def test_units_cut_over_a_cluster(prompts, gen, block, dtype, d):
    wl = small_workload(name="simt", dtype=dtype, prompt_lens=prompts, gen_len=gen, block_len=block, steps=2, hq=4,
                        hkv=2, d=d, scale_mode="inv_sqrt_d")
    _run_points(wl, "simt", seed=31, blocks=sorted({0, wl.n_blocks - 1}))
