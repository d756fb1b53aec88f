"""The stored prefix states of an advance: stored again only when one key tile no longer holds the keys of the blocks
finished since.  Walks long enough for several stores -- blocks of 16 to 64 rows, among them lengths that do not divide the
tile -- from the first block and from a later one, against a context rebuilt for every block; and a captured advance replayed
behind a build at another block than the one it was captured behind."""
import pytest
import torch

from paper_2607_16339_b200 import binding
from paper_2607_16339_b200.workloads import SyntheticSchedule, small_workload

from lacache_testlib import TOL_CACHED_VS_FULL, make_ctx, new_outputs, to_dev
from test_gpu_incremental import _state

pytestmark = pytest.mark.gpu


def _same_softmax(inc, ref, wl, sch, b):
    fixed = torch.from_numpy(sch.is_block(b) == 0).cuda()
    (m1, l1, o1), (m2, l2, o2) = _state(inc, wl), _state(ref, wl)
    has = l2[fixed] > 0
    assert torch.equal(l1[fixed] > 0, has)
    n1, n2 = ((o[fixed] / l[fixed][..., None])[has] for o, l in ((o1, l1), (o2, l2)))
    assert (n1 - n2).abs().max().item() <= TOL_CACHED_VS_FULL[wl.dtype], "block %d" % b
    e1, e2 = ((m[fixed] + torch.log(l[fixed]))[has] for m, l in ((m1, l1), (m2, l2)))
    assert (e1 - e2).abs().max().item() <= 1e-3, "block %d" % b


@pytest.mark.parametrize("block_len,n_blocks,first", [(16, 19, 0), (16, 12, 3), (24, 13, 1), (40, 8, 0), (48, 7, 2), (64, 6, 1)])
@pytest.mark.parametrize("mode", [binding.PRECISION_FP16, binding.PRECISION_SPLIT])
def test_every_block_of_a_long_walk(block_len, n_blocks, first, mode):
    wl = small_workload(name="walk", prompt_lens=(0, 141, 300), gen_len=block_len * n_blocks, block_len=block_len, steps=1, hq=4, hkv=2)
    sch = SyntheticSchedule(wl, seed=31)
    inc, ref = (make_ctx(wl, engine=binding.ENGINE_TCGEN05, precision_mode=mode) for _ in range(2))
    fin = None
    for b in range(n_blocks):
        full = [to_dev(x, wl) for x in sch.begin_block(b)]
        if b == first:
            inc.build_incremental(b, *full)
        elif b > first:
            inc.build_advance(*fin)
        if b >= first:
            ref.build(b, *full)
            torch.cuda.synchronize()
            assert inc.poll_status()[0] == 0 and ref.poll_status()[0] == 0
            _same_softmax(inc, ref, wl, sch, b)
        fin = [to_dev(x, wl) for x in sch.draw_step(b, 1)]
    inc.destroy()
    ref.destroy()


def test_captured_advance_follows_what_was_built():
    wl = small_workload(name="replay", prompt_lens=(90, 200), gen_len=256, block_len=32, steps=1, hq=4, hkv=4)
    sch = SyntheticSchedule(wl, seed=5)
    inc, ref = (make_ctx(wl, engine=binding.ENGINE_TCGEN05) for _ in range(2))
    full, fin = [], []
    for b in range(4):
        full.append([to_dev(x, wl) for x in sch.begin_block(b)])
        fin.append([to_dev(x, wl) for x in sch.draw_step(b, 1)])
    inc.build_incremental(0, *full[0])
    torch.cuda.synchronize()
    graphs = []
    for b in range(3):      # captured as a walk from block 0
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g):
            inc.build_advance(*fin[b])
        graphs.append(g)
    for start in (0, 1, 2):
        inc.build_incremental(start, *full[start])
        for g in graphs[start:]:
            g.replay()
        ref.build(3, *full[3])
        torch.cuda.synchronize()
        assert inc.poll_status()[0] == 0
        _same_softmax(inc, ref, wl, sch, 3)
    del graphs
    inc.destroy()
    ref.destroy()
