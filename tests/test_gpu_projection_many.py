"""GPU parity of the many-token projection where it can go wrong: token counts around its 128- and 256-row tiles, the
ring of operand stages shorter and longer than the reduction, an odd number of heads (half a tile of features), more
tiles than the GPU has pairs of SMs, and scattered output rows -- against the fp64 oracle."""
import numpy as np
import pytest
import torch

from paper_2607_16339_b200 import binding, workloads as W
from paper_2607_16339_b200.workloads import TokenModel

from test_gpu_tokenwise import check_qkv, make_producer, project

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("hq,hkv,d_model,n", [
    (4, 2, 64, 65), (4, 2, 64, 128), (3, 1, 128, 129), (2, 1, 448, 255), (4, 4, 512, 256), (20, 20, 128, 257),
    (3, 3, 384, 513), (24, 24, 64, 1100),
])
def test_token_counts_and_head_counts(hq, hkv, d_model, n):
    tm = TokenModel(W.small_workload(hq=hq, hkv=hkv), d_model, 500)
    prod = make_producer(tm, n)
    ids = np.random.default_rng(n).integers(0, tm.vocab, n).astype(np.int32)
    for _ in range(2):      # (the second call finds the barriers' and the ring's leftovers of another launch)
        st, msg, q, k, v, _ = project(prod, tm, n, ids=ids)
        assert st == binding.OK, msg
    check_qkv(tm, q, k, v, ids=ids, what="n=%d" % n)
    prod.destroy()


@pytest.mark.parametrize("hq,hkv,d_model,n", [
    (36, 36, 2112, 6), (36, 36, 2112, 33),       # 108 tiles on 148 SMs: more than two tiles per helper
    (40, 40, 1024, 32), (46, 46, 512, 17),       # 120; 138
    (32, 32, 1024, 32), (33, 33, 1024, 31),      # 96 and 99: two tiles per helper, and just above
])
def test_few_tokens_of_models_with_many_heads(hq, hkv, d_model, n):
    """The projection of a block's tokens on both sides of where its work is split by role, repeatedly (parts that land in
    another CTA's place show up now and then only)."""
    tm = TokenModel(W.small_workload(hq=hq, hkv=hkv), d_model, 500)
    prod = make_producer(tm, n)
    for rep in range(4):
        ids = np.random.default_rng(rep).integers(0, tm.vocab, n).astype(np.int32)
        st, msg, q, k, v, _ = project(prod, tm, n, ids=ids)
        assert st == binding.OK, msg
        check_qkv(tm, q, k, v, ids=ids, what="rep %d" % rep)
    prod.destroy()
