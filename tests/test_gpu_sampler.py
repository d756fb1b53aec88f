"""GPU parity of the sampling-stage truncation (softmax over the vocabulary on the current block's rows
only) against the fp64 oracle, through the C ABI.

Tolerance.  The token is an argmax over the stored logits themselves (no arithmetic): bit-exact, ties to
the lowest id on both sides.  The probability is 1 / sum_v exp(x_v - x_max) in fp32 with the hardware
exp2: each term carries a relative error of about |x_v - x_max| * 2^-23 from the scaled exponent plus
2^-22 from exp2, weighted by the term's share of the sum, and the fp32 sum over threads, warps and slices
adds a few 2^-24: 2e-5 relative (and absolute on the log normaliser) covers vocabularies of 1e5 entries.
"""
import numpy as np
import pytest
import torch

from oracle import sampler
from paper_2607_16339_b200 import binding
from paper_2607_16339_b200.workloads import WORKLOADS, SyntheticSchedule, small_workload

from lacache_testlib import make_ctx, to_dev

pytestmark = pytest.mark.gpu


def _built_ctx(wl, b):
    sch = SyntheticSchedule(wl, seed=4)
    for bb in range(b):
        sch.begin_block(bb)
        sch.draw_step(bb, wl.steps_per_block)
    q, k, v = sch.begin_block(b)
    ctx = make_ctx(wl)
    ctx.build(b, to_dev(q, wl), to_dev(k, wl), to_dev(v, wl))
    return ctx, sch


def _check(ctx, rows, logits_t, want_lse=True):
    n = rows.shape[0]
    conf = torch.full((n,), float("nan"), device="cuda")
    tok = torch.full((n,), -7, device="cuda", dtype=torch.int32)
    lse = torch.full((n,), float("nan"), device="cuda") if want_lse else None
    ctx.sample_block(logits_t, conf, tok, lse)
    torch.cuda.synchronize()
    st, msg = ctx.poll_status()
    assert st == 0, msg
    ref_tok, ref_conf, ref_lse = sampler.block_confidence(logits_t.float().cpu().numpy().astype(np.float64), rows)
    assert np.array_equal(tok.cpu().numpy().astype(np.int64), ref_tok)
    c = conf.cpu().numpy().astype(np.float64)
    assert np.all(np.abs(c - ref_conf) <= 2e-5 * ref_conf + 1e-30), np.abs(c / ref_conf - 1).max()
    if want_lse:
        assert np.abs(lse.cpu().numpy().astype(np.float64) - ref_lse).max() <= 2e-5 * np.maximum(1.0, np.abs(ref_lse)).max()
    return c


@pytest.mark.parametrize("dtype", [torch.bfloat16, torch.float32])
@pytest.mark.parametrize("vocab", [1, 7, 1000, 4099, 32768, 126464])
def test_block_rows_against_oracle(dtype, vocab):
    wl = small_workload(name="samp", prompt_lens=(70, 33), gen_len=64, block_len=32, steps=1, hq=2, hkv=2)
    ctx, sch = _built_ctx(wl, 1)
    g = torch.Generator(device="cuda").manual_seed(vocab)
    T = wl.total_tokens
    logits = (torch.randn(T, vocab, generator=g, device="cuda") * 4).to(dtype)
    rows = sch.block_rows(1)
    # a peaked row, a row with exact ties at the maximum, a row with masked (-inf) entries
    if vocab >= 7:
        logits[rows[0], vocab // 2] = 30.0
        logits[rows[1], [5, 3, vocab - 1]] = 25.0
        logits[rows[2], ::2] = float("-inf")
    # rows outside the block must not be read: poison them
    outside = torch.ones(T, dtype=torch.bool, device="cuda")
    outside[torch.from_numpy(rows).cuda()] = False
    logits[outside] = float("nan")
    _check(ctx, rows, logits)
    _check(ctx, rows, logits, want_lse=False)      # lse is optional; repeated calls reuse the counters
    ctx.destroy()


@pytest.mark.parametrize("rows,vocab", [(192, 50021), (96, 4097), (320, 2055)])
def test_many_rows_of_an_unaligned_vocabulary(rows, vocab):
    """Rows that start anywhere in a 16-byte vector, cut into many segments and into one."""
    wl = small_workload(name="samp-odd", prompt_lens=(5,) * (rows // 32), gen_len=32, block_len=32, steps=1, hq=2, hkv=2)
    ctx, sch = _built_ctx(wl, 0)
    g = torch.Generator(device="cuda").manual_seed(rows)
    logits = (torch.randn(wl.total_tokens, vocab, generator=g, device="cuda") * 4).to(torch.bfloat16)
    at = sch.block_rows(0)
    logits[at[0], [0, vocab - 1]] = 30.0       # the maximum at both ends of the row
    logits[at[1], :-1] = float("-inf")
    _check(ctx, at, logits)
    ctx.destroy()


@pytest.mark.parametrize("dtype", [torch.bfloat16, torch.float32])
@pytest.mark.parametrize("vocab", [7, 1000, 4099, 126464])
def test_entries_masked_with_the_lowest_value_of_the_type(dtype, vocab):
    """torch.finfo(dtype).min as a mask (finite, but its product with log2 e is not): whole batches of a lane, whole
    segments and whole rows of it, before and behind the other entries; and the largest value as a logit."""
    wl = small_workload(name="samp-min", prompt_lens=(21,), gen_len=32, block_len=16, steps=1, hq=2, hkv=2)
    ctx, sch = _built_ctx(wl, 0)
    g = torch.Generator(device="cuda").manual_seed(vocab)
    logits = (torch.randn(wl.total_tokens, vocab, generator=g, device="cuda") * 4).to(dtype)
    at, info = sch.block_rows(0), torch.finfo(dtype)
    logits[at[0], : vocab // 2] = info.min
    logits[at[1], vocab // 2:] = info.min
    logits[at[2], ::2] = info.min
    logits[at[3], : vocab - 1] = info.min          # one entry left, at the end
    logits[at[4], 1:] = info.min                   # ... at the start
    logits[at[5]] = info.min                       # none: uniform
    logits[at[6]] = info.min
    logits[at[6], ::3] = float("-inf")
    logits[at[7], vocab // 3] = info.max
    logits[at[8], vocab // 2:] = info.max
    logits[at[9], 0] = info.max * 0.7              # two that differ, both beyond 2^127
    logits[at[9], vocab - 1] = info.max * 0.8
    logits[at[10], ::2] = info.min * 0.7
    n = at.shape[0]
    conf, lse = torch.empty(n, device="cuda"), torch.empty(n, device="cuda")
    tok = torch.empty(n, device="cuda", dtype=torch.int32)
    ctx.sample_block(logits, conf, tok, lse)
    torch.cuda.synchronize()
    assert ctx.poll_status()[0] == 0
    ref_tok, ref_conf, ref_lse = sampler.block_confidence(logits.float().cpu().numpy().astype(np.float64), at)
    assert np.array_equal(tok.cpu().numpy().astype(np.int64), ref_tok)
    c, l = conf.cpu().numpy().astype(np.float64), lse.cpu().numpy().astype(np.float64)
    assert np.all(np.abs(c - ref_conf) <= 2e-5 * ref_conf), (c, ref_conf)
    assert np.all(np.abs(l - ref_lse) <= 2e-5 * np.maximum(1.0, np.abs(ref_lse))), (l, ref_lse)
    ctx.destroy()


@pytest.mark.parametrize("dtype", [torch.bfloat16, torch.float32])
@pytest.mark.parametrize("size", [1e8, 5e8, 6e8, 1e9, 1e10, 1e30, 1.6e38])
def test_entries_of_any_size_as_a_mask(dtype, size):
    """Finite masks of every size in use (the rounding of a large maximum times log2 e is itself large), and as large logits:
    below, at and above the size from which a segment is summed relative to its maximum."""
    vocab = 5003
    wl = small_workload(name="samp-mask", prompt_lens=(21,), gen_len=32, block_len=16, steps=1, hq=2, hkv=2)
    ctx, sch = _built_ctx(wl, 0)
    g = torch.Generator(device="cuda").manual_seed(3)
    logits = (torch.randn(wl.total_tokens, vocab, generator=g, device="cuda") * 4).to(dtype)
    at = sch.block_rows(0)
    logits[at[0], : vocab // 2] = -size
    logits[at[1], vocab // 2:] = -size
    logits[at[2], ::2] = -size
    logits[at[3], : vocab - 1] = -size
    logits[at[4]] = -size
    logits[at[5]] = -size
    logits[at[5], vocab // 2:] = -size * 1.02
    logits[at[6], vocab // 3] = size
    logits[at[7], ::7] = size
    logits[at[8], ::7] = size
    logits[at[8], 1] = size * 1.02
    near = torch.tensor(float(size), dtype=dtype, device="cuda")
    for k in range(40):                               # neighbouring values of the type: their differences count
        logits[at[9], 100 * k] = near
        logits[at[10], 100 * k] = -near
        near = torch.nextafter(near.float(), torch.tensor(0.0, device="cuda")).to(dtype) if dtype == torch.float32 else near * 0.99
    n = at.shape[0]
    conf, lse = torch.empty(n, device="cuda"), torch.empty(n, device="cuda")
    tok = torch.empty(n, device="cuda", dtype=torch.int32)
    ctx.sample_block(logits, conf, tok, lse)
    torch.cuda.synchronize()
    assert ctx.poll_status()[0] == 0
    ref_tok, ref_conf, ref_lse = sampler.block_confidence(logits.float().cpu().numpy().astype(np.float64), at)
    assert np.array_equal(tok.cpu().numpy().astype(np.int64), ref_tok)
    c, l = conf.cpu().numpy().astype(np.float64), lse.cpu().numpy().astype(np.float64)
    assert np.all(np.abs(c - ref_conf) <= 2e-5 * ref_conf), (c, ref_conf)
    assert np.all(np.abs(l - ref_lse) <= 2e-5 * np.maximum(1.0, np.abs(ref_lse))), (l, ref_lse)
    ctx.destroy()


def test_full_size_block_and_vocabulary():
    """The headline configuration's block (32 rows) and the large-batch extension's (8192 rows) at a
    vocabulary of 126464 entries (bf16 logits of every token would not fit for the latter: its logits
    array holds the block's rows of a smaller context with the same number of block rows)."""
    wl = WORKLOADS[2]
    ctx, sch = _built_ctx(wl, 3)
    g = torch.Generator(device="cuda").manual_seed(9)
    logits = (torch.randn(wl.total_tokens, 126464, generator=g, device="cuda") * 3).to(torch.bfloat16)
    _check(ctx, sch.block_rows(3), logits)
    ctx.destroy()
    wl = small_workload(name="samp-batch", prompt_lens=(3,) * 256, gen_len=64, block_len=32, steps=1, hq=2, hkv=2)
    ctx, sch = _built_ctx(wl, 0)
    rows = sch.block_rows(0)
    assert rows.shape[0] == 8192
    logits = (torch.randn(wl.total_tokens, 16384, generator=g, device="cuda") * 3).to(torch.bfloat16)
    _check(ctx, rows, logits)
    ctx.destroy()


def test_sample_needs_a_build_and_valid_arguments():
    wl = small_workload(name="samp-err", prompt_lens=(40,), gen_len=64, block_len=32, steps=1, hq=2, hkv=2)
    ctx = make_ctx(wl)
    logits = torch.zeros(wl.total_tokens, 64, device="cuda", dtype=torch.bfloat16)
    conf = torch.empty(32, device="cuda"); tok = torch.empty(32, device="cuda", dtype=torch.int32)
    with pytest.raises(binding.LacacheError) as e:
        ctx.sample_block(logits, conf, tok)
    assert e.value.status == binding.ERR_STATE
    sch = SyntheticSchedule(wl, seed=1)
    q, k, v = sch.begin_block(0)
    ctx.build(0, to_dev(q, wl), to_dev(k, wl), to_dev(v, wl))
    with pytest.raises(binding.LacacheError) as e:
        ctx.sample_block(logits, None, tok)
    assert e.value.status == binding.ERR_INVALID_ARG
    ctx.sample_block(logits, conf, tok)
    torch.cuda.synchronize()
    assert torch.equal(tok, torch.zeros_like(tok))          # all logits equal: the lowest id
    assert torch.allclose(conf, torch.full_like(conf, 1.0 / 64))
    ctx.destroy()
