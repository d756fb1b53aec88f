"""The fp32 engine's products, which run as products of bf16 parts that hold all bits of their operands: values that three parts do
not hold (infinities, NaN, the largest finite ones) give what fp32 arithmetic gives, in the rows and features they reach and in no other;
the range is that of fp32; and the results stay as close to fp64 as fp32 sums are, at sizes around a tile of 32 rows or keys."""
import numpy as np
import pytest
import torch

import oracle
from paper_2607_16339_b200 import binding
from paper_2607_16339_b200.workloads import SyntheticSchedule, small_workload

from lacache_testlib import make_ctx, new_outputs, to_dev

pytestmark = pytest.mark.gpu


def _run(wl, q, k, v, blk=None):
    """full recompute; and build + step of block 0 with the block's own rows"""
    ctx = make_ctx(wl)
    assert ctx.engine == binding.ENGINE_SIMT
    got = [new_outputs(wl), new_outputs(wl)]
    dq, dk, dv = (to_dev(a, wl) for a in (q, k, v))
    ctx.full_recompute(dq, dk, dv, *got[0])
    rows = torch.from_numpy(SyntheticSchedule(wl).block_rows(0)).cuda().long()
    ctx.build(0, dq, dk, dv)
    ctx.step(dq[rows].contiguous(), dk[rows].contiguous(), dv[rows].contiguous(), *got[1])
    torch.cuda.synchronize()
    assert ctx.poll_status()[0] == 0
    ctx.destroy()
    return [(o.cpu().numpy().astype(np.float64), l.cpu().numpy().astype(np.float64)) for o, l in got]


@pytest.mark.parametrize("value", [np.inf, -np.inf, np.nan, 3.4028235e38, -3.4e38])
@pytest.mark.parametrize("d", [64, 128])
def test_values_that_two_parts_do_not_hold(value, d):
    wl = small_workload(name="products", dtype="fp32", prompt_lens=(45, 30), gen_len=64, block_len=32, steps=2, hq=4, hkv=2, d=d,
                        scale_mode="inv_sqrt_d")
    sch = SyntheticSchedule(wl, seed=4)
    q, k, v = (np.array(a) for a in sch.begin_block(0))
    want, wlse = oracle.attention(q, k, v, wl.cu_seqlens, wl.rope_theta, d ** -0.5)
    tok, kh, f = 7, 1, 5                                   # a prompt token of the first sequence
    v[tok, kh, f] = value
    for out, lse in _run(wl, q, k, v):
        assert np.abs(lse - wlse).max() <= 1e-5
        hit = np.zeros(out.shape, bool)
        hit[wl.cu_seqlens[0]:wl.cu_seqlens[1], 2 * kh:2 * kh + 2, f] = True
        assert np.abs(out - want)[~hit].max() <= 1e-5       # every other row and feature: as without it
        if np.isnan(value):
            assert np.isnan(out[hit]).all()
        elif np.isinf(value):
            assert (out[hit] == value).all()
        else:                                               # p / l of the largest value: the weights are about 1 / n
            n = wl.cu_seqlens[1] - wl.cu_seqlens[0]
            assert (np.abs(out[hit] / value * n - 1) < 0.2).all()


def _exact(q, k, v, wl):
    """softmax(q k^T) v in fp64 with IEEE rules: a row that meets a NaN or a score of +inf is NaN, a score of -inf weighs nothing."""
    half, g = wl.head_dim // 2, wl.n_q_heads // wl.n_kv_heads
    f = wl.rope_theta ** (-np.arange(half) / half)
    outs = []
    for lo, hi in zip(wl.cu_seqlens, wl.cu_seqlens[1:]):
        c, s = (fn(np.arange(hi - lo)[:, None] * f)[:, None] for fn in (np.cos, np.sin))
        rot = lambda x: np.concatenate([x[..., :half] * c - x[..., half:] * s, x[..., half:] * c + x[..., :half] * s], -1)
        qq, kk, vv = rot(q[lo:hi].astype(np.float64)), rot(k[lo:hi].astype(np.float64)), v[lo:hi].astype(np.float64)
        sc = np.einsum("ihd,jhd->hij", qq, np.repeat(kk, g, 1)) * wl.head_dim ** -0.5
        p = np.exp(sc - sc.max(-1, keepdims=True))
        outs.append(np.einsum("hij,jhd->ihd", p / p.sum(-1, keepdims=True), np.repeat(vv, g, 1)))
    return np.concatenate(outs)


@pytest.mark.parametrize("value", [np.inf, -np.inf, np.nan])
@pytest.mark.parametrize("which", ["q", "k"])
@pytest.mark.parametrize("d", [64, 128])
def test_queries_and_keys_that_two_parts_do_not_hold(value, which, d):
    wl = small_workload(name="products", dtype="fp32", prompt_lens=(45, 30), gen_len=64, block_len=32, steps=2, hq=4, hkv=2, d=d,
                        scale_mode="inv_sqrt_d")
    q, k, v = (np.array(a) for a in SyntheticSchedule(wl, seed=4).begin_block(0))
    for tok in (7, 45 + 20):                               # a prompt token of the first sequence, and one of its block
        q2, k2 = q.copy(), k.copy()
        (q2 if which == "q" else k2)[tok, 1, 5] = value
        with np.errstate(invalid="ignore"):
            want = _exact(q2, k2, v, wl)
        assert np.isnan(want).any() and not np.isnan(want[wl.cu_seqlens[1]:]).any()
        for out, _ in _run(wl, q2, k2, v):
            assert np.array_equal(np.isnan(out), np.isnan(want))
            assert np.nanmax(np.abs(out - want)) <= 1e-5


@pytest.mark.parametrize("value", [np.nan, np.inf])
@pytest.mark.parametrize("prompts,block", [((50, 1), 32), ((45, 30), 32), ((3, 40), 16), ((33, 70), 64)])
@pytest.mark.parametrize("d", [64, 128])
def test_rows_of_another_sequence(prompts, block, value, d):
    """A sequence's rows, whatever they hold, reach no other: its last key tile ends where the next one's rows (in a step, rows that are just
    being written) begin, and its results are the same bits whether those are numbers or not."""
    wl = small_workload(name="products", dtype="fp32", prompt_lens=prompts, gen_len=64, block_len=block, steps=2, hq=4, hkv=2, d=d,
                        scale_mode="inv_sqrt_d")
    q, k, v = (np.array(a) for a in SyntheticSchedule(wl, seed=4).begin_block(0))
    n = wl.cu_seqlens[1]
    clean = _run(wl, q, k, v)
    q[n:], k[n:], v[n:] = value, value, value
    for (o0, l0), (o1, l1) in zip(clean, _run(wl, q, k, v)):
        assert np.array_equal(o0[:n], o1[:n]) and np.array_equal(l0[:n], l1[:n])
        assert np.isnan(o1[n:]).all()


@pytest.mark.parametrize("first,block", [(0, 32), (1, 32), (0, 16), (0, 64)])
@pytest.mark.parametrize("d", [64, 128])
def test_rows_of_the_excluded_block(first, block, d):
    """A build leaves the block's own rows out: what it is given for them reaches neither the cached state nor the steps."""
    wl = small_workload(name="products", dtype="fp32", prompt_lens=(45, 30), gen_len=64, block_len=block, steps=2, hq=4, hkv=2, d=d,
                        scale_mode="inv_sqrt_d")
    if (first + 1) * block > 64:
        pytest.skip("no such block")
    q, k, v = (np.array(a) for a in SyntheticSchedule(wl, seed=4).begin_block(0))
    rows = torch.from_numpy(SyntheticSchedule(wl).block_rows(first)).cuda().long()
    blk = [to_dev(x, wl)[rows].contiguous() for x in (q, k, v)]
    got = []
    for value in (0.0, np.nan):
        for x in (q, k, v):
            x[rows.cpu().numpy()] = value
        ctx, (out, lse) = make_ctx(wl), new_outputs(wl)
        ctx.build(first, *(to_dev(x, wl) for x in (q, k, v)))
        ctx.step(*blk, out, lse)
        got.append((out.cpu().numpy(), lse.cpu().numpy()))
        ctx.destroy()
    assert np.isfinite(got[0][0]).all()
    assert np.abs(got[0][0] - got[1][0]).max() <= 1e-5 and np.abs(got[0][1] - got[1][1]).max() <= 1e-5


@pytest.mark.parametrize("n", [33, 70])
def test_words_left_by_an_earlier_call(n):
    """The static call reads none of its scratch that it has not written: the same bits before and after a longer call of NaN."""
    g = torch.Generator().manual_seed(3)
    q, k, v = (torch.randn(200, 2, 64, generator=g).cuda() for _ in range(3))
    out, lse = torch.empty(200, 2, 64, device="cuda"), torch.empty(200, 2, device="cuda")

    def call(m, *rows):
        binding.full_recompute_static(binding.DTYPE_FP32, 2, 2, 64, 1e4, *(x[:m].contiguous() for x in rows), out[:m], lse[:m])
        torch.cuda.synchronize()
        return out[:m].clone(), lse[:m].clone()
    call(200, *(torch.zeros_like(x) for x in (q, k, v)))
    before = call(n, q, k, v)
    call(200, *(torch.full_like(x, float("nan")) for x in (q, k, v)))
    after = call(n, q, k, v)
    assert torch.isfinite(before[0]).all()
    assert torch.equal(before[0], after[0]) and torch.equal(before[1], after[1])


def test_cost_of_plain_products():
    """Units that are done once more with plain products: a build and a step where all of them are take no more than a few times as long
    (1351 us for 343 and 107 for 49 measured; 10900 and 684 where every thread took its values one at a time)."""
    wl = small_workload(name="products", dtype="fp32", prompt_lens=(2500,), gen_len=64, block_len=32, steps=2, hq=4, hkv=4, d=128,
                        scale_mode="inv_sqrt_d")
    q, k, v = (np.array(a) for a in SyntheticSchedule(wl, seed=4).begin_block(0))
    ctx, (out, lse) = make_ctx(wl), new_outputs(wl)
    rows = torch.from_numpy(SyntheticSchedule(wl).block_rows(0)).cuda().long()
    took = []
    for value in (0.0, np.nan):
        v[3, :, 5] = value
        dq, dk, dv = (to_dev(a, wl) for a in (q, k, v))
        blk = [x[rows].contiguous() for x in (dq, dk, dv)]
        for call in (lambda: ctx.build(0, dq, dk, dv), lambda: ctx.step(*blk, out, lse)):
            ts = []
            for _ in range(12):
                a, e = (torch.cuda.Event(enable_timing=True) for _ in range(2))
                a.record()
                call()
                e.record()
                torch.cuda.synchronize()
                ts.append(a.elapsed_time(e))
            took.append(sorted(ts)[6])
    ctx.destroy()
    assert took[2] <= 10 * took[0] and took[3] <= 6 * took[1], took


def test_the_range_is_that_of_fp32():
    """q and k scaled by powers of two that cancel: the same bits."""
    wl = small_workload(name="products", dtype="fp32", prompt_lens=(45, 30), gen_len=64, block_len=32, steps=2, hq=4, hkv=4, d=128,
                        scale_mode="inv_sqrt_d")
    q, k, v = (np.array(a) for a in SyntheticSchedule(wl, seed=5).begin_block(0))
    a = _run(wl, q, k, v)
    b = _run(wl, q * np.float32(2.0 ** -90), k * np.float32(2.0 ** 90), v)
    for (o0, l0), (o1, l1) in zip(a, b):
        assert np.array_equal(o0, o1) and np.array_equal(l0, l1)


def _rotated32(x, wl):
    """rows rotated as the fp32 engine does it, every product and sum rounded: what is left of an output's error is the attention's"""
    half = wl.head_dim // 2
    f = np.array([wl.rope_theta ** (-2.0 * c / wl.head_dim) for c in range(half)])
    y = np.empty_like(x)
    for lo, hi in zip(wl.cu_seqlens, wl.cu_seqlens[1:]):
        c, s = (fn(np.arange(hi - lo)[:, None] * f).astype(np.float32)[:, None] for fn in (np.cos, np.sin))
        a, b = x[lo:hi, :, :half], x[lo:hi, :, half:]
        y[lo:hi] = np.concatenate([a * c - b * s, b * c + a * s], -1)
    return y


def _attention64(q, k, v, wl):
    """output and log-sum-exp of rotated rows in fp64"""
    g, outs, lses = wl.n_q_heads // wl.n_kv_heads, [], []
    for lo, hi in zip(wl.cu_seqlens, wl.cu_seqlens[1:]):
        qq, kk, vv = (x[lo:hi].astype(np.float64) for x in (q, k, v))
        sc = np.einsum("ihd,jhd->hij", qq, np.repeat(kk, g, 1)) * wl.head_dim ** -0.5
        m = sc.max(-1, keepdims=True)
        p = np.exp(sc - m)
        outs.append(np.einsum("hij,jhd->ihd", p / p.sum(-1, keepdims=True), np.repeat(vv, g, 1)))
        lses.append((m[..., 0] + np.log(p.sum(-1))).T)
    return np.concatenate(outs), np.concatenate(lses)


def _gauss(wl, seed):
    rng = np.random.default_rng(seed)
    return [rng.standard_normal((wl.total_tokens, h, wl.head_dim)).astype(np.float32) for h in (wl.n_q_heads, wl.n_kv_heads, wl.n_kv_heads)]


def _model(d, prompts=(137, 61)):
    return small_workload(name="products", dtype="fp32", prompt_lens=prompts, gen_len=64, block_len=32, steps=2, hq=4, hkv=2, d=d,
                          scale_mode="inv_sqrt_d")


def _error_of_rounded_scores(q, k, v, wl):
    """What an output is off by, relative and in the mean, where every score is rounded four times: as the sum of two features' products
    (twice), with the scale, and as the difference to the row's maximum.  A rounding to 24 bits is off by 2^-24 / sqrt(3) of the power of two
    below the value; a score's error moves the output by its weight times its value's distance from the output."""
    g, err, norm = wl.n_q_heads // wl.n_kv_heads, 0.0, 0.0
    def rounding(x):
        return np.exp2(np.floor(np.log2(np.maximum(np.abs(x), 1e-300)))) * 2.0 ** -24 / 3 ** 0.5
    for lo, hi in zip(wl.cu_seqlens, wl.cu_seqlens[1:]):
        qq, kk, vv = (x[lo:hi].astype(np.float64) for x in (q, k, v))
        vv = np.repeat(vv, g, 1).transpose(1, 0, 2)
        sc = np.einsum("ihd,jhd->hij", qq, np.repeat(kk, g, 1)) * wl.head_dim ** -0.5 / np.log(2)
        top = sc.max(-1, keepdims=True)
        p = np.exp2(sc - top)
        p /= p.sum(-1, keepdims=True)
        out = p @ vv
        w = p ** 2 * (3 * rounding(sc) ** 2 + rounding(sc - top) ** 2) * np.log(2) ** 2
        err += (w.sum(-1) * (out ** 2).sum(-1) + np.einsum("hij,hj->hi", w, (vv ** 2).sum(-1)) - 2 * ((w @ vv) * out).sum(-1)).sum()
        norm += (out ** 2).sum()
    return (err / norm) ** 0.5


@pytest.mark.parametrize("where", ["first", "middle", "last"])
@pytest.mark.parametrize("d", [64, 128])
def test_scores_of_one_feature(where, d):
    """A score of which one feature (and the one it turns with) is all there is: every rounding of a product shows.  Operands of 22 bits
    are off by twice the sum's own roundings; the bound leaves three tenths for what else is rounded (weights, sums over keys)."""
    wl = _model(d)
    f = {"first": 0, "middle": d // 2 - 1, "last": d - 1}[where]
    for seed in range(4):
        q, k, v = _gauss(wl, seed)
        for x in (q, k):
            x[..., :f], x[..., f + 1:] = 0, 0
            x *= 8
        qr, kr = _rotated32(q, wl), _rotated32(k, wl)
        want, _ = _attention64(qr, kr, v, wl)
        most = 1.3 * _error_of_rounded_scores(qr, kr, v, wl)
        for out, _ in _run(wl, q, k, v):
            print(where, d, np.linalg.norm(out - want) / np.linalg.norm(want) / most)
            assert np.linalg.norm(out - want) <= most * np.linalg.norm(want)


@pytest.mark.parametrize("d", [64, 128])
def test_one_key_gives_its_value(d):
    """A row whose weight is all one key's returns that key's value, to the last bit."""
    wl = _model(d)
    q, k, v = _gauss(wl, 9)
    q[:], k[:] = 0, 0
    q[..., d - 1] = 64
    k[..., d - 1] = -64                                     # scores of -512 and less, but
    for lo in wl.cu_seqlens[:-1]:
        k[lo + 5, :, d - 1] = 64                            # one of +512 and less (the last feature turns by 1e-2 at most)
    for out, lse in _run(wl, q, k, v):
        for lo, hi in zip(wl.cu_seqlens, wl.cu_seqlens[1:]):
            assert np.array_equal(out[lo:hi], np.repeat(np.repeat(v[lo + 5:lo + 6], 2, 1), hi - lo, 0).astype(np.float64))


@pytest.mark.parametrize("eq,ek", [(-120, 120), (-126, 120), (-100, 60), (90, -110), (120, -120)])
@pytest.mark.parametrize("d", [64, 128])
def test_scores_of_tiny_and_huge_rows(eq, ek, d):
    """queries and keys scaled apart by powers of two, down to where parts of a split value, or the value, are subnormal: the error
    stays that of fp32 sums (the bound of the test at the end of this file), but for what the smaller side's values, which are
    multiples of 2^-149, lose themselves: the reference has the scaled values."""
    wl = _model(d, (45, 30))
    q, k, v = _gauss(wl, 5)
    q, k = q * np.float32(d ** -0.5 * 2.0 ** (-(eq + ek) // 2)), k * np.float32(d ** -0.5 * 2.0 ** ((eq + ek) // 2 - (eq + ek)))
    q, k = np.ldexp(q, eq), np.ldexp(k, ek)
    want, wlse = _attention64(_rotated32(q, wl), _rotated32(k, wl), v, wl)
    for out, lse in _run(wl, q, k, v):
        assert np.linalg.norm(out - want) <= 4.5e-7 * np.linalg.norm(want)
        assert np.abs(lse - wlse).max() <= 2e-6


@pytest.mark.parametrize("exponent", [126, 130, 140])
@pytest.mark.parametrize("d", [64, 128])
def test_subnormal_values(exponent, d):
    """values that are subnormal themselves: as close as fp32 sums, and within four roundings of a subnormal result (the two halves of a
    tile's keys, the parts of a unit, the cached state, the division: half of 2^-149 each at most)."""
    wl = _model(d, (45, 30))
    q, k, v = _gauss(wl, 6)
    q, k, v = q * np.float32(d ** -0.5), k * np.float32(d ** -0.5), np.ldexp(v, -exponent)
    want, _ = _attention64(_rotated32(q, wl), _rotated32(k, wl), v, wl)
    assert np.abs(want).max() > 2.0 ** -149
    for out, _ in _run(wl, q, k, v):
        assert (np.abs(out - want) <= 4 * 2.0 ** -149 + 2e-6 * np.abs(want).max()).all()


@pytest.mark.parametrize("d", [64, 128])
def test_tiny_probabilities(d):
    """Weights of about 2^-125 beside one of 1 whose value is zero: the result is theirs alone.  Their scores, 125 in the exponent's
    units, are rounded to 2^-17 at worst three times (the feature's product, the scale, the difference to the maximum), a weight by 2^-18.5
    ln 2 a time in the mean; the bound leaves three times that."""
    wl = _model(d, (45, 30))
    q, k, v = _gauss(wl, 7)
    q[:], k[:] = 0, 0
    q[..., d - 1] = 1
    rng = np.random.default_rng(8)
    k[..., d - 1] = -(86 + 0.5 * rng.random(k.shape[:2])) * d ** 0.5
    v = np.ldexp(v, 100)
    for lo in wl.cu_seqlens[:-1]:
        k[lo + 5, :, d - 1] = 0
        v[lo + 5] = 0
    want, _ = _attention64(_rotated32(q, wl), _rotated32(k, wl), v, wl)
    for out, _ in _run(wl, q, k, v):
        assert np.linalg.norm(out - want) <= 3 * 3 ** 0.5 * 2.0 ** -18.5 * np.log(2) * np.linalg.norm(want)


@pytest.mark.parametrize("exponent", [60, 108, 116, 122])
def test_tiny_values_keep_their_bits(exponent):
    """v scaled by a power of two down to where the low part of a split value is subnormal: the result scales with it, within the
    rounding of sums taken in another order (and of subnormal results, at most 2^-149 a value of 2^-125)."""
    wl = small_workload(name="products", dtype="fp32", prompt_lens=(45, 30), gen_len=64, block_len=32, steps=2, hq=4, hkv=4, d=128,
                        scale_mode="inv_sqrt_d")
    q, k, v = (np.array(a) for a in SyntheticSchedule(wl, seed=5).begin_block(0))
    s = 2.0 ** -exponent
    for (o0, l0), (o1, l1) in zip(_run(wl, q, k, v), _run(wl, q, k, v * np.float32(s))):
        assert np.linalg.norm(o1 / s - o0) <= 1e-6 * np.linalg.norm(o0)
        assert np.abs(l1 - l0).max() <= 2e-6      # (the order of the sums)


@pytest.mark.parametrize("prompts,gen,block", [((1,), 32, 32), ((31, 33), 32, 16), ((95, 64, 7), 64, 64), ((260,), 96, 48)])
@pytest.mark.parametrize("d", [64, 128])
def test_as_close_to_fp64_as_fp32_sums(prompts, gen, block, d):
    """Relative error (2-norm) of the output.  A sum of n fp32 products in a chain is off by about 2^-24 sqrt(n / 6) of itself, 4e-7 at 350
    keys; here a product is cut at 2^-22 (2^-24 in the mean) and sums are cut off over two steps at a time: 1.4e-7 measured, for
    chains on the CUDA cores 1.35e-7; the bound leaves three times that."""
    wl = small_workload(name="products", dtype="fp32", prompt_lens=prompts, gen_len=gen, block_len=block, steps=2, hq=4, hkv=2, d=d,
                        scale_mode="inv_sqrt_d")
    q, k, v = (np.array(a) for a in SyntheticSchedule(wl, seed=6).begin_block(0))
    want, wlse = oracle.attention(q, k, v, wl.cu_seqlens, wl.rope_theta, d ** -0.5)
    for out, lse in _run(wl, q, k, v):
        assert np.linalg.norm(out - want) <= 4.5e-7 * np.linalg.norm(want)
        assert np.abs(lse - wlse).max() <= 2e-6
