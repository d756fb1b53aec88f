"""The rotated cache on both sides of the size from which the RoPE kernel takes several heads per thread (65536 row-head
pairs), in both engines' storage: exported rows against the rotation of Eq. 1 in fp32 with the fp64-derived table.

Tolerance.  The kernel rounds each of the two products and their sum once, as the reference below does: equal up to the last
place of the table entry (2^-24 relative of |x|), then the storage format's rounding: none (fp32), 2^-12 (one fp16 plane;
2^-25 absolute below its normal range), 2^-17 (two bf16 planes).  Values are not rotated: exact in fp32, rounded once to fp16
by the tcgen05 engine (a bf16 input below 2^-14 does not fit it exactly)."""
import pytest
import torch

from paper_2607_16339_b200 import binding

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("tokens,hq,hkv", [(2730, 8, 8), (2731, 8, 8), (4097, 12, 2)])     # 65520, 65544, 65552 pairs
@pytest.mark.parametrize("dtype,d,mode,eps", [
    (torch.float32, 64, None, 2.0 ** -23),
    (torch.float32, 128, None, 2.0 ** -23),
    (torch.bfloat16, 64, None, 2.0 ** -23),
    (torch.bfloat16, 128, binding.PRECISION_FP16, 2.0 ** -11),
    (torch.bfloat16, 128, binding.PRECISION_SPLIT, 2.0 ** -16),
])
def test_rows_on_both_sides_of_the_limit(tokens, hq, hkv, dtype, d, mode, eps):
    block, theta = 16, 1.0e4
    ctx = binding.Context(binding.DTYPE_FP32 if dtype == torch.float32 else binding.DTYPE_BF16, hq, hkv, d, theta,
                          [tokens - 1000 - 2 * block, 1000 - 2 * block], 2 * block, block,
                          **({} if mode is None else dict(precision_mode=mode)))
    assert ctx.total_tokens == tokens
    g = torch.Generator(device="cuda").manual_seed(tokens + d)
    x = [torch.randn(tokens, h, d, generator=g, device="cuda").to(dtype) for h in (hq, hkv, hkv)]
    ctx.build(0, *x)
    got = [torch.full((tokens, h, d), float("nan"), device="cuda") for h in (hq, hkv, hkv)]
    ctx.export_rope_cache(*got)
    torch.cuda.synchronize()
    assert ctx.poll_status()[0] == 0
    pos = torch.cat([torch.arange(tokens - 1000), torch.arange(1000)]).double().cuda()
    ang = pos[:, None] * theta ** (-2.0 * torch.arange(d // 2, device="cuda", dtype=torch.float64) / d)
    cs, sn = torch.cos(ang).float()[:, None], torch.sin(ang).float()[:, None]
    for t, o in zip(x[:2], got[:2]):
        a, b = t.float()[..., : d // 2], t.float()[..., d // 2:]
        ref = torch.cat([a * cs - b * sn, b * cs + a * sn], dim=-1)
        size = (a.abs() + b.abs()).repeat(1, 1, 2)
        assert bool(((o - ref).abs() <= eps * size + (2.0 ** -25 if mode == binding.PRECISION_FP16 else 0.0)).all())
    assert torch.equal(got[2], x[2].float() if mode is None else x[2].half().float())
    ctx.destroy()
