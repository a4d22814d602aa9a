"""Codes of the 4-bit quantiser against the IEEE quotient, bit for bit, where
the branch-free decision could go wrong: values one unit in the last place
around the half-integers, groups of one value, scales from subnormal to the
largest, infinities and NaN (code 0), and short last groups."""
import pytest
import torch

from paper_2608_24063_gb300 import viscache as vc

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


def _codes(x, scale, lo):
    """clamp(rint((x - lo) / scale), 0, 15) in fp32; 0 for a NaN or a scale that is not positive."""
    t = torch.round((x - lo) / scale)
    t = torch.where(torch.isnan(t), torch.zeros_like(t), t.clamp(0, 15))
    return torch.where(scale > 0, t, torch.zeros_like(t)).to(torch.uint8)


def _unpack(c):
    return torch.stack([c & 15, c >> 4], dim=-1).reshape(c.shape[0], -1)


@pytest.mark.parametrize("d", [64, 128])
@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16], ids=["f32", "bf16"])
@pytest.mark.parametrize("n", [1, 31, 32, 33, 100])
def test_codes_equal_the_ieee_quotient(n, dtype, d):
    L, Hkv = 3, 2
    batch = vc.Batch([n], [8], [(1, 1)])
    prm = vc.make_params(L, 4, Hkv, d, vc.VC_BF16 if dtype == torch.bfloat16 else vc.VC_F32, h=L, m=(1, 1),
                         schedule=vc.VC_SCHED_FIXED)
    rows = L * Hkv * n
    g = torch.Generator().manual_seed(n + d)
    k = torch.randint(0, 15, (rows, d), generator=g)
    x = (k + 0.5) / 15                                      # near the half-integers of a group over [0, 1]
    x = torch.nextafter(x, x + torch.randint(-1, 2, x.shape, generator=g))
    x[torch.rand(x.shape, generator=g) < 0.1] = 0.0
    x[torch.rand(x.shape, generator=g) < 0.1] = 1.0
    seg = torch.arange(rows) // n
    x[seg == 1] = x[seg == 1] * 2.0 - 3.0
    x[seg == 2] = torch.randn(int((seg == 2).sum()), d, generator=g) * 3e37
    x[seg == 3] = torch.randn(int((seg == 3).sum()), d, generator=g) * 1e-38
    x[seg == 4] = 0.75                                      # one value: scale 0
    bad = torch.rand(x.shape, generator=g) < 0.02           # segment 5: infinities and NaN among numbers
    sp = torch.tensor([float("nan"), float("inf"), -float("inf")])[torch.randint(0, 3, x.shape, generator=g)]
    x = torch.where(bad & (seg == 5)[:, None], sp, x).to(dtype)
    kc, vcodes, kp, vp = (t.cpu() for t in vc.viscache_kv4_quantize(batch, prm, x.to(DEV), x.to(DEV)))
    xf = x.float()
    vp = vp.reshape(rows, d // 32, 2).repeat_interleave(32, dim=1)
    assert torch.equal(_unpack(vcodes.reshape(rows, -1)), _codes(xf, vp[..., 0], vp[..., 1]))
    nb = (n + 31) // 32
    kp = kp.reshape(L * Hkv, nb, d, 2).repeat_interleave(32, dim=1)[:, :n].reshape(rows, d, 2)
    assert torch.equal(_unpack(kc.reshape(rows, -1)), _codes(xf, kp[..., 0], kp[..., 1]))


@pytest.mark.parametrize("d", [64, 128])
@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16], ids=["f32", "bf16"])
@pytest.mark.parametrize("n", [1, 7, 33, 65])
@pytest.mark.parametrize("shift", [0, 1, 2])
def test_codes_of_any_alignment_give_the_same_values(shift, n, dtype, d):
    L, Hkv = 2, 3
    batch = vc.Batch([n], [8], [(1, 1)])
    prm = vc.make_params(L, 6, Hkv, d, vc.VC_BF16 if dtype == torch.bfloat16 else vc.VC_F32, h=L, m=(1, 1),
                         schedule=vc.VC_SCHED_FIXED)
    rows = L * Hkv * n
    g = torch.Generator().manual_seed(n)
    x = torch.randn(rows, d, generator=g).to(dtype).to(DEV)
    kc, vcodes, kp, vp = vc.viscache_kv4_quantize(batch, prm, x, x * 2)

    def moved(t):
        buf = torch.empty(t.numel() + 16, dtype=t.dtype, device=DEV)
        buf[shift:shift + t.numel()] = t.reshape(-1)
        return buf[shift:shift + t.numel()].view(t.shape)

    kh, vh = vc.viscache_kv4_dequantize(batch, prm, moved(kc), moved(vcodes), kp, vp, dtype=dtype)
    s = kp.reshape(L * Hkv, (n + 31) // 32, d, 2).repeat_interleave(32, dim=1)[:, :n].reshape(rows, d, 2).double()
    want = (_unpack(kc.reshape(rows, -1)).double() * s[..., 0] + s[..., 1]).float().to(dtype)
    assert torch.equal(kh.reshape(rows, d), want)
    s = vp.reshape(rows, d // 32, 2).repeat_interleave(32, dim=1).double()
    want = (_unpack(vcodes.reshape(rows, -1)).double() * s[..., 0] + s[..., 1]).float().to(dtype)
    assert torch.equal(vh.reshape(rows, d), want)
