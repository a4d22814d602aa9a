"""The 4-bit quantiser into code arrays of any alignment.

The header asks alignment of the float arrays only, so codes may start at any
byte: the same bytes must come out at every offset, and none outside the array."""
import pytest
import torch

from paper_2608_24063_gb300 import viscache as vc

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


@pytest.mark.parametrize("d", [64, 128])
@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16], ids=["f32", "bf16"])
@pytest.mark.parametrize("n", [1, 33, 70])
@pytest.mark.parametrize("k_at,v_at", [(0, 1), (1, 0), (2, 8), (15, 4), (1, 15)])
def test_same_codes_at_every_offset(k_at, v_at, n, dtype, d):
    L, Hkv = 2, 3
    batch = vc.Batch([n], [8], [(1, 1)])
    prm = vc.make_params(L, 6, Hkv, d, vc.VC_BF16 if dtype == torch.bfloat16 else vc.VC_F32, h=L, m=(1, 1),
                         schedule=vc.VC_SCHED_FIXED)
    rows = L * Hkv * n
    x = torch.randn(rows, d, generator=torch.Generator().manual_seed(n + d)).to(dtype)
    x[::7, ::5] = float("nan")                              # groups that take the slow decision too
    x = x.to(DEV)
    want = vc.viscache_kv4_quantize(batch, prm, x, x * 2)
    size, bufs = rows * d // 2, []
    for at in (k_at, v_at):
        buf = torch.full((size + 64,), 165, dtype=torch.uint8, device=DEV)
        assert buf.data_ptr() % 16 == 0
        bufs.append((buf, at, buf[at:at + size].view(rows, d // 2)))
    got = vc.viscache_kv4_quantize(batch, prm, x, x * 2,
                                   out=(bufs[0][2], bufs[1][2], torch.empty_like(want[2]), torch.empty_like(want[3])))
    for i in range(2):
        assert torch.equal(got[i], want[i])
        buf, at, _ = bufs[i]
        assert bool((buf[:at] == 165).all()) and bool((buf[at + size:] == 165).all())
    for a, b in zip(got[2:], want[2:]):
        assert torch.equal(a.view(torch.int32), b.view(torch.int32))
