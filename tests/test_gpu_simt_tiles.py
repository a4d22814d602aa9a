"""The CUDA-core passes' small and large tiles against each other, bit for bit.

One short request takes the tiles of 8 rows and 32 keys, a batch of many the
tiles of 32 rows and 64 keys; every row's and key's arithmetic is the same, so
each request of a batch must give the bits it gives alone: row counts around
the tiles (one row, odd sets), key counts around 32 and 64, both head sizes and
types, both ranking modes."""
import pytest
import torch

from paper_2608_24063_gb300 import viscache as vc

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


@pytest.mark.parametrize("mode", [vc.VC_RANK_SHARED, vc.VC_RANK_PER_LAYER], ids=["shared", "layer"])
@pytest.mark.parametrize("d,dtype", [(64, torch.float32), (128, torch.float32), (64, torch.bfloat16)])
@pytest.mark.parametrize("L,n,W", [(1, 33, 1), (2, 63, 5), (3, 64, 7), (1, 65, 16), (2, 97, 11), (1, 300, 23)])
def test_batch_equals_single(mode, d, dtype, L, n, W):
    Hq, Hkv, copies = 6, 2, 320
    g = torch.Generator().manual_seed(100 * n + d)
    q = torch.randn(L, Hq, W, d, generator=g).to(dtype).to(DEV)
    k = torch.randn(L, Hkv, n, d, generator=g).to(dtype).to(DEV)
    v = torch.randn(L, Hkv, n, d, generator=g).to(dtype).to(DEV)
    prm = vc.make_params(L, Hq, Hkv, d, vc.VC_F32 if dtype == torch.float32 else vc.VC_BF16, rank_mode=mode)

    def run(c):
        batch = vc.Batch([n] * c, [W] * c, [(1, 4)] * c)
        return vc.prunekv_compress(batch, prm, q.reshape(-1).repeat(c), k.reshape(-1).repeat(c), v.reshape(-1).repeat(c))

    one, many = run(1), run(copies)
    for a, b in zip(one, many):
        a, b = a.reshape(-1), b.reshape(-1)
        assert b.numel() == copies * a.numel()
        for i in (0, 1, copies - 1):
            assert torch.equal(a, b[i * a.numel():(i + 1) * a.numel()])
    idx = one[2].long()
    rows = k.reshape(L, Hkv, n, d)
    B, _, _ = vc.viscache_plan_budgets(L, n, 1, 4)
    o = 0
    for l in range(L):
        for h in range(Hkv):
            keep = idx[o:o + int(B[l])]
            assert torch.equal(one[0].reshape(-1, d)[o:o + int(B[l])], rows[l, h][keep])
            o += int(B[l])
