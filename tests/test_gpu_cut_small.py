"""The fused pass's cuts at the smallest token counts.

From one token on, with budgets that exist there (a fixed schedule, all layers
kept at ratio 1/1, or one layer of the parabola), the fused pass keeps what the
step entry points keep; ties and spread scores, both ranking modes, and the
CUDA-core and tensor-core passes."""
import numpy as np
import pytest
import torch

from paper_2608_24063_gb300 import viscache as vc

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


@pytest.mark.parametrize("mode", [vc.VC_RANK_SHARED, vc.VC_RANK_PER_LAYER], ids=["shared", "layer"])
@pytest.mark.parametrize("equal", [False, True], ids=["spread", "equal"])
@pytest.mark.parametrize("d,dtype", [(64, torch.float32), (128, torch.bfloat16)])
@pytest.mark.parametrize("n", [1, 2, 3, 5, 16, 31, 32])
@pytest.mark.parametrize("rr", [(1, 1), (1, 2)], ids=["all", "half"])
def test_smallest_counts(rr, n, d, dtype, equal, mode):
    L, Hq, Hkv, W = 3, 4, 2, 2
    g = torch.Generator().manual_seed(n)
    k = torch.randn(L, Hkv, n, d, generator=g)
    if equal:
        k = k[:, :, :1].expand(L, Hkv, n, d).contiguous()
    q, v = torch.randn(L, Hq, W, d, generator=g), torch.randn(L, Hkv, n, d, generator=g)
    q, k, v = (x.to(dtype).to(DEV) for x in (q, k, v))
    h, m, sched = L, (1, 1), vc.VC_SCHED_FIXED
    prm = vc.make_params(L, Hq, Hkv, d, vc.VC_F32 if dtype == torch.float32 else vc.VC_BF16, h=h, m=m, rank_mode=mode,
                         schedule=sched)
    B, Nq, _ = vc.viscache_plan_budgets_ex(L, n, rr[0], rr[1], h, m[0], m[1], sched)
    assert sum(B) > 0
    Ko, Vo, idx = vc.prunekv_compress(vc.Batch([n], [W], [rr]), prm, q, k, v)
    _, keep, drop = vc.prunekv_select(vc.prunekv_score(q, k, rank_mode=mode), B, Nq, mode)
    assert np.array_equal(idx.cpu().numpy(), keep.cpu().numpy())
    if rr == (1, 1):
        assert idx.cpu().tolist() == list(range(n)) * (L * Hkv)
    K2, V2 = vc.prunekv_fuse_compact(k, v, B, Nq, keep, drop)
    assert torch.equal(Ko, K2) and torch.equal(Vo, V2)
