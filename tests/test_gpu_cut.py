"""The fused pass's cuts against the step entry points' ranking.

prunekv_compress finds the elements at the cuts of the order without ranking
the rest; prunekv_select ranks every token.  Both must keep the same tokens,
exactly, on scores that crowd the cut search: all equal, few distinct values
(ties across every cut), a crowd of ties inside a spread, and token counts
from 1 to the library's limit, under both ranking modes."""
import numpy as np
import pytest
import torch

from paper_2608_24063_gb300 import viscache as vc

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


def _keys(kind, L, Hkv, n, d):
    g = torch.Generator().manual_seed(n * 7 + len(kind))
    distinct = {"equal": 1, "few": 5, "crowd": max(2, n // 2), "spread": n}[kind]
    rows = torch.randn(L, Hkv, distinct, d, generator=g)
    pick = torch.randint(0, distinct, (n,), generator=g)
    if kind == "crowd":
        pick[torch.rand(n, generator=g) < 0.6] = 0
    if kind == "spread":
        pick = torch.arange(n)
    return rows[:, :, pick].contiguous()


@pytest.mark.parametrize("mode", [vc.VC_RANK_SHARED, vc.VC_RANK_PER_LAYER], ids=["shared", "layer"])
@pytest.mark.parametrize("kind", ["spread", "equal", "few", "crowd"])
@pytest.mark.parametrize("n", [1, 2, 33, 1025, 5000, 16385, 65536])
def test_cuts_match_ranking(mode, kind, n):
    L, Hq, Hkv, d, W = 4, 4, 2, 64, 2
    K = _keys(kind, L, Hkv, n, d).to(DEV)
    V = torch.randn(L, Hkv, n, d, generator=torch.Generator().manual_seed(1)).to(DEV)
    Q = torch.randn(L, Hq, W, d, generator=torch.Generator().manual_seed(2)).to(DEV)
    num, den = (1, 1) if n < 3 else (1, 40)
    prm = vc.make_params(L, Hq, Hkv, d, vc.VC_F32, rank_mode=mode)
    try:
        B, Nq, _ = vc.viscache_plan_budgets(L, n, num, den)
    except vc.VisCacheError:
        return                                  # no budgets at this size, so no pass
    _, _, idx = vc.prunekv_compress(vc.Batch([n], [W], [(num, den)]), prm, Q, K, V)
    _, keep, _ = vc.prunekv_select(vc.prunekv_score(Q, K, rank_mode=mode), B, Nq, mode)
    assert np.array_equal(idx.cpu().numpy(), keep.cpu().numpy())


def test_every_layer_cuts_elsewhere():
    # 256 layers: 257 cuts a problem
    L, n = 256, 4000
    g = torch.Generator().manual_seed(3)
    K, V = (torch.randn(L, 1, n, 64, generator=g).to(DEV) for _ in range(2))
    Q = torch.randn(L, 1, 1, 64, generator=g).to(DEV)
    B, Nq, _ = vc.viscache_plan_budgets(L, n, 1, 5)
    _, _, idx = vc.prunekv_compress(vc.Batch([n], [1], [(1, 5)]), vc.make_params(L, 1, 1, 64, vc.VC_F32), Q, K, V)
    _, keep, _ = vc.prunekv_select(vc.prunekv_score(Q, K), B, Nq)
    assert torch.equal(idx, keep)
