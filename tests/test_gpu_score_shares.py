"""The column-sum pass cut into shares against whole units, bit for bit.

The fused pass cuts the (unit, layer) sequence into equal shares and adds the
layers of a cut unit afterwards; prunekv_score walks whole units.  The scores
must be the same bits, so the kept tokens must be: key counts around the
256-key units, one to many layers, window-row sets of one to five chunks
(odd counts too), both ranking modes, and batches of unequal requests."""
import numpy as np
import pytest
import torch

from paper_2608_24063_gb300 import viscache as vc

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


def _check(L, Hq, Hkv, reqs, mode):
    g = torch.Generator().manual_seed(len(reqs) * 1000 + reqs[0][0] + L)
    qs, ks, vs, want = [], [], [], []
    for n, W in reqs:
        q = torch.randn(L, Hq, W, 128, generator=g).to(torch.bfloat16).to(DEV)
        k = torch.randn(L, Hkv, n, 128, generator=g).to(torch.bfloat16).to(DEV)
        v = torch.randn(L, Hkv, n, 128, generator=g).to(torch.bfloat16).to(DEV)
        B, Nq, _ = vc.viscache_plan_budgets(L, n, 1, 4)
        _, keep, _ = vc.prunekv_select(vc.prunekv_score(q, k, rank_mode=mode), B, Nq, mode)
        qs.append(q.reshape(-1))
        ks.append(k.reshape(-1))
        vs.append(v.reshape(-1))
        want.append(keep)
    prm = vc.make_params(L, Hq, Hkv, 128, vc.VC_BF16, rank_mode=mode)
    batch = vc.Batch([n for n, _ in reqs], [w for _, w in reqs], [(1, 4)] * len(reqs))
    _, _, idx = vc.prunekv_compress(batch, prm, torch.cat(qs), torch.cat(ks), torch.cat(vs))
    assert np.array_equal(idx.cpu().numpy(), torch.cat(want).cpu().numpy())


@pytest.mark.parametrize("mode", [vc.VC_RANK_SHARED, vc.VC_RANK_PER_LAYER], ids=["shared", "layer"])
@pytest.mark.parametrize("L,n,W", [(1, 300, 16), (2, 255, 5), (4, 257, 64), (9, 1000, 33), (28, 700, 64), (28, 3000, 17),
                                   (28, 5121, 64), (40, 513, 150), (7, 20000, 20)])
def test_shares_equal_whole_units(mode, L, n, W):
    _check(L, 28, 4, [(n, W)], mode)


@pytest.mark.parametrize("mode", [vc.VC_RANK_SHARED, vc.VC_RANK_PER_LAYER], ids=["shared", "layer"])
def test_shares_of_a_batch_equal_whole_units(mode):
    _check(12, 8, 2, [(900, 10), (4000, 90), (256, 130), (2300, 33)], mode)
    _check(3, 4, 1, [(40, 1), (17, 3), (600, 64)], mode)
