"""The column-sum pass where several cuts fall on one layer, score words compared.

With fewer (unit, layer) steps than pairs of thread blocks some shares are
empty.  The fused call's scores (read from its workspace, which starts as 0xFF
bytes, so a count that is not cleared shows) must be the words prunekv_score
gives on whole units, and the kept tokens those of prunekv_select; the same for
shapes whose units are cut and none of whose shares is empty."""
import numpy as np
import pytest
import torch

from paper_2608_24063_gb300 import viscache as vc

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


def _holds(ws, words):
    """Whether the int32 words stand in the workspace at a 256-byte boundary."""
    m = words.numel()
    a = ws[:ws.numel() // 256 * 256].view(torch.int32)
    at = (a.view(-1, 64) == words[:64]).all(dim=1).nonzero().flatten() * 64
    return any(torch.equal(a[i:i + m], words) for i in at.tolist())


@pytest.mark.parametrize("L,Hkv,G,W,n", [(16, 4, 4, 64, 196), (36, 2, 8, 16, 196), (19, 1, 4, 256, 100),
                                         (16, 4, 4, 64, 256), (28, 4, 7, 64, 1500), (12, 2, 4, 30, 5000)])
def test_scores_of_cut_units_are_the_words_of_whole_units(L, Hkv, G, W, n):
    g = torch.Generator().manual_seed(L * 1000 + n)
    q, k, v = (torch.randn(L, h, m, 128, generator=g).to(torch.bfloat16).to(DEV)
               for h, m in ((G * Hkv, W), (Hkv, n), (Hkv, n)))
    scores = vc.prunekv_score(q, k)
    B, Nq, _ = vc.viscache_plan_budgets(L, n, 1, 4)
    _, keep, _ = vc.prunekv_select(scores, B, Nq)
    batch = vc.Batch([n], [W], [(1, 4)])
    prm = vc.make_params(L, G * Hkv, Hkv, 128, vc.VC_BF16)
    for _ in range(3):
        ws = torch.full((vc.prunekv_workspace_size(batch, prm),), 255, dtype=torch.uint8, device=DEV)
        _, _, idx = vc.prunekv_compress(batch, prm, q, k, v, ws=ws)
        assert np.array_equal(idx.cpu().numpy(), keep.cpu().numpy())
        assert _holds(ws, scores.view(torch.int32).flatten())
        assert vc.prunekv_get_status(ws) == vc.VC_OK
