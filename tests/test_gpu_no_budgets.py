"""Passes whose budgets are all zero, alone and in a batch with others.

A retention so small that no layer keeps a token is a valid plan: the call
succeeds, writes no rows, and the other requests of a batch get what they get
alone; both rankings, tensor-core and CUDA-core paths."""
import pytest
import torch

from paper_2608_24063_gb300 import viscache as vc

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


@pytest.mark.parametrize("mode", [vc.VC_RANK_SHARED, vc.VC_RANK_PER_LAYER], ids=["shared", "layer"])
@pytest.mark.parametrize("d,dtype", [(128, torch.bfloat16), (64, torch.float32)])
@pytest.mark.parametrize("reqs", [[(2, 1)], [(2, 1), (3, 1)], [(2, 1), (600, 25)], [(600, 25), (1, 1), (40, 25)]], ids=str)
def test_requests_without_budgets(reqs, d, dtype, mode):
    L, Hq, Hkv, W = 4, 4, 2, 3
    prm = vc.make_params(L, Hq, Hkv, d, vc.VC_BF16 if dtype == torch.bfloat16 else vc.VC_F32, rank_mode=mode)
    g = torch.Generator().manual_seed(len(reqs))
    data = [[torch.randn(L, h, m, d, generator=g).to(dtype).to(DEV) for h, m in ((Hq, W), (Hkv, n), (Hkv, n))] for n, _ in reqs]

    def run(which):
        batch = vc.Batch([reqs[i][0] for i in which], [W] * len(which), [(reqs[i][1], 100) for i in which])
        ws = torch.full((vc.prunekv_workspace_size(batch, prm),), 255, dtype=torch.uint8, device=DEV)
        out = vc.prunekv_compress(batch, prm, *(torch.cat([data[i][j].reshape(-1) for i in which]) for j in range(3)), ws=ws)
        assert vc.prunekv_get_status(ws) == vc.VC_OK
        return out

    alone = [run([i]) for i in range(len(reqs))]
    for (n, rr), (k, _, idx) in zip(reqs, alone):
        B = vc.viscache_plan_budgets(L, n, rr, 100)[0]
        assert (sum(B) == 0) == (rr == 1) and k.shape[0] == idx.shape[0] == Hkv * sum(B)
    for got, parts in zip(run(range(len(reqs))), zip(*alone)):
        assert torch.equal(got, torch.cat(parts))
