"""A captured call whose plan tables exceed the upload kernel's parameter.

The graph must hold the tables themselves, not a pointer into the call's host
memory: it is replayed on other values, after other calls have used that memory,
and must give what direct calls give."""
import pytest
import torch

from paper_2608_24063_gb300 import viscache as vc

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


@pytest.mark.parametrize("d,dtype", [(128, torch.bfloat16), (64, torch.float32)])
@pytest.mark.parametrize("n_req", [40, 70])
def test_replays_equal_direct_calls(n_req, d, dtype):
    L, Hq, Hkv = 28, 4, 2
    ns = [100 + 7 * (i % 13) for i in range(n_req)]
    batch = vc.Batch(ns, [4] * n_req, [(1, 4)] * n_req)
    prm = vc.make_params(L, Hq, Hkv, d, vc.VC_BF16 if dtype == torch.bfloat16 else vc.VC_F32)
    g = torch.Generator().manual_seed(n_req)
    new = lambda rows: torch.randn(rows, d, generator=g).to(dtype).to(DEV)
    sizes = n_req * L * Hq * 4, L * Hkv * sum(ns), L * Hkv * sum(ns)
    first, second = ([new(r) for r in sizes] for _ in range(2))
    want = [[x.clone() for x in vc.prunekv_compress(batch, prm, *v)] for v in (first, second)]
    ws = torch.full((vc.prunekv_workspace_size(batch, prm),), 255, dtype=torch.uint8, device=DEV)
    args = [x.clone() for x in first]
    out = [torch.empty_like(x) for x in want[0]]
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        vc.prunekv_compress(batch, prm, *args, *out, ws=ws)
    other = vc.Batch([50] * 90, [3] * 90, [(1, 2)] * 90)    # calls that use the host's memory again
    for _ in range(3):
        vc.prunekv_workspace_size(other, prm)
    for values, ref in ((second, want[1]), (first, want[0])):
        for a, v in zip(args, values):
            a.copy_(v)
        ws[256:].fill_(255)
        graph.replay()
        assert vc.prunekv_get_status(ws) == vc.VC_OK
        assert all(torch.equal(a, b) for a, b in zip(out, ref))
