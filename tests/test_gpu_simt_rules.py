"""The CUDA-core passes at the sizes where their tiles change, bit for bit.

A problem takes the small tiles while they leave at most half a thread block of
the large ones an SM, and pass 1 a third form (d = 64) beyond two an SM.  Each
request's arithmetic is the same in all of them, so a request alone, at the
last size of a form and at the first of the next, must give the bits it gives
in a batch of 16, which takes the forms for many blocks."""
import pytest
import torch

from paper_2608_24063_gb300 import viscache as vc

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


# blocks on 152 SMs: pass 1 (32 rows each) L * Hkv, pass 2 (64 keys each) Hkv * n / 64
@pytest.mark.parametrize("d,dtype", [(64, torch.float32), (128, torch.float32), (64, torch.bfloat16)])
@pytest.mark.parametrize("L,Hkv,n", [(19, 4, 190), (11, 7, 190), (76, 4, 70), (61, 5, 70), (2, 4, 19 * 64), (2, 7, 11 * 64),
                                     (2, 4, 19 * 64 + 1)])
def test_forms_agree_where_they_change(d, dtype, L, Hkv, n):
    W, copies = 5, 16
    g = torch.Generator().manual_seed(10 * n + L)
    q, k, v = (torch.randn(L, h, m, d, generator=g).to(dtype).to(DEV) for h, m in ((Hkv, W), (Hkv, n), (Hkv, n)))
    prm = vc.make_params(L, Hkv, Hkv, d, vc.VC_F32 if dtype == torch.float32 else vc.VC_BF16)

    def run(c):
        batch = vc.Batch([n] * c, [W] * c, [(1, 4)] * c)
        return vc.prunekv_compress(batch, prm, *(x.reshape(-1).repeat(c) for x in (q, k, v)))

    one, many = run(1), run(copies)
    for a, b in zip(one, many):
        a, b = a.reshape(-1), b.reshape(-1)
        assert b.numel() == copies * a.numel()
        for i in (0, copies - 1):
            assert torch.equal(a, b[i * a.numel():(i + 1) * a.numel()])
