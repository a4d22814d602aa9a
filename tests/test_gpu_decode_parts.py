"""Decode over batches of unequal requests, whose pairs are cut into parts.

Against the fp64 reference, and the 4-bit form against the bf16 form over the
reconstructed rows, bit for bit: a long request among short ones (text or visual
rows, so that parts end inside either), one alone, more pairs than fit at once,
requests without keys, and the workspace's size, which the parts must not
exceed (guard bytes after it)."""
import numpy as np
import pytest
import torch

from paper_2608_24063_gb300 import synth
from paper_2608_24063_gb300 import viscache as vc
from test_gpu_decode_tiles import _check, _rand

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


@pytest.mark.parametrize("d", [64, 128])
@pytest.mark.parametrize("ns,texts", [
    ([40] * 47 + [9000], [20] * 48), ([40] * 48, [20] * 30 + [7001] + [0] * 17), ([65000], [33]), ([31], [66000]),
    ([2000, 1, 40, 33] * 3, [1, 30000, 0, 5] * 3), ([640] * 79, [128] * 79), ([1, 1, 60000], [0, 0, 1])])
def test_unequal_requests(d, ns, texts):
    _check(8, 4, d, ns, texts, 5000 + len(ns) + texts[-1])


def test_request_without_keys_among_long_ones():
    # layer 1 of 2 is evicted (h = 1): text only, or no keys at all
    L, Hq, Hkv, d = 2, 8, 4, 128
    texts = [30000, 0, 5]
    batch = vc.Batch([64] * 3, [8] * 3, [(1, 2)] * 3)
    prm = vc.make_params(L, Hq, Hkv, d, vc.VC_BF16, h=1, m=(1, 1), schedule=vc.VC_SCHED_FIXED)
    rows, trows = vc.compressed_rows(batch, prm), Hkv * sum(texts)
    K, V, Kt, Vt = (_rand((n, d), 7000 + i).to(DEV) for i, n in enumerate((rows, rows, trows, trows)))
    q = _rand((3, Hq, d), 7010).to(DEV)
    need = vc.viscache_decode_workspace_size(batch, prm, texts)
    ws = torch.full((need + 4096,), 165, dtype=torch.uint8, device=DEV)
    out = vc.viscache_decode_attention(batch, prm, 1, q, K, V, Kt, Vt, texts, ws=ws[:need])
    assert bool((ws[need:] == 165).all())
    assert not out[1].any()
    for r, t0, T in ((0, 0, 30000), (2, 30000, 5)):
        k = Kt[Hkv * t0:Hkv * (t0 + T)].double().view(Hkv, T, d)
        v = Vt[Hkv * t0:Hkv * (t0 + T)].double().view(Hkv, T, d)
        p = torch.softmax(torch.einsum("gjd,gtd->gjt", q[r].double().view(Hkv, 2, d), k) / d ** 0.5, -1)
        ref = torch.einsum("gjt,gtd->gjd", p, v).reshape(Hq, d)
        err = (out[r].double() - ref).abs()
        assert bool((err <= 1e-4 * v.abs().max() + 2.0 ** -8 * ref.abs()).all())


def test_nan_and_infinite_rows_stay_in_their_request():
    ns, texts, Hq, Hkv, d = [40] * 40, [20] * 39 + [20000], 8, 4, 128
    batch = vc.Batch(ns, [8] * 40, [(1, 1)] * 40)
    prm = vc.make_params(1, Hq, Hkv, d, vc.VC_BF16, h=1, m=(1, 1), schedule=vc.VC_SCHED_FIXED)
    K, V = (_rand((Hkv * sum(ns), d), 8000 + i).to(DEV) for i in range(2))
    Kt, Vt = (_rand((Hkv * sum(texts), d), 8002 + i).to(DEV) for i in range(2))
    q = _rand((40, Hq, d), 8004).to(DEV)
    clean = vc.viscache_decode_attention(batch, prm, 0, q, K, V, Kt, Vt, texts)
    Kt[Hkv * sum(texts[:39]) + 777] = float("nan")            # KV head 0 of the long request, one part
    out = vc.viscache_decode_attention(batch, prm, 0, q, K, V, Kt, Vt, texts)
    assert torch.equal(out[:39], clean[:39])
    assert torch.isnan(out[39, :Hq // Hkv]).all() and torch.equal(out[39, Hq // Hkv:], clean[39, Hq // Hkv:])
