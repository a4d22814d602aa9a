"""GPU parity of the bf16 and 4-bit decode kernel at the edges of its tiles.

A warp takes tiles of 32 keys, visual and text rows in tiles of their own, and
a cluster of 1 to 16 thread blocks (4 warps each) shares a (request, KV head):
tile remainders, pairs with fewer tiles than warps, every cluster size, and
rows of a neighbouring segment that hold NaN.  Tolerance: as for the decode
step's other tests, 1e-4 of the largest value plus one bf16 rounding."""
from fractions import Fraction

import numpy as np
import pytest
import torch

from oracle import decode as odec
from oracle import plan as oplan
from paper_2608_24063_gb300 import synth
from paper_2608_24063_gb300 import viscache as vc

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


def _rand(shape, key):
    x = synth.normal(key, 0, int(np.prod(shape)), "cpu").view(*shape)
    return synth._round(x, torch.bfloat16)


def _check(Hq, Hkv, d, ns, texts, seed, poison=False):
    # one layer, RR = 1, m = 1: every request keeps all n rows (B = n)
    batch = vc.Batch(ns, [8] * len(ns), [(1, 1)] * len(ns))
    params = vc.make_params(1, Hq, Hkv, d, vc.VC_BF16, h=1, m=(1, 1), schedule=vc.VC_SCHED_FIXED)
    for n in ns:
        assert oplan.plan_budgets(1, n, Fraction(1), h=1, m=Fraction(1), schedule="fixed")[0] == [n]
    K, V = _rand((Hkv * sum(ns), d), seed), _rand((Hkv * sum(ns), d), seed + 1)
    trows = Hkv * sum(texts)
    Kt, Vt = _rand((max(trows, 1), d), seed + 2), _rand((max(trows, 1), d), seed + 3)
    if poison:                                  # request 1 of 3: its rows lie between the others'
        a, b = Hkv * ns[0], Hkv * (ns[0] + ns[1])
        K[a:b], V[a:b] = float("nan"), float("inf")
        a, b = Hkv * texts[0], Hkv * (texts[0] + texts[1])
        Kt[a:b], Vt[a:b] = float("nan"), float("inf")
    q = _rand((len(ns), Hq, d), seed + 4)
    dev = [x.to(DEV) for x in (K, V, Kt, Vt, q)]
    out = vc.viscache_decode_attention(batch, params, 0, dev[4], dev[0], dev[1], dev[2], dev[3], texts)
    got = out.float().cpu().numpy()
    K64, V64, Kt64, Vt64 = (x.double().numpy() for x in (K, V, Kt, Vt))
    r0 = t0 = 0
    for r, (n, T) in enumerate(zip(ns, texts)):
        if not (poison and r == 1):
            part = [x[a:a + Hkv * m].reshape(Hkv, m, d) for x, a, m in
                    ((K64, r0, n), (V64, r0, n), (Kt64, t0, T), (Vt64, t0, T))]
            ref = odec.decode_attention(q[r].double().numpy(), *part)
            vmax = max(np.abs(part[1]).max(initial=0.0), np.abs(part[3]).max(initial=0.0), 1.0)
            assert (np.abs(got[r] - ref) <= 1e-4 * vmax + 2.0 ** -8 * np.abs(ref)).all(), "request %d" % r
        r0, t0 = r0 + Hkv * n, t0 + Hkv * T
    if not poison:
        kv4 = vc.viscache_kv4_quantize(batch, params, dev[0], dev[1])
        Kh, Vh = vc.viscache_kv4_dequantize(batch, params, *kv4)
        out4 = vc.viscache_decode_attention_kv4(batch, params, 0, dev[4], kv4, dev[2], dev[3], texts)
        ref4 = vc.viscache_decode_attention(batch, params, 0, dev[4], Kh, Vh, dev[2], dev[3], texts)
        assert torch.equal(out4, ref4)


@pytest.mark.parametrize("d", [64, 128])
@pytest.mark.parametrize("n,T", [(1, 0), (1, 1), (15, 17), (16, 16), (17, 31), (31, 33), (32, 32), (33, 1), (63, 65),
                                 (129, 0), (2049, 40)])
def test_tile_remainders(d, n, T):
    _check(8, 2, d, [n], [T], 1000 + 7 * n + T)


@pytest.mark.parametrize("G", [1, 2, 3, 5, 7, 8])
def test_every_group_size(G):
    _check(3 * G, 3, 128, [300, 65], [20, 0], 2000 + G)


@pytest.mark.parametrize("n_req,n", [(1, 1800), (2, 1800), (3, 1300), (5, 900), (7, 600), (9, 500), (13, 300),
                                     (26, 150), (60, 70)])
def test_every_cluster_size(n_req, n):
    # 8 KV heads a request: 8 to 480 pairs, from the largest clusters to one block a pair
    _check(16, 8, 128, [n - 3 * (r % 7) for r in range(n_req)], [33 + r % 5 for r in range(n_req)], 3000 + n_req)


def test_neighbouring_rows_do_not_leak():
    # tiles end inside a segment whose neighbour's rows are NaN and infinite
    _check(8, 2, 128, [45, 70, 51], [13, 40, 5], 4000, poison=True)
