"""How a decode step is spread over the device (csrc/decode_plan.h), compiled for the host.

A batch of near-equal requests takes one cluster of thread blocks a (request,
KV head) pair.  Where one request is far longer than the others no warp may be
left with many times the tiles of an even spread, and the parts must cover each
pair's tiles once and fit the workspace of the 256-key splits."""
import ctypes
import os
import random
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2608_24063_gb300", "csrc")

HARNESS = """
#include "decode_plan.h"
using namespace vc;
extern "C" void plan(const long long* keys, int n_req, int Hkv, const int* fit, int* out) {
  DecodeFit f;
  for (int k = 0; k < kClusterKinds; ++k) f.n[k] = fit[k];
  int64_t tiles[512];
  for (int r = 0; r < n_req; ++r) tiles[r] = decode_tiles(keys[2 * r], keys[2 * r + 1]);
  const DecodePlan p = plan_decode(tiles, n_req, Hkv, f);
  out[0] = p.cluster;
  out[1] = p.part_tiles;
  for (int r = 0; r < n_req; ++r) {
    const int parts = p.part_tiles ? decode_parts(tiles[r], p.part_tiles) : 1;
    out[2 + 3 * r] = (int)tiles[r];
    out[3 + 3 * r] = parts;
    out[4 + 3 * r] = decode_tiles_per_part(tiles[r], parts);
  }
}
"""
SIZES = [1, 2, 3, 4, 5, 6, 7, 8, 12, 16]
FIT = [304 // c if c < 12 else {12: 20, 16: 16}[c] for c in SIZES]


@pytest.fixture(scope="module")
def plan(tmp_path_factory):
    d = tmp_path_factory.mktemp("plan")
    src, so = str(d / "plan.cpp"), str(d / "plan.so")
    with open(src, "w") as f:
        f.write(HARNESS)
    subprocess.run(["g++", "-std=c++17", "-O1", "-shared", "-fPIC", "-I", CSRC, src, "-o", so], check=True)
    fn = ctypes.CDLL(so).plan

    def call(reqs, Hkv):
        keys = (ctypes.c_longlong * (2 * len(reqs)))(*[x for r in reqs for x in r])
        out = (ctypes.c_int * (2 + 3 * len(reqs)))()
        fn(keys, len(reqs), Hkv, (ctypes.c_int * len(FIT))(*FIT), out)
        return out[0], out[1], [tuple(out[2 + 3 * r:5 + 3 * r]) for r in range(len(reqs))]

    return call


def _warp_tiles(cluster, part_tiles, reqs, Hkv):
    """Tiles of the busiest warp, and of a warp of an even spread over 304 thread blocks."""
    even = sum(t for t, _, _ in reqs) * Hkv / (304 * 4)
    if part_tiles:
        return max((min(t, per) + 3) // 4 for t, _, per in reqs), even
    return max((t + 4 * cluster - 1) // (4 * cluster) for t, _, _ in reqs), even


@pytest.mark.parametrize("n_req,keys", [(1, (2383, 512)), (16, (2383, 512)), (64, (596, 64)), (24, (7376, 900)),
                                        (80, (2400, 512)), (256, (2000, 20)), (200, (100, 20))])
def test_equal_requests_are_not_cut(plan, n_req, keys):
    assert plan([keys] * n_req, 4)[1] == 0


@pytest.mark.parametrize("reqs", [[(596, 64)] * 63 + [(596, 16384)], [(596, 64)] * 39 + [(596, 65536)],
                                  [(2383, 512)] * 15 + [(2383, 16384)], [(3500, 1 << 20)], [(1, 0)] * 255 + [(65536, 0)]])
def test_a_long_request_does_not_run_on_a_few_warps(plan, reqs):
    cluster, part, got = plan(reqs, 4)
    worst, even = _warp_tiles(cluster, part, got, 4)
    assert part > 0 and worst <= max(2 * even + 10, 17)


@pytest.mark.parametrize("seed", range(4))
def test_random_batches(plan, seed):
    rnd = random.Random(seed)
    cut = 0
    for _ in range(500):
        Hkv = rnd.choice([1, 2, 4, 8])
        reqs = [(rnd.choice([0, 1, 31, 500, 6000, 65536]) if rnd.random() < 0.4 else rnd.randrange(0, 900),
                 rnd.choice([0, 0, 5, 33, 700, 20000]) if rnd.random() < 0.4 else 64) for _ in range(rnd.choice([1, 2, 8, 40, 256]))]
        cluster, part, got = plan(reqs, Hkv)
        assert cluster in SIZES
        worst, even = _warp_tiles(cluster, part, got, Hkv)
        pairs = len(reqs) * Hkv
        if pairs <= 304:
            assert worst <= max(2 * even + 11, 17)
        if part:
            cut += 1
            assert cluster == 1
            for (t, parts, per), (B, T) in zip(got, reqs):
                assert per % 4 == 0 and parts * per >= t and 1 <= parts <= 256
                assert parts <= max(1, (B + T + 255) // 256)       # the workspace of the splits
    assert cut > 10
