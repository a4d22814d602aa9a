"""The column-sum pass's shares (csrc/score_shares.h), compiled for the host.

A pair of thread blocks takes a share of the (unit, layer) sequence.  Over all
pairs the segments must cover every layer of every unit once, none may be empty
(an empty one would count itself in a unit's arrivals without having waited
for the kernel that clears them), a unit's `parts` must be the number of its
segments, and the places of split units must be distinct and inside the
scratch region.  The shapes include those with fewer steps than pairs, where
several cuts fall on one layer."""
import ctypes
import os
import random
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2608_24063_gb300", "csrc")

HARNESS = """
#include "score_shares.h"
using namespace vc;
// req: n_req x (units2, layers, C, cw); out: rows (pair, unit, l0, l1, slot, parts); returns the rows, -1: no plan
extern "C" int plan(const int* req, int n_req, int pairs, int* cuts, int* out, int cap) {
  TcReq q[64];
  int64_t units = 0;
  int ends[64];
  for (int r = 0; r < n_req; ++r) {
    q[r] = TcReq{req[4 * r], req[4 * r + 1], req[4 * r + 2], req[4 * r + 3]};
    ends[r] = (int)(units += q[r].units2);
  }
  Shares s;
  if (!plan_shares(q, n_req, units, pairs, &s)) return -1;
  int rows = 0;
  for (int p = 0; p <= pairs; ++p) { cuts[2 * p] = s.unit[p]; cuts[2 * p + 1] = s.layer[p]; }
  for (int p = 0; p < pairs; ++p)
    for (int i = 0; i < share_segments(s, p); ++i) {
      int r = 0;
      while (r + 1 < n_req && s.unit[p] + i >= ends[r]) ++r;
      const ShareSegment d = share_segment(s, pairs, p, i, q[r].layers);
      if (rows == cap) return -2;
      int* o = out + 6 * rows++;
      o[0] = p; o[1] = d.unit; o[2] = d.l0; o[3] = d.l1; o[4] = d.slot; o[5] = d.parts;
    }
  return rows;
}
extern "C" int worth(int units2, int pairs, int per_layer) { return worth_sharing(units2, pairs, per_layer != 0); }
"""


@pytest.fixture(scope="module")
def plan(tmp_path_factory):
    d = tmp_path_factory.mktemp("shares")
    src, so = str(d / "plan.cpp"), str(d / "plan.so")
    with open(src, "w") as f:
        f.write(HARNESS)
    subprocess.run(["g++", "-std=c++17", "-O1", "-shared", "-fPIC", "-I", CSRC, src, "-o", so], check=True)
    lib = ctypes.CDLL(so)
    fn = lib.plan

    def call(reqs, pairs):
        flat = (ctypes.c_int * (4 * len(reqs)))(*[x for q in reqs for x in q])
        cap = sum(q[0] for q in reqs) + 2 * pairs + 8
        out, cuts = (ctypes.c_int * (6 * cap))(), (ctypes.c_int * (2 * pairs + 2))()
        rows = fn(flat, len(reqs), pairs, cuts, out, cap)
        assert rows != -2
        if rows < 0:
            return None, None
        return ([tuple(cuts[2 * p:2 * p + 2]) for p in range(pairs + 1)],
                [tuple(out[6 * i:6 * i + 6]) for i in range(rows)])

    call.worth = lib.worth
    return call


def _req(L, Hkv, G, W, n):
    C = (G * W + 255) // 256
    return (Hkv * ((n + 255) // 256), L, C, 16 * ((G * W + 16 * C - 1) // (16 * C)))


def _check(plan, reqs, pairs):
    """Returns the number of empty shares inside a unit, or None without a plan."""
    cuts, segs = plan(reqs, pairs)
    if cuts is None:
        return None
    layers = [q[1] for q in reqs for _ in range(q[0])]
    seen, places = {}, {}
    for p, unit, l0, l1, slot, parts in segs:
        assert 0 <= l0 < l1 <= layers[unit], "an empty segment"
        seen.setdefault(unit, []).append((l0, l1, slot, parts))
    assert sorted(seen) == list(range(len(layers)))
    for unit, parts in seen.items():
        parts.sort()
        assert [a[0] for a in parts] == [0] + [a[1] for a in parts[:-1]] and parts[-1][1] == layers[unit]
        assert {a[3] for a in parts} == {len(parts)}
        if len(parts) > 1:
            assert len({a[2] for a in parts}) == 1
            assert places.setdefault(parts[0][2], unit) == unit
            assert 0 <= parts[0][2] < min(len(layers), pairs)
    return sum(a == b and a[1] > 0 for a, b in zip(cuts, cuts[1:]))


@pytest.mark.parametrize("L,Hkv,G,W,n,empty", [(16, 4, 4, 64, 196, 12), (36, 2, 8, 16, 196, 4), (19, 1, 4, 256, 100, 47),
                                               (28, 4, 7, 64, 3136, 0), (28, 4, 7, 64, 12544, 0)])
def test_empty_shares_take_no_part(plan, L, Hkv, G, W, n, empty):
    got = _check(plan, [_req(L, Hkv, G, W, n)], 76)
    assert got >= 1 if empty else got == 0
    if L in (16, 36):
        assert got == empty


@pytest.mark.parametrize("seed", range(4))
def test_random_batches(plan, seed):
    rnd = random.Random(seed)
    empties = 0
    for _ in range(400):
        L, Hkv, G = rnd.choice([1, 2, 3, 5, 7, 16, 19, 28, 36, 80, 256]), rnd.randrange(1, 9), rnd.randrange(1, 9)
        reqs = [_req(rnd.randrange(0, L + 1) or L, Hkv, G, rnd.randrange(1, 140), rnd.choice([1, 100, 257, 900, 5000]))
                for _ in range(rnd.choice([1, 1, 2, 5, 9]))]
        empties += _check(plan, reqs, rnd.choice([1, 2, 5, 74, 76, 128])) or 0
    assert empties > 0


@pytest.mark.parametrize("units,layer,want", [(52, 0, True), (96, 0, True), (196, 0, True), (252, 0, True), (144, 0, False),
                                              (144, 1, True), (218, 0, False), (218, 1, False), (76, 0, False),
                                              (304, 0, False), (316, 0, False), (77, 0, True), (1, 0, True)])
def test_shares_where_the_last_wave_idles(plan, units, layer, want):
    assert bool(plan.worth(units, 76, layer)) == want


def test_counts_are_cleared_before_pass_2_may_start_and_read_after_the_wait():
    from test_launch_rules import _kernel_body, _sources, _strip_comments
    src = _strip_comments(_sources()["score_tc.cu"])
    lse, colsum = (_kernel_body(src, k) for k in ("score_lse_tc_kernel", "score_colsum_tc_kernel"))
    clear = lse.index("split_counts[threadIdx.x] = 0")
    assert lse.index("dep_wait()") < clear < lse.index("__syncthreads()", clear) < lse.index("dep_launch()")
    # the consumers' branch: from the register hand-over on, a wait before any use of the scratch
    consumers = colsum[colsum.index("take_registers"):]
    assert consumers.index("dep_wait()") < min(consumers.index("split_sums("), consumers.index("atomicAdd("))
