"""Host model of the fused pass's cut search (threshold_kernel, csrc/select.cu).

The search narrows, round by round, the range of composites (descending score
key, token) that holds each cut.  On scores that stand still it must find
every cut within four rounds a cut, whatever the scores (ties, NaN, infinities,
crowds).  If the scores change between rounds (past the tokens it holds in
shared memory they are read again) a cut's element can leave its range, and only
the limit on rounds ends the search: the model shows such a case, and the
kernel must have the limit and report it."""
import os
import re

import numpy as np
import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2608_24063_gb300", "csrc")
BUCKETS, CAP, POOL = 16384, 512, 8192


def composites(bits):
    u = bits.astype(np.uint64)
    neg = (u >> np.uint64(31)) != 0
    k = np.where(neg, ~u & np.uint64(0xFFFFFFFF), u | np.uint64(0x80000000))
    return [(int(x) << 16) | v for v, x in enumerate(~k & np.uint64(0xFFFFFFFF))]


def search(reads, pos, limit):
    """reads(round) gives the composites of a round; returns (cuts, rounds) or (None, limit)."""
    c = np.array(reads(0), dtype=np.uint64)
    nc, pos = len(pos), list(pos)
    lo = [int(c.min()) & ~0xFFFF] * nc
    hi = [int(c.max()) | 0xFFFF] * nc
    base = [0] * nc
    for rnd in range(limit):
        lead = next((t for t in range(nc) if pos[t] >= 0), None)
        if lead is None:
            return lo, rnd
        L, H = lo[lead], hi[lead]
        shift = max(0, (H - L).bit_length() - 14)
        c = np.array(reads(rnd), dtype=np.uint64)
        inside = c[(c >= np.uint64(L)) & (c <= np.uint64(H))]
        part = ((inside - np.uint64(L)) >> np.uint64(shift)).astype(np.int64)
        first = np.concatenate([[0], np.cumsum(np.bincount(part, minlength=BUCKETS))])
        mine = {t: int(np.searchsorted(first[:-1], pos[t] - base[t], side="right")) - 1
                for t in range(nc) if pos[t] >= 0 and lo[t] == L and hi[t] == H}
        taken, at, prev = {}, 0, None
        for t, b in mine.items():
            size = int(first[b + 1] - first[b])
            if shift and size <= CAP and prev != b:
                if at + size <= POOL:
                    taken[b] = np.sort(inside[part == b])
                at += size
            prev = b
        for t, b in mine.items():
            size = int(first[b + 1] - first[b])
            if shift == 0:
                lo[t], pos[t] = L + b, -1
            elif b in taken:
                k = pos[t] - base[t] - int(first[b])
                if 0 <= k < len(taken[b]):
                    lo[t], pos[t] = int(taken[b][k]), -1
            elif size > CAP:
                lo[t], hi[t] = L + (b << shift), min(H, L + ((b + 1) << shift) - 1)
                base[t] += int(first[b])
    return None, limit


def scores(kind, n, rng):
    if kind == "bits":
        return rng.integers(0, 2 ** 32, n, dtype=np.uint64)
    if kind == "nan":
        return np.where(rng.random(n) < 0.6, 0x7FC00000, rng.integers(0, 2 ** 32, n, dtype=np.uint64))
    if kind == "inf":
        return np.where(rng.random(n) < 0.5, 0x7F800000, 0xFF800000)
    if kind == "equal":
        return np.full(n, 0x3F800000)
    x = np.float32(0.22) + np.float32(1e-4) * rng.integers(0, 20, n).astype(np.float32)
    return x.view(np.uint32)


@pytest.mark.parametrize("kind", ["bits", "nan", "inf", "equal", "crowd"])
@pytest.mark.parametrize("n", [1, 2, 700, 5000, 65536])
def test_four_rounds_a_cut_are_enough(kind, n):
    rng = np.random.default_rng(n)
    c = composites(np.asarray(scores(kind, n, rng)))
    nq = int(rng.integers(1, n + 1))
    budgets = sorted(rng.integers(0, nq + 1, 28).tolist(), reverse=True)
    pos = [nq - 1] + [b - 1 for b in budgets]
    got, rounds = search(lambda r: c, pos, 4 * len(pos))
    assert got is not None and rounds <= 4 * len(pos)
    order = sorted(c)
    assert all(p < 0 or g == order[p] for g, p in zip(got, pos))


def test_scores_that_move_need_the_limit():
    n = 2000
    c = composites(np.full(n, 0x3F800000))
    far = composites(np.full(n, 0x3F000000))
    # after the first round narrowed the cut's range, every score lies outside it
    big = sorted(c + [x + (1 << 40) for x in c])
    got, rounds = search(lambda r: c + big if r == 0 else far, [n - 1], 1000)
    assert got is None and rounds == 1000


def test_the_kernel_has_the_limit():
    with open(os.path.join(CSRC, "select.cu")) as f:
        src = f.read()
    assert re.search(r"constexpr int kSelRounds = 4 \* kSelCuts;", src)
    assert re.search(r"for \(int round = 0; round < kSelRounds; \+\+round\)", src)
    tail = src[src.index("round < kSelRounds"):]
    assert re.search(r"if \(sm\.pos\[t\] >= 0\) set_status\(tb\.status, VC_ERR_DEVICE_INDEX\);", tail)
