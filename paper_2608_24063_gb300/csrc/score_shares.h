// How the column-sum pass cuts its (unit, layer) sequence into shares, one per
// CTA pair: the plan (host) and what a pair reads from it (host and device).
#pragma once
#include <stdint.h>

#include <algorithm>

#ifndef VC_HD
#ifdef __CUDACC__
#define VC_HD __host__ __device__ __forceinline__
#else
#define VC_HD inline
#endif
#endif

namespace vc {

constexpr int kMaxPairs2 = 128;                 // shares per launch
constexpr int kMaxSegs = 256;                   // segments per pair (descriptor table)

struct TcReq {       // one request in the column-sum pass
  int units2;        // key-tile units (Hkv * tiles, 0 when no layer is scored)
  int layers;        // layers scored
  int C, cw;         // chunks of a layer's rows, rows per chunk
};

// Share p covers (unit, layer) positions from (unit[p], layer[p]) up to
// (unit[p + 1], layer[p + 1]).  Split units are numbered by unit where there are no
// more units than shares, else by the first cut inside them.
struct Shares {
  int32_t by_unit;
  int32_t unit[kMaxPairs2 + 1];
  int16_t layer[kMaxPairs2 + 1];
};

// Units share p has layers of.  A share that ends where it begins has none: its
// CTAs take no part in any unit.
VC_HD int share_segments(const Shares& s, int p) {
  if (s.unit[p] == s.unit[p + 1] && s.layer[p] == s.layer[p + 1]) return 0;
  return s.unit[p + 1] - s.unit[p] + (s.layer[p + 1] > 0 ? 1 : 0);
}

// Segment i of share p: layers [l0, l1) of unit `unit` of Ls layers; a unit cut
// into parts > 1 segments has the place `slot` among the launch's split units.
struct ShareSegment {
  int unit, l0, l1, slot, parts;
};
VC_HD ShareSegment share_segment(const Shares& s, int npairs, int p, int i, int Ls) {
  ShareSegment d;
  d.unit = s.unit[p] + i;
  d.l0 = i == 0 ? s.layer[p] : 0;
  d.l1 = d.unit == s.unit[p + 1] ? s.layer[p + 1] : Ls;
  d.slot = 0;
  d.parts = 1;
  if (d.l0 > 0 || d.l1 < Ls) {
    // cuts a ... b - 1 lie inside the unit; those at different layers part it
    int a = i == 0 && d.l0 > 0 ? p : p + 1, b = p + 1;
    while (a > 1 && s.unit[a - 1] == d.unit && s.layer[a - 1] > 0) --a;
    while (b < npairs && s.unit[b] == d.unit && s.layer[b] > 0) ++b;
    d.slot = s.by_unit ? d.unit : a;
    d.parts = 2;
    for (int c = a + 1; c < b; ++c) d.parts += s.layer[c] != s.layer[c - 1] ? 1 : 0;
  }
  return d;
}

// The (unit, layer) sequence of pass 2 in equal shares of work for `pairs`
// pairs.  Work of a layer is its rows, with 16 a chunk for what a chunk costs
// beside them; a cut within two layers of a unit's end moves there.  False
// when a share would have more segments than the descriptor table holds
// (units of very unequal work).
inline bool plan_shares(const TcReq* req, int n_req, int64_t units2, int pairs, Shares* out) {
  int64_t total = 0;
  auto layer_work = [](const TcReq& q) { return (int64_t)q.C * (q.cw + 16); };
  for (int r = 0; r < n_req; ++r) total += (int64_t)req[r].units2 * req[r].layers * layer_work(req[r]);
  out->by_unit = units2 <= pairs;
  int r = 0;
  int64_t before = 0, unit0 = 0;               // work and units of the requests before r
  int64_t pu = 0, pl = 0;                      // previous cut
  for (int p = 0; p <= pairs; ++p) {
    int64_t cu = units2, cl = 0;
    if (p < pairs) {
      const int64_t want = total / pairs * p + total % pairs * p / pairs;
      for (; r + 1 < n_req; ++r) {
        const int64_t all = (int64_t)req[r].units2 * req[r].layers * layer_work(req[r]);
        if (before + all > want) break;
        before += all;
        unit0 += req[r].units2;
      }
      const TcReq& q = req[r];
      const int64_t work = layer_work(q), layers = std::max(q.layers, 1);
      const int64_t layer = (want - before + work / 2) / work;   // of the request, nearest
      cu = unit0 + layer / layers;
      cl = layer % layers;
      if (cl <= 2 || cl >= layers - 2) {
        if (2 * cl >= layers) ++cu;
        cl = 0;
      }
      if (cu >= units2) { cu = units2; cl = 0; }
      if (cu < pu || (cu == pu && cl < pl)) { cu = pu; cl = pl; }
    }
    out->unit[p] = (int32_t)cu;
    out->layer[p] = (int16_t)cl;
    if (p > 0 && cu - pu + 1 > kMaxSegs) return false;
    pu = cu;
    pl = cl;
  }
  return true;
}

// Whether shares pay.  They fill the last wave of whole units, but pairs that start
// inside different layers draw the window rows from the L2 at different times, and
// split units leave sums in memory (not under layer-specific ranking).  So the last
// wave has to leave a twelfth (a twentieth) of the pairs' time idle.  Whole calls, us,
// whole units | shares, by units a pair and idle part: 1.3, 37% 250 | 226; 1.9, 5%
// 319 | 326 (layer-specific 297 | 293); 2.6, 14% 462 | 452; 2.9, 4%, two ragged
// requests 761 | 796; 3.3, 17% 622 | 602.  Past four units a pair equal requests
// still gain (5.2, 14% 906 | 868; 8.3, 8% 2,026 | 1,987), ragged ones no more (5.4,
// 11% 1,082 | 1,078; layer-specific 8.2, 9% 1,158 | 1,218), so the line lies there.
constexpr int kShareUnits = 4;
inline bool worth_sharing(int64_t units2, int pairs, bool per_layer) {
  const int64_t slots = (units2 + pairs - 1) / pairs * pairs;
  return units2 <= (int64_t)kShareUnits * pairs && (slots - units2) * (per_layer ? 20 : 12) > slots;
}

// Whether a cut lies inside a unit.  Without one, and with a pair for every unit,
// whole units do the same with less to set up.
inline bool cuts_a_unit(const Shares& s, int pairs) {
  for (int p = 1; p < pairs; ++p)
    if (s.layer[p] > 0) return true;
  return false;
}

}  // namespace vc
