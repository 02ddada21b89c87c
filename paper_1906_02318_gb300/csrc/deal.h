// How a tick's slots are dealt out to blocks that take several candidates each: chunks of
// consecutive slots (whole sectors of a caller's samples and of the per-slot outputs), one
// in turn per block, since samples may come in order and long-lived ones would meet in a
// few blocks.  For device code and the host.
#pragma once

#include "basis.h"

namespace mpmi {

// The slots of a sorted unit: chunks of kUnitChunk consecutive slots, `stride` chunks
// apart, the first one number `first`.
constexpr int kUnitChunk = 8;
struct UnitSlots {
  int first, stride;
  MPMI_HD int slot(int i) const {
    return (i / kUnitChunk * stride + first) * kUnitChunk + i % kUnitChunk;
  }
};
// Unit u of n_units over n slots: chunks u, u + n_units, ...; its number of slots.
MPMI_HD int unit_count(int n, int n_units, int u) {
  const int chunks = (n + kUnitChunk - 1) / kUnitChunk;
  if (u >= chunks) return 0;
  const int mine = (chunks - u + n_units - 1) / n_units;
  return mine * kUnitChunk - ((chunks - 1) % n_units == u ? chunks * kUnitChunk - n : 0);
}

// A factorised tick's launch over n slots: one candidate per warp until every SM has 32
// warps (max_wpb), in blocks of 4 to 32 warps.
inline void fact_launch(int n, int sms, int max_wpb, int* wpb, int* grid) {
  const int per_sm = (n + sms - 1) / sms;
  *wpb = per_sm < 4 ? 4 : (per_sm < max_wpb ? per_sm : max_wpb);
  const int blocks = (n + *wpb - 1) / *wpb;
  *grid = blocks < 1 ? 1 : (blocks < sms ? blocks : sms);
}

// The share of block `first` of such a launch (n may be a shorter, device-side count): equal
// shares, at least a candidate per warp; the blocks from `stride` on have none.  While that
// is all a block gets, single slots are dealt out: chunks of eight left some blocks without
// a candidate and gave others two per warp (N = 700: 52 of 140 blocks idle, the others 8
// candidates for 5 warps).  Race car, H = 60, us: N = 500 8.4 -> 7.5, 2000 8.5 -> 7.6, 4000
// 8.9 -> 8.4; in chunks from N = 4865 on (9.4 at 5000, 16.8 at 30001).
struct FactShare {
  int first, stride, chunk;
  MPMI_HD FactShare(int n, int grid, int wpb, int block) : first(block) {
    const int even = (n + grid - 1) / grid;
    const int share = wpb > even ? wpb : even;
    const int used = (n + share - 1) / share;
    stride = used > 1 ? used : 1;
    chunk = share == wpb ? 1 : kUnitChunk;
  }
  MPMI_HD int count(int n) const {
    if (chunk > 1) return unit_count(n, stride, first);
    return n > first ? (n - first + stride - 1) / stride : 0;
  }
  MPMI_HD int slot(int i) const {
    return chunk > 1 ? UnitSlots{first, stride}.slot(i) : i * stride + first;
  }
};

}  // namespace mpmi
