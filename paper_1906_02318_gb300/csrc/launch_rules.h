// Rules on sizes that the tick launches follow, with the measurements behind them (GB300,
// 152 SMs, ticks back to back, eight states of a closed loop).  Plain host code, so that
// the lines can be checked without a GPU.
#pragma once

#include "basis.h"

namespace mpmi {

// Candidates per thread of a one-lane launch that leaves them to the library: two race
// cars past one tile for each of an SM's eight warps (H = 60, one / two, us: N = 39000 134.5
// / 116.7, 44000 139.8 / 125.3, 48000 143.2 / 128.6).
inline int one_lane_cands(int kind, long long n, int sms) {
  return kind == kCar && n > 256LL * sms ? 2 : 1;
}

// Whether a one-lane launch over n slots takes sorted units: tiles of per_warp slots, of
// which one round of the resident warps holds `warps`.  With more than ~1.6 tiles per warp
// the tiles that a warp saves by sorting outweigh drawing every candidate twice (balance
// bot, H = 50, N = 65536, 1.7 tiles, 20.8 -> 16.8 us); below, the last round's few tiles
// run alone either way (race car N = 100000, 1.3 tiles, 217 us unsorted, 225 sorted).  The
// race car also gains where every tile has a warp of its own (N = 24000 87.7 -> 84.3 us, N
// = 65536 150 -> 145 us): its warps share the shared-memory pipe, which tiles that leave
// early free.
//
// Short horizons leave little to save.  Balance bot, unsorted / sorted, us: N = 1048576 H
// = 20 90.6 / 100.0, 30 128.6 / 131.7, 34 143.8 / 140.6, 36 151.3 / 144.5; N = 90396 H = 30
// 16.5 / 18.8, 36 19.2 / 19.9, 40 19.6 / 20.4, 50 24.0 / 21.6; noisy, N = 1048576 H = 30
// 392 / 407, 40 498 / 468.  State by state (40 of them, N = 723704) sorted ticks take 1.01
// to 1.09 times the unsorted ones at H = 30 (5th to 95th percentile), 0.96 to 1.04 at 34
// and 0.94 to 1.01 at 36.  Race car, several rounds: sorting pays there too unless the
// last round is at most 3/8 full, which unsorted tiles, spread over the SMs, finish sooner
// (a unit's last tiles go to whichever warps are free, often two on one SM sub-partition):
// N = 176366 (0.27) H = 20 121.5 / 140.8, 30 175.5 / 202, 40 233 / 262, 44 257 / 277, 52
// 304 / 308, 60 350 / 332; N = 195473 (0.51) H = 20 144.7 / 141.7; N = 160737 (0.07) H = 20
// 118.9 / 122.6, 40 229 / 231, 44 252 / 249.
inline bool units_pay(int kind, int horizon, long long n, int per_warp, long long warps) {
  const long long wave = warps * per_warp;
  if (kind != kCar) return horizon >= 35 && 10 * n >= 16 * wave;
  if (10 * n < 16 * wave) return 2 * n >= wave && n <= wave;
  if (horizon > 46) return true;
  const long long last = (n + per_warp - 1) / per_warp % warps;
  return last == 0 || 8 * last > 3 * warps || (horizon > 32 && 8 * last < warps);
}

// Horizon from which a tick of S/2 < blocks <= S keeps the stream's order instead of
// starting early (S: SMs).  While the blocks of the tick before hold their SMs, an early
// grid doubles up on the idle ones; an early start gives about 2 us whatever the horizon,
// and two blocks on an SM slow each other down in every step.  How many pair up settles
// differently from run to run (both modes given where they were seen), so the lines lie
// where the slower one no longer loses much.  In order / early, us:
//   race car, K in shared memory (two lanes), 110 blocks: H = 20 16.6 / 14.3, 30 20.7 /
//     19.5 (79 blocks 18.6 or 24.7), 40 26.2 / 28.3, 60 36.5 / 41.5, 100 53.5 / 64.8;
//     noisy, 79 to 110 blocks, H = 20 22.7 / 20.5 or 25.0, 30 30.7 / 32.0, 60 53.6 / 60.9;
//     one lane, N = 19000 (149 blocks), H = 20 24.9 / 28.2; four lanes, N = 6000 29.4 / 35.1
//   eight lanes, 96 blocks: H = 60 20.6 / 18.1, 70 22.7 / 23.0, 100 28.5 / 32.1; noisy, H
//     = 40 20.6 / 19.3, 60 26.8 / 25.0, 70 30.0 / 32.7; 126 blocks: H = 40 16.6 / 14.3, 60
//     20.6 / 18.2 or 22.4, 70 22.7 / 23.5; noisy, H = 30 18.6 / 16.2, 40 22.1 / 22.7, 100
//     39.1 / 44.9
//   sixteen lanes, 96 blocks: H = 60 18.4 / 17.4, 80 20.7 / 21.7, 100 24.7 / 25.9; noisy,
//     H = 50 18.6 / 18.1, 60 20.7 / 21.3, 100 30.7 / 32.5
//   balance bot, one lane, 84 to 140 blocks: H = 60 10.5 / 8.5 to 10.8, 80 12.4 / 10.1 or
//     13.6, 90 12.5 / 13.7, 100 14.4 / 14.9; noisy, H = 30 16.3 / 15.9, 40 18.6 / 19.4, 100
//     37.0 / 40.9; noisy, four lanes, 124 blocks: H = 70 18.1 / 17.7, 80 18.6 / 19.7, 100
//     22.7 / 24.3
// On every SM or all but one (152 blocks) the balance bot loses earlier: one lane, H = 50
// 10.3 / 10.4, 60 10.4 / 12.1, 100 14.4 / 17.6 (150 blocks: H = 70 12.4 / 9.5, 90 12.5 /
// 14.0).  Its four lanes without noise never do.
inline int order_horizon(int kind, int lanes, bool k_shared, bool noise, long long grid, int sms) {
  constexpr int kNever = 1 << 30;
  if (kind == kCar) {
    if (k_shared) return noise || lanes != 2 ? 0 : 25;
    if (lanes == 16) return noise ? 55 : 75;
    return 4 * grid > 3LL * sms ? (noise ? 35 : 45) : (noise ? 50 : 65);
  }
  if (kind != kBot || (lanes > 1 && !noise)) return kNever;
  const int h = lanes > 1 ? 78 : (noise ? 35 : 85);
  return 100 * grid > 99LL * sms ? h * 2 / 3 : h;
}

// Whether a launch keeps the stream's order: `grid` of at most `resident` blocks with
// `warps_per_block` warps each over `tiles` warp-tiles, taken in strides (not sorted units).
//
// With more tiles than resident warps the first blocks take a tile more.  In order they
// spread over the SMs; early they start two to an SM as it falls free, and where the last
// round holds between a fifth and 3/8 of a round, those pairs take as long as a full
// round.  Race car, two candidates per thread, in order / early, us: N = 98558 (27 % of
// a round) H = 20 75.8 / 85.3, H = 60 209 / 235, H = 100 339 / 379; N = 89374 (15 %), H =
// 60 208.6 / 206.2; N = 108687 (40 %), H = 60 286.1 / 282.9; N = 262143 (37 %), H = 20
// 169.8 / 181.1; with noise, H = 20, N = 98558 117.0 / 114.4, N = 105275 (35 %)
// 117.1 / 132.2.  The balance bot, with K in registers, gains from the early start there too
// (H = 20, N = 450871 43.6 / 42.5).
inline bool keeps_order(int kind, int lanes, bool k_shared, bool noise, int horizon, long long grid,
                        long long resident, int warps_per_block, long long tiles, int sms) {
  const long long warps = resident * warps_per_block;
  if (resident <= sms) return false;  // an SM holds one block: none can double up
  if (tiles > warps) {
    const long long last = tiles % warps;
    return kind == kCar && lanes == 1 && k_shared && 10 * last > (noise ? 3 : 2) * warps &&
           8 * last <= 3 * warps;
  }
  if (2 * grid <= sms) return false;
  // grids past S blocks: only the race car's one-lane shapes where an SM holds more blocks
  // than an even spread gives it (blocks of 64 threads, N = 19000, H = 60 65.3 / 75.0; two
  // candidates per thread, N = 24000, H = 20 35.2 / 31.8)
  if (grid > sms)
    return k_shared && lanes == 1 && horizon >= 25 && (grid + sms - 1) / sms < resident / sms;
  return horizon >= order_horizon(kind, lanes, k_shared, noise, grid, sms);
}

// Which of its other launch shapes an untuned server takes for a batch of that many slots:
// 0 eight lanes, 1 two lanes, 2 two candidates per thread, -1 the initial one (one lane),
// for which the batch has `tiles` warp-tiles on `warps` resident warps.
// Race cars, submit to collect, us.  One session, H = 60: N = 1000 103 -> 65 and N = 3000
// 103 -> 69 with eight lanes, N = 6000 102 -> 78 and N = 18000 135 -> 99 with two.  Where the
// one-lane tiles need a second round, two lanes save it (256 slots per SM, seven sessions,
// 1219 tiles on 1216 warps 190 / 151; three sessions, 1216 tiles 136 / 147; 275 slots per
// SM, four mixes: 226 / 191 / 185 / 187 -> 176 / 177 / 146 / 173) until theirs is full (420:
// 209 / 233 / 176 / 225 -> 197 / 227 / 165 / 216).  Past that sessions of one horizon lose
// (450: 234 / 222 -> 250 / 240; 505: 234 / 228 -> 255 / 245), mixed ones, whose short
// sessions make room, gain up to 512 (470: 246 / 234 -> 236 / 210; 505: 336 / 213 -> 337 /
// 202).  Two candidates per thread: see serve_alts.
inline int serve_alt(int kind, long long slots, long long tiles, long long warps, bool mixed,
                     int sms) {
  if (kind != kCar) return -1;
  if (slots < 32LL * sms) return 0;
  if (slots < 128LL * sms || (tiles > warps && slots < (mixed ? 512LL : 432LL) * sms)) return 1;
  return slots >= 1200LL * sms ? 2 : -1;
}

// Whether a served batch takes sorted units: `horizon` is its longest, `wave` the slots of
// one tile per resident warp.  A unit costs barriers, and its blocks end the last round
// together where strided tiles spread it.  Unsorted / sorted, us, submit to collect; the
// first two of each row mix N and H, the last two are sessions of one N and H = 60:
//   race cars, one candidate per thread, below two tiles per warp: 93k slots 245 / 274; at
//     2.15 tiles 289 / 251, 276 / 262, 297 / 322, 279 / 309; 2.3: 307 / 309, 247 / 262, 298
//     / 326, 286 / 311; 3.1: 401 / 365, 377 / 351, 391 / 414, 373 / 364; 3.9: 418 / 346, 427
//     / 389, 436 / 435, 416 / 406.  What sorting saves grows with the horizon, so batches
//     without long ones stay unsorted.
//   balance bots: 4.1 tiles 117 / 119, 105 / 108, 121 / 135, 102 / 114; 4.5: 96 / 104, 123 /
//     128, 127 / 138, 103 / 116; 4.7: 116 / 115, 109 / 108, 128 / 130, 106 / 109, one N and
//     H = 100 131 / 117; 5.1: 99 / 100, 115 / 114, 140 / 134, 116 / 108; 5.9: 128 /
//     116, 132 / 120, 148 / 139, 123 / 113; H = 30: 7.0 109 / 117, 9.8 136 / 144.
inline bool serve_units_pay(int kind, int cands, int horizon, long long slots, long long wave) {
  if (kind == kCar) return slots >= 2 * wave && (cands > 1 || horizon > 64);
  return horizon >= 35 && 5 * slots >= 23 * wave;
}

}  // namespace mpmi
