"""The host rules on sizes that the tick launches follow (launch_rules.h), at the sizes
where both sides were measured."""
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_1906_02318_gb300", "csrc")
HEAD = r"""
#include <stdio.h>
#include "launch_rules.h"
using namespace mpmi;
static int failed = 0;
#define EXPECT(want, call)                                             \
  do {                                                                 \
    if ((want) != (call)) failed = printf("line %d: %s\n", __LINE__, #call); \
  } while (0)
"""


def _run(tmp_path, body):
    gxx = shutil.which("g++")
    if gxx is None:
        pytest.skip("no g++")
    (tmp_path / "rules.cpp").write_text(HEAD + body + "  return failed != 0;\n}\n")
    exe = tmp_path / "rules"
    subprocess.run([gxx, "-std=c++17", "-O1", "-Wall", "-Wno-unused-function", "-I", CSRC,
                    str(tmp_path / "rules.cpp"), "-o", str(exe)], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout


def test_launches_keep_the_streams_order_where_that_is_faster(tmp_path):
    _run(tmp_path, r"""
// kind, lanes, noise, H, blocks: grids of up to one 128-thread block per SM
static bool one(int kind, int lanes, bool noise, int H, int blocks) {
  return keeps_order(kind, lanes, kind == kCar && lanes < 8, noise, H, blocks, 304, 4, 4 * blocks,
                     152);
}
// race car, one lane, two candidates per thread, two blocks per SM
static bool rounds(long long n) {
  return keeps_order(kCar, 1, true, false, 60, 304, 304, 4, (n + 63) / 64, 152);
}
int main() {
  // balance bot
  EXPECT(false, one(kBot, 1, false, 50, 128));
  EXPECT(false, one(kBot, 1, false, 80, 116));
  EXPECT(true, one(kBot, 1, false, 100, 84));
  EXPECT(true, one(kBot, 1, false, 100, 132));
  EXPECT(true, one(kBot, 1, false, 60, 152));
  EXPECT(false, one(kBot, 1, false, 65, 148));
  EXPECT(false, one(kBot, 1, false, 30, 152));
  EXPECT(false, one(kBot, 1, false, 100, 76));
  EXPECT(false, one(kBot, 1, false, 100, 153));
  EXPECT(true, one(kBot, 1, true, 50, 112));
  EXPECT(false, one(kBot, 1, true, 20, 112));
  EXPECT(false, one(kBot, 4, false, 100, 152));
  EXPECT(false, one(kBot, 4, true, 50, 124));
  EXPECT(true, one(kBot, 4, true, 90, 124));
  // race car
  EXPECT(false, one(kCar, 2, false, 20, 110));
  EXPECT(true, one(kCar, 2, false, 30, 79));
  EXPECT(true, one(kCar, 2, true, 20, 79));
  EXPECT(true, one(kCar, 2, true, 40, 110));
  EXPECT(false, one(kCar, 8, false, 60, 104));
  EXPECT(true, one(kCar, 8, false, 60, 126));
  EXPECT(false, one(kCar, 8, false, 40, 126));
  EXPECT(true, one(kCar, 8, false, 80, 96));
  EXPECT(true, one(kCar, 8, true, 60, 126));
  EXPECT(false, one(kCar, 16, false, 60, 112));
  EXPECT(true, one(kCar, 16, false, 100, 112));
  EXPECT(true, one(kCar, 16, true, 60, 112));
  EXPECT(false, one(kCar, 16, true, 40, 112));
  // several rounds of tiles: the last one between 1/5 and 3/8 full
  EXPECT(false, rounds(77824));
  EXPECT(false, rounds(89374));
  EXPECT(true, rounds(98558));
  EXPECT(true, rounds(105275));
  EXPECT(false, rounds(108687));
  EXPECT(false, keeps_order(kCar, 1, true, true, 20, 304, 304, 4, (98558 + 63) / 64, 152));
  EXPECT(true, keeps_order(kCar, 1, true, true, 20, 304, 304, 4, (105275 + 63) / 64, 152));
  EXPECT(false, keeps_order(kBot, 1, false, false, 20, 456, 456, 4, 4 * 456 + 600, 152));
  EXPECT(true, one(kCar, 1, false, 20, 149));
  EXPECT(true, keeps_order(kCar, 1, true, false, 60, 297, 608, 2, 594, 152));
  EXPECT(false, keeps_order(kCar, 2, true, false, 60, 257, 304, 4, 1028, 152));
  EXPECT(false, keeps_order(kCar, 4, true, false, 60, 188, 608, 4, 750, 152));
  // an SM that holds one block has nothing to double up
  EXPECT(false, keeps_order(kCar, 1, true, false, 60, 152, 152, 8, 1563, 152));
  EXPECT(false, keeps_order(kCar, 2, true, false, 60, 128, 152, 8, 1024, 152));
""")


def test_sorted_units_where_they_pay(tmp_path):
    _run(tmp_path, r"""
// balance bot (blocks of 256, one per SM) and race car, two candidates per thread
static bool bot(int H, long long n) { return units_pay(kBot, H, n, 32, 8 * 152); }
static bool car(int H, long long n) { return units_pay(kCar, H, n, 64, 8 * 152); }
int main() {
  EXPECT(false, bot(20, 1048576));
  EXPECT(false, bot(30, 1048576));
  EXPECT(true, bot(36, 1048576));
  EXPECT(true, bot(50, 65536));
  EXPECT(false, bot(50, 60000));
  EXPECT(true, car(60, 65536));
  EXPECT(true, car(20, 65536));
  EXPECT(false, car(60, 100000));
  EXPECT(true, car(60, 176366));
  EXPECT(false, car(20, 176366));
  EXPECT(false, car(44, 176366));
  EXPECT(false, car(20, 262143));
  EXPECT(true, car(20, 195473));
  EXPECT(true, car(20, 155648));
  EXPECT(true, car(44, 160737));
  EXPECT(false, car(20, 160737));
  EXPECT(true, units_pay(kCar, 60, 24000, 32, 8 * 152));
""")


def test_served_batches_take_the_faster_shape(tmp_path):
    _run(tmp_path, r"""
// one lane per candidate: 32 slots a tile, eight warps an SM; `ragged` more tiles
static int car(int per_sm, bool mixed = false, int ragged = 0) {
  return serve_alt(kCar, 152LL * per_sm, 152LL * per_sm / 32 + ragged, 8 * 152, mixed, 152);
}
int main() {
  EXPECT(0, car(20));
  EXPECT(1, car(100));
  EXPECT(-1, car(200));
  EXPECT(-1, car(256));
  EXPECT(1, car(256, false, 3));
  EXPECT(1, car(470, true));
  EXPECT(1, car(505, true));
  EXPECT(-1, car(520, true));
  EXPECT(1, car(275));
  EXPECT(1, car(420));
  EXPECT(-1, car(450));
  EXPECT(-1, car(505));
  EXPECT(-1, car(1000));
  EXPECT(2, car(1250));
  EXPECT(-1, serve_alt(kBot, 100, 4, 8 * 152, false, 152));
  // one tile per warp: 256 slots per SM, a tile of two candidates per thread 512
  EXPECT(true, serve_units_pay(kCar, 1, 100, 550 * 152, 256 * 152));
  EXPECT(false, serve_units_pay(kCar, 1, 60, 550 * 152, 256 * 152));
  EXPECT(false, serve_units_pay(kCar, 1, 60, 800 * 152, 256 * 152));
  EXPECT(false, serve_units_pay(kCar, 1, 100, 500 * 152, 256 * 152));
  EXPECT(true, serve_units_pay(kCar, 2, 60, 1250 * 152, 512 * 152));
  EXPECT(false, serve_units_pay(kBot, 1, 60, 1078 * 152, 256 * 152));
  EXPECT(false, serve_units_pay(kBot, 1, 60, 1150 * 152, 256 * 152));
  EXPECT(true, serve_units_pay(kBot, 1, 60, 1250 * 152, 256 * 152));
  EXPECT(false, serve_units_pay(kBot, 1, 30, 2500 * 152, 256 * 152));
""")


def test_candidates_per_thread_of_one_lane_shapes(tmp_path):
    _run(tmp_path, r"""
int main() {
  EXPECT(1, one_lane_cands(kCar, 38912, 152));
  EXPECT(2, one_lane_cands(kCar, 39000, 152));
  EXPECT(1, one_lane_cands(kBot, 1048576, 152));
""")
