"""The rules by which the roles of a thread block agree on its work units (csrc/ts_units.h), run on the host.

The two warps of a row pair meet on a barrier that has no time limit, so after a time-out, when all
other waits end early and the K loader is no longer held back, they must still meet equally often and
read the same unit. A small simulation steps the K loader and both warps in random order, lets a
wait run out at a random moment, and compares what the warps did."""
import os
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(HERE, "..", "paper_2512_03416_b200", "csrc")

HARNESS = r"""
#include "ts_units.h"
#include <cstdio>
#include <cstdlib>
#include <random>
using namespace ts;
// argv[1]: 1 = the K loader goes on after a failure, 2 = the second warp goes by its own record
int main(int argc, char** argv) {
  const int broken = atoi(argv[1]);
  for (unsigned seed = 0; seed < 4000; ++seed) {
    std::mt19937 rng(seed);
    auto roll = [&](int n) { return (int)(rng() % (unsigned)n); };
    const int n_units = 1 + roll(60), tile_tokens = 32, x = roll(2), fail_at = roll(400);
    UnitRec ring[kSchedRing] = {};
    int published = 0, taken = 0;
    bool failed = false, closed = false;
    int k[2] = {0, 0}, phase[2] = {0, 0}, read_w[2] = {-2, -2}, posted = -2;
    long meets[2] = {0, 0};
    for (int t = 0; phase[0] != 9 || phase[1] != 9; ++t) {
      if (t > 100000) return printf("seed %u: the warps wait for each other\n", seed), 1;
      failed = failed || t >= fail_at;
      const int who = failed ? roll(6) : roll(3);               // after a failure the K loader is the quickest
      if (who >= 2) {                                            // K loader
        const bool held_back = !failed && published > (k[0] < k[1] ? k[0] : k[1]) + 2;
        if (closed || held_back) continue;
        const int w = next_unit(failed && broken != 1, false, 0, n_units, [&]() { return taken++; });
        UnitRec r = {};
        r.w = -1;
        if (w < n_units) { r.w = w; r.q_count = 1 + (w * 7) % (2 * tile_tokens); r.ctx = (w * 131) % 900; }
        closed = r.w < 0;
        ring[published++ % kSchedRing] = r;
        continue;
      }
      const UnitRec r = ring[k[who] % kSchedRing];
      const PfUnit u = unit_shape(r, tile_tokens);
      if (who == 0 && phase[0] == 0) {                           // first warp: is there a unit, how many blocks
        if (published <= k[0] && !failed) continue;
        const bool have = published > k[0] && r.w >= 0;
        posted = posted_blocks(have, u, x);
        read_w[0] = have ? r.w : -1;
        phase[0] = 1;
      } else if (who == 1 && phase[0] == 1 && phase[1] == 0) {   // they have met; second warp reads the record
        read_w[1] = posted < 0 ? -1 : r.w;
        if (read_w[0] != read_w[1]) return printf("seed %u: units %d and %d\n", seed, read_w[0], read_w[1]), 1;
        const int mine = broken == 2 && failed && posted >= 0 ? posted_blocks(r.w >= 0, unit_shape(ring[(k[1] + 1) % kSchedRing], tile_tokens), x) : posted;
        ++meets[0]; ++meets[1];
        meets[0] += posted > 0 ? posted + 2 : posted == 0; meets[1] += mine > 0 ? mine + 2 : mine == 0;
        if (meets[0] != meets[1]) return printf("seed %u: %ld and %ld meetings\n", seed, meets[0], meets[1]), 1;
        for (int i = 0; i < 2; ++i) { phase[i] = posted < 0 ? 9 : 0; ++k[i]; }
      }
    }
  }
  return 0;
}
"""


@pytest.fixture(scope="module")
def harness(tmp_path_factory):
    d = tmp_path_factory.mktemp("ring")
    src, exe = d / "ring.cpp", d / "ring"
    src.write_text(HARNESS)
    subprocess.check_call(["g++", "-std=c++17", "-O1", "-I", CSRC, "-o", str(exe), str(src)])
    return str(exe)


def test_the_warps_of_a_pair_meet_equally_often_after_a_time_out(harness):
    r = subprocess.run([harness, "0"], capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stdout


@pytest.mark.parametrize("broken", ["1", "2"], ids=["loader-goes-on", "second-warp-on-its-own"])
def test_the_simulation_sees_the_mistakes(harness, broken):
    assert subprocess.run([harness, broken], capture_output=True, timeout=300).returncode == 1
