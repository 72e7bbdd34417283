"""The rings of key and value tiles in the whole-item attention kernel, walked on the host: a model of their barriers whose copies
land in any order and whose producer and streams run in any interleaving, on the index arithmetic the kernel is compiled from.
No stream may pass its wait for a tile whose stage does not hold that tile, no copy may overwrite a tile that is still read, and
every walk ends."""
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

MODEL = r"""
#include <cstdio>
#include <cstdlib>
#include <random>
#include <vector>
#include "paper_2503_23367_b200/csrc/attention_ring.h"

// The oracle's own planted mistake: one full barrier per stage although the streams take the tiles in turn.
template <int STAGES> struct SharedBarriers {
  static constexpr int kFull = STAGES;
  static int stage(int j) { return j % STAGES; }
  static int full(int j) { return j % STAGES; }
  static unsigned full_parity(int j) { return (j / STAGES) & 1; }
  static unsigned empty_parity(int j) { return ((j / STAGES) & 1) ^ 1; }
};

struct Barrier {   // phases completed so far; a wait on a parity is over when the phase in progress has the other one
  unsigned done = 0;
  int arrivals = 0;
  bool passes(unsigned parity) const { return ((done + 1) & 1) == parity; }
};

template <class Ring, int STAGES, int STREAMS> int walk(int tiles, int streams, unsigned seed) {
  std::mt19937 rng(seed);
  std::vector<Barrier> full(Ring::kFull), empty(STAGES);
  std::vector<int> holds(STAGES, -1), busy(STAGES, 0);   // tile in a stage (-2: a copy is writing it); its readers
  std::vector<int> flight;
  int produced = 0;
  std::vector<int> next(streams), reading(streams, -1);
  for (int t = 0; t < streams; ++t) next[t] = STREAMS > 1 ? t : 0;
  const int readers = STREAMS > 1 ? 1 : streams;         // arrivals an empty barrier takes
  for (int step = 0; step < 400 * (tiles + 4); ++step) {
    bool over = produced == tiles && flight.empty();
    for (int t = 0; t < streams; ++t) over = over && next[t] >= tiles && reading[t] < 0;
    if (over) return 0;
    switch (rng() % 3) {
      case 0: {   // the producer requests the next tile
        const int j = produced;
        if (j < tiles && empty[Ring::stage(j)].passes(Ring::empty_parity(j))) {
          if (busy[Ring::stage(j)]) return 1;            // overwritten under a reader
          holds[Ring::stage(j)] = -2;
          flight.push_back(j);
          ++produced;
        }
        break;
      }
      case 1: {   // some copy lands
        if (flight.empty()) break;
        const size_t i = rng() % flight.size();
        const int j = flight[i];
        flight.erase(flight.begin() + i);
        holds[Ring::stage(j)] = j;
        ++full[Ring::full(j)].done;
        break;
      }
      default: {  // a stream moves on
        const int t = rng() % streams;
        if (reading[t] >= 0) {
          const int s = Ring::stage(reading[t]);
          --busy[s];
          if (++empty[s].arrivals == readers) { empty[s].arrivals = 0; ++empty[s].done; }
          reading[t] = -1;
        } else if (next[t] < tiles && full[Ring::full(next[t])].passes(Ring::full_parity(next[t]))) {
          const int j = next[t];
          if (holds[Ring::stage(j)] != j) return 2;      // let through before its tile was there
          ++busy[Ring::stage(j)];
          reading[t] = j;
          next[t] += STREAMS;
        }
      }
    }
  }
  return 3;                                              // stuck
}

template <class Ring, int STAGES, int STREAMS> int worst(int streams) {
  for (int tiles = 1; tiles <= 20; ++tiles)
    for (unsigned seed = 0; seed < 400; ++seed) {
      const int r = walk<Ring, STAGES, STREAMS>(tiles, streams, 1000 * tiles + seed);
      if (r) return r;
    }
  return 0;
}

int main() {
  // the builds of the kernel: 128-wide heads 2 stages (shared tiles) or 3 (in turn), 64-wide heads 4 stages
  printf("%d %d %d %d %d %d ", worst<fv::TileRing<2, 1>, 2, 1>(2), worst<fv::TileRing<2, 1>, 2, 1>(1), worst<fv::TileRing<4, 1>, 4, 1>(2),
         worst<fv::TileRing<4, 1>, 4, 1>(1), worst<fv::TileRing<3, 2>, 3, 2>(2), worst<fv::TileRing<4, 2>, 4, 2>(2));
  printf("%d %d\n", worst<SharedBarriers<3>, 3, 2>(2), worst<SharedBarriers<4>, 4, 2>(2));
}
"""


@pytest.fixture(scope="module")
def verdicts(tmp_path_factory):
    d = tmp_path_factory.mktemp("ring")
    src, exe = str(d / "ring.cpp"), str(d / "ring")
    with open(src, "w") as f:
        f.write(MODEL)
    subprocess.run(["g++", "-std=c++17", "-O2", "-I", ROOT, src, "-o", exe], check=True)
    return [int(v) for v in subprocess.run([exe], check=True, capture_output=True, text=True).stdout.split()]


def test_no_stream_passes_its_wait_before_its_tile_has_landed(verdicts):
    assert verdicts[:6] == [0] * 6


def test_the_model_finds_a_full_barrier_shared_by_two_streams(verdicts):
    assert verdicts[6] == 2                    # three stages: tile j - 3 belongs to the other stream
    assert verdicts[7] == 0                    # four stages: tile j - 4 is the stream's own


def test_the_kernel_takes_its_ring_from_the_model_s_header():
    """One producer and one consumer expression per ring, none of them spelled out beside the header."""
    text = open(os.path.join(ROOT, "paper_2503_23367_b200", "csrc", "attention.cu")).read()
    whole = text[text.index("attention_whole_kernel("):text.index("bool make_tmap_rows")]
    assert "using Ring = TileRing<NS, ONE_TILE ? 2 : 1>" in whole
    assert "% NS" not in whole and "/ NS" not in whole
