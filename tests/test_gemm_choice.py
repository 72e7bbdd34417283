"""The rule that picks a GEMM's tile, compiled for the host from the launcher's own header."""
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
PROGRAM = r"""
#include <cstdio>
#include "paper_2503_23367_b200/csrc/gemm_choice.h"
int main() {
  int M, N, K, hd, clusters;
  while (scanf("%d %d %d %d %d", &M, &N, &K, &hd, &clusters) == 5) {
    const fv::TileChoice t = fv::pick_tile(M, N, K, 148, hd, clusters);
    printf("%d %d %d\n", t.bn, (int)t.pair, t.slices);
  }
}
"""


@pytest.fixture(scope="module")
def pick(tmp_path_factory):
    d = tmp_path_factory.mktemp("choice")
    src, exe = str(d / "choice.cpp"), str(d / "choice")
    with open(src, "w") as f:
        f.write(PROGRAM)
    subprocess.run(["g++", "-std=c++17", "-O1", "-I", ROOT, src, "-o", exe], check=True)

    def run(shapes, clusters=1):
        text = "\n".join(" ".join(map(str, (*s, clusters))) for s in shapes)
        out = subprocess.run([exe], input=text, check=True, capture_output=True, text=True).stdout
        return [tuple(map(int, line.split())) for line in out.splitlines()]

    return run


def _one_cta_cost(bn, M, N, K):
    fixed, per_round, per_kb = {128: (3.63, 0.81, 0.214), 192: (3.53, 1.79, 0.251), 256: (2.87, 2.28, 0.343)}[bn]
    ctas = -(-M // 128) * -(-N // bn)
    return fixed + -(-ctas // 148) * (per_round + -(-K // 64) * per_kb)


def _cost(bn, pair, M, N, K):
    fixed, per_round, per_kb = {(64, 0): (3.17, 0.42, 0.151), (128, 0): (3.63, 0.81, 0.214), (192, 0): (3.53, 1.79, 0.251), (256, 0): (2.87, 2.28, 0.343),
                                (128, 1): (5.09, 1.11, 0.168), (256, 1): (6.47, 1.55, 0.292)}[bn, pair]
    ctas = -(-M // (256 if pair else 128)) * -(-N // bn)
    return fixed + -(-ctas // (74 if pair else 148)) * (per_round + -(-K // 64) * per_kb)


@pytest.mark.parametrize("C", [256, 1024, 1920, 2048])
def test_rows_of_a_map_take_the_cheapest_tile_that_is_no_cluster(pick, C):
    seen = set()
    for K in (C, 4 * C):
        shapes = [(M, C, K, 0) for M in range(128, 6600, 37)]
        for (M, _, _, _), (bn, pair, slices) in zip(shapes, pick(shapes, clusters=0)):
            assert slices == 1
            every = [(b, 0) for b in (64, 128, 192, 256)] + ([(128, 1), (256, 1)] if M > 256 else [])
            assert _cost(bn, pair, M, C, K) <= min(_cost(*t, M, C, K) for t in every) + 1e-6, (M, K, bn, pair)
            seen.add((bn, pair))
    if C == 2048:
        assert seen == {(64, 0), (128, 0), (192, 0), (256, 0), (128, 1), (256, 1)}         # every build of that epilogue is in use


@pytest.mark.parametrize("C,head_dim", [(256, 64), (512, 64), (1024, 64), (1024, 128), (1536, 128), (1920, 64), (2048, 128)])
def test_projection_with_head_norms_or_rotation_takes_the_cheapest_tile_it_may_use(pick, C, head_dim):
    rows = list(range(1, 4000, 13))
    allowed = [bn for bn in (128, 192, 256) if bn % head_dim == 0]
    for M, (bn, pair, slices) in zip(rows, pick([(M, 3 * C, C, head_dim) for M in rows])):
        assert bn in allowed and not pair and slices == 1
        assert _one_cta_cost(bn, M, 3 * C, C) <= min(_one_cta_cost(b, M, 3 * C, C) for b in allowed) + 1e-6, (M, bn)


def test_clusters_only_while_all_their_ctas_run_at_once(pick):
    shapes = [(M, N, K, 0) for M in (1, 40, 129, 256, 400, 820, 1640, 3277) for N in (64, 1024, 2048, 6144, 8192) for K in (256, 512, 2048, 8192)]
    seen = set()
    for (M, N, K, _), (bn, pair, slices) in zip(shapes, pick(shapes)):
        seen.add((pair, slices > 1))
        if slices > 1:
            assert not pair and K >= 512 and -(-M // 128) * -(-N // bn) * slices <= 148
        if pair:
            assert M > 256
    assert seen == {(0, False), (0, True), (1, False)}
