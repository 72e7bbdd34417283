// Which GEMM kernel and tile a shape takes.  Host code only, apart from the launcher so that the rule can be checked without a GPU.
#pragma once

namespace fv {

// Kernel and tile for a shape.  Measured on B200 (launches replayed from a CUDA graph, so that the host does not pace
// them, weights rotating through HBM), one launch costs about
//     fixed + rounds x (per_round + k-blocks x per_kblock)
// where rounds = ceil(CTAs / SMs), or pairs / half the SMs.  A k-block of a 128-wide tile is paced by the operand loads (an SM takes
// in about 110 bytes per clock, whatever the tile), the wider tiles by the MMAs themselves; wider tiles and CTA pairs win by needing
// fewer rounds and less L2 traffic per flop.  Where tiles leave SMs idle, the CTAs of a cluster share a tile's K (2 or 4 slices,
// gemm_cluster.cu); those only compete while all their CTAs run at once.
struct TileChoice { int bn; bool pair; int slices; };   // slices 1: no cluster
// head_dim > 0: the QKV projection with head norms or rotation, whose epilogue exists for one-CTA tiles of at least 128 columns that hold
// whole heads; only those are compared.  (Taking the cheapest of all and widening it until it was allowed: blocks of 820 and 1024 rows at C 2048 with 128-wide
// heads 133 and 139 us, now 129 and 135; 3249 rows at C 1024 193 -> 187.)
// clusters false: the residual epilogue that writes rows of a map, which clusters do not have.
inline TileChoice pick_tile(int M, int N, int K, int sms, int head_dim = 0, bool clusters = true) {
  const int num_kb = (K + 63) / 64;
  struct Cand { int bn; bool pair; int slices; double fixed_us, round_us, kb_us; };
  // Least-squares fits over M 36 ... 3277 x the four projection shapes of 1024-, 1920- and 2048-wide blocks, every candidate forced.  On
  // that sweep the choice costs 0.3 % over the best candidate on average (10 % at worst, 0.5 us); e.g. (us) N 2048 K 8192: M 400 64-wide
  // 23.0, 128 x 2 24.5; M 820 pair of 128 27.7, 128-wide 31.7, 192-wide 35.5; N 1024 K 4096: M 400 64 x 2 9.9, 128 x 4 11.4; M 816 64-wide
  // 12.8, 128 x 2 14.5; N 2048 K 2048 M 3277 192-wide 24.6, 128-wide 30.4.
  const Cand cand[10] = {{128, false, 1, 3.63, 0.81, 0.214}, {192, false, 1, 3.53, 1.79, 0.251}, {256, false, 1, 2.87, 2.28, 0.343},
                         {256, true, 1, 6.47, 1.55, 0.292}, {128, true, 1, 5.09, 1.11, 0.168}, {64, false, 1, 3.17, 0.42, 0.151},
                         {64, false, 4, 3.79, 0.0, 0.228}, {64, false, 2, 3.48, 0.0, 0.196},
                         {128, false, 4, 5.75, 0.0, 0.304}, {128, false, 2, 5.38, 0.0, 0.295}};
  TileChoice best{128, false, 1};
  double best_cost = 1e30;
  for (const Cand& c : cand) {
    if (c.pair && M <= 256) continue;
    if (!clusters && c.slices > 1) continue;
    if (head_dim > 0 && (c.pair || c.slices > 1 || c.bn < 128 || c.bn % head_dim)) continue;
    const int rows = c.pair ? 256 : 128;
    const int slots = c.pair ? sms / 2 : sms;
    const long ctas = (long)((M + rows - 1) / rows) * ((N + c.bn - 1) / c.bn) * c.slices;
    if (c.slices > 1 && (ctas > slots || num_kb < 8)) continue;
    const long rounds = (ctas + slots - 1) / slots;
    const double cost = c.fixed_us + (double)rounds * (c.round_us + (num_kb + c.slices - 1) / c.slices * c.kb_us);
    if (cost < best_cost - 1e-9) { best_cost = cost; best = TileChoice{c.bn, c.pair, c.slices}; }
  }
  return best;
}

// Rows of a map on 64-wide tiles: whether to take the build that leaves room on its SMs for the restoration of the map's other rows.  It costs such a GEMM some
// 0.5 us (112 registers against 158) and pays once that restoration outlasts what runs in front of the GEMM.  The line lies at 4 million elements of other rows: over 443 steps of
// 130 ... 800 kept rows, C 256 ... 2048, maps of 24 x 24 ... 128 x 128, below it the step is up to 2.9 % shorter without, above it 1 ... 12 % shorter with (at worst 1 % longer).
inline bool gemm_leaves_room(int M, int rows_per_image, int map_tokens, int N) {
  return (double)(M / rows_per_image) * (map_tokens - rows_per_image) * N > 4e6;
}

}  // namespace fv
