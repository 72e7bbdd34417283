// Index arithmetic of the whole-item attention kernel's rings of key and value tiles, apart from the kernel so that the
// protocol can be walked on the host with copies that land in any order.
//
// A full barrier is waited on by the parity of its phase, which tells a phase apart only from its neighbours: a waiter that has
// not seen the phase before the one it wants to end may be let through by the phase before that.  So every waiter must see EVERY phase of
// the barriers it waits on.  Where the streams share all tiles each of them does, and tile j uses the barrier of its
// stage.  Where they take the tiles in turn (stream = tile mod STREAMS) a barrier must only ever carry tiles of one stream: the
// number of full barriers is a multiple of STREAMS, twice the stages when these are odd, and tile j uses barrier j mod that number.
// The empty barriers have one waiter, the producer, which waits on every phase of each.  (The added barriers cost nothing that shows: 16 heads of 128,
// 820 queries x 7245 keys 58 -> 59 us, 1024 x 2410 23 -> 22, 576 x 1386 15 -> 15.)
#pragma once

#if defined(__CUDACC__)
#define FV_RING_FN __host__ __device__ __forceinline__ static constexpr
#else
#define FV_RING_FN static constexpr
#endif

namespace fv {

// STAGES tiles in flight; STREAMS 1: every stream works on every tile, 2: two streams take the tiles in turn.
template <int STAGES, int STREAMS> struct TileRing {
  static constexpr int kFull = STAGES % STREAMS == 0 ? STAGES : STAGES * STREAMS;   // full barriers
  static_assert(kFull % STREAMS == 0 && kFull % STAGES == 0, "a full barrier belongs to one stream and to one stage");
  FV_RING_FN int stage(int j) { return j % STAGES; }
  FV_RING_FN int full(int j) { return j % kFull; }
  FV_RING_FN unsigned full_parity(int j) { return (unsigned)(j / kFull) & 1u; }            // the consumer's wait for tile j
  FV_RING_FN unsigned empty_parity(int j) { return ((unsigned)(j / STAGES) & 1u) ^ 1u; }   // the producer's wait before tile j
};

}  // namespace fv
