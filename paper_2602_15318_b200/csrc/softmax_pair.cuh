// How the two softmax warps that share a row (verification, one row block) keep the same reference maximum.
//
// They work through the piece's tiles apart from one another, each on its own half of a tile's keys.  Two things have to hold
// whatever the timing: nobody waits for a partner that does not come, and the results do not depend on who came first.
//
// A warp *passes* tile j when it has looked at its scores; where one of them has outgrown its row's reference the row's maximum in this
// half is the warp's own new reference, posted as it passes.  Then it makes P of the tile.  It *settles* the tile when its
// partner has passed it too: the row's reference is now the larger of the two, and P, the sums and this warp's half of the
// accumulator follow where they were made with another one.  It passes the next tile and hands P over only behind that.  So
// both look at tile j + 1 with one reference, a function of the scores up to tile j, and every P and every accumulator goes through the
// same roundings in every order of events.  Neither is ever more than one tile ahead, and P held back until then costs nothing: the product
// needs the partner's half as well.  Nobody waits for what waits for him: the scores of tile j stand behind the product of tile j - 3,
// whose P both hand over when they have passed tile j - 2, and a partner passes tile j - 1 without this warp's P of it.
// What a warp posts lies there until its partner has read it: with a move in each of two tiles in a row it waits for that.
// The piece's first tile, in which nearly every row gets its reference, is the exception: there both wait for one another at a
// barrier before they pass.
#pragma once
#include <stdint.h>

namespace sparrow {
namespace tc {

// The posted word: tiles passed; whether the last of them is settled (posted only where the partner's move was read for that); and
// whether references moved in the last of them (bit 0) and in the one before (bit 1).
__host__ __device__ __forceinline__ int pair_word(int passed, bool settled, uint32_t moved) { return 8 * passed + (settled ? 4 : 0) + (int)(moved & 3u); }
__host__ __device__ __forceinline__ int pair_passed(int word) { return word >> 3; }
// Tile j is passed and nothing moved: as good as settled.
__host__ __device__ __forceinline__ bool pair_quiet(int word, int j) { return pair_passed(word) > j && (word & 3) == 0; }
// Did references move in tile j?  (Of a partner that has passed it, by a warp that has not passed the next.)
__host__ __device__ __forceinline__ bool pair_moved(int word, int j)
{
    const int later = pair_passed(word) - (j + 1);
    return later < 2 && ((word >> later) & 1) != 0;
}
// Tile j is settled: what was posted for it has been read.
__host__ __device__ __forceinline__ bool pair_settled(int word, int j) { return pair_passed(word) > j + 1 || (pair_passed(word) == j + 1 && (word & 4) != 0); }

}  // namespace tc
}  // namespace sparrow
