// Which 128-token tiles a block of the persistent bidirectional kernels walks.
//
// The tiles of all units ((batch, head) pairs) form one list, unit after unit.  stream: block i takes the i-th of equally long
// ranges of that list, wherever they cut a unit; a unit's pieces are then numbered by the blocks that hold them.  Otherwise
// every unit is cut into `per_unit` pieces of `piece` tiles (the last one shorter), and blocks take whole pieces.
#pragma once
#include <stdint.h>

struct TileWork {
  int units, tiles;          // tiles per unit
  int piece, per_unit;       // pieces (not stream)
  int stream;
  int slots;                 // places per unit in the array of partial results
};

struct TileIter {
  int c, end;                // position in the list of tiles (stream) or pieces
  int bh, tile0, ntiles, idx, blk, nblk;
  // the blocks that hold tile t of a stream
  static __host__ __device__ int block_of(const TileWork& w, int64_t t, int nblk) {
    return (int)(((t + 1) * nblk - 1) / ((int64_t)w.units * w.tiles));
  }
  __host__ __device__ void begin(const TileWork& w, int block, int blocks) {
    const int64_t n = w.stream ? (int64_t)w.units * w.tiles : (int64_t)w.units * w.per_unit;
    blk = block;
    nblk = blocks;
    c = (int)(n * block / blocks);
    end = (int)(n * (block + 1) / blocks);
    bh = tile0 = ntiles = idx = 0;
  }
  // the next tile: tile0 + idx of unit bh; false at the end
  __host__ __device__ bool next(const TileWork& w) {
    if (idx + 1 < ntiles) { idx++; return true; }
    return next_piece(w);
  }
  // the next piece: ntiles tiles from tile0 on
  __host__ __device__ bool next_piece(const TileWork& w) {
    if (c >= end) { ntiles = 0; return false; }
    idx = 0;
    if (w.stream) {
      bh = c / w.tiles;
      tile0 = c % w.tiles;
      ntiles = w.tiles - tile0 < end - c ? w.tiles - tile0 : end - c;
      c += ntiles;
    } else {
      bh = c / w.per_unit;
      const int p = c % w.per_unit;
      tile0 = p * w.piece;
      ntiles = w.tiles - tile0 < w.piece ? w.tiles - tile0 : w.piece;
      c++;
    }
    return true;
  }
  __host__ __device__ bool first() const { return idx == 0; }
  __host__ __device__ bool last() const { return idx + 1 >= ntiles; }
  // where the partial result of the piece goes
  __host__ __device__ int slot(const TileWork& w) const {
    return bh * w.slots + (w.stream ? blk - block_of(w, (int64_t)bh * w.tiles, nblk) : tile0 / w.piece);
  }
  __host__ __device__ int tile() const { return tile0 + idx; }
};
// number of partial results of unit bh
static __host__ __device__ inline int work_pieces(const TileWork& w, int bh, int nblk) {
  if (!w.stream) return w.per_unit;
  return TileIter::block_of(w, (int64_t)(bh + 1) * w.tiles - 1, nblk) - TileIter::block_of(w, (int64_t)bh * w.tiles, nblk) + 1;
}
// the unit that the end of block i's range of a stream cuts, or -1: it cuts none, or block i - 1's end cuts the same one
static __host__ __device__ inline int cut_unit(const TileWork& w, int i, int nblk) {
  const int64_t n = (int64_t)w.units * w.tiles, c = n * (i + 1) / nblk;
  const int unit = (int)(c / w.tiles);
  const int64_t start = (int64_t)unit * w.tiles;
  return c == start || n * i / nblk > start ? -1 : unit;
}
