// The chunk records of the FP32 step (bsb_simt.cu).  A chunk is 8 of the 128 columns of one
// FP32 tile.  A graph's tiles outgrow 32-bit chunk offsets from 2^20 tiles (64 GiB) on, so a
// record counts from the first tile of its row tile: 31 bits hold 2^20 tiles of one row
// tile, a block of 2^27 vertices, beyond any tile storage.  The row tile's own offset is
// 64-bit.  Plain C++ (no CUDA types), so a host compiler checks it at tile counts that need
// no memory.
#pragma once

#include <stdint.h>

#ifdef __CUDACC__
#define QH_CHUNK_FN __host__ __device__ __forceinline__
#else
#define QH_CHUNK_FN static inline
#endif

namespace qh {

constexpr int F32_TILE = 128;
constexpr int F_COLS = 8;  // columns of a chunk: one 32-byte sector of x
constexpr int F_TILE_CHUNKS = F32_TILE / F_COLS;

// Chunk c (0 .. F_TILE_CHUNKS - 1) of tile e (0 .. n_hi - 1) of a row tile.
QH_CHUNK_FN int32_t f32_chunk(int32_t e, int32_t c) {
  return e * (F32_TILE * F32_TILE / F_COLS) + c;
}

// The first chunk of a row tile whose first tile is f32_begin, and the address of a record's
// first column.  The form matters to the compiler: 80 reads at R = 32 / hifi-region at
// R = 1,024 take 2.09 / 59.4 us a step with this one, 2.13 / 59.1 with a pointer to the row
// tile, 2.17 / 62.0 with an offset from here added to the tiles' address by the caller.
QH_CHUNK_FN int64_t f32_row_chunk(int32_t f32_begin) {
  return (int64_t)f32_begin * (F32_TILE * F32_TILE / F_COLS);
}
QH_CHUNK_FN const float* f32_chunk_at(const float* tiles, int64_t row_chunk, int32_t rec) {
  return tiles + (row_chunk + rec) * F_COLS;
}

}  // namespace qh
