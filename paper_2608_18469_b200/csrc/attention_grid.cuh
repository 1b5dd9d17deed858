// Blocks of the attention kernels: one per (tile of 128 rows, sequence, head), in one grid dimension with the tile as the
// slowest index, so that all heads' long walks start first.  (Three dimensions would hold at most 65535 tiles, sequences
// of 8.4 M positions, or as many sequences.)
#pragma once

namespace erase {

constexpr long long ATTN_MAX_BLOCKS = 0x7fffffffLL;

__host__ __device__ inline long long attn_blocks(int heads, int batch, int tiles) { return (long long)heads * batch * tiles; }

struct AttnPlace { int tile, seq, head; };
__host__ __device__ inline AttnPlace attn_place(unsigned block, unsigned heads, unsigned batch) {
  const unsigned r = block / heads;
  return AttnPlace{(int)(r / batch), (int)(r % batch), (int)(block % heads)};
}

}  // namespace erase
