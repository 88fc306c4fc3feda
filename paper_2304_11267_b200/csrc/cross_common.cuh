// Tile geometry shared by the attention kernels.
#pragma once

namespace sd_attn {

constexpr int TILE_M = 128;          // query rows per tile = TMEM lanes
constexpr int CHUNK_COLS = 64;       // 16-bit elements per 128-byte swizzled row
constexpr int CHUNK_ROW_BYTES = 128;

}  // namespace sd_attn
