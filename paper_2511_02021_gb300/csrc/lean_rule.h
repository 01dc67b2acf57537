// Which form of the lean mixed column a state runs (host code only; the forms are in lean_column.h
// and give the same bits).
#pragma once
#include <cstddef>
#include <cstdint>

namespace icon {

// launch forms (the tile of kind K_MX_LEAN: lanes 2, block one of these): blocks of four or eight
// warps per 32 columns, the rule below, one column per thread with loads one or two levels ahead
enum { LEAN_TILE4 = 6, LEAN_TILE8 = 8, LEAN_RULE = 9, LEAN_COLUMN1 = 10, LEAN_COLUMN2 = 12 };

constexpr int kLeanPitch = 33;             // shared row pitch: conflict-free by columns and by levels
inline size_t lean_tile_bytes(int N, bool topo) {
  return (size_t)N * kLeanPitch * (sizeof(double) + 3 * sizeof(float)) +
         (topo ? (size_t)(N + 1) * kLeanPitch * sizeof(float) : 0);
}

// By tiles of 32 columns per SM and by how many of them an SM holds: a tile takes 660 bytes of
// shared memory per level (792 over terrain), so five blocks of four warps up to 69 levels (57),
// two blocks of eight warps up to 175 (145), one beyond. Up to three tiles per SM eight warps shorten
// a tile's parallel parts, at any number of levels (R2B3/180: 130 us a launch, mean of the stages,
// against 254 one column per thread; over terrain 225 against 327). Up to eight: four warps a tile
// while all of them are resident at once (R2B4/60: 64 against 99; terrain R2B4/57: 99 against 125);
// then, on flat levels, eight warps while an SM holds two (R2B4/128: 174 against 205 by columns and
// 225 with four warps; R2B4/174: 236 against 287; over terrain the columns are level or ahead, R2B4/58:
// 127 against 143, R2B4/128: 274 against 265). With one tile at a time, or more tiles, the warps of
// columns fill the SMs better (R2B4/180: 290 against 328 and 457; terrain R2B4/256: 543 against 766
// and 1297; R2B5/90: 250 / 295 against 273 / 397).
inline int lean_form_for(int64_t cells, int N, bool topo, int sms, size_t shared_per_sm, size_t reserved_per_block) {
  const int64_t tiles = (cells + 31) / 32;
  if (tiles <= 3 * (int64_t)sms) return LEAN_TILE8;
  if (tiles <= 8 * (int64_t)sms) {
    const int64_t fit = (int64_t)(shared_per_sm / (lean_tile_bytes(N, topo) + reserved_per_block));
    const int64_t four = fit < 5 ? fit : 5;              // 102 registers: five blocks of four warps
    if (tiles <= four * sms) return LEAN_TILE4;
    if (!topo && fit >= 2) return LEAN_TILE8;
  }
  return topo ? LEAN_COLUMN1 : LEAN_COLUMN2;
}

}  // namespace icon
