// Which form of the morphing forward transform a call takes (morph_api.cu).
#pragma once

namespace fftenkf {

constexpr int kMorphTX = 64;        // nodes of a tile along x
constexpr int kMorphThreads = 256;  // threads of a CTA

enum MorphForm { kMorphGather, kMorphTiles8, kMorphTiles16 };

// Tiles of 16 rows from one wave of 8 CTAs per SM on; 8 rows below (256^2, K = 4: 15 us, 17 with 16 rows); no
// tiles where they hardly pay their halo and padding: up to three CTAs of nodes per SM (62 x 173, K = 9: 11 us,
// 13 with tiles), or less than 60 % of the tiles' columns on the grid (2400 x 65, K = 6: 40 us, 42 with tiles;
// 1692 x 77, 60 %: 35.5 both).  Tiles stay ahead for displacements beyond their halo (2048^2, K = 4, M = 2, up
// to 3, 10 and 30 cells: 286, 441 and 1244 us; gathers 496, 788 and 1417).
inline MorphForm morph_form(int ny, int nx, int K, int sms) {
  const long long tiles_x = (nx + (long long)kMorphTX - 1) / kMorphTX;
  if ((long long)ny * nx * K <= 3LL * sms * kMorphThreads || 5LL * nx < 3 * kMorphTX * tiles_x) return kMorphGather;
  return tiles_x * ((ny + 15) / 16) * K >= 8LL * sms ? kMorphTiles16 : kMorphTiles8;
}

}  // namespace fftenkf
