// Tile plans of the one-barrier solves: plain arithmetic on sizes, no GPU needed.
#pragma once
#include <algorithm>
#include <cstddef>
#include <cstdint>

namespace ccm {

constexpr int kFusedTilesMax = 512;    // tiles of a launch, at most (two per SM)
constexpr int kResidentCells = 128;    // cells of a built-in resident tile, at least about
constexpr int kFusedRows = 32;         // rows of a resident tile that one thread takes, at most (bits of its masks)

// Mailbox slots of a resident plan (16 bytes each): the ring of every tile, twice.
inline size_t fused_mail_slots(int nx, int TX, int TY, int ntiles) {
  return (size_t)2 * (size_t)ntiles * 2 * (size_t)(TY + std::min(TX, nx));
}

// Tile shape for at most `blocks` blocks: TX a power of two in 32..max_tx, as many tile rows as
// the blocks allow while a tile keeps about min_cells cells and the plan needs no more than
// max_slots mailbox slots (wide flat tiles have the longest rings: a width takes fewer and taller
// ones until its rings fit, and is skipped where none fits); the shape with the smallest largest
// tile wins (then the shortest ring).  One block per tile; *ntiles = 0 if there is no such shape.
inline void fused_tiles(int nx, int ny, int blocks, int* TX, int* TY, int* nbx, int* ntiles, int min_cells = 512,
                        int max_tx = 512, size_t max_slots = SIZE_MAX) {
  long long best = -1, best_ring = 0;
  *ntiles = 0;
  for (int tx = 32; tx <= max_tx; tx *= 2) {
    const int bxn = (nx + tx - 1) / tx;
    if (bxn > blocks) continue;
    const int wx = std::min(tx, nx);
    const int min_ty = (min_cells + wx - 1) / wx;
    int byn = std::max(1, std::min(blocks / bxn, (ny + min_ty - 1) / min_ty));
    auto height = [&](int rows) { return (ny + rows - 1) / rows; };
    auto tiles = [&](int ty) { return bxn * ((ny + ty - 1) / ty); };
    while (byn > 1 && fused_mail_slots(nx, tx, height(byn), tiles(height(byn))) > max_slots) --byn;
    const int ty = height(byn);
    if (fused_mail_slots(nx, tx, ty, tiles(ty)) > max_slots) continue;
    const long long cells = (long long)wx * ty, ring = 2LL * (wx + ty);
    if (best < 0 || cells < best || (cells == best && ring < best_ring)) {
      best = cells;
      best_ring = ring;
      *TX = tx;
      *TY = ty;
      *nbx = bxn;
      *ntiles = tiles(ty);
    }
  }
}

// Computing threads of a plan's blocks, the same whether its tiles are resident or not (so that
// both run the same additions in the same order): one or two cells per thread on small tiles,
// whose iteration is paced by its barriers and block sums; 512 where the FP64 pipe sets the pace;
// 256 where two blocks of an SM share it (their threads then have registers enough).
inline int fused_threads(int TX, int TY, int ntiles, int sms) {
  const int cells = TX * TY;
  if (cells <= 256 && TX <= 128) return 128;
  if (TX <= 256 && (cells <= 1024 || (ntiles > sms && cells <= 2048))) return 256;
  return 512;
}

// Dynamic shared memory of a tile with its vectors resident (f2): x~, p, s, w, r~ with its
// one-cell frame (two of them with `defer`), the ring's s, the coefficients of every cell
// (`dcache`) or of nt listed cells (`lcache`), a list of up to one entry per cell.
inline size_t resident_smem(int TX, int TY, int nt, bool dcache, bool defer, bool lcache) {
  const size_t txy = (size_t)TX * (size_t)TY;
  return sizeof(double) * (4 * txy + (defer ? 2 : 1) * ((size_t)TX + 2) * ((size_t)TY + 2) +
                           2 * ((size_t)TX + (size_t)TY) + (dcache ? 5 * txy : 0) + (lcache ? 5 * (size_t)nt : 0)) +
         sizeof(int) * txy;
}
inline size_t fused_resident_smem_min(int TX, int TY) { return resident_smem(TX, TY, 0, false, false, false); }

// The most slots any resident plan of a grid can need, a caller's included (whose tiles may be higher
// than the grid): every tile width and height that shared memory could hold, up to kFusedTilesMax tiles.
inline size_t fused_mail_slots_max(int nx, int ny) {
  size_t most = 0;
  for (int tx = 32; tx <= 512; tx *= 2)
    for (int ty = 1; fused_resident_smem_min(tx, ty) <= 227 * 1024; ++ty) {
      const long long tiles = (long long)((nx + tx - 1) / tx) * ((ny + ty - 1) / ty);
      if (tiles <= kFusedTilesMax) most = std::max(most, fused_mail_slots(nx, tx, ty, (int)tiles));
    }
  return most;
}

}  // namespace ccm
