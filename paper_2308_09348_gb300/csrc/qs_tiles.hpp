// qs_tiles.hpp -- the kinds of shots of a batch and the sizes of their work
// items.  Plain C++: the rules are checked on the CPU against the workspace's
// slots.
#pragma once

#include <cstdint>

#include "qs_layout.hpp"

namespace qs {

// The kinds of shots, each with its own kernel (so that each keeps its own
// register budget, block and tile size) over one (shot, tile) schedule: the
// quantum model, the classical closed form, and the shots with a model
// variant (the per-cell focus, cycle-resolved chi).
enum { kKindQfp = 0, kKindLL = 1, kKindVar = 2, kKinds = 3 };

// Tile sizes (samples per work item) when the caller leaves them open, by the
// number of samples of each kind of shot, which k_bscan counts: the kinds run
// one after the other, and a few shots of one kind among many of another are
// to spread over the chip as well.  The smallest is one step of a 256-thread
// CTA.  The SM count is the full chip's, so that the workspace's slots
// (open_tiles) can be counted on the host without a device.
enum { kTileFixed = 0, kTileForward = 1, kTileAdjoint = 2 };
// powers of two, by their exponents (shifts: one thread of k_bscan does this,
// and a chain of 64-bit divisions takes 2 us)
constexpr int kMinTile = 9, kMaxTile = 13, kTopTile = 14;
constexpr int64_t kTileSms = 152;

// The largest tile from 2^t up to 2^most that leaves `leave` full ones.
QS_LAYOUT int grow_tile(int t, int most, int64_t total, int64_t leave) {
  while (t < most && total >> (t + 1) >= leave) ++t;
  return t;
}

// Forward: the largest power of two up to 8192 that leaves sixteen tiles per
// resident CTA (four per SM), so that the last round is short: 8.0e6 samples
// of the quantum model in 400 shots 5.49 ms with 512 against 5.65 with 2048,
// 7.1e5 in 40 shots 0.62 against 0.93, 80000 in 16 shots 0.25 against 0.52.
// A classical tile costs more to set up than to evaluate (at 512 samples:
// clearing and merging the spectrum), so those shots take the largest tile
// up to 16384 that leaves two per resident CTA (three per SM): a sweep of 256
// shots over 1e5 samples 149 us with 16384, 171 with 8192, 311 with 2048
// (548 one sample per thread; 130 us with everything below), 8.0e6 samples in
// 400 shots 124 us with 8192.  With a smoothed spectrum the deposits cost as
// much as a quantum sample's cells, and they take the first rule's tile (1000
// shots of 20000 samples 1583 us with 2048, 1723 with 8192; 256 shots of 20000
// 486 with 512, 701 with 8192); at least half as many samples as smoothed
// bins, up to 2048, for the clearing and merging of long spectra.
constexpr int64_t kForwardTiles = 16 * 4 * kTileSms;

// The variants' kernel has two CTAs per SM, and a tile costs it more: those
// shots take the largest tile up to 2048 that leaves eight per resident CTA
// (256 shots of 20000 samples x 128 cells, us with 512, 1024, 2048, 4096:
// per-cell focus 1416, 1312, 1314, 1317, cycle-resolved 1473, 1390, 1332, 1379,
// classical with the per-cell focus 690, 588, 549, 536; 64 shots of 160000:
// 2682, 2434, 2411, 2439 and 2808, 2645, 2554, 2574; with 512 cells 8965, 8853,
// 8842, 9034; 64 of 20000: 387, 369, 402, 457 and 404, 400, 421, 491).
QS_LAYOUT int forward_tile(int kind, int64_t total, int smooth_bins) {
  if (kind == kKindVar) return grow_tile(kMinTile, 11, total, 8 * 2 * kTileSms);
  int t = grow_tile(kMinTile, kMaxTile, total, kForwardTiles);
  if (kind == kKindQfp) return t;
  if (smooth_bins == 0) return grow_tile(t, kTopTile, total, 2 * 3 * kTileSms);
  while (t < 11 && 2 << t < smooth_bins) ++t;
  return t;
}

// Adjoint: the largest power of two up to 8192 that leaves sixteen tiles per
// CTA (one per SM), and at least one step of its 512 threads (1024 samples:
// 2^20 samples in 64 shots 1.45 ms, 1.60 with 2048).
QS_LAYOUT int adjoint_tile(int64_t total) {
  return grow_tile(kMinTile + 1, kMaxTile, total, 16 * kTileSms);
}

// With a caller's grid fewer CTAs than the chip holds may be there, and one
// step per tile leaves an SM with a single CTA idle at every edge: at least the
// largest tile up to 2048 that leaves sixteen to each of them (152 CTAs, 256
// shots of 20000 samples, quantum model: 1825 us with 512, 1515 with 2048).
QS_LAYOUT int grid_tile(int64_t total, int grid) {
  return grow_tile(kMinTile, 11, total, 16 * (int64_t)grid);
}

// The tiles (exponents) of the kinds, given their numbers of samples: by the
// rule, then doubled, the kind with the most tiles first, until they fit the
// workspace's slots (one more per shot is reserved for its last tile).
QS_LAYOUT void choose_tiles(int rule, int grid, const int64_t (&total)[kKinds],
                                    int smooth_bins, int64_t slots, int (&tile)[kKinds]) {
  const int64_t all = total[0] + total[1] + total[2];
  for (int k = 0; k < kKinds; ++k) {
    tile[k] = rule == kTileAdjoint ? adjoint_tile(all) : forward_tile(k, total[k], smooth_bins);
    if (rule == kTileForward && grid > 0) {
      const int t = grid_tile(total[k], grid);
      if (t > tile[k]) tile[k] = t;
    }
  }
  for (;;) {
    // tiles in units of 2^-kTopTile, exact: every tile divides 2^kTopTile
    int64_t sum = 0, most = -1;
    int big = -1;
    for (int k = 0; k < kKinds; ++k) {
      const int64_t u = total[k] << (kTopTile - tile[k]);
      sum += u;
      if (tile[k] < kTopTile && u > most) {
        most = u;
        big = k;
      }
    }
    if (sum >> kTopTile <= slots || big < 0) return;
    ++tile[big];
  }
}

// Samples over all shots: a sweep (shared samples) evaluates all of them for
// every shot.
inline int64_t total_samples(int32_t n_shots, int64_t n, bool shared) {
  if (!shared) return n;
  return n > INT64_MAX / n_shots ? INT64_MAX : n * n_shots;
}

// Tile slots when the tile size is open (choose_tiles keeps within them): the
// rules stop below 2 kForwardTiles tiles, or at kMaxTile; every shot may add
// one that is not full.  It never falls with `total`, so a workspace made for
// more samples serves fewer.  (A slot per 512 samples would be four times those of a
// fixed tile of 2048: 29 GB for 4096 shots over 5e7 samples, here 1.8.)
inline int64_t open_tiles(int32_t n_shots, int64_t total) {
  const int64_t few = total >> kMinTile, many = total >> kMaxTile;
  const int64_t most = many > 2 * kForwardTiles ? many : 2 * kForwardTiles;
  return (few < most ? few : most) + n_shots + 1;
}

// Slots with which any open batch of these numbers fits: tiles of 2^kTopTile.
inline int64_t least_tiles(int32_t n_shots, int64_t n, bool shared) {
  const int64_t top = (int64_t)1 << kTopTile;
  return shared ? (int64_t)n_shots * ((n + top - 1) / top) + 1 : n / top + n_shots + 1;
}

}  // namespace qs
