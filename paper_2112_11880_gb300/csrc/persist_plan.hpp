// Plan of a persistent solver kernel (persist.cuh): the rounds of its grid and
// the layout of a block's dynamic shared memory.  Host arithmetic only.
#pragma once

#include <stddef.h>
#include <stdint.h>

#include <algorithm>

namespace helm {

// Polls after which a wait of the grid barrier gives up.  A poll is a round trip to
// L2: 0.228 us on one block, 0.237 on 304 (measured at 2070 MHz), so no wait ends
// before 2 s of the kernel's own running time (time during which the GPU runs
// another process does not count).
constexpr int kBarrierPolls = 9 << 20;

// Dynamic shared memory of a block:
//   table (where it fits): per round and owner warp its slice (-1: none) and that
//     slice's position, per round and owner thread the row's length; without it
//     the kernel works them out at every product (unsplit kernels only);
//   exchange (split): the helper warps' partial row sums (complex128);
//   nown vectors of rounds x owner threads elements.
constexpr size_t kRoundTabBytes = 32, kExchangeBytes = 16;

struct PLayout {
  int32_t rounds, split, nown;
  int32_t warps;                     // owner warps
  int32_t tab;                       // the table is there
  int32_t tlen_at, xchg_at, own_at;  // bytes from the start
  int32_t own_len;                   // elements of an own vector
};

// Rounds of `grid` blocks of `warps` owner warps over the slices of n rows.  One
// at least: a split kernel reads the first round's entry whatever n is (without
// rows it says that there is no slice).
inline int32_t persist_rounds(int32_t n, int grid, int warps) {
  const int64_t nsl = (static_cast<int64_t>(n) + 31) / 32, W = static_cast<int64_t>(grid) * warps;
  return static_cast<int32_t>(std::max<int64_t>((nsl + W - 1) / W, 1));
}

// The offsets for L's rounds, warps, split, tab and nown; returns the bytes in all.
inline size_t persist_layout(PLayout* L, size_t elem) {
  const size_t rounds = static_cast<size_t>(L->rounds), warps = static_cast<size_t>(L->warps);
  const size_t tlen = L->tab ? rounds * warps * kRoundTabBytes : 0;
  const size_t xchg = tlen + (L->tab ? rounds * warps * 32 * sizeof(int32_t) : 0);
  const size_t own = xchg + static_cast<size_t>(L->split - 1) * warps * 32 * kExchangeBytes;
  L->tlen_at = static_cast<int32_t>(tlen);
  L->xchg_at = static_cast<int32_t>(xchg);
  L->own_at = static_cast<int32_t>(own);
  L->own_len = static_cast<int32_t>(rounds * warps * 32);
  return own + static_cast<size_t>(L->nown) * rounds * warps * 32 * elem;
}

// Shared memory a block may take, of `bps` blocks per SM that have `per_sm` bytes
// between them: `reserved` and `fixed` (static) bytes go off each.  What the blocks of
// an SM leave of its 256 kB is its L1, and each of a warp's gathers from scattered
// columns holds a line of it while in flight; own vectors in shared memory gain 1 % at
// most, a small L1 costs up to a factor of two.  So all blocks of an SM stay within
// kPersistSmem, unless the columns of neighbouring rows are neighbours (`near`: the
// matrix lies on few diagonals) and a block has the SM to itself.
// Measured (us per iteration with 16 / 48 / 112 / 227 kB per SM): 27 random columns a
// row, BiCGStab, n = 300,007 114 / 112 / 113 / 192, 400,009 141 / 141 / 143 / 251,
// 1,600,003 477 / 478 / 505 / 1205; TFQMR, 200,003 90 / 88 / 89 / 141; meshes,
// BiCGStab, 120x60x50 120 / 121 / 122 / 121, 200x100x80 466 / 468 / 472 / 469;
// BiCGStab(2), 120x60x50 271 / 268 / 271 / 268.
constexpr size_t kPersistSmem = 100 * 1024;
inline size_t persist_room(size_t per_sm, size_t optin, size_t reserved, size_t fixed, int bps, bool near) {
  const size_t sm = near && bps == 1 ? per_sm : std::min(per_sm, kPersistSmem);
  const size_t block = std::min(sm / bps - reserved, optin);
  return block > fixed ? block - fixed : 0;
}

// The layout on a grid of `grid` blocks of `owners` owner threads, `split` warps
// a slice: the table, dropped where it does not fit (two blocks per SM of 16 warps:
// from 20 rounds on, 3 million unknowns), and as many of `want` own vectors of
// `elem` bytes as `room` bytes hold.  *bytes is what it takes; false when it does
// not fit.  Without the table (27 entries a row, us per BiCGStab iteration, graph /
// persistent): 7.2 million unknowns 1,997 / 1,909, 9 million 2,471 / 2,361, 10.5
// million 2,880 / 2,758; with it, 6.5 million: 1,798 / 1,750.
inline bool persist_plan(int32_t n, int grid, int owners, int split, int want, size_t elem, size_t room, PLayout* L,
                         size_t* bytes) {
  L->warps = owners / 32;
  L->rounds = persist_rounds(n, grid, L->warps);
  L->split = split;
  L->nown = 0;
  L->tab = 1;
  if (persist_layout(L, elem) > room && split == 1) L->tab = 0;
  if (persist_layout(L, elem) > room) return false;
  L->nown = want;
  while (persist_layout(L, elem) > room) --L->nown;
  *bytes = persist_layout(L, elem);
  return true;
}

// Longest row up to which HELM_LAUNCH_AUTO runs a solve as a persistent kernel; the
// graph beyond.  A product lasts as long as its longest row's chain of loads, and
// the graph's pipeline is deeper (four entries a stage against three, or two on the
// large shape).
// Measured (one long row of L entries among rows of five; us per iteration,
// persistent / graph; before persistent kernels):
//   large shape, n = 1,000,000: BiCGStab L = 128 224 / 238 (234), 192 267 / 274
//     (274), 256 314 / 310 (312), 1024 835 / 735 (791); TFQMR 192 280 / 268 (318),
//     1024 852 / 736 (831); BiCGStab(2) 192 542 / 545 (660), 1024 1591 / 1471 (1652);
//   complex64, n = 240,000: L = 64 50 / 56 (57), 128 67 / 67 (67), 192 90 / 83 (82),
//     1024 336 / 249 (259);
//   mid, n = 100,000: L = 1024 BiCGStab 384 / 352 (408), TFQMR 385 / 399 (434),
//     BiCGStab(2) 836 / 729 (915): ahead of what was at every length.
// A warp takes a row in each of its rounds, and a step has to stay well inside the
// time that a wait lasts: above 2^18 entries in all the graph (0.34 us an entry, 1.1 s
// a product of a row of 3.3 million; an entry with an imaginary part another 1 us).
inline int32_t persist_max_row(bool large, bool c64, int32_t rounds) {
  return c64 ? 128 : large ? 192 : (1 << 18) / rounds;
}

}  // namespace helm
