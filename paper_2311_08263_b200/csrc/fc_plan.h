// Integer arithmetic of the launch plans and of the waits, without CUDA types (the tests compile it with the host compiler).
#pragma once
#include <cstddef>
#include <mutex>

#ifdef __CUDACC__
#define FC_HD __host__ __device__ inline
#else
#define FC_HD inline
#endif

namespace fc {

// A ring of `stages` stages into which `issued` copies have been requested, copy j into stage j % stages: the parity of the phase that
// the last copy into `stage` completes (stage < issued).
FC_HD unsigned int last_copy_parity(int issued, int stages, int stage) { return (unsigned int)((issued - 1 - stage) / stages) & 1u; }

// x / n == x * reciprocal(n) >> 32 while x * (n - 1) < 2^32.
inline unsigned int reciprocal(int n) { return n == 1 ? 0u : (unsigned int)((0x100000000ull + (unsigned)n - 1) / (unsigned)n); }
FC_HD int quotient(int x, unsigned int inv) { return inv ? (int)((unsigned long long)(unsigned)x * inv >> 32) : x; }

// Column ranges that `units` units are cut into for tiles of at most `tile` units on each of `clusters` clusters, and whether the
// reciprocals that find the ranges' bounds are exact for that many (units of 16: a vocabulary below 1,070,000 on 33 clusters, 660,000 on 16).
inline int column_ranges(int units, int clusters, int tile) { return ((units + clusters - 1) / clusters + tile - 1) / tile; }
inline bool ranges_exact(int units, int clusters, int tile) {
  const long long parts = column_ranges(units, clusters, tile);
  return parts * units * (parts - 1) < (1ll << 32);
}

// Share of the one-writer projections' ring stages that is weights: a stage takes two k-blocks of a tile however few of its 8 x 16 weight
// rows the tile has.  shape: pairs (weight rows, k) of a layer's n matrices.
inline double stage_fill(const int (*shape)[2], int n, int clusters) {
  double bytes = 0, room = 0;
  for (int i = 0; i < n; ++i) {
    bytes += (double)shape[i][0] * shape[i][1];
    room += (double)column_ranges(shape[i][0] / 16, clusters, 8) * 128 * clusters * shape[i][1];
  }
  return bytes / room;
}

// Where the one-writer projections are faster than the chained launch, by how full their stages are, a layer's weight bytes, the rows and
// (up to 16 rows) the cached keys.
// Measured, a step, chained launch -> one writer, us (layer MB, fill; 1.1B, 7B whole, others 2 to 8 layers).  Full stages, up to 32 rows
// always: 7B (405, .92) 1 row 2869 -> 2638, 40 rows 4564 -> 4383, 64 rows 4521 -> 4133; 1070 MB, .81: 1 row 649 -> 644, 16 728 -> 655; 1711, .92:
// 678 -> 648, 770 -> 664.  From 33 rows the activations' loads grow with the stages: 625, .84: 40 rows 790 -> 791, 64 850 -> 812; 906, .82: 775 ->
// 857, 812 -> 890; 1070, .81: 911 -> 997.  Stages half to two thirds full: 294, .58: 1 row 345 -> 395, 16 396 -> 426, 32 499 -> 451, 40 527 -> 618;
// 402, .59: 406 -> 508, 456 -> 517, 571 -> 551, 629 -> 767; 510, .68: 468 -> 548, 531 -> 556, 648 -> 591, 696 -> 810; 567, .65: 515 -> 571, 580 ->
// 576, 696 -> 640, 738 -> 919; 13B (634, .69): 553 -> 582, 8 rows 593 -> 587, 16 624 -> 593, 32 738 -> 658, 40 797 -> 942; 721, .72: 482 -> 499, 539 ->
// 508, 629 -> 556, 662 -> 781.  Small layers, where the chained launch's latency counts: 1.1B (88, .47) 1 row 47 -> 43 a layer, 40 rows 83 -> 73;
// 170, .62: 379 -> 398, 436 -> 406, 571 -> 427, 622 -> 589; 201, .73: 71 -> 60 a layer, 105 -> 98.
// Where the chained launch would have the fused attention kernel in front of it (`fused`: few units), the short kernel's lead grows with the
// cached keys.  Up to 16 rows, 1000 / 3000 / 5000 / 8000 keys, chained -> one writer, 4 layers: 402 MB, 1 row 426 -> 498, 508 -> 523, 559 -> 552, 623 -> 588,
// 8 rows 452 -> 500, 532 -> 525, 584 -> 552, 649 -> 589, 16 rows 475 -> 505, 562 -> 530; 510 MB, 1 row 486 -> 537, 569 -> 556, 8 rows 521 -> 537, 608 -> 560;
// 13B, 1 row 565 -> 591, 642 -> 616, 708 -> 645, 800 -> 681, 8 rows 607 -> 595, 688 -> 620.  The line is a plane through these crossings.
inline bool one_writer_pays(double fill, long long layer_bytes, int rows, int cached, bool fused) {
  if (layer_bytes < 210000000 || (rows > 16 && rows <= 32)) return true;
  const bool full = fill >= 0.74;
  if (rows > 16) return full && layer_bytes < 750000000;
  if (full || (rows > 8 && layer_bytes >= 550000000)) return true;
  long long over = layer_bytes > 400000000 ? (layer_bytes - 400000000) / 100000 : 0;
  if (over > 2000) over = 2000;                    // 721 MB, .72: 1 row 1000 keys 492 -> 506, 3000 521 -> 524, 5000 552 -> 547
  return fused && cached >= 4000 - 150 * rows - over;
}

// Key splits of the short attention (the CTAs of a unit, one cluster): `units` units of (sequence, kv head, 16 queries), `tiles` key tiles
// for the `warps` warps of a CTA.  fit(splits, deep): clusters that run at the same time, with one CTA per SM and the whole ring of tiles
// (deep) or with two per SM and half of it.  Either cut is taken back until all clusters run at once: clusters do not cross groups of SMs, and
// what does not fit is a second round.
template <typename Fit>
void short_plan(int tiles, long long units, int head_dim, int warps, int n_sms, Fit fit, int &splits, bool &deep) {
  const int most = tiles < 8 * warps ? (tiles + warps - 1) / warps : 8;
  auto cut = [&](long long slots, bool d) {
    int s = (int)(slots / units < most ? slots / units : most);
    while (s > 1 && units > fit(s, d)) --s;
    return s > 1 ? s : 1;
  };
  splits = cut(n_sms, true);
  deep = units * splits <= n_sms;
  // Two CTAs per SM where one leaves a warp more than two tiles: always at head_dim 64 (half the bytes per tile), at 128 where it makes three or
  // more of one or two.
  if (tiles > 2 * warps * splits) {
    const int half = cut(2ll * n_sms, false);
    if (half > splits && units * half > n_sms && (head_dim == 64 || (splits <= 2 && half >= 3))) { splits = half; deep = false; }
  }
}

// Key splits of the streaming attention: the fewest rounds of clusters times a CTA's length in tile times, where start, query loads and merge
// cost about as much as six tiles.  fit(splits): clusters that run at the same time.  spare: where all run at once, a thirty-second more
// has to fit.
template <typename Fit>
int stream_splits(int tiles, long long units, bool spare, Fit fit) {
  long long best = 0;
  int ns = 1;
  for (int s = 1; s <= 8 && s <= tiles; ++s) {
    const long long n = fit(s);
    const long long rounds = spare && s > 1 && units <= n && units + units / 32 > n ? 2 : (units + n - 1) / n;
    const long long cost = rounds * ((tiles + s - 1) / s + 6 + (s > 1 ? 2 : 0));
    if (s == 1 || cost < best) { best = cost; ns = s; }
  }
  return ns;
}

// A limit per device that only rises (a kernel's dynamic shared memory), set and remembered by one thread at a time: a thread that sets
// a lower one after another has remembered its higher one would have that one's next launch refused.
struct RisingLimit {
  std::mutex m;
  size_t done[64] = {0};
  template <typename Set>
  auto raise(int dev, size_t bytes, Set set) -> decltype(set(bytes)) {      // set: 0 is success
    std::lock_guard<std::mutex> lock(m);
    if (bytes <= done[dev]) return (decltype(set(bytes)))0;
    auto e = set(bytes);
    if (e == (decltype(e))0) done[dev] = bytes;
    return e;
  }
};

}  // namespace fc
