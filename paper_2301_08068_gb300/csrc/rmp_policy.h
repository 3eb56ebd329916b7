// rmp_policy.h -- launch policy of the evaluation kernels: host-only decisions taken from
// the ray count, the context's knobs and the measured occupancy (direction cells, segments
// per ray, threads per CTA, grid size, voxel-box use).  No CUDA calls, so the rules can be
// checked on a machine without a GPU.
#pragma once

#include <algorithm>
#include <cmath>
#include <cstdint>

#include "rmp_internal.h"

namespace rmp {

// Launch knobs of a context (rmp_tune_set): -1 / 0 select the library's choice.
struct Tuning {
  // log2 segments per ray, ray order, threads per CTA, voxel boxes
  int lg_segs = -1, ray_order = 0, block = 0, cells = -1;
};

// Coherent ray order: residue classes modulo M = 2^a 3^b are direction cells (see the
// kernel's ray_of_slot).  Cells hold >= 32 rays so a warp spans at most two of them, about
// n/48 cells, shaped close to square on the sphere (3^b ~ pi 2^a).
inline void pick_ray_cells(uint32_t n, EvalConsts* k) {
  // candidates M = 2^a 3^b with 32 M <= n, scored in log2 units with one logarithm per call:
  // |log2 M - log2(n / 48)| + 0.5 |log2(3^b / (pi 2^a))|
  const double L3 = 1.5849625007211562, LPI = 1.6514961294723187;   // log2 3, log2 pi
  const double lt = std::log2(std::max(n / 48.0, 1.0));
  uint64_t best = 1;
  double best_score = 1e300;
  for (int a = 0; a <= 24; ++a) {
    uint64_t m = 1ull << a;
    for (int b = 0; b <= 15 && m * 32ull <= n; ++b, m *= 3ull) {
      const double score = std::fabs(a + b * L3 - lt) + 0.5 * std::fabs(b * L3 - LPI - a);
      if (score < best_score) {
        best_score = score;
        best = m;
      }
    }
  }
  k->perm_M = (uint32_t)best;
  k->perm_Q = n / k->perm_M;
  k->perm_R = n % k->perm_M;
}

// Segments per ray of a single-state evaluation left to the library: as many (up to 32,
// kMaxSingleLgSegs) as keep the launch within one wave of 256-thread CTAs (`wave256`
// threads), since the evaluation lasts as long as its longest ray's serial march and
// segments shorten it while the extra threads still find free SMs (measured, device time, hashed
// 40 m map: 1024 rays 14.3 / 11.2 / 10.1 / 9.4 / 9.3 us with 1 / 4 / 8 / 16 / 32 segments, 4096
// rays 14.6 / 11.1 / 10.6 / 10.1 with 1 / 4 / 8 / 16, 16384 rays 13.9 / 13.0 / 12.1 with 1 / 2 / 4,
// 32768 rays 14.4 / 13.7 with 1 / 2, 65536 rays, past one wave with 2, 15.0 / 19.3; dense 64^3 map
// 1024 rays 11.0 / 9.8 / 9.4 / 8.9 / 9.1).  Without a wave size (0) the ray-count rule of
// make_consts stays.
constexpr uint32_t kMaxSingleLgSegs = 5;
inline void auto_segments(const Tuning& t, uint32_t n, uint64_t wave256, EvalConsts* k) {
  if (t.lg_segs >= 0 || wave256 == 0) return;
  uint32_t lg = kMaxSingleLgSegs;
  while (lg > 0 && ((uint64_t)n << lg) > wave256) --lg;
  k->lg_segs = lg;
}

// The voxel boxes' rule from when a box was looked up beside the voxel walk: as tuned, or only
// with 4 or more segments per ray.  No launch uses it any more (the box field replaces the
// walk, and is faster for every segment count); tests/launch_policy_check.cpp still builds it.
inline void single_state_cells(int tune_cells, const EvalConsts& k, DevMap* dm) {
  if (tune_cells == 1) return;
  if (tune_cells == 0 || k.lg_segs < 2) dm->cells = nullptr;
}

// n_threads: rays (or points) times segments per ray.  Threads per CTA: the tuned value, or
// (automatic) 256 when the whole launch fits in one wave of 256-thread CTAs (`wave256` threads:
// fewer CTA partials, and more registers for its slowest warps: 65536 rays 15.0 us, 17.3 with
// 128) and 128 otherwise, held to fewer registers so that more warps fit an SM (262144 rays on the
// 40 m map 27.8 us, 31.2 with 256; on the 100 m map 28.0 and 31.8).
inline void launch_shape(const Tuning& t, uint64_t n_threads, uint64_t wave256, int* block,
                  int* grid) {
  int b = t.block;
  if (b == 0) b = (wave256 > 0 && n_threads <= wave256) ? 256 : 128;
  uint64_t g = (n_threads + b - 1) / b;
  if (g > (uint64_t)kMaxGrid) g = kMaxGrid;
  if (g < 1) g = 1;
  *block = b;
  *grid = (int)g;
}

// Whether a map gets a box field of `bytes`: up to kMaxBoxFieldBytes, from memory the context's
// pool holds already (`room`) or while a sixteenth of the device's memory stays free beside it.  At
// 4 KB per occupied block the field is by far the largest part of a map, and one that a map can
// do without (65536 rays on the 40 m map 15.5 us with it, 44 without, 52 by the voxel walk before
// it): it is never the reason why another map, or another library, finds no memory.
inline bool box_field_fits(uint64_t bytes, uint64_t room, uint64_t free_bytes,
                           uint64_t total_bytes) {
  if (bytes > kMaxBoxFieldBytes) return false;
  return bytes <= room || (free_bytes >= bytes && free_bytes - bytes >= total_bytes / 16);
}

// What the context's pool keeps reserved: the bytes its maps hold and, free, as much as the largest
// upload so far took, so that a map of that size can be replaced again and again without mapping
// pages (at most 2 GiB of it: past that a refresh is long for its build, 9 ns an occupied block,
// and a context should not sit on the memory), and 64 MiB more for pieces left of other sizes.
// Upload and release with 64 MiB kept in all / by this rule: 100 m map (89 MB) 608 / 507 us, dense
// 512^3 of walls (174 MB) 1013 / 765, floor of 2048 x 2048 x 64 (319 MB) 1753 / 1244, the 40 m map (35 MB)
// beside three resident ones 515 / 397.
constexpr uint64_t kPoolKeepMore = 64ull << 20, kPoolKeepMost = 2ull << 30;
inline uint64_t pool_keep(uint64_t live, uint64_t largest) {
  return live + (largest < kPoolKeepMost ? largest : kPoolKeepMost) + kPoolKeepMore;
}

// Scans: threads per CTA the tuned value or (automatic) 256, and at most 512 threads per
// SM, each thread striding over several points, so that large scans are reduced from few
// CTA partials (measured, device time: 4096 / 65536 / 262144 points 5.7 / 8.1 / 9.7 us with
// 128-thread CTAs and 4 per SM, 5.7 / 6.3 / 8.1 us with 256 and 2 per SM).
inline void scan_shape(const Tuning& t, int sm_count, uint64_t n, int* block, int* grid) {
  const int b = t.block != 0 ? t.block : 256;
  const uint64_t cap = (uint64_t)(512 / b) * (uint64_t)(sm_count > 0 ? sm_count : 1);
  uint64_t g = (n + b - 1) / b;
  if (g > cap) g = cap;
  if (g < 1) g = 1;
  *block = b;
  *grid = (int)g;
}

}  // namespace rmp
