// Item order and slot rings of the tiled fused Myrtle form (myrtle_tiled.cu),
// written once for the device and for plain C++ (the CPU tests compile this
// header with g++ and enumerate whole queues).
//
// A queue holds blocks of 64x64 pairs first, then blocks of 32x32 pairs.
// Pair g's stage 0 is cut into tasks_per_pair(side) tasks; the items are all
// stage-0 tasks, block by block, with the stage-1 task of pair k merged LAG
// stage-0 tasks after k's last one (after all of them near the end).  Each
// image side owns a ring of S slots; pair g's slot was last used by pair
// g - S of the same side.  Functions take any struct Q with the fields
//   n, R[b], nt0[b], g0[b] (first pair of block b, g0[n] = G),
//   f0[b] (first stage-0 task of block b, f0[n] = T0), G, G64, T0, LAG, S[2];
// split_tail also split[b], wn[b] and p0[b].
#pragma once

#include <math.h>
#include <stdint.h>

#if defined(__CUDACC__)
#define NK_SCHED_HD __host__ __device__ inline
#else
#define NK_SCHED_HD inline
#endif

namespace nkf {
namespace sched {

// stage-0 tasks of a pair: 2 bands x 4 shift-t_y groups x 8 shift-t_x groups
// at 64x64, 1 x 2 x 4 at 32x32
NK_SCHED_HD constexpr int tasks_per_pair(int side) { return side == 64 ? 64 : 8; }

template <class Q>
NK_SCHED_HD int block_of_pair(const Q& q, int64_t g) {
  int b = 0;
  while (b + 1 < q.n && g >= q.g0[b + 1]) ++b;
  return b;
}

// n / d for n >= 0, d > 0: 32-bit where it fits (a 64-bit division is about
// a hundred dependent instructions on the device, on the one thread that
// decodes an item)
NK_SCHED_HD int64_t quot(int64_t n, int64_t d) {
  if (((n | d) >> 32) == 0) return (int64_t)((uint32_t)n / (uint32_t)d);
  return n / d;
}

// Linear pair index -> (i, j) of a block; the upper triangle row by row when
// symmetric.  The row's square root is FP32 with exact integer corrections:
// an FP64 root and its division, by every thread of a CTA, took 5 % of the
// FP64 pipe, which is 1/64 as wide as the FP32 one.
NK_SCHED_HD void pair_of(int64_t idx, int64_t na, int64_t nb, int sym, int64_t* i, int64_t* j) {
  if (!sym) {
    *i = quot(idx, nb);
    *j = idx - *i * nb;
    return;
  }
  const int64_t w = 2 * na + 1;
  int64_t r = (int64_t)(0.5f * ((float)w - sqrtf((float)(w * w - 8 * idx))));
  if (r < 0) r = 0;
  if (r > na - 1) r = na - 1;
  while (r > 0 && r * na - r * (r - 1) / 2 > idx) --r;
  while (r + 1 < na && (r + 1) * na - (r + 1) * r / 2 <= idx) ++r;
  *i = r;
  *j = r + (idx - (r * na - r * (r - 1) / 2));
}

// stage-0 task index k -> block, pair, task within the pair
template <class Q>
NK_SCHED_HD void stage0_of(const Q& q, int64_t k, int* b, int64_t* g, int* sub) {
  int bb = 0;
  while (bb + 1 < q.n && k >= q.f0[bb + 1]) ++bb;
  const int64_t x = k - q.f0[bb], d = quot(x, q.nt0[bb]);
  *b = bb;
  *g = q.g0[bb] + d;
  *sub = (int)(x - d * q.nt0[bb]);
}

// position of pair k's stage-1 task in the item order
template <class Q>
NK_SCHED_HD int64_t stage1_pos(const Q& q, int64_t k) {
  const int b = block_of_pair(q, k);
  int64_t x = q.f0[b] + (k - q.g0[b] + 1) * q.nt0[b] + q.LAG;
  if (x > q.T0) x = q.T0;
  return x + k;
}

// item m -> stage-1 task of pair *k (returns 1) or stage-0 task *k (0)
template <class Q>
NK_SCHED_HD int decode(const Q& q, bool two, int64_t m, int64_t* k) {
  if (!two) {
    *k = m;
    return 0;
  }
  // lo = number of stage-1 tasks at positions <= m.  Pair g0 + x of block b
  // sits at min(f0 + (x + 1) nt0 + LAG, T0) + g0 + x, which is at most m iff
  // x (nt0 + 1) <= m - f0 - nt0 - LAG - g0 or x <= m - T0 - g0.  (A search
  // over the pairs took 14 dependent steps of 64-bit arithmetic at 13,000
  // pairs; claiming and decoding an item took 6,400 cycles of a CTA.)
  int64_t lo = 0;
  for (int b = 0; b < q.n; ++b) {
    const int64_t d = m - q.f0[b] - q.nt0[b] - q.LAG - q.g0[b];
    const int64_t y = m - q.T0 - q.g0[b];
    int64_t x = d < 0 ? -1 : quot(d, q.nt0[b] + 1);
    if (y > x) x = y;
    if (x < 0) break;
    const int64_t last = q.g0[b + 1] - q.g0[b] - 1;
    if (x < last) {
      lo = q.g0[b] + x + 1;
      break;
    }
    lo = q.g0[b + 1];
  }
  if (lo > 0 && stage1_pos(q, lo - 1) == m) {
    *k = lo - 1;
    return 1;
  }
  *k = m - lo;
  return 0;
}

// ring (0: 64x64, 1: 32x32) and slot of pair g of block b; *prev = the pair
// that used the slot before (-1: none)
template <class Q>
NK_SCHED_HD int64_t slot(const Q& q, int b, int64_t g, int* ring, int64_t* prev) {
  const int r = q.R[b] == 64 ? 0 : 1;
  const int64_t ord = r == 0 ? g : g - q.G64;
  *ring = r;
  *prev = ord >= q.S[r] ? g - q.S[r] : -1;
  return ord - quot(ord, q.S[r]) * q.S[r];
}

// Lag and ring sizes of a launch of `grid` CTAs: stage-1 tasks come LAG =
// two waves after their pair's last stage-0 task; order alone needs
// S >= LAG / tasks + 1, and one more LAG between a slot's stage-1 task and
// its next user lets that task finish before it is waited for.  `tensors`
// pooled tensors per slot and global-average sums per pair (2 for the NTK:
// K and Theta).
struct Plan {
  int64_t LAG;
  int S[2];
  int64_t slot_floats[2], ring_off[2];
  uint64_t slot_bytes, bytes;
};

inline Plan make_plan(bool two, const int* R, const int64_t* npairs, int n, int grid, int tensors = 1) {
  Plan p = {};
  p.LAG = 2 * (int64_t)grid;
  int64_t G = 0;
  bool has[2] = {false, false};
  int64_t pairs[2] = {0, 0};
  for (int b = 0; b < n; ++b) {
    has[R[b] == 64 ? 0 : 1] = true;
    pairs[R[b] == 64 ? 0 : 1] += npairs[b];
    G += npairs[b];
  }
  const int side[2] = {64, 32};
  int64_t off = 0;
  for (int r = 0; r < 2; ++r) {
    const int nt = tasks_per_pair(side[r]);
    const int64_t R1 = side[r] / 2;
    p.S[r] = 1;
    if (two && has[r]) {
      // no more slots than pairs: they are cleared before each launch, 40 MB
      // of them at 32x32 whatever the block's size
      const int64_t S = (2 * p.LAG + nt - 1) / nt + 2;
      p.S[r] = (int)(S < pairs[r] ? S : pairs[r] > 0 ? pairs[r] : 1);
    }
    p.slot_floats[r] = (two && has[r]) ? tensors * R1 * R1 * R1 * R1 : 0;
    p.ring_off[r] = off;
    off += p.S[r] * p.slot_floats[r];
  }
  p.slot_bytes = (uint64_t)off * sizeof(float);
  p.bytes = p.slot_bytes + (uint64_t)G * (2 * sizeof(int) + tensors * sizeof(double)) + 64;
  return p;
}

// A single block whose items fill a few waves of the grid and a part of one:
// the pairs of that part get their tasks cut into two or four items (at most
// one warp task a warp), so that the last wave is as long as its share of the
// work.  An item's staging, claim and fence, about 0.12 of a whole task's time,
// are paid by each part: cut only where that is less than what the wave saves.
// One 32x32 image against 1, 8, 100, 200: 93.5, 104.9, 253, 429 us uncut, 51.0,
// 55.3, 254, 410 cut.  `rounds`: warp tasks of a warp in a whole task.  np: the
// blocks' pairs.  True if it cut: the last block's own parameters are the first's.
template <class Q_>
inline bool split_tail(Q_& Q, int64_t* np, int grid, int rounds) {
  if (Q.n != 1) return false;
  const int nt = Q.nt0[0];
  const int64_t full = Q.T0 / grid, rest = Q.T0 - full * grid;
  if (rest == 0 || full >= 24) return false;  // a wave in 24 is not worth it
  const int64_t main = full * grid / nt, tail = Q.G - main;
  int parts = 1;
  double best = 0.9;  // the partial wave as it is takes 1
  for (int n = 2; n <= rounds; n *= 2) {
    const int64_t waves = (tail * nt * n + grid - 1) / grid;
    const double cost = (double)waves * (0.88 / n + 0.12) - (double)(tail * nt - rest) / grid;
    if (cost < best) {
      best = cost;
      parts = n;
    }
  }
  if (parts == 1) return false;
  const int b = main > 0 ? 1 : 0;
  Q.n = b + 1;
  Q.R[b] = Q.R[0];
  Q.p0[b] = main;
  Q.split[b] = parts;
  Q.wn[b] = Q.wn[0] / parts;
  Q.nt0[b] = nt * parts;
  Q.g0[b] = main;
  Q.f0[b] = main * nt;
  Q.g0[b + 1] = Q.G;
  Q.f0[b + 1] = Q.T0 = main * nt + tail * nt * parts;
  if (b) np[0] = main;
  np[b] = tail;
  return true;
}

}  // namespace sched
}  // namespace nkf
