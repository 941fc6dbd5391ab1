// Tiled fused Myrtle NNGP blocks (NK_PREC_MIXED) for 64x64 images, and for
// queues that mix 64x64 and 32x32 blocks in one persistent launch: the kernel
// templates (instantiated per activation by myrtle_tiled.cu, ReLU, and
// myrtle_tiled_erf.cu, Erf).
//
// Same arithmetic as the super-plane kernel (myrtle_fused.cuh): K_1 from the
// channel contraction, the diagonal 3x3 stencil streamed along the rows of a
// super-plane t = (t_y, t_x) (pairs (p, p') with p' = (p + t) mod R), the
// arc-cosine ReLU map with the scale factors folded into the p-side tables,
// 2x2 pooling into the next stage's super-planes, and the global average.
//
// What changes at 64x64: the pooled stage-1 tensor holds R1^4 = 32^4 floats
// (4 MB) per pair and the per-pair tables of both images (x and the per-layer
// self-variances of the 64x64 stage) no longer fit one CTA's shared memory.
// So a pair is cut into independent stage-0 tasks and one stage-1 task:
//
//  * stage-0 task = (row band of B = 32 rows, group of TY = 16 shifts t_y,
//    group of TX = 8 shifts t_x), 64 or 32 warp tasks of one t_x and two or
//    four t_y each.  A
//    band streams its rows plus N0 halo rows on each inner side (the halo
//    outputs are recomputed, not exchanged); the p-side tables cover the
//    band's rows, the p'-side tables the window of rows (r + t_y) mod R and
//    columns (c + t_x) mod R it touches.  At 64x64 with two stage-0 layers
//    the tables take 200 KB; 64 tasks a pair.
//  * the pooled output goes into a per-pair slot in global memory (L2
//    resident: a ring of S slots) by vector atomic adds; rows are paired in
//    registers, columns too when t_x is even.
//  * stage-1 task = the whole R1 = 32 stage of the pair on one CTA, rows read
//    from the slot (L2, bypassing L1) and cleared for the slot's next pair,
//    the last layer reduced into the global average and K written.
//
// Scheduling (tiled_schedule.h): one or two persistent CTAs per SM pull
// items from a global counter.  The items are the stage-0 tasks of every
// pair, block by block, with the stage-1 task of pair k merged in LAG
// stage-0 items (about two waves of the grid) after the last stage-0 task of
// k, so that it rarely waits for them.  The 64x64 and the 32x32 pairs each
// own a ring of S_R slots; a stage-0 task of pair g waits until the slot's
// previous user, pair g - S_R, has been cleared by its stage-1 task, which
// S_R >= LAG / (tasks per pair) + 1 puts earlier in the order (S_R = 2 LAG /
// (tasks per pair) + 2 puts it a LAG earlier, so that it is normally done).
// Every wait is on an item claimed earlier, so the earliest unfinished item
// never waits and the queue drains.  Waits are bounded: on a timeout the
// kernel raises NK_DEV_TIMEOUT and an abort flag that makes every CTA stop
// taking items.  The bound is the handle's wait limit (nk_set_wait_limit;
// 2^22 polls, seconds, by default).
//
// What bounds it: instruction issue and the latency of 16 warps an SM, not
// the FP32 pipe (a 48-image symmetric 32x32 block, 1176 pairs: issue 61 %,
// FP32 pipe 56 %, shared memory 67 % of their peaks).  The arithmetic is
// packed (f32x2) over two super-planes per lane.  A 160-image symmetric block
// of 32x32 images: 31.9 ms scalar with one super-plane per lane, 27.6 ms
// packed, 26.9 ms with maps that give J / pi, 25.6 ms with items decoded in
// closed form and stage-1 rows loaded further ahead, 23.6 ms with running
// addresses, 23.2 with the warps' tasks counted down (item0); 30 images of
// 64x64 symmetric: 20.1 -> 14.7 ms.  More warps do
// not help: at 80 or 64 registers the pipeline spills inside the stream (42
// ms); a form without barriers between items, warps drawing on two sets of
// tables, ran at the same issue rate with longer code (29 ms).
#pragma once

#include <algorithm>

#include "myrtle_fused.cuh"
#include "nk_f32x2.cuh"
#include "tiled_schedule.h"

namespace nkf {
namespace tiled {

// Threads per CTA: 512 with one CTA per SM wherever 64x64 blocks are present
// (their tables take 200 KB); 256 with two CTAs per SM for 32x32-only
// launches (106 KB each), so that one CTA's table staging and barriers
// overlap the other's row streams.
constexpr int MAX_WARPS = 16;
constexpr int NT32 = 256;

// Row split at image side R: a row of a super-plane is cut into NQ parts of
// COLS columns; a lane holds one part of TWO super-planes, t_y and t_y + 1
// (t_y even), packed as f32x2, and a warp the NQ parts of TYP such pairs
// (lane = part * TYP + pair: neighbouring lanes of one part read the same
// p-side entry, and a 16-byte load whose neighbouring lanes agree takes two
// passes of the shared-memory pipe; with the equal lanes 16 apart it takes
// four, measured).
template <int R_, int COLS_>
struct Cut {
  static constexpr int R = R_, COLS = COLS_;
  static constexpr int NQ = R / COLS, TYP = 32 / NQ;
  static_assert(R % COLS == 0 && NQ >= 8 && NQ <= 32 && 2 * TYP <= R, "row split");
  // p-side rows, one stretch per part: the x entries (float4) take COLS + 1
  // (odd: a quarter-warp's parts fall on distinct banks), the factor pairs
  // (float2, read two at a time) COLS, or 6 for four columns, for the same
  // reason.
  static constexpr int XST = COLS + 1, XROW = NQ * XST;
  static constexpr int PST = COLS == 4 ? 6 : COLS, PROW = NQ * PST;
};

// p'-side rows of `ncol` columns, column-phase major: column c at
// (c mod COLS) NPH + c / COLS, so that for a fixed k the parts of a row read
// consecutive entries.  A half-warp's float2 loads (a quarter-warp's float4
// loads) take 32 / TYP words of each of TYP rows that are two rows apart; the
// row strides put those rows on different banks.
template <class C, int ncol>
struct QRow {
  static constexpr int NPH = (ncol + C::COLS - 1) / C::COLS;
  static constexpr int N = C::COLS * NPH;
  // factor rows (float2): 4 Q = (32 / TYP) odd mod 32; x' rows (float4): 8 X likewise
  static constexpr int Q = C::TYP == 4 ? (N % 4 <= 2 ? N / 4 * 4 + 2 : N / 4 * 4 + 6)
                                       : (C::TYP == 2 ? (N + 3) / 8 * 8 + 4 : N);
  static constexpr int X = C::TYP == 4 ? N | 1 : (C::TYP == 2 ? (N % 4 <= 2 ? N / 4 * 4 + 2 : N / 4 * 4 + 6) : N);
  static_assert(Q >= N && X >= N, "row strides");
  static_assert(C::TYP == 1 || ((4 * Q) % (32 / C::TYP) == 0 && (4 * Q) / (32 / C::TYP) % 2 == 1), "factor banks");
  static_assert(C::TYP == 1 || ((8 * X) % (32 / C::TYP) == 0 && (8 * X) / (32 / C::TYP) % 2 == 1), "x' banks");
  static __host__ __device__ constexpr int pos(int c) { return (c % C::COLS) * NPH + c / C::COLS; }
};

// Stage-0 tiling at image side R.
template <int R, int COLS>
struct G0 : Cut<R, COLS> {
  using C = Cut<R, COLS>;
  static constexpr int B = 32;  // rows of a band
  static constexpr int NB = R / B;
  static constexpr int TY = 16, TX = 8;
  static constexpr int NTY = R / TY, NTX = R / TX;
  static constexpr int NT0 = NB * NTY * NTX;   // stage-0 tasks per pair
  static constexpr int YW = TY / (2 * C::TYP);  // warps per t_x within a task
  static constexpr int WT = TX * YW;           // warp tasks per CTA task
  static constexpr int SQ = R + TX - 1;        // p'-side window columns
  using W = QRow<C, SQ>;
  static_assert(R % B == 0 && COLS % 2 == 0 && YW * 2 * C::TYP == TY, "tiling");
  static_assert(NT0 == sched::tasks_per_pair(R), "task count of the item order (tiled_schedule.h)");
};

template <int R, int N, int COLS>
struct L0 : G0<R, COLS> {
  using G = G0<R, COLS>;
  using W = typename G::W;
  static constexpr int HALO = (G::NB > 2 ? 2 : (G::NB == 2 ? 1 : 0)) * N;
  static constexpr int NRP = G::B + HALO;  // streamed rows of a band (at most)
  static constexpr int NRQ = NRP + G::TY - 1;
  static constexpr int PL = NRP * G::PROW;  // p-side layer stride (elements)
  static constexpr int QL = NRQ * W::Q;     // p'-side layer stride of the q tables
  static constexpr size_t xs_off = 0;
  static constexpr size_t xq_off = xs_off + (size_t)NRP * G::XROW * 16;
  static constexpr size_t p_off = xq_off + (size_t)NRQ * W::X * 16;
  static constexpr size_t q_off = p_off + (size_t)N * PL * 8;
  static constexpr size_t bytes = q_off + (size_t)N * QL * 8;
  static_assert(p_off % 16 == 0 && PL % 2 == 0 && (COLS == 1 || G::PROW % 2 == 0), "16-byte factor loads");
};

// Columns per lane of stage 0.  Two columns of two super-planes fill the 128
// registers that 512 threads an SM leave; four take 168 (192 threads, two
// CTAs): 11 % fewer instructions, but 16 warp tasks over 6 warps, the same
// time on the headline (23.65 and 23.68 ms for a 160-image symmetric block).
constexpr int COLS0 = 2;

// Columns per lane of the later stages (side R1 = R / 2, then R1 / 2).
template <int R1>
struct Cols1 {
  static constexpr int v = R1 >= 32 ? 4 : (R1 == 16 ? 2 : 1);
};

// Stage-1 (and stage-2) tables at side R1 (full images, p' side doubled along
// rows and columns).
template <int R1, int N>
struct L1 : Cut<R1, Cols1<R1>::v> {
  using C = Cut<R1, Cols1<R1>::v>;
  using W = QRow<C, 2 * R1>;
  static constexpr int PL = R1 * C::PROW, QL = 2 * R1 * W::Q;
  static constexpr size_t p_off = 0;
  static constexpr size_t q_off = (size_t)N * PL * 8;
  static constexpr size_t bytes = q_off + (size_t)N * QL * 8;
  static constexpr int WPT = R1 / (2 * C::TYP);  // warps per t_x
  // p-side position of pixel e
  static __host__ __device__ constexpr int at(int e) {
    return e / R1 * C::PROW + e % R1 / C::COLS * C::PST + e % R1 % C::COLS;
  }
  static_assert(PL % 2 == 0, "16-byte factor loads");
};

struct TiledParams {
  int n;                          // blocks, 64x64 first
  int R[QUEUE_MAX];               // image side of each block (64 or 32)
  int nt0[QUEUE_MAX];             // stage-0 items per pair of each block: its tasks x split
  int split[QUEUE_MAX];           // items that a stage-0 task is cut into (split_tail)
  int wn[QUEUE_MAX];              // warp tasks of an item
  int64_t p0[QUEUE_MAX];          // first pair of the block in the B[b] it is a part of
  int64_t g0[QUEUE_MAX + 1];      // first pair index of each block
  int64_t f0[QUEUE_MAX + 1];      // first stage-0 task index of each block
  FusedParams B[QUEUE_MAX];
  int64_t G;                      // pairs
  int64_t G64;                    // pairs of 64x64 blocks (they come first)
  int64_t T0;                     // stage-0 tasks
  int64_t nitems;                 // T0 + G (stage 1 of two-stage nets) or T0
  int64_t LAG;                    // stage-0 tasks between a pair's last one and its stage-1 task
  int S[2];                       // slot rings of the 64x64 and the 32x32 pairs
  int64_t ring_off[2];            // first float of each ring
  int64_t slot_floats[2];         // (R / 2)^4
  float* slots;
  int* cnt0;                      // [G] finished stage-0 tasks
  int* done1;                     // [G] stage 1 finished (slot cleared)
  double* gacc;                   // [G] global-average sums (single-stage nets)
  unsigned long long* next;       // item counter
  int* abort_flag;
  unsigned int* dstatus;
  long long wait_limit;           // polls (~0.25-1 us each) before a wait gives up
};

__device__ __forceinline__ void red_v2(float* a, float x, float y) {
  asm volatile("red.global.add.v2.f32 [%0], {%1, %2};" ::"l"(a), "f"(x), "f"(y) : "memory");
}
// Loads from a shared-memory byte address (volatile: they stay between the
// barriers around them).
__device__ __forceinline__ float2 lds64(unsigned a) {
  float2 v;
  asm volatile("ld.shared.v2.f32 {%0, %1}, [%2];" : "=f"(v.x), "=f"(v.y) : "r"(a));
  return v;
}
__device__ __forceinline__ float4 lds128(unsigned a) {
  float4 v;
  asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "r"(a));
  return v;
}
// 1 where a != b, else 0
__device__ __forceinline__ float set_ne(float a, float b) {
  float r;
  asm("set.ne.f32.f32 %0, %1, %2;" : "=f"(r) : "f"(a), "f"(b));
  return r;
}
template <int BYTES>
__device__ __forceinline__ void cp_async(unsigned dst, const void* src) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], %2;" ::"r"(dst), "l"(src), "n"(BYTES) : "memory");
}
__device__ __forceinline__ void st_shared(unsigned dst, float v) {
  asm volatile("st.shared.f32 [%0], %1;" ::"r"(dst), "f"(v) : "memory");
}
__device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_all;" ::: "memory"); }
__device__ __forceinline__ int ld_acquire(const int* p) {
  int v;
  asm volatile("ld.acquire.gpu.global.s32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}

// Thread 0: waits until *p >= v.  False on abort or timeout (which raises
// the abort flag and NK_DEV_TIMEOUT).
__device__ inline bool wait_geq(const TiledParams& Q, const int* p, int v) {
  for (long long it = 0;; ++it) {
    if (ld_acquire(p) >= v) return true;
    if (*(volatile int*)Q.abort_flag) return false;
    if (it > Q.wait_limit) {
      atomicOr(Q.dstatus, NK_DEV_TIMEOUT);
      atomicExch(Q.abort_flag, 1);
      return false;
    }
    __nanosleep(256);
  }
}

// Loads COLS consecutive floats of a row of each of a lane's two super-planes
// from a slot (L2 only) and clears them.  SH: the rows are in this CTA's
// shared memory (the stage-2 tile of a three-stage net, cleared before each
// stage-1 task): plain loads.
template <int COLS>
__device__ __forceinline__ void take1(float* p, float (&v)[COLS]) {
  if constexpr (COLS == 4) {
    const float4 u = __ldcg(reinterpret_cast<const float4*>(p));
    v[0] = u.x; v[1] = u.y; v[2] = u.z; v[3] = u.w;
    __stcg(reinterpret_cast<float4*>(p), make_float4(0.f, 0.f, 0.f, 0.f));
  } else if constexpr (COLS == 2) {
    const float2 u = __ldcg(reinterpret_cast<const float2*>(p));
    v[0] = u.x; v[1] = u.y;
    __stcg(reinterpret_cast<float2*>(p), make_float2(0.f, 0.f));
  } else {
#pragma unroll
    for (int k = 0; k < COLS; ++k) {
      v[k] = __ldcg(p + k);
      __stcg(p + k, 0.f);
    }
  }
}
template <int COLS, bool SH>
__device__ __forceinline__ void take_row(float* p, size_t to_hi, f2 (&v)[COLS]) {
  if constexpr (SH) {
#pragma unroll
    for (int k = 0; k < COLS; ++k) v[k] = f2_make(p[k], p[to_hi + k]);
  } else {
    float a[COLS], b[COLS];
    take1<COLS>(p, a);
    take1<COLS>(p + to_hi, b);
#pragma unroll
    for (int k = 0; k < COLS; ++k) v[k] = f2_make(a[k], b[k]);
  }
}

// Horizontal 3-tap sum of one row part of both super-planes.  e[k] (k =
// 0..COLS) is the 0/1 factor of the coupling between local columns k-1 and k:
// 0 across the image border and across the column cut, so e[0] / e[COLS] also
// gate the values of lanes that have no neighbouring part (their own).
template <int COLS, int TYP>
__device__ __forceinline__ void hsum2(const f2 (&A)[COLS], f2 (&Hc)[COLS], const f2 (&e)[COLS + 1]) {
  const f2 fromL =
      f2_make(__shfl_up_sync(FULL, f2_lo(A[COLS - 1]), TYP), __shfl_up_sync(FULL, f2_hi(A[COLS - 1]), TYP));
  const f2 fromR = f2_make(__shfl_down_sync(FULL, f2_lo(A[0]), TYP), __shfl_down_sync(FULL, f2_hi(A[0]), TYP));
#pragma unroll
  for (int k = 0; k < COLS; ++k) {
    const f2 l = (k == 0) ? fromL : A[k > 0 ? k - 1 : 0];
    const f2 r = (k == COLS - 1) ? fromR : A[k + 1 < COLS ? k + 1 : 0];
    Hc[k] = f2_fma(e[k + 1], r, f2_fma(e[k], l, A[k]));
  }
}

// ---------------------------------------------------------------------------
// A band of rows [s0, s1) of the super-planes (t_y, t_x) and (t_y + 1, t_x),
// t_y even, rows [b0, b1) output; the two super-planes are the halves of
// f32x2 values.  Row stream as in the super-plane kernel: at step t the input
// row t enters layer 0 and layer j finishes row t - j - 1; rows before b0 are
// the halo (their outputs are discarded), and a band that ends at the image
// border drains the pipeline with the zero row below.
//   L:    the table layout (Cut members, W the p'-side rows, PL, QL).
//   SEED: input rows are the channel contraction (stage 0), else they are
//         taken from a slot in global memory (stage 1).
//   GAP:  the last layer feeds the global average, else the pooled scatter
//         into the slot of the next stage.
//   NTK:  a tangent row B (the neural tangent kernel's Theta, NTK
//         parameterisation) streams beside the NNGP row A through the same
//         stencil: a conv gives Theta = a S(Theta_t) + K (K with its bias; at
//         the first conv Theta_t = 0, so Theta = K), the ReLU gives Theta_t =
//         Theta (pi - arccos c) / (2 pi), and the layer's folded factor (a /
//         (2 pi), / 16 before a pool) scales B as it scales A, without the
//         sqrt(q q') that A's map carries.  Pools and the global average act
//         on both; the slot holds K's pooled tensor, then Theta's.
//   SHIN: input rows come from shared memory (the stage-2 tile), not a slot.
//   OWN:  the pooled output is a shared-memory tile that this warp alone
//         writes (one column per lane, all of t_y in the warp): plain adds.
//
// Why two t_y per lane: the second super-plane's p' row r + t_y + 1 is the
// first one's at the next row, so a lane loads one new p' row per step and
// keeps it for the next, and both share the p-side loads: half the
// shared-memory traffic per pixel pair.  The products of a p-side and a
// p'-side factor are scalar (the second operands of the two halves sit in
// different rows' registers); everything after them is packed.  An even t_y
// with the odd one above it also pools in registers: rows of both go to
// T_y = t_y / 2 in one add, only the odd one's odd rows to T_y + 1, and no
// lane of a warp branches.
// ---------------------------------------------------------------------------
template <class L, int N, bool SEED, bool GAP, bool BIAS, int ACT, bool NTK = false, bool SHIN = false,
          bool OWN = false>
struct Band {
  using W = typename L::W;
  static constexpr int R = L::R, COLS = L::COLS;
  static constexpr int R1 = R / 2;
  static constexpr int CT = NTK ? COLS : 1;  // tangent row width (1: unused)
  static constexpr int NTL = NTK ? N : 1;
  // Input rows in flight.  A slot row is a round trip to L2 (700 cycles and
  // more under load) against about 100 of a row's arithmetic: with one row
  // ahead a 16x16 stage-1 task took as long as a stage-0 task of three times
  // its work.
  static constexpr int PF = SEED || SHIN ? 1 : (COLS * (NTK ? 2 : 1) <= 2 ? 4 : 2);
  static constexpr size_t HI = (size_t)R * R * R;  // a slot's distance from t_y to t_y + 1
  int t_x, t_y;         // t_y: of the low half
  int s0, s1, b0;
  f2 E[COLS + 1];
  f2 Hp[N][COLS], Pp[N][COLS], acc[COLS];
  f2 nx[PF][COLS];      // input rows on their way (later stages)
  f2 HpT[NTL][CT], PpT[NTL][CT], accT[CT], nxT[PF][CT];  // the tangent row's pipeline
  float2 qh[N][COLS];   // p' factors of the row the low half finishes next
  float4 wh[SEED ? COLS : 1];  // p' x of the row the low half reads next
  // Shared-memory byte addresses of this lane's entries for step t, moved on
  // by whole rows once or twice per loop turn; rows within a turn and the
  // layers' tables are immediate offsets (index arithmetic per load was a
  // quarter of the stream's instructions).
  unsigned xa, pa;                 // p side: x and factors of row t
  unsigned xqa[SEED ? COLS : 1];   // p' side: x and factors of row t + t_y + 1
  unsigned qa[COLS];
  float* in;            // stage-1 input super-plane in its slot (row stride R)
  float* inT;           // its tangent (NTK)
  float* out;           // pooled output: row b0 / 2, T_x = t_x / 2, T_y = t_y / 2 of the slot
  long dT;              // from K's pooled tensor to Theta's (NTK)
  int dU, dO;           // from T_y to the next one, from T_x to the next one
  float cut;            // row cut: p' wraps between rows cut - 1 and cut of the low half
  const float* fth;     // folded factor of each layer of this stage (NTK)
  bool dg;              // NTK: the low half is the diagonal super-plane t = (0, 0) of an image with itself
  float b;
  float ge, geT;        // rounding errors of the rows' sums (add_row)

  // the tangent row enters layer j (not the first conv of stage 0)
  template <int j>
  static constexpr bool tin() { return NTK && !(SEED && j == 0); }

  // D: rows from the row of the addresses; SLOT: t mod PF
  template <int D, int SLOT>
  __device__ __forceinline__ void input_row(int t, f2 (&A)[COLS], f2 (&B)[CT]) {
    if constexpr (SEED) {
#pragma unroll
      for (int k = 0; k < COLS; ++k) {
        const float4 u = lds128(xa + (D * L::XROW + k) * 16), w = wh[k], v = lds128(xqa[k] + D * W::X * 16);
        A[k] = f2_make(fmaf(u.x, w.x, fmaf(u.y, w.y, u.z * w.z)), fmaf(u.x, v.x, fmaf(u.y, v.y, u.z * v.z)));
        wh[k] = v;
      }
    } else {
#pragma unroll
      for (int k = 0; k < COLS; ++k) A[k] = nx[SLOT][k];
      if constexpr (NTK) {
#pragma unroll
        for (int k = 0; k < COLS; ++k) B[k] = nxT[SLOT][k];
      }
      if (t + PF < R) {
        take_row<COLS, SHIN>(in + (t + PF) * R, HI, nx[SLOT]);
        if constexpr (NTK) take_row<COLS, SHIN>(inT + (t + PF) * R, HI, nxT[SLOT]);
      }
    }
  }

  // layer j at step t (row t - j) finishes row t - j - 1; tf = (float)t
  template <int j, int D, bool FIN>
  __device__ __forceinline__ void layer(float tf, f2 (&A)[COLS], f2 (&B)[CT]) {
    f2 Hc[COLS], HcT[CT];
    hsum2<COLS, L::TYP>(A, Hc, E);
    if constexpr (tin<j>()) hsum2<COLS, L::TYP>(B, HcT, E);
    // 0 across the row cut: the low half's lies between rows cut - 1 and cut,
    // the high half's a row earlier
    f2 e;
    if constexpr (R >= 64) {
      // fewer instructions than two compares (64x64: 15.5 -> 15.0 ms); at
      // 32x32 the pair of compares is the faster by 1 %
      const f2 dd = f2_sub(f2_dup(tf - (float)j), f2_make(cut, cut - 1.f));
      e = f2_make(fminf(fabsf(f2_lo(dd)), 1.f), fminf(fabsf(f2_hi(dd)), 1.f));
    } else {
      e = f2_make(set_ne(tf, cut + (float)j), set_ne(tf, cut + (float)(j - 1)));
    }
    if (FIN) finish<j, D>(e, Hc, HcT, A, B);
#pragma unroll
    for (int k = 0; k < COLS; ++k) {
      Pp[j][k] = f2_fma(e, Hp[j][k], Hc[k]);
      Hp[j][k] = Hc[k];
    }
    if constexpr (tin<j>()) {
#pragma unroll
      for (int k = 0; k < COLS; ++k) {
        PpT[j][k] = f2_fma(e, HpT[j][k], HcT[k]);
        HpT[j][k] = HcT[k];
      }
    }
  }

  template <int j, int D>
  __device__ __forceinline__ void finish(f2 e, const f2 (&Hc)[COLS], const f2 (&HcT)[CT], f2 (&A)[COLS],
                                         f2 (&B)[CT]) {
    constexpr unsigned po = (unsigned)((j * L::PL + (D - j - 1) * L::PROW) * 8);
    constexpr unsigned qo = (unsigned)((j * L::QL + (D - j - 1) * W::Q) * 8);
    float2 pv[COLS];
    if constexpr (COLS % 2 == 0) {
#pragma unroll
      for (int k = 0; k < COLS; k += 2) {
        const float4 v = lds128(pa + po + k * 8);
        pv[k] = make_float2(v.x, v.y);
        pv[k + 1] = make_float2(v.z, v.w);
      }
    } else {
#pragma unroll
      for (int k = 0; k < COLS; ++k) pv[k] = lds64(pa + po + k * 8);
    }
#pragma unroll
    for (int k = 0; k < COLS; ++k) {
      f2 K = f2_fma(e, Hc[k], Pp[j][k]);
      if constexpr (BIAS) K = f2_add(K, f2_dup(b));
      const float2 p = pv[k], q0 = qh[j][k], q1 = lds64(qa[k] + qo);
      qh[j][k] = q1;
      constexpr bool SIGNED = ACT == NK_ACT_ERF || (SEED && j == 0);  // correlations may be negative
      const f2 aa = f2_make(p.x * q0.x, p.x * q1.x), c = SIGNED ? f2_mul(K, aa) : f2_mul_sat(K, aa);
      f2 J;
      if constexpr (ACT == NK_ACT_ERF)
        J = nk_asin_2(c);  // Erf: (2/pi) asin(c), 2/pi folded into the p side
      else
        J = SIGNED ? nk_Jpi_2(c) : nk_Jpi01_2(c);
      const f2 sq = f2_make(p.y * q0.y, p.y * q1.y);
      A[k] = f2_mul(sq, J);
      if constexpr (NTK) {
        f2 T = K;
        if constexpr (tin<j>()) T = f2_add(T, f2_fma(e, HcT[k], PpT[j][k]));
        // pi - arccos c; a zero self-variance on either side gives a zero
        // derivative kernel.  Its slope is infinite at c = 1, where an FP32
        // c short of 1 by d moves it by sqrt(2 d); the pixel pairs (p, p) of
        // an image with itself have c = 1 exactly and take pi.
        const f2 as = f2_add(nk_asin_2(c), f2_dup(NK_HALF_PI_F));
        const f2 dJ = f2_make(f2_lo(sq) != 0.f ? (dg ? NK_PI_F : f2_lo(as)) : 0.f,
                              f2_hi(sq) != 0.f ? f2_hi(as) : 0.f);
        B[k] = f2_mul(f2_mul(T, dJ), f2_dup(fth[j]));
      }
    }
  }

  template <int j, int D>
  __device__ __forceinline__ void finish_last(f2 (&A)[COLS], f2 (&B)[CT]) {
    f2 Hz[COLS], HzT[CT];
#pragma unroll
    for (int k = 0; k < COLS; ++k) Hz[k] = f2_dup(0.f);
#pragma unroll
    for (int k = 0; k < CT; ++k) HzT[k] = f2_dup(0.f);
    finish<j, D>(f2_dup(0.f), Hz, HzT, A, B);
  }

  // adds one pooled row part at `aE` (T_x = t_x / 2)
  __device__ __forceinline__ void scatter(float* aE, const float (&v)[COLS]) const {
    if constexpr (COLS == 1) {
      // one column a lane: its parity decides where an odd t_x's goes
      const bool odd = ((threadIdx.x & 31) / L::TYP) & 1;
      atomicAdd((t_x & 1) && odd ? aE + dO : aE, v[0]);
    } else if (!(t_x & 1)) {
      if constexpr (COLS == 4) {
        red_v2(aE, v[0] + v[1], v[2] + v[3]);
      } else {
#pragma unroll
        for (int k = 0; k < COLS; k += 2) atomicAdd(aE + k / 2, v[k] + v[k + 1]);
      }
    } else {
      // even pixel columns keep T_x, odd ones go to the next T_x
      float* aO = aE + dO;
      if constexpr (COLS == 4) {
        red_v2(aE, v[0], v[2]);
        red_v2(aO, v[1], v[3]);
      } else {
#pragma unroll
        for (int k = 0; k < COLS; k += 2) {
          atomicAdd(aE + k / 2, v[k]);
          atomicAdd(aO + k / 2, v[k + 1]);
        }
      }
    }
  }

  // the even row (a0) and the odd row (a1) of a pooled row, of both
  // super-planes: the even t_y's rows and the odd one's even row pool into
  // T_y = t_y / 2, the odd one's odd row into the next T_y
  __device__ __forceinline__ void pool_rows(float* o, const f2 (&a0)[COLS], const f2 (&a1)[COLS]) const {
    float v[COLS], w[COLS];
#pragma unroll
    for (int k = 0; k < COLS; ++k) {
      v[k] = (f2_lo(a0[k]) + f2_lo(a1[k])) + f2_hi(a0[k]);
      w[k] = f2_hi(a1[k]);
    }
    scatter(o, v);
    scatter(o + dU, w);
  }

  // OWN: the column pairs of an even t_x meet by a shuffle, the odd t_y's odd
  // row goes to the lane of the next T_y, and each cell has one lane
  __device__ __forceinline__ void pool_own(float* o, f2 a0, f2 a1) const {
    static_assert(!OWN || (COLS == 1 && 2 * L::TYP == R), "one warp holds every t_y of its t_x");
    const int lane = threadIdx.x & 31, tyl = lane % L::TYP, q = lane / L::TYP;
    float v = (f2_lo(a0) + f2_lo(a1)) + f2_hi(a0);
    v += __shfl_sync(FULL, f2_hi(a1), q * L::TYP + ((tyl + L::TYP - 1) % L::TYP));
    const float w = v + __shfl_xor_sync(FULL, v, L::TYP);
    float* t = o + ((q & 1) ? dO : 0);
    if (t_x & 1)
      *t += v;
    else if (!(q & 1))
      *o += w;
    __syncwarp();
  }

  // Adds a row to a global average: at most four values in FP32 (stage 0 of
  // 32x32 and 64x64 images, and rows cut into four columns), two elsewhere, then
  // FP64.  The two halves' sum is split exactly (TwoSum) and its errors summed in
  // FP32 until the band's end: an FP64 addition or conversion more a row takes
  // 1 x 200 images of 32x32 from 438 to 447 us, and the NTK of 80 from 11.62 to
  // 11.69 ms.  At R = 32 (stage 1 of 64x64) the error's register costs more than
  // its addition (30 symmetric images 14.89 and 14.66 ms).
  __device__ __forceinline__ static void add_row(const f2* A, double& sum, float& err) {
    f2 s = A[0];
#pragma unroll
    for (int k = 1; k < COLS; ++k) s = f2_add(s, A[k]);
    if constexpr (COLS == 1 || (SEED && R >= 32)) {
      sum += (double)(f2_lo(s) + f2_hi(s));
    } else {
      const float a = f2_lo(s), b = f2_hi(s), t = __fadd_rn(a, b), z = __fsub_rn(t, a);
      const float e = __fadd_rn(__fsub_rn(a, __fsub_rn(t, z)), __fsub_rn(b, z));
      sum += (double)t;
      if constexpr (R >= 32)
        sum += (double)e;
      else
        err += e;
    }
  }

  template <int PAR>
  __device__ __forceinline__ void output(const f2 (&A)[COLS], const f2 (&B)[CT], double& gap, double& gapT) {
    if constexpr (GAP) {
      add_row(A, gap, ge);
      if constexpr (NTK) add_row(B, gapT, geT);
    } else if constexpr (PAR == 0) {
#pragma unroll
      for (int k = 0; k < COLS; ++k) acc[k] = A[k];
      if constexpr (NTK) {
#pragma unroll
        for (int k = 0; k < COLS; ++k) accT[k] = B[k];
      }
    } else if constexpr (OWN) {
      pool_own(out, acc[0], A[0]);
      out += R1;
    } else {
      pool_rows(out, acc, A);
      if constexpr (NTK) pool_rows(out + dT, accT, B);
      out += R1;
    }
  }

  template <int j0, int j1, int D>
  __device__ __forceinline__ void layers_fin(float tf, f2 (&A)[COLS], f2 (&B)[CT]) {
    if constexpr (j0 < j1) {
      layer<j0, D, true>(tf, A, B);
      layers_fin<j0 + 1, j1, D>(tf, A, B);
    }
  }

  // the addresses of step t + n
  __device__ __forceinline__ void advance(int n) {
    pa += n * L::PROW * 8;
    if constexpr (SEED) xa += n * L::XROW * 16;
#pragma unroll
    for (int k = 0; k < COLS; ++k) {
      qa[k] += n * W::Q * 8;
      if constexpr (SEED) xqa[k] += n * W::X * 16;
    }
  }

  // pipeline fill, step s0 + T for T < N: layers 0..T-1 finish rows, layer T
  // receives its first row s0
  template <int T>
  __device__ __forceinline__ void fill(float tf) {
    if constexpr (T < N) {
      f2 A[COLS], B[CT];
      input_row<T, T % PF>(s0 + T, A, B);
      layers_fin<0, T, T>(tf, A, B);
      layer<T, T, false>(tf, A, B);
      fill<T + 1>(tf + 1.f);
    }
  }

  // step t + I, the addresses at step t; SLOT: t mod PF; an output row's
  // parity is that of I
  template <int I, int SLOT>
  __device__ __forceinline__ void steady(int t, float tf, double& gap, double& gapT) {
    f2 A[COLS], B[CT];
    input_row<I, SLOT>(t + I, A, B);
    layers_fin<0, N, I>(tf + (float)I, A, B);
    output<I & 1>(A, B, gap, gapT);
  }

  // drain, step R + D, the addresses at step R
  template <int D>
  __device__ __forceinline__ void drain(double& gap, double& gapT) {
    if constexpr (D < N) {
      f2 A[COLS], B[CT];
      finish_last<D, D>(A, B);
      layers_fin<D + 1, N, D>((float)(R + D), A, B);
      output<((R + D - N) & 1)>(A, B, gap, gapT);
      drain<D + 1>(gap, gapT);
    }
  }

  // steady steps t + I .. t + M - 1, t = N mod the steps of a ring
  template <int I, int M>
  __device__ __forceinline__ void steps(int t, float tf, double& gap, double& gapT) {
    if constexpr (I < M) {
      steady<I, (N + I) % PF>(t, tf, gap, gapT);
      steps<I + 1, M>(t, tf, gap, gapT);
    }
  }

  __device__ __forceinline__ void run(double& gap, double& gapT) {
    ge = geT = 0.f;
#pragma unroll
    for (int j = 0; j < N; ++j)
#pragma unroll
      for (int k = 0; k < COLS; ++k) {
        Hp[j][k] = Pp[j][k] = f2_dup(0.f);
        qh[j][k] = lds64(qa[k] + (j * L::QL - W::Q) * 8);
      }
    if constexpr (NTK) {
#pragma unroll
      for (int j = 0; j < N; ++j)
#pragma unroll
        for (int k = 0; k < CT; ++k) HpT[j][k] = PpT[j][k] = f2_dup(0.f);
    }
    if constexpr (SEED) {
#pragma unroll
      for (int k = 0; k < COLS; ++k) wh[k] = lds128(xqa[k] - W::X * 16);
    } else {
#pragma unroll
      for (int i = 0; i < PF; ++i) {
        take_row<COLS, SHIN>(in + i * R, HI, nx[i]);
        if constexpr (NTK) take_row<COLS, SHIN>(inT + i * R, HI, nxT[i]);
      }
    }
    int t = s0 + N;
    float tf = (float)s0;
    fill<0>(tf);
    advance(N);
    tf += (float)N;
    if constexpr (SEED) {
      // halo rows: computed, not output (b0 - s0 is 0 or N)
      for (; t < b0 + N; ++t) {
        f2 A[COLS], B[CT];
        input_row<0, 0>(t, A, B);
        layers_fin<0, N, 0>(tf, A, B);
        advance(1);
        tf += 1.f;
      }
      // output rows from b0 (even) in pairs
#pragma unroll 1
      for (; t + 1 < s1; t += 2) {
        steady<0, 0>(t, tf, gap, gapT);
        steady<1, 0>(t, tf, gap, gapT);
        advance(2);
        tf += 2.f;
      }
      if (t < s1) {
        steady<0, 0>(t, tf, gap, gapT);
        advance(1);
      }
    } else {
      // all rows (s0 = b0 = 0, s1 = R), a ring of input rows at a time
      constexpr int STEP = PF > 2 ? PF : 2;
      for (; t + STEP <= R; t += STEP) {
        steps<0, STEP>(t, tf, gap, gapT);
        advance(STEP);
        tf += (float)STEP;
      }
      steps<0, (R - N) % STEP>(t, tf, gap, gapT);
      advance((R - N) % STEP);
    }
    if (s1 == R) drain<0>(gap, gapT);
    if constexpr (GAP && COLS > 1 && R < 32) {
      gap += (double)ge;
      if constexpr (NTK) gapT += (double)geT;
    }
  }
};

// 0/1 factors of the couplings between local columns k-1 and k of a row part
// (0 across the image border and the super-plane's column cut).
template <int COLS>
__device__ __forceinline__ void edges(f2 (&e)[COLS + 1], int R, int t_x, int q) {
  const int c0 = q * COLS;
  const int kc = (t_x == 0) ? -100 : R - 1 - t_x;
#pragma unroll
  for (int k = 0; k <= COLS; ++k) {
    const int lc = c0 + k - 1;
    e[k] = f2_dup(((lc < 0) || (lc + 1 > R - 1) || (lc == kc)) ? 0.f : 1.f);
  }
}

__device__ __forceinline__ float4 ld_x(const float* p, int C, float s) {
  return make_float4(p[0] * s, C > 1 ? p[1] * s : 0.f, C > 2 ? p[2] * s : 0.f, 0.f);
}

// An item of the queue, decoded by one thread for its CTA.
struct Item {
  int64_t g;       // pair
  int64_t i, j;    // its row and column in the block
  float* slot;     // its slot (two-stage nets)
  int kind;        // 0: stage-0 task `sub`, 1: stage-1 task, -1: the queue is empty
  int b, sub;      // block; stage-0 task within the pair
  int w0, nw;      // its first warp task, warp tasks of each warp
};

// Slot of pair g (block b) in its resolution's ring, and the pair that used
// it before (-1: none).
__device__ __forceinline__ float* slot_of(const TiledParams& Q, int b, int64_t g, int64_t* prev) {
  int r;
  const int64_t k = sched::slot(Q, b, g, &r, prev);
  return Q.slots + Q.ring_off[r] + k * Q.slot_floats[r];
}

// Theta of the NTK: K + sw2 mean(Theta_t), i.e. the GAP scale applied to the
// sum of both global-average sums (K's bias added once).
__device__ __forceinline__ void store_theta(const FusedParams& P, int64_t i, int64_t j, double tot) {
  const float v = (float)(P.out_scale * tot + P.out_bias);
  P.Th[i * P.ldk + j] = v;
  if (P.sym && i != j) P.Th[j * P.ldk + i] = v;
}

// ---------------------------------------------------------------------------
// Stage-0 task `sub` of pair g (block b): its tables, its warp tasks.
// ---------------------------------------------------------------------------
template <int R, int N0, int N1, bool BIAS, int ACT, bool NTK>
struct Stage0 {
  using L = L0<R, N0, COLS0>;
  using G = typename L::G;
  using W = typename L::W;
  static constexpr bool TWO = N1 > 0;
  static constexpr int WT = G::WT;  // warp tasks
  using BT = Band<L, N0, true, !TWO, BIAS, ACT, NTK>;

  struct Rows {
    int s0, s1, b0, ty0, tx0;
  };
  static __device__ __forceinline__ Rows rows(int sub) {
    Rows w;
    w.b0 = sub / (G::NTY * G::NTX) * G::B;
    w.s0 = w.b0 - N0 > 0 ? w.b0 - N0 : 0;
    w.s1 = w.b0 + G::B + N0 < R ? w.b0 + G::B + N0 : R;
    w.ty0 = (sub / G::NTX) % G::NTY * G::TY;
    w.tx0 = sub % G::NTX * G::TX;
    return w;
  }

  // The task's tables, by NT threads of which this is number `tid`.
  template <int NT>
  static __device__ __forceinline__ void load(const TiledParams& Q, const Item& it, unsigned char* smem, int tid) {
    const FusedParams& P = Q.B[it.b];
    const int64_t ia = P.a0 + it.i, ib = P.b0 + it.j;
    const Rows o = rows(it.sub);
    float4* xs = reinterpret_cast<float4*>(smem + L::xs_off);
    float4* xq = reinterpret_cast<float4*>(smem + L::xq_off);
    float2* pt = reinterpret_cast<float2*>(smem + L::p_off);
    float2* qt = reinterpret_cast<float2*>(smem + L::q_off);
    const int C = P.C;
    const float* xa = P.Xa + ia * (int64_t)R * R * C;
    const float* xb = P.Xb + ib * (int64_t)R * R * C;
    const float2* qa = reinterpret_cast<const float2*>(P.qsa) + ia * P.nq;
    const float2* qb = reinterpret_cast<const float2*>(P.qsb) + ib * P.nq;
    const float2* qb0[N0];
#pragma unroll
    for (int l = 0; l < N0; ++l) qb0[l] = qb + P.qoff[l];
    // p' window: copied as it is, asynchronously, so that all of it is in
    // flight at once (loads held in registers were a round trip to memory per
    // pixel of a thread: 11 a task).  32-bit offsets, stepped without divisions.
    const int nrow = o.s1 - o.s0 + G::TY - 1;
    int wr = tid / G::SQ, wc = tid % G::SQ;
    while (wr < nrow) {
      const int px = ((o.s0 + o.ty0 + wr) & (R - 1)) * R + ((o.tx0 + wc) & (R - 1));
      const int pc = W::pos(wc);  // column position in a window row
      const unsigned xd = smem_u32(xq) + 16u * (wr * W::X + pc);
      const float* xsrc = xb + px * C;
#pragma unroll
      for (int ch = 0; ch < 3; ++ch) {
        if (ch < C)
          cp_async<4>(xd + 4 * ch, xsrc + ch);
        else
          st_shared(xd + 4 * ch, 0.f);
      }
      const unsigned qd = smem_u32(qt) + 8u * (wr * W::Q + pc);
#pragma unroll
      for (int l = 0; l < N0; ++l) cp_async<8>(qd + 8u * (l * L::QL), qb0[l] + px);
      wr += NT / G::SQ;
      wc += NT % G::SQ;
      if (wc >= G::SQ) {
        wc -= G::SQ;
        ++wr;
      }
    }
    // p side: scaled on the way
    const int np = (o.s1 - o.s0) * R;
    for (int e = tid; e < np; e += NT) {
      const int row = e / R, c = e % R;
      const int part = c / G::COLS, k = c % G::COLS;
      xs[row * G::XROW + part * G::XST + k] = ld_x(xa + (o.s0 * R + e) * C, C, P.xscale);
#pragma unroll
      for (int l = 0; l < N0; ++l) {
        const float2 v = qa[P.qoff[l] + o.s0 * R + e];
        pt[l * L::PL + row * G::PROW + part * G::PST + k] = make_float2(v.x, v.y * P.foldp[l]);
      }
    }
    cp_async_wait();
  }

  // Warp task w of the task; adds to this lane's global-average sums.
  static __device__ __forceinline__ void warp_task(const TiledParams& Q, const Item& it, unsigned char* smem, int w,
                                                   int lane, double& gap, double& gapT) {
    const FusedParams& P = Q.B[it.b];
    const Rows o = rows(it.sub);
    const int q = lane / G::TYP, tyl = lane % G::TYP;  // row part, pair of t_y
    constexpr long R1 = R / 2;
    BT T;
    const int txl = w / G::YW;
    const int tyw = 2 * ((w % G::YW) * G::TYP + tyl);  // t_y - ty0
    T.t_x = o.tx0 + txl;
    T.t_y = o.ty0 + tyw;
    T.s0 = o.s0;
    T.s1 = o.s1;
    T.b0 = o.b0;
    edges<G::COLS>(T.E, R, T.t_x, q);
    const unsigned sm = smem_u32(smem);
    T.xa = sm + L::xs_off + q * G::XST * 16;
    T.pa = sm + L::p_off + q * G::PST * 8;
#pragma unroll
    for (int k = 0; k < G::COLS; ++k) {
      const int c = q + W::pos(txl + k);
      T.xqa[k] = sm + L::xq_off + ((tyw + 1) * W::X + c) * 16;
      T.qa[k] = sm + L::q_off + ((tyw + 1) * W::Q + c) * 8;
    }
    T.in = nullptr;
    T.inT = nullptr;
    T.cut = (float)(R - T.t_y);
    // pooled output (single-stage nets have none)
    const int Ty = T.t_y >> 1, Tx = T.t_x >> 1;
    T.out = TWO ? it.slot + ((Ty * R1 + Tx) * R1 + o.b0 / 2) * R1 + q * (G::COLS / 2) : nullptr;
    T.dT = R1 * R1 * R1 * R1;  // the tangent's pooled tensor follows
    T.dU = (((Ty + 1) & (R1 - 1)) - Ty) * (int)(R1 * R1 * R1);
    T.dO = ((((T.t_x + 1) >> 1) & (R1 - 1)) - Tx) * (int)(R1 * R1);
    T.fth = P.fold;
    T.dg = NTK && P.Xa == P.Xb && P.a0 + it.i == P.b0 + it.j && T.t_x == 0 && T.t_y == 0;
    T.b = P.sb2;
    T.run(gap, gapT);
  }

  // One thread, once every warp task is done and its writes are ordered
  // before this: counts the task; in a single-stage net (sum, sumT: the
  // task's share of the global averages) the pair's last task writes K.
  static __device__ __forceinline__ void publish(const TiledParams& Q, const Item& it, double sum, double sumT) {
    const int64_t g = it.g;
    if constexpr (TWO) {
      __threadfence();
      atomicAdd(Q.cnt0 + g, 1);
    } else {
      atomicAdd(Q.gacc + g, sum);
      if constexpr (NTK) atomicAdd(Q.gacc + Q.G + g, sumT);
      __threadfence();
      const int old = atomicAdd(Q.cnt0 + g, 1);
      if (old == Q.nt0[it.b] - 1) {
        __threadfence();
        const FusedParams& P = Q.B[it.b];
        const double tk = atomicAdd(Q.gacc + g, 0.0);
        store_entry(P, it.i, it.j, tk);
        if constexpr (NTK) store_theta(P, it.i, it.j, tk + atomicAdd(Q.gacc + Q.G + g, 0.0));
      }
    }
  }
};

// ---------------------------------------------------------------------------
// Stage-1 task of pair g: the whole R1 stage, then K.  Shared memory: its
// tables, then (three-stage nets) the pooled stage-2 tile of K (and of Theta)
// and the stage-2 tables.
// ---------------------------------------------------------------------------
template <int R1, int N1, int N2, bool NTK>
struct L1x {
  static constexpr int R2 = R1 / 2;
  static constexpr size_t tile_off = (L1<R1, N1>::bytes + 15) / 16 * 16;
  static constexpr size_t tile_floats = N2 > 0 ? (size_t)R2 * R2 * R2 * R2 : 0;
  static constexpr size_t tab2_off = tile_off + (NTK ? 2 : 1) * tile_floats * 4;
  static constexpr size_t bytes = tab2_off + (N2 > 0 ? L1<R2, N2>::bytes : 0);
};

template <int R1, int N0, int N1, bool BIAS, int ACT, bool NTK, int N2 = 0>
struct Stage1 {
  using L = L1<R1, N1>;
  using W = typename L::W;
  using X1 = L1x<R1, N1, N2, NTK>;
  static constexpr int WT = R1 * L::WPT;  // warp tasks
  static constexpr int R2 = R1 / 2;
  // stage 1 feeds the global average (two-stage nets) or pools into the
  // stage-2 tile in shared memory (three-stage nets)
  using BT = Band<L, N1, false, N2 == 0, BIAS, ACT, NTK>;
  static_assert(WT % MAX_WARPS == 0, "every warp takes the same number of tasks");
  static_assert(N2 == 0 || BT::COLS == 2, "the pooled adds into the shared tile use generic atomics (COLS == 2)");

  // Tables of N layers from layer Lr0 of the net at side L_::R.
  template <class L_, int NT, int N>
  static __device__ __forceinline__ void tables(const FusedParams& P, int Lr0, const float2* qa, const float2* qb,
                                                unsigned char* smem, int tid) {
    using W_ = typename L_::W;
    constexpr int S = L_::R;
    float2* pt = reinterpret_cast<float2*>(smem + L_::p_off);
    float2* qt = reinterpret_cast<float2*>(smem + L_::q_off);
    for (int l = 0; l < N; ++l) {
      const int Lr = Lr0 + l;
      const float f = P.foldp[Lr];
      for (int e = tid; e < S * S; e += NT) {
        const float2 v = qa[P.qoff[Lr] + e];
        pt[l * L_::PL + L_::at(e)] = make_float2(v.x, v.y * f);
        const float2 u = qb[P.qoff[Lr] + e];
        const int row = e / S, col = e % S;
        float2* d = qt + l * L_::QL + row * W_::Q;
        d[W_::pos(col)] = u;
        d[W_::pos(col + S)] = u;
        d[S * W_::Q + W_::pos(col)] = u;
        d[S * W_::Q + W_::pos(col + S)] = u;
      }
    }
  }

  template <int NT>
  static __device__ __forceinline__ void load(const TiledParams& Q, const Item& it, unsigned char* smem, int tid) {
    const FusedParams& P = Q.B[it.b];
    const float2* qa = reinterpret_cast<const float2*>(P.qsa) + (P.a0 + it.i) * P.nq;
    const float2* qb = reinterpret_cast<const float2*>(P.qsb) + (P.b0 + it.j) * P.nq;
    tables<L, NT, N1>(P, N0, qa, qb, smem, tid);
    if constexpr (N2 > 0) {
      // stage-2 tables, and the stage-2 tile(s) cleared for this pair's pooled adds
      tables<L1<R2, N2>, NT, N2>(P, N0 + N1, qa, qb, smem + X1::tab2_off, tid);
      float* tile = reinterpret_cast<float*>(smem + X1::tile_off);
      for (size_t e = tid; e < (NTK ? 2 : 1) * X1::tile_floats; e += NT) tile[e] = 0.f;
    }
  }

  template <class BT_>
  static __device__ __forceinline__ void common(const TiledParams& Q, const Item& it, BT_& T, int R_, int fth) {
    const FusedParams& P = Q.B[it.b];
    T.s0 = 0;
    T.s1 = R_;
    T.b0 = 0;
    T.xa = 0;
    T.cut = (float)(R_ - T.t_y);
    T.fth = P.fold + fth;
    T.dg = NTK && P.Xa == P.Xb && P.a0 + it.i == P.b0 + it.j && T.t_x == 0 && T.t_y == 0;
    T.b = P.sb2;
  }

  static __device__ __forceinline__ void warp_task(const TiledParams& Q, const Item& it, unsigned char* smem,
                                                   int task, int lane, double& gap, double& gapT) {
    const int q = lane / L::TYP, tyl = lane % L::TYP;
    float* tile = N2 > 0 ? reinterpret_cast<float*>(smem + X1::tile_off) : nullptr;
    BT T;
    T.t_x = task / L::WPT;
    T.t_y = 2 * ((task % L::WPT) * L::TYP + tyl);
    common(Q, it, T, R1, N0);
    edges<L::COLS>(T.E, R1, T.t_x, q);
    T.in = it.slot + ((size_t)(T.t_y * R1 + T.t_x) * R1) * R1 + q * L::COLS;
    T.inT = NTK ? T.in + (size_t)R1 * R1 * R1 * R1 : nullptr;
    // pooled output into the stage-2 tile (three-stage nets)
    const int Ty = T.t_y >> 1, Tx = T.t_x >> 1;
    T.out = N2 > 0 ? tile + ((Ty * R2 + Tx) * R2) * R2 + q * (L::COLS / 2) : nullptr;
    T.dT = (long)X1::tile_floats;
    T.dU = (((Ty + 1) & (R2 - 1)) - Ty) * (R2 * R2 * R2);
    T.dO = ((((T.t_x + 1) >> 1) & (R2 - 1)) - Tx) * (R2 * R2);
    const unsigned sm = smem_u32(smem);
    T.pa = sm + L::p_off + q * L::PST * 8;
#pragma unroll
    for (int k = 0; k < L::COLS; ++k) T.qa[k] = sm + L::q_off + ((T.t_y + 1) * W::Q + q + W::pos(T.t_x + k)) * 8;
    T.run(gap, gapT);
  }

  // Stage 2 of a three-stage net, from the pooled tile.
  static __device__ __forceinline__ void warp_task2(const TiledParams& Q, const Item& it, unsigned char* smem,
                                                    int task, int lane, double& gap, double& gapT) {
    using L2 = L1<R2, N2>;
    using W2 = typename L2::W;
    using BT2 = Band<L2, N2, false, true, BIAS, ACT, NTK, true>;
    const int q2 = lane / L2::TYP, tyl2 = lane % L2::TYP;
    float* tile = reinterpret_cast<float*>(smem + X1::tile_off);
    BT2 T;
    T.t_x = task / L2::WPT;
    T.t_y = 2 * ((task % L2::WPT) * L2::TYP + tyl2);
    common(Q, it, T, R2, N0 + N1);
    edges<L2::COLS>(T.E, R2, T.t_x, q2);
    T.in = tile + ((size_t)(T.t_y * R2 + T.t_x) * R2) * R2 + q2 * L2::COLS;
    T.inT = NTK ? T.in + X1::tile_floats : nullptr;
    T.out = nullptr;
    T.dT = 0;
    T.dU = T.dO = 0;
    const unsigned sm = smem_u32(smem) + (unsigned)X1::tab2_off;
    T.pa = sm + L2::p_off + q2 * L2::PST * 8;
#pragma unroll
    for (int k = 0; k < L2::COLS; ++k) T.qa[k] = sm + L2::q_off + ((T.t_y + 1) * W2::Q + q2 + W2::pos(T.t_x + k)) * 8;
    T.run(gap, gapT);
  }
  static constexpr int WT2 = N2 > 0 ? R2 * L1<R2, N2 == 0 ? 1 : N2>::WPT : 0;

  // One thread, once every warp task is done: K (and Theta), and the cleared
  // slot is released.
  static __device__ __forceinline__ void publish(const TiledParams& Q, const Item& it, double sum, double sumT) {
    const FusedParams& P = Q.B[it.b];
    store_entry(P, it.i, it.j, sum);
    if constexpr (NTK) store_theta(P, it.i, it.j, sum + sumT);
    __threadfence();
    atomicExch(Q.done1 + it.g, 1);
  }
};

// Sums of a CTA's lanes, valid in thread 0 after the barrier inside.
template <bool NTK, int NT>
__device__ __forceinline__ void cta_sums(double* red, double gap, double gapT, double* s, double* sT) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) gap += __shfl_xor_sync(FULL, gap, o);
  if (lane == 0) red[warp] = gap;
  if constexpr (NTK) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) gapT += __shfl_xor_sync(FULL, gapT, o);
    if (lane == 0) red[MAX_WARPS + warp] = gapT;
  }
  __syncthreads();
  *s = *sT = 0.0;
  if (threadIdx.x == 0) {
    for (int w = 0; w < NT / 32; ++w) *s += red[w];
    if constexpr (NTK)
      for (int w = 0; w < NT / 32; ++w) *sT += red[MAX_WARPS + w];
  }
}

// A whole item by all NT threads of the CTA.  The warps' tasks are counted
// down, and stage 0 steps through a copy of the item: with the bound of a loop
// over w alive across the row stream, the stream was 2 to 4 % slower (160
// symmetric 32x32 images 23.6 ms and 23.2, NTK of 80 11.9 and 11.6, 30 of 64x64
// 15.3 to 15.9 and 14.7).
template <class S0, int NT, bool NTK>
__device__ __forceinline__ void item0(const TiledParams& Q, const Item& it, unsigned char* smem, double* red) {
  S0::template load<NT>(Q, it, smem, threadIdx.x);
  __syncthreads();
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  double gap = 0.0, gapT = 0.0, s = 0.0, sT = 0.0;
  Item t = it;
  for (int n = it.nw; n > 0; --n, t.w0 += NT / 32) S0::warp_task(Q, t, smem, t.w0 + warp, lane, gap, gapT);
  // publish the task's atomic adds: the barrier orders every thread's adds
  // before thread 0's fence, which releases them together with the count
  if constexpr (S0::TWO)
    __syncthreads();
  else
    cta_sums<NTK, NT>(red, gap, gapT, &s, &sT);
  if (threadIdx.x == 0) S0::publish(Q, it, s, sT);
}
template <class S1, int NT, bool NTK, int N2>
__device__ __forceinline__ void item1(const TiledParams& Q, const Item& it, unsigned char* smem, double* red) {
  S1::template load<NT>(Q, it, smem, threadIdx.x);
  __syncthreads();
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  double gap = 0.0, gapT = 0.0, s, sT;
  int w = warp;
  for (int n = S1::WT / (NT / 32); n > 0; --n, w += NT / 32) S1::warp_task(Q, it, smem, w, lane, gap, gapT);
  if constexpr (N2 > 0) {
    // stage 2 from the pooled tile, on the same CTA
    __syncthreads();
    for (int w = warp; w < S1::WT2; w += NT / 32) S1::warp_task2(Q, it, smem, w, lane, gap, gapT);
  }
  cta_sums<NTK, NT>(red, gap, gapT, &s, &sT);
  if (threadIdx.x == 0) S1::publish(Q, it, s, sT);
}

template <int N0, int N1, int RMAX, bool NTK = false, int N2 = 0>
struct Smem {
  static_assert(N2 == 0 || RMAX == 32, "three-stage nets: 32x32 images only");
  template <int R>
  using S0 = L0<R, N0, COLS0>;
  static constexpr size_t s0 = RMAX == 64 ? std::max(S0<64>::bytes, S0<32>::bytes) : S0<32>::bytes;
  static constexpr size_t s1 =
      N1 > 0 ? (RMAX == 64 ? std::max(L1<32, N1>::bytes, L1<16, N1>::bytes) : L1x<16, N1, N2, NTK>::bytes) : 0;
  static constexpr size_t tables = std::max(s0, s1);
  static constexpr size_t red = (NTK ? 2 : 1) * MAX_WARPS * 8;  // per-warp global-average sums
  static constexpr size_t bytes = tables + red + (sizeof(Item) + 15) / 16 * 16;
};

// Thread 0: takes the next item of the queue and waits for what it depends
// on: a stage-0 task for the stage-1 task of its slot's previous pair, a
// stage-1 task for its pair's stage-0 tasks.  An aborted wait ends the queue
// for this CTA.
template <bool TWO>
__device__ inline void claim(const TiledParams& Q, Item* out) {
  Item it;
  it.kind = -1;
  const long long m = *(volatile int*)Q.abort_flag ? (long long)Q.nitems : (long long)atomicAdd(Q.next, 1ull);
  if (m < Q.nitems) {
    int64_t k;
    it.kind = sched::decode(Q, TWO, m, &k);
    if (it.kind == 0) {
      sched::stage0_of(Q, k, &it.b, &it.g, &it.sub);
      const int t = it.sub / Q.split[it.b];
      it.w0 = (it.sub - t * Q.split[it.b]) * Q.wn[it.b];
      it.nw = Q.wn[it.b] / ((int)blockDim.x / 32);
      it.sub = t;
    } else {
      it.g = k;
      it.b = sched::block_of_pair(Q, k);
      it.sub = it.w0 = it.nw = 0;
    }
    const FusedParams& P = Q.B[it.b];
    sched::pair_of(it.g - Q.g0[it.b] + Q.p0[it.b], P.na, P.nb, P.sym, &it.i, &it.j);
    it.slot = nullptr;
    if constexpr (TWO) {
      int64_t prev;
      it.slot = slot_of(Q, it.b, it.g, &prev);
      bool ok = true;
      if (it.kind == 1)
        ok = wait_geq(Q, Q.cnt0 + it.g, Q.nt0[it.b]);
      else if (prev >= 0)
        ok = wait_geq(Q, Q.done1 + prev, 1);
      if (!ok) it.kind = -1;
    }
  }
  *out = it;
}

// NTK instantiations carry the tangent rows (twice the pipeline registers)
// in the same launch shapes (at 128 registers they spill a few bytes).
template <int N0, int N1, bool BIAS, int NT, int RMAX, int ACT, bool NTK = false, int N2 = 0>
__global__ void __launch_bounds__(NT, 512 / NT) k_myrtle_tiled(const __grid_constant__ TiledParams Q) {
  extern __shared__ __align__(16) unsigned char smem[];
  using SM = Smem<N0, N1, RMAX, NTK, N2>;
  constexpr bool TWO = N1 > 0;
  double* red = reinterpret_cast<double*>(smem + SM::tables);
  Item* item = reinterpret_cast<Item*>(smem + SM::tables + SM::red);
  for (;;) {
    if (threadIdx.x == 0) claim<TWO>(Q, item);
    __syncthreads();
    const Item it = *item;
    if (it.kind < 0) break;
    if (it.kind == 0) {
      if constexpr (RMAX == 64) {
        if (Q.R[it.b] == 64)
          item0<Stage0<64, N0, N1, BIAS, ACT, NTK>, NT, NTK>(Q, it, smem, red);
        else
          item0<Stage0<32, N0, N1, BIAS, ACT, NTK>, NT, NTK>(Q, it, smem, red);
      } else {
        item0<Stage0<32, N0, N1, BIAS, ACT, NTK>, NT, NTK>(Q, it, smem, red);
      }
    } else if constexpr (TWO) {
      if constexpr (RMAX == 64) {
        if (Q.R[it.b] == 64)
          item1<Stage1<32, N0, N1, BIAS, ACT, NTK>, NT, NTK, 0>(Q, it, smem, red);
        else
          item1<Stage1<16, N0, N1, BIAS, ACT, NTK>, NT, NTK, 0>(Q, it, smem, red);
      } else {
        item1<Stage1<16, N0, N1, BIAS, ACT, NTK, N2>, NT, NTK, N2>(Q, it, smem, red);
      }
    }
    // the next item's staging overwrites the tables
    __syncthreads();
  }
}

template <int N0, int N1, bool BIAS, int NT, int RMAX, int ACT, bool NTK = false, int N2 = 0>
cudaError_t launch_t(TiledParams& Q, const int64_t* npairs, int sm_count, void* ws, size_t ws_bytes,
                     cudaStream_t st) {
  using SM = Smem<N0, N1, RMAX, NTK, N2>;
  auto kern = k_myrtle_tiled<N0, N1, BIAS, NT, RMAX, ACT, NTK, N2>;
  constexpr size_t smem = SM::bytes;
  constexpr int tensors = NTK ? 2 : 1;
  static bool attr_set[64] = {false};
  static int per_sm[64] = {0};
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) dev = 0;
  if (!attr_set[dev]) {
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    int nb = 0;
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, kern, NT, smem);
    if (e != cudaSuccess) return e;
    per_sm[dev] = nb > 0 ? nb : 1;
    attr_set[dev] = true;
  }
  const int grid = std::max(1, sm_count * per_sm[dev]);
  constexpr bool TWO = N1 > 0;
  int64_t np[QUEUE_MAX];
  for (int b = 0; b < Q.n; ++b) np[b] = npairs[b];
  if (sched::split_tail(Q, np, grid, Q.wn[0] / (NT / 32))) Q.B[Q.n - 1] = Q.B[0];
  const sched::Plan p = sched::make_plan(TWO, Q.R, np, Q.n, grid, tensors);
  if (p.bytes > ws_bytes) return cudaErrorInvalidValue;
  Q.LAG = p.LAG;
  Q.nitems = Q.T0 + (TWO ? Q.G : 0);
  const size_t G = (size_t)Q.G;
  char* c = reinterpret_cast<char*>(ws);
  for (int r = 0; r < 2; ++r) {
    Q.S[r] = p.S[r];
    Q.slot_floats[r] = p.slot_floats[r];
    Q.ring_off[r] = p.ring_off[r];
  }
  Q.slots = reinterpret_cast<float*>(c);
  Q.gacc = reinterpret_cast<double*>(c + p.slot_bytes);
  Q.cnt0 = reinterpret_cast<int*>(c + p.slot_bytes + tensors * G * sizeof(double));
  Q.done1 = Q.cnt0 + G;
  Q.next = reinterpret_cast<unsigned long long*>(c + p.slot_bytes + G * (2 * sizeof(int) + tensors * sizeof(double)));
  Q.abort_flag = reinterpret_cast<int*>(Q.next + 1);
  cudaError_t e = cudaMemsetAsync(ws, 0, p.bytes, st);
  if (e != cudaSuccess) return e;
  kern<<<grid, NT, smem, st>>>(Q);
  return cudaGetLastError();
}

// Fills the queue description shared by every instantiation.  False when a
// block is not 64x64 or 32x32 or 64x64 blocks do not come first.
inline bool make_queue(TiledParams& Q, int64_t* np, const int* R, const FusedParams* B, int n,
                       unsigned int* dstatus, long long wait_limit) {
  Q = TiledParams{};
  Q.n = n;
  Q.g0[0] = 0;
  Q.f0[0] = 0;
  for (int b = 0; b < n; ++b) {
    if (R[b] != 64 && R[b] != 32) return false;
    if (b > 0 && R[b] > R[b - 1]) return false;  // 64x64 blocks first
    Q.R[b] = R[b];
    Q.nt0[b] = R[b] == 64 ? sched::tasks_per_pair(64) : sched::tasks_per_pair(32);
    Q.split[b] = 1;
    Q.wn[b] = R[b] == 64 ? G0<64, COLS0>::WT : G0<32, COLS0>::WT;
    Q.B[b] = B[b];
    np[b] = B[b].npairs;
    Q.g0[b + 1] = Q.g0[b] + B[b].npairs;
    Q.f0[b + 1] = Q.f0[b] + B[b].npairs * Q.nt0[b];
    if (R[b] == 64) Q.G64 = Q.g0[b + 1];
  }
  Q.G = Q.g0[n];
  Q.T0 = Q.f0[n];
  Q.dstatus = dstatus;
  Q.wait_limit = wait_limit;
  return true;
}

// The instantiations of one activation: stage patterns (2,1,0) (1) (1,1),
// with and without the bias, 256-thread 32x32-only or 512-thread launches.
template <int ACT>
cudaError_t launch_act(const int c[3], bool bias, TiledParams& Q, const int64_t* np, int sm_count, void* ws,
                       size_t ws_bytes, cudaStream_t st) {
  const bool only32 = Q.G64 == 0;
#define NK_T(a, b_)                                                                                    \
  if (c[0] == a && c[1] == b_) {                                                                       \
    if (only32)                                                                                        \
      return bias ? launch_t<a, b_, true, NT32, 32, ACT>(Q, np, sm_count, ws, ws_bytes, st)            \
                  : launch_t<a, b_, false, NT32, 32, ACT>(Q, np, sm_count, ws, ws_bytes, st);          \
    return bias ? launch_t<a, b_, true, 512, 64, ACT>(Q, np, sm_count, ws, ws_bytes, st)              \
                : launch_t<a, b_, false, 512, 64, ACT>(Q, np, sm_count, ws, ws_bytes, st);            \
  }
  NK_T(2, 1) NK_T(1, 0) NK_T(1, 1)
#undef NK_T
  return cudaErrorNotSupported;
}

}  // namespace tiled
}  // namespace nkf
