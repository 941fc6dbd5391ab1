// Fused Myrtle NNGP blocks (NK_PREC_MIXED, ReLU) of 16x16 and 8x8 images: the
// packed row stream of the tiled form (myrtle_tiled.cuh: Band) with a whole
// pair on one CTA (16x16) or on one warp (8x8), so that no pooled tensor, task
// queue or cluster barrier passes between CTAs.
//
//  * 16x16: one CTA of 256 threads a pair, two CTAs an SM.  Stage 0 pools with
//    atomic adds into a 16 KB slot of the CTA's own in L2 (shared memory has
//    no native FP32 add), stage 1 takes its rows from there, and an 8x8
//    stage's pooled tensor (256 values) stays in shared memory.
//  * 8x8: one warp a pair; the warp alone writes its pooled tile, so plain
//    adds serve and a warp synchronisation is all that separates stages.
//  * Stages of side 4 and 2 (256 and 16 pixel pairs) go entry by entry, with
//    the pool as a gather.
//
// Issue bound like the tiled form.  Against the cluster kernel, (2,1,0) with a
// bias: 16x16 one pair 49 -> 40 us, 32,768 pairs 8.72 -> 4.43 ms; 8x8 one pair
// 26 -> 24 us (launch), 32,768 pairs 2.25 -> 0.336 ms (24 warps used to share
// an 8x8 pair).
#pragma once

#include "myrtle_tiled.cuh"

namespace nkf {
namespace small {

using tiled::Band;
using tiled::cp_async;
using tiled::cp_async_wait;
using tiled::Cut;
using tiled::edges;
using tiled::ld_x;
using tiled::QRow;
using tiled::st_shared;

// Tables of a banded stage of N layers at side R (p' side doubled along rows
// and columns), with the x entries when it is the first (SEED).
template <int R, int N, bool SEED>
struct LS : Cut<R, (R == 16 ? 2 : 1)> {
  using C = Cut<R, (R == 16 ? 2 : 1)>;
  using W = QRow<C, 2 * R>;
  static constexpr int PL = R * C::PROW, QL = 2 * R * W::Q;
  static constexpr size_t xs_off = 0;
  static constexpr size_t xq_off = SEED ? (size_t)R * C::XROW * 16 : 0;
  static constexpr size_t p_off = xq_off + (SEED ? (size_t)2 * R * W::X * 16 : 0);
  static constexpr size_t q_off = p_off + (size_t)N * PL * 8;
  static constexpr size_t bytes = (q_off + (size_t)N * QL * 8 + 15) / 16 * 16;
  static constexpr int WPT = R / (2 * C::TYP);  // warp tasks per t_x
};

// Tables of an entry-by-entry stage: factor pairs of both sides per pixel.
template <int R, int N>
struct LE {
  static constexpr size_t bytes = (size_t)2 * N * R * R * 8;
};

// Copies a banded stage's tables (layers Lr0 ..) by NT threads.
template <class L, int NT, int N, bool SEED>
__device__ __forceinline__ void load_banded(const FusedParams& P, int Lr0, int64_t ia, int64_t ib,
                                            unsigned char* smem, int tid) {
  constexpr int R = L::R;
  using W = typename L::W;
  const float2* qa = reinterpret_cast<const float2*>(P.qsa) + ia * P.nq;
  const float2* qb = reinterpret_cast<const float2*>(P.qsb) + ib * P.nq;
  float4* xs = reinterpret_cast<float4*>(smem + L::xs_off);
  float2* pt = reinterpret_cast<float2*>(smem + L::p_off);
  const unsigned xq = smem_u32(smem) + (unsigned)L::xq_off, qt = smem_u32(smem) + (unsigned)L::q_off;
  const int C = P.C;
  for (int e = tid; e < R * R; e += NT) {
    const int row = e / R, c = e % R;
#pragma unroll
    for (int d = 0; d < 4; ++d) {  // the four copies of a p' entry
      const int rr = row + (d >> 1) * R, pc = W::pos(c + (d & 1) * R);
      if constexpr (SEED) {
        const unsigned xd = xq + 16u * (rr * W::X + pc);
        const float* src = P.Xb + (ib * R * R + e) * C;
#pragma unroll
        for (int ch = 0; ch < 3; ++ch) {
          if (ch < C)
            cp_async<4>(xd + 4 * ch, src + ch);
          else
            st_shared(xd + 4 * ch, 0.f);
        }
      }
#pragma unroll
      for (int l = 0; l < N; ++l)
        cp_async<8>(qt + 8u * (l * L::QL + rr * W::Q + pc), qb + P.qoff[Lr0 + l] + e);
    }
    const int part = c / L::COLS, k = c % L::COLS;
    if constexpr (SEED)
      xs[row * L::XROW + part * L::XST + k] = ld_x(P.Xa + (ia * R * R + e) * C, C, P.xscale);
#pragma unroll
    for (int l = 0; l < N; ++l) {
      const float2 v = qa[P.qoff[Lr0 + l] + e];
      pt[l * L::PL + row * L::PROW + part * L::PST + k] = make_float2(v.x, v.y * P.foldp[Lr0 + l]);
    }
  }
}

template <int R, int NT, int N>
__device__ __forceinline__ void load_entries(const FusedParams& P, int Lr0, int64_t ia, int64_t ib, float2* t,
                                             int tid) {
  const float2* qa = reinterpret_cast<const float2*>(P.qsa) + ia * P.nq;
  const float2* qb = reinterpret_cast<const float2*>(P.qsb) + ib * P.nq;
  for (int e = tid; e < N * R * R; e += NT) {
    const int l = e / (R * R), p = e - l * R * R;
    const float2 v = qa[P.qoff[Lr0 + l] + p];
    t[e] = make_float2(v.x, v.y * P.foldp[Lr0 + l]);
    t[N * R * R + e] = qb[P.qoff[Lr0 + l] + p];
  }
}

// The band fields that a table layout fixes (super-planes t_y, t_y + 1 = the
// halves, t_x; part q of a row).
template <class L, bool SEED, class BT>
__device__ __forceinline__ void set_band(BT& T, const unsigned char* smem, int t_x, int t_y, int q, float b) {
  using W = typename L::W;
  const unsigned sm = smem_u32(smem);
  T.t_x = t_x;
  T.t_y = t_y;
  T.s0 = 0;
  T.s1 = L::R;
  T.b0 = 0;
  edges<L::COLS>(T.E, L::R, t_x, q);
  T.xa = sm + (unsigned)L::xs_off + q * L::XST * 16;
  T.pa = sm + (unsigned)L::p_off + q * L::PST * 8;
#pragma unroll
  for (int k = 0; k < L::COLS; ++k) {
    const int c = q + W::pos(t_x + k);
    if constexpr (SEED) T.xqa[k] = sm + (unsigned)L::xq_off + ((t_y + 1) * W::X + c) * 16;
    T.qa[k] = sm + (unsigned)L::q_off + ((t_y + 1) * W::Q + c) * 8;
  }
  T.cut = (float)(L::R - t_y);
  T.in = nullptr;
  T.inT = nullptr;
  T.out = nullptr;
  T.dT = 0;
  T.dU = T.dO = 0;
  T.fth = nullptr;
  T.dg = false;
  T.b = b;
}

// Pooled output of super-planes (t_y, t_x) in a tile [T_y][T_x][I][K] of side H.
template <int H, int COLS, class BT>
__device__ __forceinline__ void set_out(BT& T, float* tile, int q) {
  const int Ty = T.t_y >> 1, Tx = T.t_x >> 1;
  T.out = tile + ((Ty * H + Tx) * H) * H + q * COLS / 2;
  T.dU = (((Ty + 1) & (H - 1)) - Ty) * (H * H * H);
  T.dO = ((((T.t_x + 1) >> 1) & (H - 1)) - Tx) * (H * H);
}

// N layers on a tile [t_y][t_x][i][k] of side R by the calling NT threads,
// ping-pong with `tmp` of the same size; sync() orders them.  Returns the
// tile that holds the last layer's output.
template <int R, int N, int NT, bool BIAS, class Sync>
__device__ __forceinline__ float* entry_layers(float* tile, float* tmp, const float2* tab, float b, int tid,
                                               Sync sync) {
  for (int l = 0; l < N; ++l) {
    const float2* pt = tab + l * R * R;
    const float2* qt = pt + N * R * R;
    for (int e = tid; e < R * R * R * R; e += NT) {
      const int k = e % R, i = e / R % R, tx = e / (R * R) % R, ty = e / (R * R * R);
      const int i2 = (i + ty) & (R - 1), k2 = (k + tx) & (R - 1);
      float s = 0.f;
#pragma unroll
      for (int dy = -1; dy <= 1; ++dy)
#pragma unroll
        for (int dx = -1; dx <= 1; ++dx)
          if (i + dy >= 0 && i + dy < R && i2 + dy >= 0 && i2 + dy < R && k + dx >= 0 && k + dx < R && k2 + dx >= 0 &&
              k2 + dx < R)
            s += tile[e + dy * R + dx];
      if constexpr (BIAS) s += b;
      const float2 p = pt[i * R + k], q = qt[i2 * R + k2];
      const float c = __saturatef(s * (p.x * q.x));
      tmp[e] = (p.y * q.y) * f2_lo(nk_Jpi01_2(f2_make(c, c)));
    }
    sync();
    float* t = tile;
    tile = tmp;
    tmp = t;
  }
  return tile;
}

// 2x2 pool of both pixels: a tile of side R to one of side R / 2 (the factor
// 1/16 is in the layer's fold).
template <int R, int NT>
__device__ __forceinline__ void entry_pool(const float* in, float* out, int tid) {
  constexpr int H = R / 2;
  for (int e = tid; e < H * H * H * H; e += NT) {
    const int K = e % H, I = e / H % H, Tx = e / (H * H) % H, Ty = e / (H * H * H);
    const int I2 = (I + Ty) & (H - 1), K2 = (K + Tx) & (H - 1);
    float s = 0.f;
#pragma unroll
    for (int a = 0; a < 4; ++a)
#pragma unroll
      for (int c = 0; c < 4; ++c) {
        const int i = 2 * I + (a >> 1), k = 2 * K + (a & 1), i2 = 2 * I2 + (c >> 1), k2 = 2 * K2 + (c & 1);
        s += in[((((i2 - i) & (R - 1)) * R + ((k2 - k) & (R - 1))) * R + i) * R + k];
      }
    out[e] = s;
  }
}

__device__ __forceinline__ double warp_total(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(FULL, v, o);
  return v;
}

// --------------------------------------------------------------------------
// 8x8: one warp a pair.
// --------------------------------------------------------------------------
constexpr int W8 = 4;  // warps of a CTA

template <int N0, int N1, int N2>
struct Smem8 {
  using L = LS<8, N0, true>;
  static constexpr size_t tile_off = L::bytes;  // side 4: two tiles of 256, then side 2: two of 16
  static constexpr size_t t1_off = tile_off + (N1 > 0 ? (2 * 256 + 2 * 16) * 4 : 0);
  static constexpr size_t t2_off = t1_off + LE<4, N1>::bytes;
  static constexpr size_t bytes = (t2_off + LE<2, N2>::bytes + 15) / 16 * 16;
};

template <int N0, int N1, int N2, bool BIAS>
__global__ void __launch_bounds__(32 * W8, 4) k_myrtle_small8(const __grid_constant__ FusedParams P) {
  extern __shared__ __align__(16) unsigned char raw[];
  using S = Smem8<N0, N1, N2>;
  using L = typename S::L;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  unsigned char* smem = raw + warp * S::bytes;
  float* tile = reinterpret_cast<float*>(smem + S::tile_off);
  float2* t1 = reinterpret_cast<float2*>(smem + S::t1_off);
  float2* t2 = reinterpret_cast<float2*>(smem + S::t2_off);
  auto sync = [] { __syncwarp(); };
  const int q = lane / L::TYP, tyl = lane % L::TYP;
  for (int64_t g = (int64_t)blockIdx.x * W8 + warp; g < P.npairs; g += (int64_t)gridDim.x * W8) {
    int64_t i, j;
    sched::pair_of(g, P.na, P.nb, P.sym, &i, &j);
    const int64_t ia = P.a0 + i, ib = P.b0 + j;
    __syncwarp();
    load_banded<L, 32, N0, true>(P, 0, ia, ib, smem, lane);
    if constexpr (N1 > 0) {
      load_entries<4, 32, N1>(P, N0, ia, ib, t1, lane);
      if constexpr (N2 > 0) load_entries<2, 32, N2>(P, N0 + N1, ia, ib, t2, lane);
      for (int e = lane; e < 256; e += 32) tile[e] = 0.f;
    }
    cp_async_wait();
    __syncwarp();
    double gap = 0.0, gapT = 0.0;
#pragma unroll 1
    for (int t_x = 0; t_x < 8; ++t_x) {
      Band<L, N0, true, N1 == 0, BIAS, NK_ACT_RELU, false, false, (N1 > 0)> T;
      set_band<L, true>(T, smem, t_x, 2 * tyl, q, P.sb2);
      if constexpr (N1 > 0) set_out<4, 1>(T, tile, q);
      T.run(gap, gapT);
      __syncwarp();
    }
    if constexpr (N1 > 0) {
      const float* o = entry_layers<4, N1, 32, BIAS>(tile, tile + 256, t1, P.sb2, lane, sync);
      if constexpr (N2 > 0) {
        float* u = tile + 512;
        entry_pool<4, 32>(o, u, lane);
        __syncwarp();
        o = entry_layers<2, N2, 32, BIAS>(u, u + 16, t2, P.sb2, lane, sync);
        gap = lane < 16 ? (double)o[lane] : 0.0;
      } else {
        for (int e = lane; e < 256; e += 32) gap += (double)o[e];
      }
    }
    gap = warp_total(gap);
    if (lane == 0) store_entry(P, i, j, gap);
  }
}

// --------------------------------------------------------------------------
// 16x16: one CTA a pair.
// --------------------------------------------------------------------------
constexpr int NT16 = 256;

template <int N0, int N1, int N2>
struct Smem16 {
  using L = LS<16, N0, true>;
  using M = LS<8, N1 == 0 ? 1 : N1, false>;
  static constexpr size_t m_off = L::bytes;
  static constexpr size_t tile_off = m_off + (N1 > 0 ? M::bytes : 0);  // side 4: two tiles of 256
  static constexpr size_t t2_off = tile_off + (N2 > 0 ? 2 * 256 * 4 : 0);
  static constexpr size_t red_off = t2_off + LE<4, N2>::bytes;
  static constexpr size_t bytes = red_off + NT16 / 32 * 8;
};

template <int N0, int N1, int N2, bool BIAS>
__global__ void __launch_bounds__(NT16, 2) k_myrtle_small16(const __grid_constant__ FusedParams P, float* slots) {
  extern __shared__ __align__(16) unsigned char smem[];
  using S = Smem16<N0, N1, N2>;
  using L = typename S::L;
  using M = typename S::M;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  float* slot = slots + (size_t)blockIdx.x * 4096;  // zero between pairs
  float* tile = reinterpret_cast<float*>(smem + S::tile_off);
  float2* t2 = reinterpret_cast<float2*>(smem + S::t2_off);
  double* red = reinterpret_cast<double*>(smem + S::red_off);
  auto sync = [] { __syncthreads(); };
  const int q = lane / L::TYP, tyl = lane % L::TYP;
  for (int64_t g = blockIdx.x; g < P.npairs; g += gridDim.x) {
    int64_t i, j;
    sched::pair_of(g, P.na, P.nb, P.sym, &i, &j);
    const int64_t ia = P.a0 + i, ib = P.b0 + j;
    load_banded<L, NT16, N0, true>(P, 0, ia, ib, smem, tid);
    if constexpr (N1 > 0) load_banded<M, NT16, N1, false>(P, N0, ia, ib, smem + S::m_off, tid);
    if constexpr (N2 > 0) {
      load_entries<4, NT16, N2>(P, N0 + N1, ia, ib, t2, tid);
      tile[tid] = 0.f;
    }
    cp_async_wait();
    __syncthreads();
    double gap = 0.0, gapT = 0.0;
#pragma unroll 1
    for (int w = warp; w < 16 * L::WPT; w += NT16 / 32) {
      Band<L, N0, true, N1 == 0, BIAS, NK_ACT_RELU> T;
      set_band<L, true>(T, smem, w / L::WPT, 2 * ((w % L::WPT) * L::TYP + tyl), q, P.sb2);
      if constexpr (N1 > 0) set_out<8, 2>(T, slot, q);
      T.run(gap, gapT);
    }
    if constexpr (N1 > 0) {
      __threadfence();  // the pooled adds, before the CTA's stage 1 reads them
      __syncthreads();
#pragma unroll 1
      for (int t_x = warp; t_x < 8; t_x += NT16 / 32) {
        const int mq = lane / M::TYP, mt = lane % M::TYP;
        Band<M, N1, false, N2 == 0, BIAS, NK_ACT_RELU> T;
        set_band<M, false>(T, smem + S::m_off, t_x, 2 * mt, mq, P.sb2);
        T.in = slot + ((T.t_y * 8 + t_x) * 8) * 8 + mq;
        if constexpr (N2 > 0) set_out<4, 1>(T, tile, mq);
        T.run(gap, gapT);
      }
      if constexpr (N2 > 0) {
        __syncthreads();
        const float* o = entry_layers<4, N2, NT16, BIAS>(tile, tile + 256, t2, P.sb2, tid, sync);
        gap = (double)o[tid];
      } else {
        __threadfence();  // the slot's clears, before the next pair's adds
      }
    }
    gap = warp_total(gap);
    if (lane == 0) red[warp] = gap;
    if constexpr (N2 > 0) __threadfence();
    __syncthreads();  // also: the next pair's tables overwrite this one's
    if (tid == 0) {
      double s = 0.0;
      for (int w = 0; w < NT16 / 32; ++w) s += red[w];
      store_entry(P, i, j, s);
    }
    __syncthreads();
  }
}

}  // namespace small
}  // namespace nkf
