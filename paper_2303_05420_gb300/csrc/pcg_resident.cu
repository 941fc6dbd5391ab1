// One CG run of nk_pcg_solve (FP32 products, Jacobi or no preconditioner) with
// K held in the shared memory of the whole GPU, all of it or the rows that
// fit: a cooperative kernel, one CTA
// per SM, each owning nr = ceil(N / SMs) rows of K and of every vector.
//
// Why: at N of a few thousand an iteration's work is a microsecond (16 MB of
// K at N = 2048, 42 M multiply-adds), but as four launches replayed from a
// graph it took 36: K came from L2 each time and 10 MB of row-split partial
// sums went through it twice.  Here K is read once per run, a row's product
// sums stay on its SM, and what an iteration costs is crossing the chip.
//
// Textbook CG needs three crossings an iteration, about 3 us each: the sum that
// beta takes, the direction, (p, A p).  Where a warp has one block of columns
// and one group of right-hand sides (KEEP: N up to about 2,700 and 16 columns,
// 10 from N = 2,049 on) two do: z = M r is published together with (r, z) and
// (r, r), and after that crossing every SM forms the direction p = z + beta
// p_old on its own, its old one still in the lanes' registers.  It is the same
// FP32 operation on the same values everywhere, so the p that the rows' owners
// add to x is the p of the product.  Elsewhere the owners publish p.
//
// CG with one reduction (Chronopoulos and Gear: A p and (p, A p) by recurrences)
// has two crossings everywhere and was faster (12.7 us an iteration at N = 2048,
// 10 columns, and 13.3 here), but with FP32 products its recurrences drift: at
// kappa = 7e7 (1000 points, Gaussian kernel) (p, A p) came out negative and
// the solve diverged where this form converges as the graph-replayed run does.
// Flags in place of the barriers (a warp waiting for the CTAs that own its
// columns, a column for its own counter) were slower, 18 us: every word has 152
// pollers.
//
// Matvec: a warp owns 128 columns; a lane holds p at 8 of them for half of a
// group of right-hand sides (2 RH <= 16 of them) in registers, as f32x2 over
// column pairs, and meets every row of the CTA with two 16-byte loads.  A
// row's sums over a warp's 128 columns are eight-column sums added in an FP32
// butterfly that folds 16 (row, right-hand side) values at once (15 shuffles,
// not 80); the warps' sums are added in two floats (TwoSum) and go on in FP64.
// Short FP32 runs, then wider: as in k_matvec, whose runs are 32 to 256
// products long.  x, r, A p, scalars and dot products are FP64; the direction is
// the FP32 one that the product takes (with an FP64 p and its FP32 copy, as in
// the graph-replayed run, x and r drift apart by the copy's rounding: 600 points,
// kappa 4e6, products in FP32 alone, residual 1.3e-3 there and 1.1e-3 here).  gl
// lanes (a power of two, at least nr) hold a column's rows, so several columns share a
// warp's FP64 instructions, each of which takes its scheduler 64 cycles.
//
// Every SM reads the same sums, so all take the same decisions.  Waits are
// bounded; one that runs out sets *status and ends the kernel.
#include <algorithm>

#include "nk_common.cuh"
#include "nk_f32x2.cuh"
#include "pcg_resident.h"

namespace {

struct Args {
  const float* K;
  int64_t ldk;
  int N, R, nr, npad, groups;
  int res;              // rows of each CTA held in shared memory
  int gl;               // lanes of a column: a power of two, nr of them used
  int vec;              // K rows are 16-byte aligned
  const double* B;
  const double* minv;
  double* X;
  float* P;             // published z (KEEP) or p, see p_index
  double* sums;         // [3 slots][R][4]: (r, z), (r, r), (p, A p), unused
  unsigned* bar;        // barrier count; bar[1]: status
  long long polls;      // bound of a barrier's wait
  double lam, tol2;
  double tol2_long;     // in place of tol2 from iteration NK_LONG_RUN on
  int maxit;
  double* iters;        // [R] iterations of each column
};

// Element (i, r) of the published vector: right-hand sides in groups of
// 2 RH, within a group blocks of 8 columns x RH sides per (8-column block,
// half), which is what a lane loads.
template <int RH>
__device__ __forceinline__ int64_t p_index(int npad, int i, int r) {
  const int g = r / (2 * RH), q = r - g * 2 * RH;
  return (int64_t)g * npad * 2 * RH + (((i >> 3) * 2 + q / RH) * RH + q % RH) * 8 + (i & 7);
}

// A barrier of all CTAs, in two halves: arrive() by all threads (everything
// that they wrote is then on its way), of which the last warp's first thread
// counts the CTA in and waits, while other warps may go on with work of their
// own; leave() by all threads, false if the wait ran out.
struct GridBarrier {
  unsigned* bar;
  long long polls;  // bound of a wait
  unsigned target;
  bool ok;
  // also: whether `flag` holds in any thread of the CTA
  __device__ int arrive(int flag) {
    target += gridDim.x;
    const int any = __syncthreads_or(flag);
    ok = true;
    if (threadIdx.x == blockDim.x - 32) {
      __threadfence();
      atomicAdd(bar, 1u);
      ok = false;
      for (long long k = 0; k < polls && !ok; ++k) {
        unsigned v;
        asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(bar) : "memory");
        ok = (int)(v - target) >= 0;
      }
      if (!ok) atomicExch(bar + 1, 1u);
    }
    return any;
  }
  __device__ bool leave() { return __syncthreads_and(ok) != 0; }
};

__device__ __forceinline__ void red_add(double* p, double v) {
  asm volatile("red.relaxed.gpu.global.add.f64 [%0], %1;" ::"l"(p), "d"(v) : "memory");
}

__device__ __forceinline__ void two_sum(float& s, float& c, float p) {
  const float t = __fadd_rn(s, p);
  const float z = __fsub_rn(t, s);
  c = __fadd_rn(c, __fadd_rn(__fsub_rn(s, __fsub_rn(t, z)), __fsub_rn(p, z)));
  s = t;
}

// STREAM: rows from a.res on are read from memory in every product.
// KEEP: a warp has one block of columns and one group of right-hand sides, and
// its lanes keep their p in registers.
template <int RH, int MAXT, bool STREAM, bool KEEP>
__global__ void __launch_bounds__(MAXT, 1) k_cg_resident(const __grid_constant__ Args a) {
  extern __shared__ __align__(16) unsigned char smem[];
  constexpr int RC = 16 / RH, V = RC * RH;  // rows a butterfly folds; its values (<= 16)
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, T = blockDim.x;
  const int N = a.N, R = a.R, npad = a.npad, cbs = npad / 128;
  const int row0 = blockIdx.x * a.nr, nrow = min(a.nr, N - row0);
  const int res = STREAM ? min(a.res, nrow) : nrow;
  float* Ks = reinterpret_cast<float*>(smem);  // [res][npad]
  // vectors, [R][nr]; an element is touched by its own thread only
  double* x = reinterpret_cast<double*>(Ks + (size_t)a.res * npad);
  double* rv = x + a.nr * R;
  double* p = rv + a.nr * R;
  double* q = p + a.nr * R;
  double* mi = q + a.nr * R;                              // [nr]
  float* pf = reinterpret_cast<float*>(mi + a.nr);        // [R][nr]: p again, and z
  float* zf = pf + a.nr * R;
  float* part = zf + a.nr * R;                            // [cbs][nr * 2 RH]
  const int pstride = a.nr * 2 * RH;
  // this thread's row and its first column; the columns repeat every cstep
  const int ri = lane & (a.gl - 1), col0 = warp * (32 / a.gl) + lane / a.gl, cstep = (T >> 5) * (32 / a.gl);
  int c_its = 0;      // column `lane`, warp 0: its iterations
  double c_bb = 0.0;  // and (b, b)
  // per column: alpha, 1 / (r, z), tol^2 (b, b), beta, whether it goes on
  __shared__ double s_al[32], s_inv[32], s_lim[32];
  __shared__ float s_be[32];
  __shared__ int s_on[32];
  GridBarrier gb = {a.bar, a.polls, 0, true};

  for (int i = 0; i < res; ++i) {
    const float* src = a.K + (int64_t)(row0 + i) * a.ldk;
    float* dst = Ks + (size_t)i * npad;
    for (int c = 4 * tid; c < npad; c += 4 * T) {
      float4 v;
      if (a.vec && c + 3 < N) {
        v = __ldg(reinterpret_cast<const float4*>(src + c));
      } else {
        v.x = c < N ? __ldg(src + c) : 0.f;
        v.y = c + 1 < N ? __ldg(src + c + 1) : 0.f;
        v.z = c + 2 < N ? __ldg(src + c + 2) : 0.f;
        v.w = c + 3 < N ? __ldg(src + c + 3) : 0.f;
      }
      *reinterpret_cast<float4*>(dst + c) = v;
    }
  }
  for (int i = tid; i < nrow; i += T) mi[i] = a.minv[row0 + i];
  if (tid < 32) {
    s_inv[tid] = s_lim[tid] = 0.0;
    s_on[tid] = tid < R;
  }
  __syncthreads();

  // sum over a column's lanes (every lane of the warp takes part)
  auto col_sum = [&](double v) {
    for (int o = a.gl >> 1; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
  };
  // z = M r (published with KEEP); (r, z) and (r, r) go to slot `slot`
  auto publish = [&](int r, bool mine, int slot) {
    double rz = 0.0, rr = 0.0;
    if (mine) {
      const int e = r * a.nr + ri;
      const double rn = rv[e], zn = mi[ri] * rn;
      zf[e] = (float)zn;
      if constexpr (KEEP) __stcg(a.P + p_index<RH>(npad, row0 + ri, r), zf[e]);
      rz = rn * zn;
      rr = rn * rn;
    }
    // both sums in one butterfly: the upper half of the lanes takes (r, r)
    const int o = a.gl >> 1;
    double* out = a.sums + ((size_t)slot * R + min(r, R - 1)) * 4;
    if (o == 0) {
      if (mine) {
        red_add(out, rz);
        red_add(out + 1, rr);
      }
      return;
    }
    const bool up = (ri & o) != 0;
    double v = (up ? rr : rz) + __shfl_xor_sync(0xffffffffu, up ? rz : rr, o);
    for (int x = o >> 1; x > 0; x >>= 1) v += __shfl_xor_sync(0xffffffffu, v, x);
    if (r < R && (ri & (o - 1)) == 0) red_add(out + (up ? 1 : 0), v);
  };

  for (int cw = warp * (32 / a.gl), r = col0; cw < R; cw += cstep, r += cstep) {  // cw: the warp's first column
    const bool mine = r < R && ri < nrow;
    if (mine) {
      const int e = r * a.nr + ri;
      x[e] = 0.0;
      pf[e] = 0.f;
      rv[e] = a.B[(int64_t)(row0 + ri) * R + r];
    }
    publish(r, mine, 0);
  }

  // a lane's columns and right-hand sides of the published vector, block cb, group g
  const int cg = lane >> 1, half = lane & 1;
  auto at = [&](int g, int cb) {
    return (int64_t)g * npad * 2 * RH + ((int64_t)((cb * 16 + cg) * 2 + half) * RH) * 8;
  };
  auto load = [&](const float* from, int h, f2 (&v)[4]) {
    const float4 a = __ldcg(reinterpret_cast<const float4*>(from) + 2 * h);
    const float4 b = __ldcg(reinterpret_cast<const float4*>(from) + 2 * h + 1);
    v[0] = f2_make(a.x, a.y);
    v[1] = f2_make(a.z, a.w);
    v[2] = f2_make(b.x, b.y);
    v[3] = f2_make(b.z, b.w);
  };
  f2 P2[RH][4];
#pragma unroll
  for (int h = 0; h < RH; ++h) P2[h][0] = P2[h][1] = P2[h][2] = P2[h][3] = f2_dup(0.f);

  for (int it = 0;; ++it) {
    gb.arrive(0);
    if (!gb.leave()) return;
    // with registers to spare, z is on its way while the sums are
    constexpr bool EARLY = KEEP && RH <= 5 && MAXT <= 512;
    f2 Z2[EARLY ? RH : 1][4];
    if constexpr (EARLY) {
      if (warp < cbs) {
#pragma unroll
        for (int h = 0; h < RH; ++h) load(a.P + at(0, warp), h, Z2[h]);
      }
    }
    double* sums = a.sums + (size_t)(it % 3) * R * 4;
    // every warp: the columns that go on (the same everywhere), and their beta;
    // sums of squares compare as their bits do (a NaN stops its column)
    double rz = 0.0;
    int on = 0;
    if (lane < R) {
      const long long rr = __double_as_longlong(__ldcg(sums + lane * 4 + 1));
      rz = __ldcg(sums + lane * 4);
      on = s_on[lane] && (it == 0 || (rr > __double_as_longlong(s_lim[lane]) && rr <= 0x7ff0000000000000ll));
    }
    if (!__any_sync(0xffffffffu, on) || it == a.maxit) break;
    const float beta = lane < R ? (float)(rz * s_inv[lane]) : 0.f;
    if (warp == 0) s_be[lane] = beta;
    if constexpr (!KEEP) {
      __syncthreads();
      for (int r = col0; r < R; r += cstep) {
        const int e = r * a.nr + ri;
        if (ri < nrow) __stcg(a.P + p_index<RH>(npad, row0 + ri, r), pf[e] = fmaf(s_be[r], pf[e], zf[e]));
      }
      gb.arrive(0);
      if (!gb.leave()) return;
    }
    // A p and (p, A p), A = K + lam I
    for (int g = 0; g < a.groups; ++g) {
      for (int cb = warp; cb < cbs; cb += T >> 5) {
#pragma unroll
        for (int h = 0; h < RH; ++h) {
          if constexpr (KEEP) {
            f2 z[4];
            if constexpr (EARLY) {
#pragma unroll
              for (int c = 0; c < 4; ++c) z[c] = Z2[h][c];
            } else {
              load(a.P + at(g, cb), h, z);
            }
            const f2 be = f2_dup(__shfl_sync(0xffffffffu, beta, half * RH + h));
#pragma unroll
            for (int c = 0; c < 4; ++c) P2[h][c] = f2_fma(be, P2[h][c], z[c]);
          } else {
            load(a.P + at(g, cb), h, P2[h]);
          }
        }
        const int c0 = cb * 128 + cg * 8;
        float* out = part + (size_t)cb * pstride;
        // the RC rows from i0 on (clamped to the last): eight columns each
        auto rows = [&](int i0, const float4 (&ka)[RC], const float4 (&kb)[RC], int end) {
          float v[16];
#pragma unroll
          for (int e = V; e < 16; ++e) v[e] = 0.f;
#pragma unroll
          for (int q = 0; q < RC; ++q) {
            const f2 k0 = f2_make(ka[q].x, ka[q].y), k1 = f2_make(ka[q].z, ka[q].w), k2 = f2_make(kb[q].x, kb[q].y),
                     k3 = f2_make(kb[q].z, kb[q].w);
#pragma unroll
            for (int h = 0; h < RH; ++h) {
              f2 t = f2_mul(k0, P2[h][0]);
              t = f2_fma(k1, P2[h][1], t);
              t = f2_fma(k2, P2[h][2], t);
              t = f2_fma(k3, P2[h][3], t);
              v[q * RH + h] = f2_lo(t) + f2_hi(t);
            }
          }
          // fold over the 16 column blocks: lane (cg, half) ends with value cg
#pragma unroll
          for (int w = 8; w > 0; w >>= 1) {
            const bool up = (cg & w) != 0;
#pragma unroll
            for (int e = 0; e < w; ++e) {
              const float keep = up ? v[e + w] : v[e], send = up ? v[e] : v[e + w];
              v[e] = keep + __shfl_xor_sync(0xffffffffu, send, 2 * w);
            }
          }
          const int i = i0 + cg / RH;
          if (cg < V && i < end) out[i * 2 * RH + half * RH + cg % RH] = v[0];
        };
        for (int i0 = 0; i0 < res; i0 += RC) {
          float4 ka[RC], kb[RC];
#pragma unroll
          for (int q = 0; q < RC; ++q) {
            const float* k = Ks + (size_t)min(i0 + q, res - 1) * npad + c0;
            ka[q] = *reinterpret_cast<const float4*>(k);
            kb[q] = *reinterpret_cast<const float4*>(k + 4);
          }
          rows(i0, ka, kb, res);
        }
        if constexpr (STREAM) {
          auto fetch = [&](int i0, float4 (&ka)[RC], float4 (&kb)[RC]) {
#pragma unroll
            for (int q = 0; q < RC; ++q) {
              const float* k = a.K + (int64_t)(row0 + min(i0 + q, nrow - 1)) * a.ldk + c0;
              if (a.vec && c0 + 7 < N) {
                ka[q] = __ldg(reinterpret_cast<const float4*>(k));
                kb[q] = __ldg(reinterpret_cast<const float4*>(k + 4));
              } else {
                float t[8];
#pragma unroll
                for (int c = 0; c < 8; ++c) t[c] = c0 + c < N ? __ldg(k + c) : 0.f;
                ka[q] = make_float4(t[0], t[1], t[2], t[3]);
                kb[q] = make_float4(t[4], t[5], t[6], t[7]);
              }
            }
          };
          float4 a0[RC], b0[RC], a1[RC], b1[RC];
          if (res < nrow) fetch(res, a0, b0);
          for (int i0 = res; i0 < nrow; i0 += 2 * RC) {
            if (i0 + RC < nrow) fetch(i0 + RC, a1, b1);
            rows(i0, a0, b0, nrow);
            if (i0 + RC < nrow) {
              if (i0 + 2 * RC < nrow) fetch(i0 + 2 * RC, a0, b0);
              rows(i0 + RC, a1, b1, nrow);
            }
          }
        }
      }
      __syncthreads();
      const int r0 = g * 2 * RH;
      for (int cw = warp * (32 / a.gl), r = col0; cw < R; cw += cstep, r += cstep) {
        const bool mine = r >= r0 && r < min(R, r0 + 2 * RH) && ri < nrow;
        double pq = 0.0;
        if (mine) {
          float t = 0.f, c = 0.f;
          for (int w = 0; w < cbs; ++w) two_sum(t, c, part[(size_t)w * pstride + ri * 2 * RH + r - r0]);
          const int e = r * a.nr + ri;
          if constexpr (KEEP) pf[e] = fmaf(s_be[r], pf[e], zf[e]);  // as in the product
          const double pd = (double)pf[e], qn = fma(a.lam, pd, (double)t + (double)c);
          p[e] = pd;
          q[e] = qn;
          pq = qn * pd;
        }
        pq = col_sum(pq);
        if (mine && ri == 0) red_add(sums + r * 4 + 2, pq);
      }
      if (g + 1 < a.groups) __syncthreads();  // the partial sums are written again
    }
    gb.arrive(0);
    // off the path to the next sums: the reciprocal that the next beta takes
    if (warp == 0) {
      if (on) s_inv[lane] = fabs(rz) > 1e-300 ? 1.0 / rz : 0.0;
      if (it == 0 && lane < R) {
        c_bb = __ldcg(sums + lane * 4 + 1);
        s_lim[lane] = a.tol2 * c_bb;
      }
      if (it == NK_LONG_RUN) s_lim[lane] = a.tol2_long * c_bb;
      s_on[lane] = on;
      c_its += on;
    }
    if (!gb.leave()) return;
    // alpha by one lane a column: an FP64 division costs a warp the same for
    // one lane as for 32
    if (tid < R) {
      const double pq = __ldcg(sums + tid * 4 + 2);
      s_al[tid] = pq != 0.0 ? rz / pq : 0.0;
      // slot it + 2 was last read before the sums just met
      if (blockIdx.x == 0)
        for (int q = 0; q < 3; ++q) __stcg(a.sums + ((size_t)((it + 2) % 3) * R + tid) * 4 + q, 0.0);
    }
    __syncthreads();
    // x, r and the next z
    for (int cw = warp * (32 / a.gl), r = col0; cw < R; cw += cstep, r += cstep) {
      const bool mine = r < R && ri < nrow;
      if (mine && s_on[r]) {
        const double al = s_al[r];
        const int e = r * a.nr + ri;
        x[e] = fma(al, p[e], x[e]);
        rv[e] = fma(-al, q[e], rv[e]);
      }
      publish(r, mine, (it + 1) % 3);
    }
  }
  for (int r = col0; r < R; r += cstep) {
    if (ri < nrow) a.X[(int64_t)(row0 + ri) * R + r] = x[r * a.nr + ri];
  }
  if (blockIdx.x == 0 && tid < R) a.iters[tid] = (double)c_its;
}

struct Shape {
  int rh, nr, res, gl, grid, npad, groups, threads;
  size_t smem;
  bool ok;
};

// All rows in shared memory up to N of about 2,700.  Beyond, up to 32 rows a
// CTA (a column's lanes; N = 4,864), the rows that fit stay and the others are
// read in every product, mostly from L2 (K is 81 MB at N = 4500): 34.0 ms with
// graph replays and 12.6 here at N = 4500, 10 columns, tol 1e-10; at N = 3000,
// 20 columns 32.5 and 10.6.
Shape shape_of(int64_t N, int R, int sm) {
  Shape s = {};
  if (N < 1 || N > (int64_t)32 * sm || N > 8192 || R < 1 || R > 32 || sm < 1) return s;
  s.nr = (int)((N + sm - 1) / sm);
  s.grid = (int)((N + s.nr - 1) / s.nr);
  s.npad = (int)((N + 127) / 128 * 128);
  s.gl = 1;
  while (s.gl < s.nr) s.gl *= 2;
  const int cbs = s.npad / 128;
  for (int stream = 0; stream < 2 && !s.ok; ++stream) {
    if (!stream && s.npad > 3072) continue;
    // a warp a block of 128 columns; streamed, two to four of them, and at most
    // 12 warps, for the registers that hold the next rows
    s.threads = stream ? 32 * std::max(8, (cbs + (cbs + 11) / 12 - 1) / ((cbs + 11) / 12)) : std::max(256, s.npad / 4);
    // right-hand sides a lane holds: half of a group, at most 8 (5 where the
    // block needs more than 512 threads)
    const int cap = s.threads > 512 ? 5 : 8;
    const int sizes[] = {1, 2, 4, 5, 8};
    s.groups = (R + 2 * cap - 1) / (2 * cap);
    for (int v : sizes) {
      if (stream && v < 4) continue;  // the next rows' registers: 16 / v of them are in flight
      s.rh = v;
      if (2 * v * s.groups >= R) break;
    }
    const size_t fixed = ((size_t)4 * s.nr * R + s.nr) * 8 + ((size_t)2 * s.nr * R + (size_t)cbs * s.nr * 2 * s.rh) * 4;
    const size_t room = (size_t)226 * 1024, row = (size_t)s.npad * 4;
    if (fixed > room) continue;
    s.res = (int)std::min<size_t>(s.nr, (room - fixed) / row);
    s.smem = fixed + s.res * row;
    s.ok = stream || s.res == s.nr;
  }
  return s;
}

template <int RH, int MAXT, bool STREAM, bool KEEP>
cudaError_t launch(const Args& a, const Shape& s, cudaStream_t st) {
  auto kern = k_cg_resident<RH, MAXT, STREAM, KEEP>;
  const cudaError_t e = nk_smem_optin(kern, s.smem);
  if (e != cudaSuccess) return e;
  void* args[] = {const_cast<Args*>(&a)};
  return cudaLaunchCooperativeKernel(kern, dim3((unsigned)s.grid), dim3((unsigned)s.threads), args, s.smem, st);
}

// The workspace: barrier, status, sums; the published vector follows.
size_t carve(int R, char* w, Args* a) {
  const size_t sums = 256, P = sums + ((size_t)12 * R * 8 + 255) / 256 * 256;
  if (a) {
    a->bar = reinterpret_cast<unsigned*>(w);
    a->sums = reinterpret_cast<double*>(w + sums);
    a->P = reinterpret_cast<float*>(w + P);
  }
  return P;
}

}  // namespace

size_t nk_cg_resident_bytes(int64_t N, int R, int sm) {
  const Shape s = shape_of(N, R, sm);
  if (!s.ok) return 0;
  return carve(R, nullptr, nullptr) + (size_t)s.groups * s.npad * 2 * s.rh * 4;
}

cudaError_t nk_cg_resident(const float* K, int64_t ldk, int64_t N, int R, const double* B, const double* minv,
                           double* X, double lam, double tol, double tol_long, int maxit, double* iters, void* ws,
                           int sm, long long polls, cudaStream_t st) {
  const Shape s = shape_of(N, R, sm);
  if (!s.ok) return cudaErrorNotSupported;
  Args a = {};
  a.K = K;
  a.ldk = ldk;
  a.N = (int)N;
  a.R = R;
  a.nr = s.nr;
  a.npad = s.npad;
  a.groups = s.groups;
  a.res = s.res;
  a.vec = ldk % 4 == 0 && (reinterpret_cast<uintptr_t>(K) & 15) == 0;
  a.B = B;
  a.minv = minv;
  a.X = X;
  a.gl = s.gl;
  carve(R, reinterpret_cast<char*>(ws), &a);
  a.polls = polls;
  a.lam = lam;
  a.tol2 = tol * tol;
  a.tol2_long = tol_long * tol_long;
  a.maxit = maxit;
  a.iters = iters;
  // barrier, sums and the padding of the published vector
  cudaError_t e = cudaMemsetAsync(ws, 0, nk_cg_resident_bytes(N, R, sm), st);
  if (e != cudaSuccess) return e;
  if (s.res < s.nr) {
    switch (s.rh) {
      case 4: return launch<4, 384, true, false>(a, s, st);
      case 5: return launch<5, 384, true, false>(a, s, st);
      default: return launch<8, 384, true, false>(a, s, st);
    }
  }
  if (s.threads > 512) {
    if (s.groups > 1) return s.rh == 4 ? launch<4, 768, false, false>(a, s, st) : launch<5, 768, false, false>(a, s, st);
    switch (s.rh) {
      case 1: return launch<1, 768, false, true>(a, s, st);
      case 2: return launch<2, 768, false, true>(a, s, st);
      case 4: return launch<4, 768, false, true>(a, s, st);
      default: return launch<5, 768, false, true>(a, s, st);
    }
  }
  if (s.groups > 1) return s.rh == 5 ? launch<5, 512, false, false>(a, s, st) : launch<8, 512, false, false>(a, s, st);
  switch (s.rh) {
    case 1: return launch<1, 512, false, true>(a, s, st);
    case 2: return launch<2, 512, false, true>(a, s, st);
    case 4: return launch<4, 512, false, true>(a, s, st);
    case 5: return launch<5, 512, false, true>(a, s, st);
    default: return launch<8, 512, false, true>(a, s, st);
  }
}
