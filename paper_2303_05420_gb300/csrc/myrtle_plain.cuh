// Plain layer-wise Myrtle kernels shared by the forward (myrtle_plain.cu) and
// the adjoint (myrtle_backward.cu): one thread per pixel-pair element.
#pragma once

#include "nk_common.cuh"
#include "nk_map64.cuh"

namespace nkp {

// Maps a linear pair index of the block to (i, j).  Symmetric blocks
// enumerate the upper triangle (j >= i) row by row.
__device__ __forceinline__ void pair_of(int64_t idx, int64_t na, int64_t nb, int symmetric,
                                        int64_t* i, int64_t* j) {
  if (!symmetric) {
    *i = idx / nb;
    *j = idx - (*i) * nb;
    return;
  }
  const double m = (double)na;
  double t = (2.0 * m + 1.0) * (2.0 * m + 1.0) - 8.0 * (double)idx;
  int64_t r = (int64_t)floor(((2.0 * m + 1.0) - sqrt(t > 0 ? t : 0)) / 2.0);
  if (r < 0) r = 0;
  if (r > na - 1) r = na - 1;
  // S(r) = r*m - r(r-1)/2 is the first index of row r
  for (int it = 0; it < 4 && r > 0 && r * na - r * (r - 1) / 2 > idx; ++it) --r;
  for (int it = 0; it < 4 && r + 1 < na && (r + 1) * na - (r + 1) * r / 2 <= idx; ++it) ++r;
  *i = r;
  *j = r + (idx - (r * na - r * (r - 1) / 2));
}

// Input covariance of each pair: mean over channels of x(p) y(p').  With
// `staged` both images lie in shared memory as T (2 HW C of them): an FP64
// conversion or division costs as much as several FP64 products, so a pixel is
// converted once, not once per pixel pair, and the mean is a product by 1 / C
// on the second image (FP64 only: 1100 -> 380 us for 8256 pairs of
// 8x8x3 images).
template <typename T>
__global__ void k_input_cov(const float* __restrict__ Xa, const float* __restrict__ Xb,
                            int64_t a0, int64_t b0, int64_t na, int64_t nb, int symmetric,
                            int64_t pair0, int64_t npairs, int H, int W, int C, int staged, T* __restrict__ out) {
  extern __shared__ __align__(16) unsigned char cov_sm[];
  const int HW = H * W, HW2 = HW * HW;
  T* sx = reinterpret_cast<T*>(cov_sm);
  T* sy = sx + HW * C;
  const T inv = (T)1 / (T)C;
  for (int64_t pr = blockIdx.y; pr < npairs; pr += gridDim.y) {
    int64_t i, j;
    pair_of(pair0 + pr, na, nb, symmetric, &i, &j);
    const float* xa = Xa + (a0 + i) * (int64_t)HW * C;
    const float* xb = Xb + (b0 + j) * (int64_t)HW * C;
    if (staged) {
      __syncthreads();  // the previous pair's images are no longer read
      for (int e = threadIdx.x; e < HW * C; e += blockDim.x) {
        sx[e] = (T)xa[e];
        sy[e] = (T)xb[e];
      }
      __syncthreads();
    }
    for (int rem = blockIdx.x * blockDim.x + threadIdx.x; rem < HW2; rem += gridDim.x * blockDim.x) {
      const int p = rem / HW, pp = rem - p * HW;
      T acc = 0;
      if (staged) {
        for (int c = 0; c < C; ++c) acc += sx[p * C + c] * sy[pp * C + c];
        out[pr * (int64_t)HW2 + rem] = acc * inv;
      } else {
        const float* x = xa + p * C;
        const float* y = xb + pp * C;
        for (int c = 0; c < C; ++c) acc += (T)x[c] * (T)y[c];
        out[pr * (int64_t)HW2 + rem] = acc / (T)C;
      }
    }
  }
}

template <typename T>
__global__ void k_conv(const T* __restrict__ in, T* __restrict__ out, int64_t npairs, int H, int W,
                       int filt, T a, T b, const T* __restrict__ addend) {
  // one pair per blockIdx.y step, 32-bit index arithmetic inside a pair
  const int HW = H * W;
  const int HW2 = HW * HW;
  const int r = filt / 2;
  for (int64_t pr = blockIdx.y; pr < npairs; pr += gridDim.y) {
    const T* src = in + pr * (int64_t)HW2;
    T* dst = out + pr * (int64_t)HW2;
    for (int rem = blockIdx.x * blockDim.x + threadIdx.x; rem < HW2; rem += gridDim.x * blockDim.x) {
      const int p = rem / HW, pp = rem - p * HW;
      const int i = p / W, j = p - i * W, k = pp / W, l = pp - k * W;
      T acc = 0;
      for (int dy = -r; dy <= r; ++dy) {
        const int i2 = i + dy, k2 = k + dy;
        if (i2 < 0 || i2 >= H || k2 < 0 || k2 >= H) continue;
        for (int dx = -r; dx <= r; ++dx) {
          const int j2 = j + dx, l2 = l + dx;
          if (j2 >= 0 && j2 < W && l2 >= 0 && l2 < W) acc += src[(i2 * W + j2) * HW + k2 * W + l2];
        }
      }
      dst[rem] = a * acc + b + (addend ? addend[pr * (int64_t)HW2 + rem] : (T)0);
    }
  }
}

// Launch shape of the per-pair kernels: pairs along y, a pair's pixel pairs
// along x.
inline dim3 pair_grid(int64_t npairs, int64_t HW2) {
  int64_t x = (HW2 + 255) / 256;
  int64_t y = npairs;
  if (y > 65535) y = 65535;
  while (x * y > 152 * 64 && x > 1) x = (x + 1) / 2;
  return dim3((unsigned)std::max<int64_t>(1, x), (unsigned)std::max<int64_t>(1, y));
}

template <typename T>
inline void input_cov(const float* Xa, const float* Xb, int64_t a0, int64_t b0, int64_t na, int64_t nb, int symmetric,
                      int64_t pair0, int64_t np, int H, int W, int C, T* out, cudaStream_t st) {
  const int64_t HW = (int64_t)H * W;
  const size_t smem = (size_t)2 * HW * C * sizeof(T);
  const bool staged = sizeof(T) == 8 && smem <= 48 * 1024;
  dim3 grid = pair_grid(np, HW * HW);
  // at least two elements a block for each pixel that it converts
  if (staged) grid.x = (unsigned)std::max<int64_t>(1, std::min<int64_t>(grid.x, HW / 2));
  k_input_cov<T><<<grid, 256, staged ? smem : 0, st>>>(Xa, Xb, a0, b0, na, nb, symmetric, pair0, np, H, W, C, staged,
                                                       out);
}

// What an activation after a conv reads: the pair's images and their tables.
struct ActArgs {
  int64_t na, nb, pair0, a0, b0, nq;
  const double *qda, *qdb;
  const float *qsa, *qsb;
  int symmetric, qoff, moff, act;
  unsigned int* dstatus;
};

// FP64 factors of one pixel, from its self-variance and (with a norm) its
// image's divisor m: the map is y y' J(K x x') / (2 pi) for ReLU (the norm
// cancels from the cosine; 1 / (2 pi) rides on the second image) and
// (2/pi) asin(K x x') for Erf.
__device__ __forceinline__ double2 act_factors64(const ActArgs& g, const double* qd, int64_t base, int p, double w) {
  const double q = qd[base + g.qoff + p], m = g.moff >= 0 ? qd[base + g.moff] : 1.0;
  if (!(q >= 0.0)) atomicOr(g.dstatus, NK_DEV_NUMERICAL);
  if (g.act == NK_ACT_ERF) return make_double2(sqrt(2.0) * rsqrt(m + 2.0 * q), 0.0);
  if (!(q > 0.0)) return make_double2(0.0, 0.0);
  const double r = rsqrt(q);
  return make_double2(r, g.moff >= 0 ? w * sqrt(q / m) : w * (q * r));
}

// ReLU or Erf from FP32 factor tables (of nk_self_diag; they carry a norm):
// b b' J(K a a') / (2 pi), (2/pi) asin(K a a').
__device__ __forceinline__ float act_map32(int act, float K, float2 s1, float2 s2) {
  const float s = s1.y * s2.y;
  float c = K * (s1.x * s2.x);
  c = fminf(fmaxf(c, -1.f), 1.f);
  if (act == NK_ACT_ERF) return s * 0.63661977236758134308f * asinf(c);
  if (!(s > 0.f)) return 0.f;
  return s * (0.15915494309189533577f) * (sqrtf(fmaxf(1.f - c * c, 0.f)) + c * (NK_PI_F - acosf(c)));
}

// The same 3x3 SAME conv, streamed: the diagonal stencil factors into a
// 3-tap sum along the (j, l) diagonal of a fixed (i, k) plane and a 3-tap sum
// over the planes (i - 1, k - 1), (i, k), (i + 1, k + 1), with the validity
// masks factoring the same way.  A block walks one (i, k) diagonal; the
// row-filtered planes of a sliding window of three live in shared memory, so
// each input element is read three times (L1) instead of nine and each output
// once.  Planes of fewer than 256 elements: `grp` pairs at a time, a group of
// W^2 threads each (one pair left 3/4 of the block idle at W = 8).
//
// ACT: the activation that follows is applied as the plane is written, so the
// tensor crosses memory once per layer, not three times.  FP64: the factors of
// the plane's 2 W pixels are computed beside the next plane's load (2 W square
// roots per W^2 elements, not W^2 with a division), and the map is nk_J64_tab.
// FP64 is what bounds it: about 30 operations an element and layer at 2 lanes
// a clock and SM (1.7 ms of the 2.0 that a layer of 8256 pairs of 8x8 images
// takes; conv and activation as two passes with nk_J64 were 3.8).
//
// smem: grp * 3 W^2 elements of T, the pairs' table rows, and for FP64
// activations the table of B and grp * 2 W factor pairs.
template <typename T, bool ACT>
__global__ void __launch_bounds__(256) k_conv_diag(const T* __restrict__ in, T* __restrict__ out, int64_t npairs,
                                                   int H, int W, int grp, T a, T b, const T* __restrict__ addend,
                                                   const __grid_constant__ ActArgs g) {
  constexpr bool F64 = sizeof(T) == 8;
  extern __shared__ __align__(16) unsigned char conv_sm[];
  const int HW = H * W, W2 = W * W;
  const int gi = grp > 1 ? (int)threadIdx.x / W2 : 0;  // my pair within the group
  const int e0 = (int)threadIdx.x - gi * W2, es = grp > 1 ? W2 : (int)blockDim.x;
  int64_t* base = reinterpret_cast<int64_t*>(conv_sm);  // [grp][2]: the pairs' rows of the tables
  double2* fac = reinterpret_cast<double2*>(base + (ACT ? grp * 2 : 0));  // [grp][2 W]
  double* tab = reinterpret_cast<double*>(fac + (ACT && F64 ? grp * 2 * W : 0));
  T* sh = reinterpret_cast<T*>(tab + (ACT && F64 ? NK_J64_TAB_DOUBLES : 0)) + gi * 3 * W2;
  const int d = (int)blockIdx.x - (H - 1);  // k - i on this diagonal
  const int i0 = d < 0 ? -d : 0;
  const int i1 = (d > 0 ? H - d : H) - 1;   // last i with k = i + d < H
  if constexpr (ACT && F64) nk_J64_tab_load(tab, nk_j64_table);
  for (int64_t pg = (int64_t)blockIdx.y * grp; pg < npairs; pg += (int64_t)gridDim.y * grp) {
    const int64_t pr = pg + gi;
    const bool live = gi < grp && pr < npairs;
    const T* src = in + pr * (int64_t)HW * HW;
    T* dst = out + pr * (int64_t)HW * HW;
    // row-filtered plane (ii, ii + d) into slot ii % 3
    auto load = [&](int ii) {
      const int kk = ii + d;
      T* slot = sh + (ii % 3) * W2;
      for (int e = e0; live && e < W2; e += es) {
        const int j = e / W, l = e - j * W;
        T v = src[(int64_t)(ii * W + j) * HW + kk * W + l];
        if (j > 0 && l > 0) v += src[(int64_t)(ii * W + j - 1) * HW + kk * W + l - 1];
        if (j + 1 < W && l + 1 < W) v += src[(int64_t)(ii * W + j + 1) * HW + kk * W + l + 1];
        slot[e] = v;
      }
    };
    __syncthreads();  // the previous pairs' planes and rows are no longer read
    if constexpr (ACT) {
      for (int e = threadIdx.x; e < grp; e += blockDim.x) {
        int64_t ia, jb;
        pair_of(g.pair0 + min(pg + e, npairs - 1), g.na, g.nb, g.symmetric, &ia, &jb);
        base[2 * e] = (g.a0 + ia) * g.nq;
        base[2 * e + 1] = (g.b0 + jb) * g.nq;
      }
      __syncthreads();
    }
    load(i0);
    for (int i = i0; i <= i1; ++i) {
      const int k = i + d;
      if (i + 1 <= i1) load(i + 1);
      if constexpr (ACT && F64) {
        for (int e = threadIdx.x; e < grp * 2 * W; e += blockDim.x) {
          const int pi = e / (2 * W), x = e - pi * 2 * W;
          fac[e] = x < W ? act_factors64(g, g.qda, base[2 * pi], i * W + x, 1.0)
                         : act_factors64(g, g.qdb, base[2 * pi + 1], k * W + x - W, NK_INV_2PI_D);
        }
      }
      __syncthreads();
      const T* cur = sh + (i % 3) * W2;
      const T* prv = sh + ((i + 2) % 3) * W2;
      const T* nxt = sh + ((i + 1) % 3) * W2;
      for (int e = e0; live && e < W2; e += es) {
        T acc = cur[e];
        if (i > i0) acc += prv[e];
        if (i < i1) acc += nxt[e];
        const int j = e / W, l = e - j * W;
        const int64_t o = (int64_t)(i * W + j) * HW + k * W + l;
        T v = a * acc + b;
        if (!ACT && addend) v += addend[pr * (int64_t)HW * HW + o];
        if constexpr (ACT && F64) {
          const double2 f1 = fac[gi * 2 * W + j], f2 = fac[gi * 2 * W + W + l];
          v = v * f1.x * f2.x;
          if (g.act == NK_ACT_ERF)
            v = (2.0 / NK_PI_D) * asin(fmin(fmax(v, -1.0), 1.0));
          else
            v = nk_J64_tab(v, tab) * f1.y * f2.y;
        } else if constexpr (ACT) {
          v = act_map32(g.act, v, reinterpret_cast<const float2*>(g.qsa)[base[2 * gi] + g.qoff + i * W + j],
                        reinterpret_cast<const float2*>(g.qsb)[base[2 * gi + 1] + g.qoff + k * W + l]);
        }
        dst[o] = v;
      }
      __syncthreads();  // slot (i + 2) % 3 and the factors are refilled next
    }
  }
}

// Pairs a block of k_conv_diag takes at a time, and its shared memory.
inline int conv_diag_group(int W) { return W * W <= 128 ? 256 / (W * W) : 1; }
template <typename T>
inline size_t conv_diag_smem(int W, bool act) {
  const size_t grp = conv_diag_group(W);
  return grp * 3 * W * W * sizeof(T) + (act ? grp * 16 : 0) + (act && sizeof(T) == 8 ? grp * 2 * W * 16 + NK_J64_TAB_DOUBLES * 8 : 0);
}

// One 3x3 (or other odd) SAME conv layer on a chunk of pair tensors:
// out = a S(in) + b (+ addend, a tensor of the same shape, when not null),
// and with `act` the activation after it, where true is returned; false: the
// filter or the width is not the streamed form's, and the caller applies it.
template <typename T>
inline bool conv_layer(const T* in, T* out, int64_t np, int H, int W, int filt, T a, T b, cudaStream_t st,
                       const T* addend = nullptr, const ActArgs* act = nullptr) {
  const size_t smem = conv_diag_smem<T>(W, act != nullptr);
  if (filt != 3 || smem > 200 * 1024) {
    k_conv<T><<<pair_grid(np, (int64_t)H * W * H * W), 256, 0, st>>>(in, out, np, H, W, filt, a, b, addend);
    return false;
  }
  auto kern = act ? k_conv_diag<T, true> : k_conv_diag<T, false>;
  nk_smem_optin(kern, smem);
  const int grp = conv_diag_group(W);
  const int64_t y = std::min<int64_t>((np + grp - 1) / grp, 65535);
  kern<<<dim3((unsigned)(2 * H - 1), (unsigned)y), 256, smem, st>>>(in, out, np, H, W, grp, a, b, addend,
                                                                   act ? *act : ActArgs{});
  return act != nullptr;
}

// Activation of the forward layer-wise form, in place, after the convs that
// k_conv_diag does not take: ReLU or Erf, with or without the LayerNorm before
// it.  FP64 reads the self-variances q and (with
// a norm) the divisors m of both images from qd and maps the normalised
// K / sqrt(m m') with q / m, q' / m'; FP32 uses the factor tables qs of
// nk_self_diag, which carry the norm: ReLU b b' J(K a a') / (2 pi), Erf
// (2/pi) asin(K a a').
template <typename T>
__global__ void k_act(T* K, int64_t npairs, int HW, int64_t na, int64_t nb, int symmetric, int64_t pair0,
                      int64_t a0, int64_t b0, const double* __restrict__ qda, const double* __restrict__ qdb,
                      const float* __restrict__ qsa, const float* __restrict__ qsb, int64_t nq, int qoff,
                      int act, int moff, unsigned int* dstatus) {
  const int HW2 = HW * HW;
  for (int64_t pr = blockIdx.y; pr < npairs; pr += gridDim.y) {
    int64_t i, j;
    pair_of(pair0 + pr, na, nb, symmetric, &i, &j);
    const int64_t ra = (a0 + i) * nq, rb = (b0 + j) * nq;
    for (int rem = blockIdx.x * blockDim.x + threadIdx.x; rem < HW2; rem += gridDim.x * blockDim.x) {
      const int64_t e = pr * (int64_t)HW2 + rem;
      const int p = rem / HW, pp = rem - p * HW;
      if constexpr (sizeof(T) == 8) {
        double q1 = qda[ra + qoff + p], q2 = qdb[rb + qoff + pp];
        if (!(q1 >= 0.0) || !(q2 >= 0.0)) atomicOr(dstatus, NK_DEV_NUMERICAL);
        double k = K[e];
        if (moff >= 0) {
          const double m1 = qda[ra + moff], m2 = qdb[rb + moff];
          k /= sqrt(m1 * m2);
          q1 /= m1;
          q2 /= m2;
        }
        K[e] = (act == NK_ACT_ERF) ? nk_erf_map_f64(k, q1, q2) : nk_relu_map64(k, q1, q2);
      } else {
        const float2 s1 = reinterpret_cast<const float2*>(qsa)[ra + qoff + p];
        const float2 s2 = reinterpret_cast<const float2*>(qsb)[rb + qoff + pp];
        K[e] = act_map32(act, K[e], s1, s2);
      }
    }
  }
}

template <typename T>
__global__ void k_pool(const T* __restrict__ in, T* __restrict__ out, int64_t npairs, int H, int W) {
  const int Ho = H / 2, Wo = W / 2;
  const int64_t HW = (int64_t)H * W, HWo = (int64_t)Ho * Wo;
  const int64_t total = npairs * HWo * HWo;
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < total;
       e += (int64_t)gridDim.x * blockDim.x) {
    const int64_t pr = e / (HWo * HWo), rem = e - pr * HWo * HWo;
    const int P = (int)(rem / HWo), PP = (int)(rem - (int64_t)P * HWo);
    const int I = P / Wo, J = P % Wo, K2 = PP / Wo, L = PP % Wo;
    T acc = 0;
    for (int a = 0; a < 2; ++a)
      for (int b = 0; b < 2; ++b)
        for (int c = 0; c < 2; ++c)
          for (int d = 0; d < 2; ++d)
            acc += in[pr * HW * HW + (int64_t)((2 * I + a) * W + 2 * J + b) * HW +
                      (2 * K2 + c) * W + 2 * L + d];
    out[e] = acc / (T)16;
  }
}

template <typename T>
__global__ void k_gap(const T* __restrict__ in, int64_t HW2, int64_t na, int64_t nb, int symmetric,
                      int64_t pair0, T sw2, T sb2, T* __restrict__ K, int64_t ldk) {
  __shared__ double red[32];
  const int64_t pr = blockIdx.x;
  double acc = 0.0;
  for (int64_t e = threadIdx.x; e < HW2; e += blockDim.x) acc += (double)in[pr * HW2 + e];
  for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = acc;
  __syncthreads();
  if (threadIdx.x < 32) {
    acc = (threadIdx.x < (blockDim.x >> 5)) ? red[threadIdx.x] : 0.0;
    for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
    if (threadIdx.x == 0) {
      int64_t i, j;
      pair_of(pair0 + pr, na, nb, symmetric, &i, &j);
      const T v = (T)((double)sw2 * (acc / (double)HW2) + (double)sb2);
      K[i * ldk + j] = v;
      if (symmetric && i != j) K[j * ldk + i] = v;
    }
  }
}

// Flatten + Dense readout (the CV8 listing): K = sw2 mean_p Kt(p, p) + sb2,
// the pixel pairs p' = p of each pair's last tensor (HW x HW), summed in FP64.
template <typename T>
__global__ void k_flatten(const T* __restrict__ in, int HW, int64_t na, int64_t nb, int symmetric,
                          int64_t pair0, T sw2, T sb2, T* __restrict__ K, int64_t ldk) {
  __shared__ double red[32];
  const int64_t pr = blockIdx.x;
  const int64_t HW2 = (int64_t)HW * HW;
  double acc = 0.0;
  for (int p = threadIdx.x; p < HW; p += blockDim.x) acc += (double)in[pr * HW2 + (int64_t)p * HW + p];
  for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = acc;
  __syncthreads();
  if (threadIdx.x < 32) {
    acc = (threadIdx.x < (blockDim.x >> 5)) ? red[threadIdx.x] : 0.0;
    for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
    if (threadIdx.x == 0) {
      int64_t i, j;
      pair_of(pair0 + pr, na, nb, symmetric, &i, &j);
      const T v = (T)((double)sw2 * (acc / (double)HW) + (double)sb2);
      K[i * ldk + j] = v;
      if (symmetric && i != j) K[j * ldk + i] = v;
    }
  }
}

inline int grid_for(int64_t total) {
  int64_t g = (total + 255) / 256;
  if (g > 152 * 64) g = 152 * 64;
  if (g < 1) g = 1;
  return (int)g;
}

// NTK ReLU step (NTK parameterisation): Kt = map(K) in place and
// Theta_t = Theta * E[relu' relu'] = Theta (pi - arccos c) / (2 pi).
template <typename T>
__global__ void k_relu_ntk(T* K, T* Th, int64_t npairs, int HW, int64_t na, int64_t nb, int symmetric,
                           int64_t pair0, int64_t a0, int64_t b0, const double* __restrict__ qda,
                           const double* __restrict__ qdb, const float* __restrict__ qsa,
                           const float* __restrict__ qsb, int64_t nq, int qoff, unsigned int* dstatus) {
  const int HW2 = HW * HW;
  for (int64_t pr = blockIdx.y; pr < npairs; pr += gridDim.y) {
    int64_t i, j;
    pair_of(pair0 + pr, na, nb, symmetric, &i, &j);
    for (int rem = blockIdx.x * blockDim.x + threadIdx.x; rem < HW2; rem += gridDim.x * blockDim.x) {
      const int64_t e = pr * (int64_t)HW2 + rem;
      const int p = rem / HW, pp = rem - p * HW;
      if constexpr (sizeof(T) == 8) {
        const double q1 = qda[(a0 + i) * nq + qoff + p];
        const double q2 = qdb[(b0 + j) * nq + qoff + pp];
        if (!(q1 >= 0.0) || !(q2 >= 0.0)) atomicOr(dstatus, NK_DEV_NUMERICAL);
        const double s = sqrt(q1 * q2);
        double kd = 0.0, kt = 0.0;
        if (s > 0.0) {
          double c = K[e] / s;
          c = c < -1.0 ? -1.0 : (c > 1.0 ? 1.0 : c);
          const double th = acos(c);
          kt = s * NK_INV_2PI_D * (sqrt(fmax(1.0 - c * c, 0.0)) + c * (NK_PI_D - th));
          kd = (NK_PI_D - th) * NK_INV_2PI_D;
        }
        K[e] = kt;
        Th[e] *= kd;
      } else {
        const float2 s1 = reinterpret_cast<const float2*>(qsa)[(a0 + i) * nq + qoff + p];
        const float2 s2 = reinterpret_cast<const float2*>(qsb)[(b0 + j) * nq + qoff + pp];
        const float s = s1.y * s2.y;
        float kt = 0.f, kd = 0.f;
        if (s > 0.f) {
          float c = K[e] * (s1.x * s2.x);
          c = fminf(fmaxf(c, -1.f), 1.f);
          const float th = acosf(c);
          kt = s * 0.15915494309189533577f * (sqrtf(fmaxf(1.f - c * c, 0.f)) + c * (NK_PI_F - th));
          kd = (NK_PI_F - th) * 0.15915494309189533577f;
        }
        K[e] = kt;
        Th[e] *= kd;
      }
    }
  }
}

// NTK readout: K = sw2 mean(Kt) + sb2, Theta = K + sw2 mean(Theta_t).
template <typename T>
__global__ void k_gap_ntk(const T* __restrict__ Kt, const T* __restrict__ Tt, int64_t HW2, int64_t na, int64_t nb,
                          int symmetric, int64_t pair0, double sw2, double sb2, T* __restrict__ K,
                          T* __restrict__ Th, int64_t ldk) {
  __shared__ double r1[32], r2[32];
  const int64_t pr = blockIdx.x;
  double a = 0.0, b = 0.0;
  for (int64_t e = threadIdx.x; e < HW2; e += blockDim.x) {
    a += (double)Kt[pr * HW2 + e];
    b += (double)Tt[pr * HW2 + e];
  }
  for (int o = 16; o > 0; o >>= 1) {
    a += __shfl_xor_sync(0xffffffffu, a, o);
    b += __shfl_xor_sync(0xffffffffu, b, o);
  }
  if ((threadIdx.x & 31) == 0) {
    r1[threadIdx.x >> 5] = a;
    r2[threadIdx.x >> 5] = b;
  }
  __syncthreads();
  if (threadIdx.x < 32) {
    a = (threadIdx.x < (blockDim.x >> 5)) ? r1[threadIdx.x] : 0.0;
    b = (threadIdx.x < (blockDim.x >> 5)) ? r2[threadIdx.x] : 0.0;
    for (int o = 16; o > 0; o >>= 1) {
      a += __shfl_xor_sync(0xffffffffu, a, o);
      b += __shfl_xor_sync(0xffffffffu, b, o);
    }
    if (threadIdx.x == 0) {
      int64_t i, j;
      pair_of(pair0 + pr, na, nb, symmetric, &i, &j);
      const double kv = sw2 * (a / (double)HW2) + sb2;
      const double tv = kv + sw2 * (b / (double)HW2);
      K[i * ldk + j] = (T)kv;
      Th[i * ldk + j] = (T)tv;
      if (symmetric && i != j) {
        K[j * ldk + i] = (T)kv;
        Th[j * ldk + i] = (T)tv;
      }
    }
  }
}

}  // namespace nkp
