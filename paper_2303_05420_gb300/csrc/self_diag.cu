// nk_self_diag: per-pixel self-variances q_l(p) = K_l(p, p; x, x) in FP64, by
// the banded self recursion of self_planes.cuh.
//
// Activations: ReLU (arc-cosine map) or Erf, E[erf(u) erf(v)] =
// (2/pi) asin(2 K / sqrt((1 + 2 q)(1 + 2 q'))).  With a LayerNorm between
// conv and activation (the tuned Myrtle listing), the layer's band is divided
// by m = mean_p q(p) of this image before the activation, which then sees
// the self-variances q / m (the infinite-width limit of normalising over
// pixels and channels); m is written after the layer's q values.
//
// What bounds it: the FP64 pipe (two lanes an SM and cycle) for many images,
// launches and one CTA's share of it for a few.  One CTA used to carry all
// planes of an image through all layers, both halves of them and with acos,
// two square roots and a division a map: 0.53 ms for one 32x32 image of
// Myrtle-5 and 4.0 ms for ten of Myrtle-10.  Now a first image against 200
// held ones (self-variances and block) takes 0.477 ms where it took 0.963.
#include "self_planes.cuh"

#include <algorithm>

namespace {

// The D = 0 planes of stage s: q of each layer, its factor tables, and the
// stage's output plane 0; rows of band blockIdx.y of image blockIdx.x.  A whole
// 32x32 plane keeps one SM's FP64 pipe busy for 15 us a stage, so few images
// are cut into row bands with halos, like the other planes (a norm needs the
// whole plane's mean: one band), and the divisions that are none (by C, by
// m = 1) are left out: they were half of the operations.
template <bool STORE>
__global__ void __launch_bounds__(512)
k_self_center(SelfGeom G, int s, int bands, double sw2, double sb2, const float* __restrict__ X, SelfBufs Bf,
              double* __restrict__ qd, float* __restrict__ qs, unsigned int* dstatus) {
  extern __shared__ double sh[];
  const NkGeom& g = G.g;
  const int H = g.Hs[s], W = g.Ws[s], HW = H * W, C = g.C, fr = g.filter / 2;
  const int tid = threadIdx.x, bd = blockDim.x;
  const int64_t img = blockIdx.x;
  const NkBand o = nk_band(H, bands, blockIdx.y, fr * g.convs[s]);
  const int rows = o.hi - o.lo, ne = rows * W, p0 = o.lo * W;  // element e is pixel p0 + e
  double* A = sh;
  double* B = sh + ne;
  double* red = B + ne;  // [33]: warp sums, then m
  const double a_conv = sw2 / (double)(g.filter * g.filter), invC = 1.0 / (double)C;
  if (s == 0) {
    const float* x = X + img * (int64_t)HW * C;
    for (int e = tid; e < ne; e += bd) {
      double v = 0.0;
      for (int c = 0; c < C; ++c) {
        const double u = (double)x[(p0 + e) * C + c];
        v += u * u;
      }
      A[e] = v * invC;
    }
  } else {
    const double* Tp = Bf.T[(s - 1) & 1] + img * G.tmax;
    for (int e = tid; e < ne; e += bd) A[e] = nk_pooled_at(g, s, Tp, 0, 0, o.lo + e / W, e % W);
  }
  for (int k = 0; k < g.convs[s]; ++k) {
    const int layer = G.layer0[s] + k, off = g.layer_qoff[layer];
    __syncthreads();
    nk_rows3(A, B, rows, W, fr);
    __syncthreads();
    for (int e = tid; e < ne; e += bd) A[e] = a_conv * nk_cols3(B, e, e / W, rows, W, fr) + sb2;
    // LayerNorm divisor m = mean_p q(p) (1 without a norm)
    double m = 1.0;
    if (g.norm == NK_NORM_LAYER) {
      double t = 0.0;
      for (int e = tid; e < ne; e += bd) t += A[e];
      for (int x = 16; x > 0; x >>= 1) t += __shfl_xor_sync(0xffffffffu, t, x);
      if ((tid & 31) == 0) red[tid >> 5] = t;
      __syncthreads();
      if (tid == 0) {
        t = 0.0;
        for (int w = 0; w < (bd >> 5); ++w) t += red[w];
        t /= (double)HW;
        if (qd) qd[img * (int64_t)g.nq + g.nq_base + layer] = t;
        if (qs) reinterpret_cast<float2*>(qs)[img * (int64_t)g.nq + g.nq_base + layer] = make_float2(0.f, 0.f);
        if (!(t > 0.0)) {
          atomicOr(dstatus, NK_DEV_NUMERICAL);
          t = 1.0;  // results are flagged; keep them finite
        }
        red[32] = t;
      }
      __syncthreads();
      m = red[32];
    }
    for (int e = tid; e < ne; e += bd) {
      const int p = p0 + e;
      const bool mine = p >= o.i0 * W && p < o.i1 * W;
      const double q = A[e], qm = m == 1.0 ? q : q / m;
      double t = q;  // post-activation
      if (g.act == NK_ACT_ERF)
        t = nk_erf_map_f64(qm, qm, qm);
      else if (g.act == NK_ACT_RELU)
        t = q > 0.0 ? 0.5 * qm : 0.0;
      A[e] = t;
      if (!mine) continue;
      if (qd) qd[img * (int64_t)g.nq + off + p] = q;
      if (!(q >= 0.0)) atomicOr(dstatus, NK_DEV_NUMERICAL);
      if constexpr (STORE) Bf.store[img * G.store_total + G.store_off[layer] + p] = q;
      double2 ab = make_double2(0.0, 0.0);
      if (g.act == NK_ACT_ERF) {
        ab = make_double2(sqrt(2.0 / (m + 2.0 * q)), 1.0);
      } else if (q > 0.0) {
        ab.x = rsqrt(q);
        ab.y = m == 1.0 ? q * ab.x : sqrt(qm);
      }
      Bf.tab[img * (int64_t)g.nq_base + off + p] = ab;
      if (qs) reinterpret_cast<float2*>(qs)[img * (int64_t)g.nq + off + p] = make_float2((float)ab.x, (float)ab.y);
    }
  }
  if (s < g.last_act_stage) {
    double* T = Bf.T[s & 1] + img * G.tmax;
    __syncthreads();
    for (int e = tid + (o.i0 - o.lo) * W; e < (o.i1 - o.lo) * W; e += bd) T[p0 + e] = A[e];
  }
}

// Plane h = blockIdx.y + 1 of stage s, rows of band blockIdx.x, of image
// blockIdx.z: all layers of the stage in shared memory.  Rows next to a cut
// are wrong by one row more with each layer; the halo (a row a layer) keeps
// them out of the band's own.
template <bool STORE>
__global__ void __launch_bounds__(256)
k_self_planes(SelfGeom G, int s, int bands, double sw2, double sb2, const float* __restrict__ X, SelfBufs Bf) {
  extern __shared__ double sh[];
  __shared__ double jtab[NK_J64_TAB_DOUBLES];
  const NkGeom& g = G.g;
  const int H = g.Hs[s], W = g.Ws[s], HW = H * W, C = g.C, fr = g.filter / 2, r = g.radius[s];
  const int tid = threadIdx.x, bd = blockDim.x;
  const int h = blockIdx.y + 1;
  const int64_t img = blockIdx.z;
  int dy, dx;
  nk_plane_offset(h, r, &dy, &dx);
  const NkBand o = nk_band(H, bands, blockIdx.x, fr * g.convs[s]);
  const int rows = o.hi - o.lo, ne = rows * W;
  double* A = sh;
  double* B = sh + ne;
  nk_J64_tab_load(jtab, nk_j64_table);
  const double a_conv = sw2 / (double)(g.filter * g.filter), invC = 1.0 / (double)C;
  // K_0(p, p + D) = (1/C) sum_c x[p, c] x[p + D, c], or the pooled planes
  for (int e = tid; e < ne; e += bd) {
    const int i = o.lo + e / W, j = e % W;
    double v = 0.0;
    if (i + dy >= 0 && i + dy < H && j + dx >= 0 && j + dx < W) {
      if (s == 0) {
        const float* u = X + (img * (int64_t)HW + i * W + j) * C;
        const float* w = u + (dy * W + dx) * C;
        for (int c = 0; c < C; ++c) v += (double)u[c] * (double)w[c];
        v *= invC;
      } else {
        v = nk_pooled_at(g, s, Bf.T[(s - 1) & 1] + img * G.tmax, dy, dx, i, j);
      }
    }
    A[e] = v;
  }
  for (int k = 0; k < g.convs[s]; ++k) {
    const int layer = G.layer0[s] + k;
    const double2* tab = Bf.tab + img * (int64_t)g.nq_base + g.layer_qoff[layer];
    // with a norm the map's factors carry it, the identity does not occur there
    __syncthreads();
    nk_rows3(A, B, rows, W, fr);
    __syncthreads();
    for (int e = tid; e < ne; e += bd) {
      const int er = e / W, i = o.lo + er, j = e % W, p = i * W + j;
      // entries whose p + D leaves the image stay zero
      if (i + dy < 0 || i + dy >= H || j + dx < 0 || j + dx >= W) continue;
      double v = a_conv * nk_cols3(B, e, er, rows, W, fr) + sb2;
      if constexpr (STORE) {
        if (i >= o.i0 && i < o.i1)
          Bf.store[img * G.store_total + G.store_off[layer] + (int64_t)h * HW + p] = v;
      }
      const double2 f = tab[p], f2 = tab[p + dy * W + dx];
      if (g.act == NK_ACT_RELU)
        v = nk_J64_tab(v * f.x * f2.x, jtab) * (f.y * NK_INV_2PI_D) * f2.y;
      else if (g.act == NK_ACT_ERF)
        v = (2.0 / NK_PI_D) * asin(fmin(fmax(v * (f.x * f2.x), -1.0), 1.0));
      A[e] = v;
    }
  }
  __syncthreads();
  double* T = Bf.T[s & 1] + img * G.tmax + (int64_t)h * HW;
  for (int e = tid; e < (o.i1 - o.i0) * W; e += bd) T[o.i0 * W + e] = A[(o.i0 - o.lo) * W + e];
}

}  // namespace

size_t nk_self_buf_bytes(const SelfGeom& G, int64_t m, bool store) {
  return (size_t)m * ((2 * G.tmax + 2 * G.g.nq_base + (store ? G.store_total : 0)) * sizeof(double)) + 1024;
}

SelfBufs nk_self_carve(const SelfGeom& G, int64_t m, bool store, void* ws) {
  SelfBufs B = {};
  char* w = reinterpret_cast<char*>(ws);
  auto take = [&](size_t n) {
    char* p = w;
    w += (n + 255) / 256 * 256;
    return p;
  };
  B.tab = reinterpret_cast<double2*>(take((size_t)m * G.g.nq_base * sizeof(double2)));
  B.T[0] = reinterpret_cast<double*>(take((size_t)m * G.tmax * sizeof(double)));
  B.T[1] = reinterpret_cast<double*>(take((size_t)m * G.tmax * sizeof(double)));
  B.store = store ? reinterpret_cast<double*>(w) : nullptr;
  return B;
}

int nk_self_bands(int H, int W, int64_t planes, int halo, int arrays, int sm) {
  int bands = 1;
  while (2 * bands * 8 <= H && planes * bands < 2 * sm) bands *= 2;
  // shared memory: more bands if a band's arrays do not fit
  auto bytes = [&](int b) {
    return (size_t)arrays * std::min(H, (H + b - 1) / b + 2 * halo) * W * sizeof(double);
  };
  while (bytes(bands) > 220 * 1024 && bands < H) ++bands;
  return bands;
}

cudaError_t nk_self_forward(const SelfGeom& G, double sw2, double sb2, const float* X, int64_t m, double* qd,
                            float* qs, const SelfBufs& B, int sm, unsigned int* dstatus, cudaStream_t st,
                            int64_t* launches) {
  const NkGeom& g = G.g;
  const bool store = B.store != nullptr;
  for (int s = 0; s <= g.last_act_stage; ++s) {
    const int halo = g.filter / 2 * g.convs[s];
    const int cb = g.norm == NK_NORM_LAYER ? 1 : nk_self_bands(g.Hs[s], g.Ws[s], m, halo, 2, sm);
    const int crows = cb == 1 ? g.Hs[s] : std::min(g.Hs[s], (g.Hs[s] + cb - 1) / cb + 2 * halo);
    const size_t csm = (2 * (size_t)crows * g.Ws[s] + 33) * sizeof(double);
    auto kc = store ? k_self_center<true> : k_self_center<false>;
    cudaError_t e = nk_smem_optin(kc, csm);
    if (e != cudaSuccess) return e;
    ++*launches;
    kc<<<dim3((unsigned)m, (unsigned)cb), 512, csm, st>>>(G, s, cb, sw2, sb2, X, B, qd, qs, dstatus);
    if (G.nh[s] > 1) {
      const int bands = nk_self_bands(g.Hs[s], g.Ws[s], m * (G.nh[s] - 1), halo, 2, sm);
      const int rows = std::min(g.Hs[s], (g.Hs[s] + bands - 1) / bands + 2 * halo);
      const size_t psm = 2 * (size_t)rows * g.Ws[s] * sizeof(double);
      auto kp = store ? k_self_planes<true> : k_self_planes<false>;
      e = nk_smem_optin(kp, psm);
      if (e != cudaSuccess) return e;
      ++*launches;
      kp<<<dim3((unsigned)bands, (unsigned)(G.nh[s] - 1), (unsigned)m), 256, psm, st>>>(G, s, bands, sw2, sb2, X, B);
    }
    e = cudaGetLastError();
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

// Images a pass: the buffers within 128 MB (at least 64 images, grid.z at most).
static int64_t self_chunk(const SelfGeom& G, int64_t n) {
  const int64_t per = (int64_t)nk_self_buf_bytes(G, 1, false);
  return std::min<int64_t>(std::min<int64_t>(n, 32768), std::max<int64_t>(64, ((int64_t)128 << 20) / per));
}

size_t nk_self_diag_ws_bytes(const NkGeom& g, int64_t n) {
  const SelfGeom G = nk_self_geom(g);
  return nk_self_buf_bytes(G, self_chunk(G, n), false);
}

cudaError_t nk_launch_self_diag(const NkGeom& g, double sw2, double sb2, const float* X, int64_t n, double* qd,
                                float* qs, void* ws, int sm, unsigned int* dstatus, cudaStream_t st,
                                int64_t* launches) {
  if (n <= 0 || g.last_act_stage < 0) return cudaSuccess;
  const SelfGeom G = nk_self_geom(g);
  const int64_t chunk = self_chunk(G, n);
  const SelfBufs B = nk_self_carve(G, chunk, false, ws);
  for (int64_t i = 0; i < n; i += chunk) {
    const int64_t m = std::min(chunk, n - i);
    const cudaError_t e = nk_self_forward(G, sw2, sb2, X + i * (int64_t)g.Hs[0] * g.Ws[0] * g.C, m,
                                          qd + i * (int64_t)g.nq, qs ? qs + 2 * i * (int64_t)g.nq : nullptr, B, sm,
                                          dstatus, st, launches);
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}
