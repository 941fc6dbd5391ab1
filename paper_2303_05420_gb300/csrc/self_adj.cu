// Adjoint of the banded self recursion (self_planes.cuh) that produces
// q_l(p), FP64: given dq_l(p) of every activation layer, accumulates dX and
// the sigma sums.  ReLU networks without a norm.
//
// The forward planes are recomputed with every layer's pre-activation kept.
// Reverse, stage by stage from the last: the carried planes D != 0 run back
// through the stage's layers on their own (map adjoint, conv adjoint), each
// writing per layer what its maps owe to q(p); then the D = 0 plane, whose
// gradient at each layer takes those sums and the external dq.  The D = 0
// plane's own map is q / 2.  A carried plane stands for both halves, so its
// q-terms, sigma sums and input gradients count twice.  The previous stage
// gathers the pool adjoint as it loads.
//
// One CTA used to carry an image through all of this with two FP64 atomic
// adds per map: 9.1 ms for ten 32x32 images of Myrtle-10 as for a hundred and
// fifty.  With the forward's, gradients of a Myrtle-10 block of 10 support
// images against 30 targets went from 36.7 to 12.1 ms.  Bounded by the FP64 pipe (two lanes an SM and cycle) or, for a few
// images, by eleven dependent launches.
#include "self_planes.cuh"

#include <algorithm>

namespace {

struct AdjBufs {
  double* G[2];  // [m][tmax]: gradient of a stage's input planes, by stage parity
  double* hq;    // [m][store_total]: a layer's q-terms per plane h and pixel (plane 0 unused)
};

// Pool adjoint: the gradient of the post-activation (u, u + D) of stage s - 1
// is stage s's input gradient at the one pooled pair that holds it, / 16.
__device__ __forceinline__ double unpooled_at(const NkGeom& g, int s, const double* Gs, int dy, int dx, int ui,
                                              int uj) {
  const int H = g.Hs[s], W = g.Ws[s], r = g.radius[s];
  const int ay = ui & 1, ax = uj & 1, I = ui >> 1, J = uj >> 1;
  const int by = (dy + ay) & 1, bx = (dx + ax) & 1;
  const int ey = (dy + ay - by) / 2, ex = (dx + ax - bx) / 2;
  if (ey < -r || ey > r || ex < -r || ex > r || I + ey < 0 || I + ey >= H || J + ex < 0 || J + ex >= W) return 0.0;
  return nk_plane_at(Gs, H * W, W, r, ey, ex, I * W + J) * (1.0 / 16.0);
}

// Block sums of the sigma terms, added to the outputs.
__device__ __forceinline__ void add_sigma(double lsw, double lsb, double sw2, double* dsw2, double* dsb2,
                                          double* red) {
  for (int o = 16; o > 0; o >>= 1) {
    lsw += __shfl_xor_sync(0xffffffffu, lsw, o);
    lsb += __shfl_xor_sync(0xffffffffu, lsb, o);
  }
  const int w = threadIdx.x >> 5, nw = blockDim.x >> 5;
  if ((threadIdx.x & 31) == 0) {
    red[w] = lsw;
    red[nw + w] = lsb;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    double a = 0.0, b = 0.0;
    for (int i = 0; i < nw; ++i) {
      a += red[i];
      b += red[nw + i];
    }
    atomicAdd(dsw2, a / sw2);
    atomicAdd(dsb2, b);
  }
}

// Plane h = blockIdx.y + 1 of stage s (s before the last, whose only plane is
// D = 0), band blockIdx.x, image blockIdx.z.  The halo is a row a layer, and
// |dy| more for the q-terms of the partner pixels.
__global__ void __launch_bounds__(256)
k_self_adj_planes(SelfGeom G, int s, int bands, double sw2, double sb2, SelfBufs Bf, AdjBufs Ab,
                  double* __restrict__ dsw2, double* __restrict__ dsb2) {
  extern __shared__ double sh[];
  __shared__ double red[16];
  __shared__ double djtab[NK_J64_TAB_DOUBLES];
  const NkGeom& g = G.g;
  const int H = g.Hs[s], W = g.Ws[s], HW = H * W, fr = g.filter / 2, r = g.radius[s];
  const int tid = threadIdx.x, bd = blockDim.x;
  const int h = blockIdx.y + 1;
  const int64_t img = blockIdx.z;
  int dy, dx;
  nk_plane_offset(h, r, &dy, &dx);
  const NkBand o = nk_band(H, bands, blockIdx.x, fr * g.convs[s] + r);
  const int rows = o.hi - o.lo, ne = rows * W, dD = dy * W + dx;
  double* Dg = sh;        // gradient of the layer's post-activation
  double* E = sh + ne;    // of its pre-activation
  double* Q = E + ne;     // its q-terms
  const double a_conv = sw2 / (double)(g.filter * g.filter);
  const double* Gn = Ab.G[(s + 1) & 1] + img * G.tmax;
  double lsw = 0.0, lsb = 0.0;
  nk_J64_tab_load(djtab, nk_dj64_table);
  for (int e = tid; e < ne; e += bd) {
    const int i = o.lo + e / W, j = e % W;
    const bool in = i + dy >= 0 && i + dy < H && j + dx >= 0 && j + dx < W;
    Dg[e] = in ? unpooled_at(g, s + 1, Gn, dy, dx, i, j) : 0.0;
  }
  for (int k = g.convs[s] - 1; k >= 0; --k) {
    const int layer = G.layer0[s] + k;
    const double* Kst = Bf.store + img * G.store_total + G.store_off[layer] + (int64_t)h * HW;
    double* hq = Ab.hq + img * G.store_total + G.store_off[layer] + (int64_t)h * HW;
    const double2* tab = Bf.tab + img * (int64_t)g.nq_base + g.layer_qoff[layer];
    __syncthreads();
    for (int e = tid; e < ne; e += bd) {
      const int i = o.lo + e / W, j = e % W, p = i * W + j;
      double ev = 0.0, qv = 0.0;
      if (i + dy >= 0 && i + dy < H && j + dx >= 0 && j + dx < W) {
        const double2 f = tab[p], f2 = tab[p + dD];
        const double aa = f.x * f2.x, bb = f.y * f2.y, K = Kst[p], gk = Dg[e] * NK_INV_2PI_D;
        if (bb > 0.0) {
          // e = g J' / (2 pi); the map's q-derivative is (Kt - K J' / (2 pi))
          // / (2 q), and sqrt(q q') J - K J' = sqrt(q q') sqrt(1 - c^2)
          double dJ, sn;
          nk_dJ64_tab(K * aa, djtab, &dJ, &sn);
          ev = gk * dJ;
          qv = gk * (bb * sn);
        }
        if (i >= o.i0 && i < o.i1) {
          lsw += ev * (K - sb2);
          lsb += ev;
        }
      }
      E[e] = ev;
      Q[e] = qv;
    }
    __syncthreads();
    // q-terms of pixel p as the first pixel of (p, p + D) and as the second of
    // (p - D, p); both halves of the pair of planes: twice h / (2 q)
    for (int e = tid; e < (o.i1 - o.i0) * W; e += bd) {
      const int i = o.i0 + e / W, j = e % W, p = i * W + j, x = (i - o.lo) * W + j;
      double v = Q[x];
      if (i - dy >= 0 && i - dy < H && j - dx >= 0 && j - dx < W) v += Q[x - dD];
      const double a = tab[p].x;
      hq[p] = v * (a * a);  // 1 / q, 0 where q = 0
    }
    nk_rows3(E, Dg, rows, W, fr);
    __syncthreads();
    for (int e = tid; e < ne; e += bd) {
      const int er = e / W, i = o.lo + er, j = e % W;
      const bool in = i + dy >= 0 && i + dy < H && j + dx >= 0 && j + dx < W;
      E[e] = in ? a_conv * nk_cols3(Dg, e, er, rows, W, fr) : 0.0;
    }
    double* t = Dg;
    Dg = E;
    E = t;
  }
  __syncthreads();
  double* Go = Ab.G[s & 1] + img * G.tmax + (int64_t)h * HW;
  for (int e = tid; e < (o.i1 - o.i0) * W; e += bd) Go[o.i0 * W + e] = Dg[(o.i0 - o.lo) * W + e];
  add_sigma(2.0 * lsw, 2.0 * lsb, sw2, dsw2, dsb2, red);
}

// The D = 0 plane of stage s, rows of band blockIdx.y of image blockIdx.x (a
// pixel's q-terms are 24 loads and FP64 sums a layer).
template <typename T>
__global__ void __launch_bounds__(512)
k_self_adj_center(SelfGeom G, int s, int bands, double sw2, double sb2, SelfBufs Bf, AdjBufs Ab,
                  const T* __restrict__ dq, double* __restrict__ dsw2, double* __restrict__ dsb2) {
  extern __shared__ double sh[];
  __shared__ double red[32];
  const NkGeom& g = G.g;
  const int H = g.Hs[s], W = g.Ws[s], HW = H * W, fr = g.filter / 2;
  const int tid = threadIdx.x, bd = blockDim.x;
  const int64_t img = blockIdx.x;
  const NkBand o = nk_band(H, bands, blockIdx.y, fr * g.convs[s]);
  const int rows = o.hi - o.lo, ne = rows * W, p0 = o.lo * W;  // element x is pixel p0 + x
  double* E = sh;
  double* B = sh + ne;
  const double a_conv = sw2 / (double)(g.filter * g.filter);
  double lsw = 0.0, lsb = 0.0;
  for (int x = tid; x < ne; x += bd)
    E[x] = s < g.last_act_stage
               ? unpooled_at(g, s + 1, Ab.G[(s + 1) & 1] + img * G.tmax, 0, 0, o.lo + x / W, x % W)
               : 0.0;
  for (int k = g.convs[s] - 1; k >= 0; --k) {
    const int layer = G.layer0[s] + k, off = g.layer_qoff[layer];
    const double* q = Bf.store + img * G.store_total + G.store_off[layer];
    const double* hq = Ab.hq + img * G.store_total + G.store_off[layer];
    __syncthreads();
    for (int x = tid; x < ne; x += bd) {
      const int p = p0 + x;
      double e = q[p] > 0.0 ? 0.5 * E[x] : 0.0;
#pragma unroll 8
      for (int h = 1; h < G.nh[s]; ++h) e += hq[(int64_t)h * HW + p];
      e += (double)dq[img * (int64_t)g.nq + off + p];
      if (p >= o.i0 * W && p < o.i1 * W) {
        lsw += e * (q[p] - sb2);
        lsb += e;
      }
      E[x] = e;
    }
    __syncthreads();
    nk_rows3(E, B, rows, W, fr);
    __syncthreads();
    for (int x = tid; x < ne; x += bd) E[x] = a_conv * nk_cols3(B, x, x / W, rows, W, fr);
  }
  __syncthreads();
  double* Go = Ab.G[s & 1] + img * G.tmax;
  for (int x = tid + (o.i0 - o.lo) * W; x < (o.i1 - o.lo) * W; x += bd) Go[p0 + x] = E[x];
  add_sigma(lsw, lsb, sw2, dsw2, dsb2, red);
}

// dX += the input covariances' adjoint: K_0(p, p + D) = (1/C) x[p] . x[p + D]
// over all planes, gathered per pixel.
template <typename T>
__global__ void __launch_bounds__(256)
k_self_adj_input(SelfGeom G, const float* __restrict__ X, int64_t m, AdjBufs Ab, T* __restrict__ dX) {
  const NkGeom& g = G.g;
  const int H = g.Hs[0], W = g.Ws[0], HW = H * W, C = g.C, r = g.radius[0];
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < m * HW; e += (int64_t)gridDim.x * blockDim.x) {
    const int64_t img = e / HW;
    const int p = (int)(e - img * HW), i = p / W, j = p % W;
    const double* Gs = Ab.G[0] + img * G.tmax;
    const float* x = X + img * (int64_t)HW * C;
    for (int c0 = 0; c0 < C; c0 += 4) {
      double acc[4] = {0.0, 0.0, 0.0, 0.0};
      for (int h = 0; h < G.nh[0]; ++h) {
        int dy, dx;
        nk_plane_offset(h, r, &dy, &dx);
        const int d = dy * W + dx;
        const bool fw = i + dy >= 0 && i + dy < H && j + dx >= 0 && j + dx < W;
        const bool bw = h > 0 && i - dy >= 0 && i - dy < H && j - dx >= 0 && j - dx < W;
        const double gf = fw ? Gs[(int64_t)h * HW + p] : 0.0, gb = bw ? Gs[(int64_t)h * HW + p - d] : 0.0;
        for (int c = 0; c < 4 && c0 + c < C; ++c) {
          if (fw) acc[c] += gf * (double)x[(int64_t)(p + d) * C + c0 + c];
          if (bw) acc[c] += gb * (double)x[(int64_t)(p - d) * C + c0 + c];
        }
      }
      for (int c = 0; c < 4 && c0 + c < C; ++c) {
        T* o = dX + (img * (int64_t)HW + p) * C + c0 + c;
        *o = (T)((double)*o + acc[c] * (2.0 / (double)C));
      }
    }
  }
}

// Images a pass: the buffers within 512 MB, at least 16.
int64_t adj_chunk(const SelfGeom& G, int64_t n) {
  const int64_t per = (int64_t)nk_self_buf_bytes(G, 1, true) + (2 * G.tmax + G.store_total) * (int64_t)sizeof(double);
  return std::min<int64_t>(std::min<int64_t>(n, 32768), std::max<int64_t>(16, ((int64_t)512 << 20) / per));
}

}  // namespace

size_t nk_self_adj_ws_bytes(const NkGeom& g, int64_t n) {
  const SelfGeom G = nk_self_geom(g);
  const int64_t m = adj_chunk(G, n);
  return nk_self_buf_bytes(G, m, true) + (size_t)m * (2 * G.tmax + G.store_total) * sizeof(double) + 4 * 256;
}

template <typename T>
cudaError_t nk_launch_self_adj(const NkGeom& g, double sw2, double sb2, const float* X, int64_t n, const T* dq,
                               T* dX, double* dsw2, double* dsb2, void* ws, int sm, unsigned int* dstatus,
                               cudaStream_t st, int64_t* launches) {
  if (n <= 0 || g.last_act_stage < 0) return cudaSuccess;
  const SelfGeom G = nk_self_geom(g);
  const int64_t chunk = adj_chunk(G, n);
  const SelfBufs B = nk_self_carve(G, chunk, true, ws);
  char* w = reinterpret_cast<char*>(ws) + (nk_self_buf_bytes(G, chunk, true) + 255) / 256 * 256;
  AdjBufs A;
  for (int i = 0; i < 2; ++i) {
    A.G[i] = reinterpret_cast<double*>(w);
    w += ((size_t)chunk * G.tmax * sizeof(double) + 255) / 256 * 256;
  }
  A.hq = reinterpret_cast<double*>(w);
  const int64_t px = (int64_t)g.Hs[0] * g.Ws[0] * g.C;
  for (int64_t i = 0; i < n; i += chunk) {
    const int64_t m = std::min(chunk, n - i);
    cudaError_t e = nk_self_forward(G, sw2, sb2, X + i * px, m, nullptr, nullptr, B, sm, dstatus, st, launches);
    if (e != cudaSuccess) return e;
    for (int s = g.last_act_stage; s >= 0; --s) {
      const int H = g.Hs[s], W = g.Ws[s];
      if (G.nh[s] > 1) {
        const int halo = g.filter / 2 * g.convs[s] + g.radius[s];
        const int bands = nk_self_bands(H, W, m * (G.nh[s] - 1), halo, 3, sm);
        const size_t psm = 3 * (size_t)std::min(H, (H + bands - 1) / bands + 2 * halo) * W * sizeof(double);
        e = nk_smem_optin(k_self_adj_planes, psm);
        if (e != cudaSuccess) return e;
        ++*launches;
        k_self_adj_planes<<<dim3((unsigned)bands, (unsigned)(G.nh[s] - 1), (unsigned)m), 256, psm, st>>>(
            G, s, bands, sw2, sb2, B, A, dsw2, dsb2);
      }
      const int chalo = g.filter / 2 * g.convs[s], cb = nk_self_bands(H, W, m, chalo, 2, sm);
      const size_t csm = 2 * (size_t)(cb == 1 ? H : std::min(H, (H + cb - 1) / cb + 2 * chalo)) * W * sizeof(double);
      e = nk_smem_optin(k_self_adj_center<T>, csm);
      if (e != cudaSuccess) return e;
      ++*launches;
      k_self_adj_center<T><<<dim3((unsigned)m, (unsigned)cb), 512, csm, st>>>(G, s, cb, sw2, sb2, B, A,
                                                                             dq + i * (int64_t)g.nq, dsw2, dsb2);
    }
    if (dX) {
      ++*launches;
      const int64_t blocks = (m * g.Hs[0] * g.Ws[0] + 255) / 256;
      k_self_adj_input<T><<<(unsigned)std::min<int64_t>(blocks, 16 * (int64_t)sm), 256, 0, st>>>(G, X + i * px, m, A,
                                                                                                dX + i * px);
    }
    e = cudaGetLastError();
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

template cudaError_t nk_launch_self_adj<float>(const NkGeom&, double, double, const float*, int64_t, const float*,
                                               float*, double*, double*, void*, int, unsigned int*, cudaStream_t,
                                               int64_t*);
template cudaError_t nk_launch_self_adj<double>(const NkGeom&, double, double, const float*, int64_t, const double*,
                                                double*, double*, double*, void*, int, unsigned int*, cudaStream_t,
                                                int64_t*);
