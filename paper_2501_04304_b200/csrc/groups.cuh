// Calibration of one layer (Sec. 3.3, Eq. 4 - Eq. 7): extrema reductions on the GPU,
// dimension choice and K-means grouping on the host, padded code layout, per-timestep tables.
#pragma once

#include <algorithm>
#include <cmath>
#include <numeric>

#include "common.cuh"

struct dgq_groups {
  int C = 0, P = 0, bits = 8, dim = DGQ_DIM_CHANNEL, G = 1, R = 1, T = 1, K_pad = 0;
  double D_channel = 0.0, D_pixel = 0.0;
  std::vector<int32_t> col_group, row_group, perm, group_off;  // perm[K_pad], group_off[G+1]
  std::vector<float> scale, inv_scale;                          // [T][R][G]
  std::vector<int32_t> zp;                                      // [T][R][G]
  std::vector<char> filled;                                     // [T]
  int device = 0;
  // device copies, one allocation
  unsigned char* d_slab = nullptr;
  int16_t* d_perm = nullptr;          // [K_pad], -1 = padding
  uint8_t* d_chunk_group = nullptr;   // [K_pad / 16] group of every 16-code chunk
  int32_t* d_row_group = nullptr;     // [P]
  int32_t* d_col_group = nullptr;     // [C]
  float* d_scale = nullptr;           // [T][R][G], then d_inv_scale and d_zp of the same shape
  float* d_inv_scale = nullptr;
  int32_t* d_zp = nullptr;
  int* d_cell = nullptr;              // scratch of a calibration: minima and maxima [2][R][G] as ordered integers
};

namespace dgq {

// ------------------------------------------------------------------ kernels
// Running range of eight neighbouring columns.  NaN never wins a packed minimum or maximum.
struct Range8 {
  __half2 lo[4], hi[4];
  __device__ __forceinline__ void reset() {
    const __half2 inf = __half2half2(__ushort_as_half(0x7C00)), ninf = __half2half2(__ushort_as_half(0xFC00));
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      lo[i] = inf;
      hi[i] = ninf;
    }
  }
  __device__ __forceinline__ void add(const uint4& x) {
    const __half2* h = reinterpret_cast<const __half2*>(&x);
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      lo[i] = __hmin2(lo[i], h[i]);
      hi[i] = __hmax2(hi[i], h[i]);
    }
  }
  __device__ __forceinline__ float min_of(int i) const { return __half2float(i & 1 ? __high2half(lo[i >> 1]) : __low2half(lo[i >> 1])); }
  __device__ __forceinline__ float max_of(int i) const { return __half2float(i & 1 ? __high2half(hi[i >> 1]) : __low2half(hi[i >> 1])); }
};
// Columns 8 v .. 8 v + 7 of a row; a last vector that the matrix does not fill is completed with NaN.
__device__ __forceinline__ uint4 load8(const __half* row, int v, int C) {
  if (v * 8 + 8 <= C) return __ldg(reinterpret_cast<const uint4*>(row) + v);
  uint16_t h[8];
#pragma unroll
  for (int i = 0; i < 8; ++i) h[i] = v * 8 + i < C ? __half_as_ushort(row[v * 8 + i]) : (uint16_t)0x7FFF;
  return make_uint4(h[0] | (uint32_t)h[1] << 16, h[2] | (uint32_t)h[3] << 16, h[4] | (uint32_t)h[5] << 16, h[6] | (uint32_t)h[7] << 16);
}

// The calibration reductions read 16 bytes per thread and load, CAL_ROWS rows per block: with one 2-byte load per
// row and thread and 128 rows per block a 4096 x 640 recording kept 32 blocks busy for 128 dependent steps each.
constexpr int CAL_ROWS = 32;
constexpr int CAL_THREADS = 256;

// Per-channel extrema (Eq. 4, d = channel): a thread walks the rows of its block over eight columns.
__global__ void channel_extrema_kernel(const __half* __restrict__ X, int64_t n_rows, int C, int64_t ld,
                                       int* __restrict__ ch_min, int* __restrict__ ch_max) {
  const int64_t r0 = (int64_t)blockIdx.x * CAL_ROWS;
  const int rows = (int)min((int64_t)CAL_ROWS, n_rows - r0);
  for (int v = threadIdx.x; v * 8 < C; v += CAL_THREADS) {
    Range8 x;
    x.reset();
#pragma unroll 8
    for (int r = 0; r < rows; ++r) x.add(load8(X + (r0 + r) * ld, v, C));
#pragma unroll
    for (int i = 0; i < 8; ++i)
      if (v * 8 + i < C) {
        atomicMin(&ch_min[v * 8 + i], float_to_ordered(x.min_of(i)));
        atomicMax(&ch_max[v * 8 + i], float_to_ordered(x.max_of(i)));
      }
  }
}

// Per-pixel extrema (Eq. 4, d = pixel): one warp per row, pooled over samples at index row mod P.
__global__ void pixel_extrema_kernel(const __half* __restrict__ X, int64_t n_rows, int C, int64_t ld, int P,
                                     int* __restrict__ px_min, int* __restrict__ px_max) {
  const int lane = threadIdx.x & 31;
  const int64_t warp = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int64_t n_warps = ((int64_t)gridDim.x * blockDim.x) >> 5;
  for (int64_t r = warp; r < n_rows; r += n_warps) {
    Range8 x;
    x.reset();
#pragma unroll 4
    for (int v = lane; v * 8 < C; v += 32) x.add(load8(X + r * ld, v, C));
    float lo = INFINITY, hi = -INFINITY;
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      lo = fminf(lo, x.min_of(i));
      hi = fmaxf(hi, x.max_of(i));
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      lo = fminf(lo, __shfl_xor_sync(0xffffffffu, lo, o));
      hi = fmaxf(hi, __shfl_xor_sync(0xffffffffu, hi, o));
    }
    if (lane == 0) {
      atomicMin(&px_min[r % P], float_to_ordered(lo));
      atomicMax(&px_max[r % P], float_to_ordered(hi));
    }
  }
}

// Extrema of every (pixel group, channel group) cell (the x of Eq. 6).  A thread keeps the running range of eight
// columns and flushes it into the block's cells when the row's pixel group changes; the block's cells go to
// global memory once.
__global__ void cell_extrema_kernel(const __half* __restrict__ X, int64_t n_rows, int C, int64_t ld, int P,
                                    const int32_t* __restrict__ row_group, const int32_t* __restrict__ col_group, int G,
                                    int n_cells, int* __restrict__ cell_min, int* __restrict__ cell_max) {
  extern __shared__ int cells[];  // [2][n_cells]
  for (int i = threadIdx.x; i < n_cells; i += CAL_THREADS) {
    cells[i] = INT_MAX;
    cells[n_cells + i] = INT_MIN;
  }
  __syncthreads();
  const int64_t r0 = (int64_t)blockIdx.x * CAL_ROWS;
  const int rows = (int)min((int64_t)CAL_ROWS, n_rows - r0);
  for (int v = threadIdx.x; v * 8 < C; v += CAL_THREADS) {
    Range8 x;
    x.reset();
    auto flush = [&](int rg) {
#pragma unroll
      for (int i = 0; i < 8; ++i)
        if (v * 8 + i < C) {
          const int cell = rg * G + __ldg(col_group + v * 8 + i);
          atomicMin(&cells[cell], float_to_ordered(x.min_of(i)));
          atomicMax(&cells[n_cells + cell], float_to_ordered(x.max_of(i)));
        }
      x.reset();
    };
    int cur = __ldg(row_group + r0 % P);
#pragma unroll 8
    for (int r = 0; r < rows; ++r) {
      const int rg = __ldg(row_group + (r0 + r) % P);
      if (rg != cur) {
        flush(cur);
        cur = rg;
      }
      x.add(load8(X + (r0 + r) * ld, v, C));
    }
    flush(cur);
  }
  __syncthreads();
  for (int i = threadIdx.x; i < n_cells; i += CAL_THREADS) {
    if (cells[i] != INT_MAX) atomicMin(&cell_min[i], cells[i]);
    if (cells[n_cells + i] != INT_MIN) atomicMax(&cell_max[i], cells[n_cells + i]);
  }
}

// n minima followed by n maxima
__global__ void fill_extrema_kernel(int* p, int n) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < 2 * n) p[i] = i < n ? INT_MAX : INT_MIN;
}

// ------------------------------------------------------------------ host: grouping
// K-means on the 2-D points (min_i, max_i) (Sec. 3.3, "K groups based on their range"), made
// deterministic: vectors ranked by width (stable), centroid k starts at rank floor((2k+1)n/(2K)),
// nearest centroid with ties to the lowest k, means summed in index order in fp64, stop when the
// assignment repeats or after 100 rounds, empty clusters dropped, groups renumbered by ascending
// centroid width.
static std::vector<int> kmeans_ranges(const std::vector<double>& vmin, const std::vector<double>& vmax, int K) {
  const int n = (int)vmin.size();
  K = std::max(1, std::min(K, n));
  std::vector<int> order(n);
  std::iota(order.begin(), order.end(), 0);
  std::stable_sort(order.begin(), order.end(), [&](int a, int b) {
    return vmax[a] - vmin[a] < vmax[b] - vmin[b];
  });
  std::vector<double> cx(K), cy(K);
  for (int k = 0; k < K; ++k) {
    int i = order[(int)(((int64_t)(2 * k + 1) * n) / (2 * K))];
    cx[k] = vmin[i];
    cy[k] = vmax[i];
  }
  std::vector<int> labels(n, -1), next(n);
  for (int it = 0; it < 100; ++it) {
    // Squares and their sum are rounded one by one (host code is compiled without contraction).  Centroids outside,
    // a block of points inside: the inner loop is a select without a carried dependency, two points per
    // instruction.
    constexpr int BLOCK = 64;
    for (int i0 = 0; i0 < n; i0 += BLOCK) {
      const int m = std::min(BLOCK, n - i0);
      const double *x = &vmin[i0], *y = &vmax[i0];
      double bd[BLOCK], best[BLOCK];
      for (int i = 0; i < m; ++i) {
        const double dx = x[i] - cx[0], dy = y[i] - cy[0];
        bd[i] = dx * dx + dy * dy;
        best[i] = 0.0;
      }
      for (int k = 1; k < K; ++k) {
        const double ck = cx[k], dk = cy[k], label = (double)k;
        for (int i = 0; i < m; ++i) {
          const double dx = x[i] - ck, dy = y[i] - dk;
          const double d = dx * dx + dy * dy;
          best[i] = d < bd[i] ? label : best[i];
          bd[i] = d < bd[i] ? d : bd[i];
        }
      }
      for (int i = 0; i < m; ++i) next[i0 + i] = (int)best[i];
    }
    if (next == labels) break;
    labels = next;
    std::vector<double> sx(K, 0.0), sy(K, 0.0);
    std::vector<int> cnt(K, 0);
    for (int i = 0; i < n; ++i) {
      sx[labels[i]] += vmin[i];
      sy[labels[i]] += vmax[i];
      cnt[labels[i]]++;
    }
    for (int k = 0; k < K; ++k)
      if (cnt[k]) {
        cx[k] = sx[k] / cnt[k];
        cy[k] = sy[k] / cnt[k];
      }
  }
  std::vector<int> used;
  {
    std::vector<char> has(K, 0);
    for (int i = 0; i < n; ++i) has[labels[i]] = 1;
    for (int k = 0; k < K; ++k)
      if (has[k]) used.push_back(k);
  }
  std::stable_sort(used.begin(), used.end(), [&](int a, int b) {
    return cy[a] - cx[a] < cy[b] - cx[b];
  });
  std::vector<int> remap(K, -1);
  for (size_t j = 0; j < used.size(); ++j) remap[used[j]] = (int)j;
  for (int i = 0; i < n; ++i) labels[i] = remap[labels[i]];
  return labels;
}

// Vectors whose width exceeds tau x the median width (median of an even count = mean of the middle two).
static std::vector<char> explicit_outliers(const std::vector<double>& vmin, const std::vector<double>& vmax,
                                           double tau) {
  const int n = (int)vmin.size();
  std::vector<double> w(n);
  for (int i = 0; i < n; ++i) w[i] = vmax[i] - vmin[i];
  std::vector<double> s = w;
  std::sort(s.begin(), s.end());
  double med = (n & 1) ? s[n / 2] : 0.5 * (s[n / 2 - 1] + s[n / 2]);
  std::vector<char> out(n);
  for (int i = 0; i < n; ++i) out[i] = w[i] > tau * med;
  return out;
}

static std::vector<int> group_vectors(const std::vector<double>& vmin, const std::vector<double>& vmax, int K,
                                      int outlier_mode, double tau) {
  if (outlier_mode == DGQ_OUTLIER_KMEANS) return kmeans_ranges(vmin, vmax, K);
  const int n = (int)vmin.size();
  std::vector<char> out = explicit_outliers(vmin, vmax, tau);
  std::vector<double> rmin, rmax;
  std::vector<int> ridx;
  for (int i = 0; i < n; ++i)
    if (!out[i]) {
      rmin.push_back(vmin[i]);
      rmax.push_back(vmax[i]);
      ridx.push_back(i);
    }
  std::vector<int> labels(n, 0);
  int g_rest = 0;
  if (!ridx.empty()) {
    std::vector<int> lr = kmeans_ranges(rmin, rmax, K);
    for (size_t j = 0; j < ridx.size(); ++j) {
      labels[ridx[j]] = lr[j];
      g_rest = std::max(g_rest, lr[j] + 1);
    }
  }
  for (int i = 0; i < n; ++i)
    if (out[i]) labels[i] = g_rest;
  return labels;
}

// ------------------------------------------------------------------ host: object plumbing
constexpr int GROUP_MIN_PAD = 8;

static void groups_free_device(dgq_groups* g) { pool_free(g->d_slab); }

// Padded, group-contiguous code layout: members of each group in ascending channel order, every
// group padded to a multiple of DGQ_K_ATOM positions with at least GROUP_MIN_PAD padding positions.
// The padding carries the cell's zero-point as its code; the weight side stores -wsum spread over
// those positions, so the integer product already contains the zero-point term of Eq. 1.

static dgq_status groups_build_layout(dgq_groups* g, cudaStream_t stream) {
  g->group_off.assign(g->G + 1, 0);
  g->perm.clear();
  for (int k = 0; k < g->G; ++k) {
    g->group_off[k] = (int32_t)g->perm.size();
    for (int c = 0; c < g->C; ++c)
      if (g->col_group[c] == k) g->perm.push_back(c);
    for (int i = 0; i < GROUP_MIN_PAD; ++i) g->perm.push_back(-1);
    while (g->perm.size() % DGQ_K_ATOM) g->perm.push_back(-1);
  }
  g->K_pad = (int)g->perm.size();
  g->group_off[g->G] = g->K_pad;
  const size_t tn = (size_t)g->T * g->R * g->G;
  // One allocation and one upload for everything but the tables, which groups_upload_tables sends; every part
  // starts on a 256-byte boundary.
  size_t bytes = 0;
  auto part = [&](size_t n) {
    const size_t at = bytes;
    bytes += (n + 255) & ~size_t(255);
    return at;
  };
  const size_t o_perm = part(g->K_pad * sizeof(int16_t)), o_chunk = part(g->K_pad / 16);
  const size_t o_row = part(g->P * sizeof(int32_t)), o_col = part(g->C * sizeof(int32_t)), upload = bytes;
  const size_t o_tab = part(3 * tn * sizeof(float)), o_cell = part(2 * (size_t)g->R * g->G * sizeof(int));
  std::vector<unsigned char> h(upload, 0);
  int16_t* perm16 = reinterpret_cast<int16_t*>(h.data() + o_perm);
  uint8_t* cg = h.data() + o_chunk;
  for (int p = 0; p < g->K_pad; ++p) perm16[p] = (int16_t)g->perm[p];
  for (int k = 0; k < g->G; ++k)
    for (int p = g->group_off[k]; p < g->group_off[k + 1]; p += 16) cg[p / 16] = (uint8_t)k;
  std::memcpy(h.data() + o_row, g->row_group.data(), g->P * sizeof(int32_t));
  std::memcpy(h.data() + o_col, g->col_group.data(), g->C * sizeof(int32_t));
  DGQ_CUDA_OK(cudaGetDevice(&g->device));
  DGQ_CUDA_OK(pool_alloc(reinterpret_cast<void**>(&g->d_slab), bytes, stream));
  g->d_perm = reinterpret_cast<int16_t*>(g->d_slab + o_perm);
  g->d_chunk_group = g->d_slab + o_chunk;
  g->d_row_group = reinterpret_cast<int32_t*>(g->d_slab + o_row);
  g->d_col_group = reinterpret_cast<int32_t*>(g->d_slab + o_col);
  g->d_scale = reinterpret_cast<float*>(g->d_slab + o_tab);
  g->d_inv_scale = g->d_scale + tn;
  g->d_zp = reinterpret_cast<int32_t*>(g->d_inv_scale + tn);
  g->d_cell = reinterpret_cast<int*>(g->d_slab + o_cell);
  DGQ_CUDA_OK(cudaMemcpyAsync(g->d_slab, h.data(), upload, cudaMemcpyHostToDevice, stream));
  DGQ_CUDA_OK(cudaStreamSynchronize(stream));
  return DGQ_OK;
}

static dgq_status groups_upload_tables(dgq_groups* g, cudaStream_t stream) {
  const size_t tn = (size_t)g->T * g->R * g->G;
  std::vector<float> h(3 * tn);
  std::copy(g->scale.begin(), g->scale.end(), h.begin());
  std::copy(g->inv_scale.begin(), g->inv_scale.end(), h.begin() + tn);
  std::memcpy(h.data() + 2 * tn, g->zp.data(), tn * sizeof(int32_t));
  DGQ_CUDA_OK(cudaMemcpyAsync(g->d_scale, h.data(), h.size() * sizeof(float), cudaMemcpyHostToDevice, stream));
  DGQ_CUDA_OK(cudaStreamSynchronize(stream));
  return DGQ_OK;
}

}  // namespace dgq

// ------------------------------------------------------------------ C ABI
extern "C" dgq_status dgq_calibrate_groups(const dgq_calib_config* cfg, const void* X_cal, int64_t n_rows, int C,
                                           int64_t ld, int timestep, dgq_groups** inout, void* stream_) {
  using namespace dgq;
  if (!cfg || !X_cal || !inout || n_rows <= 0 || C <= 0) return DGQ_ERR_INVALID_ARG;
  if (cfg->act_bits < 2 || cfg->act_bits > 8 || cfg->n_groups < 1 || cfg->n_groups >= DGQ_MAX_GROUPS)
    return DGQ_ERR_INVALID_ARG;
  if (cfg->n_timesteps < 1 || timestep < 0 || timestep >= cfg->n_timesteps) return DGQ_ERR_INVALID_ARG;
  const int P = cfg->rows_per_sample;
  if (P <= 0 || n_rows % P != 0) return DGQ_ERR_INVALID_ARG;
  if (cfg->dim_select < DGQ_DIM_AUTO || cfg->dim_select > DGQ_DIM_BOTH) return DGQ_ERR_INVALID_ARG;
  if (cfg->outlier_mode != DGQ_OUTLIER_KMEANS && cfg->outlier_mode != DGQ_OUTLIER_EXPLICIT)
    return DGQ_ERR_INVALID_ARG;
  if (ld < C) return DGQ_ERR_INVALID_ARG;
  if (!aligned16(X_cal) || (ld % 8) != 0) return DGQ_ERR_ALIGNMENT;
  if (C > 8192) return DGQ_ERR_UNSUPPORTED;
  cudaStream_t stream = (cudaStream_t)stream_;
  const __half* X = (const __half*)X_cal;
  dgq_groups* g = *inout;
  const bool fresh = (g == nullptr);
  if (!fresh && (g->C != C || g->P != P || g->T != cfg->n_timesteps || g->bits != cfg->act_bits))
    return DGQ_ERR_INVALID_ARG;

  const unsigned n_blocks = (unsigned)((n_rows + CAL_ROWS - 1) / CAL_ROWS);
  dgq_status st = DGQ_OK;
  std::vector<double> cmin, cmax, pmin, pmax;  // (fresh only) ranges of the channels and of the pixel positions

  if (fresh) {
    int* d_ext = nullptr;  // minima of the C channels and P pixels, then their maxima
    const int n_ext = C + P;
    DGQ_CUDA_OK(pool_alloc(reinterpret_cast<void**>(&d_ext), 2 * (size_t)n_ext * sizeof(int), stream));
    fill_extrema_kernel<<<(2 * n_ext + 255) / 256, 256, 0, stream>>>(d_ext, n_ext);
    channel_extrema_kernel<<<n_blocks, CAL_THREADS, 0, stream>>>(X, n_rows, C, ld, d_ext, d_ext + n_ext);
    const int pb = (int)std::min<int64_t>((n_rows + 7) / 8, 148 * 8);
    pixel_extrema_kernel<<<pb, 256, 0, stream>>>(X, n_rows, C, ld, P, d_ext + C, d_ext + n_ext + C);
    g_launches += 3;
    std::vector<int> ext(2 * (size_t)n_ext);
    if (cudaMemcpyAsync(ext.data(), d_ext, ext.size() * sizeof(int), cudaMemcpyDeviceToHost, stream) != cudaSuccess ||
        cudaStreamSynchronize(stream) != cudaSuccess)
      st = DGQ_ERR_CUDA;
    cudaFreeAsync(d_ext, stream);
    if (st != DGQ_OK) return st;
    auto range = [&](int first, int n) {
      std::vector<double> v(n);
      for (int i = 0; i < n; ++i) v[i] = ordered_to_float(ext[first + i]);
      return v;
    };
    cmin = range(0, C);
    pmin = range(C, P);
    cmax = range(n_ext, C);
    pmax = range(n_ext + C, P);
    // Eq. 4
    auto spread = [](const std::vector<double>& v) {
      return *std::max_element(v.begin(), v.end()) - *std::min_element(v.begin(), v.end());
    };
    const double Dc = spread(cmax) + spread(cmin), Dp = spread(pmax) + spread(pmin);
    int dim = cfg->dim_select;
    if (dim == DGQ_DIM_AUTO) dim = (Dc >= Dp) ? DGQ_DIM_CHANNEL : DGQ_DIM_PIXEL;  // Eq. 5, tie -> channel
    g = new dgq_groups();
    g->C = C;
    g->P = P;
    g->bits = cfg->act_bits;
    g->T = cfg->n_timesteps;
    g->dim = dim;
    g->D_channel = Dc;
    g->D_pixel = Dp;
    g->col_group.assign(C, 0);
    g->row_group.assign(P, 0);
    if (dim == DGQ_DIM_CHANNEL || dim == DGQ_DIM_BOTH) {
      std::vector<int> l = group_vectors(cmin, cmax, cfg->n_groups, cfg->outlier_mode, cfg->outlier_tau);
      g->col_group.assign(l.begin(), l.end());
    }
    if (dim == DGQ_DIM_PIXEL || dim == DGQ_DIM_BOTH) {
      std::vector<int> l = group_vectors(pmin, pmax, cfg->n_groups, cfg->outlier_mode, cfg->outlier_tau);
      g->row_group.assign(l.begin(), l.end());
    }
    g->G = *std::max_element(g->col_group.begin(), g->col_group.end()) + 1;
    g->R = *std::max_element(g->row_group.begin(), g->row_group.end()) + 1;
    const size_t tn = (size_t)g->T * g->R * g->G;
    g->scale.assign(tn, 1.0f);
    g->inv_scale.assign(tn, 1.0f);
    g->zp.assign(tn, 0);
    g->filled.assign(g->T, 0);
    st = groups_build_layout(g, stream);
    if (st != DGQ_OK) {
      groups_free_device(g);
      delete g;
      return st;
    }
  }

  // Eq. 6 per cell from this timestep's rows
  const int n_cells = g->R * g->G;
  std::vector<int> cell(2 * (size_t)n_cells, INT_MIN);  // minima, then maxima, as ordered integers
  if (fresh && (g->R == 1 || g->G == 1)) {
    // grouped along one dimension: a cell's range is that of its channels (or pixel positions), which are at hand
    std::fill(cell.begin(), cell.begin() + n_cells, INT_MAX);
    const bool by_channel = g->R == 1;
    const std::vector<int32_t>& group = by_channel ? g->col_group : g->row_group;
    const std::vector<double>&lo = by_channel ? cmin : pmin, &hi = by_channel ? cmax : pmax;
    for (size_t i = 0; i < group.size(); ++i) {
      cell[group[i]] = std::min(cell[group[i]], float_to_ordered((float)lo[i]));
      cell[n_cells + group[i]] = std::max(cell[n_cells + group[i]], float_to_ordered((float)hi[i]));
    }
  } else {
    fill_extrema_kernel<<<(2 * n_cells + 255) / 256, 256, 0, stream>>>(g->d_cell, n_cells);
    cell_extrema_kernel<<<n_blocks, CAL_THREADS, 2 * n_cells * sizeof(int), stream>>>(
        X, n_rows, C, ld, P, g->d_row_group, g->d_col_group, g->G, n_cells, g->d_cell, g->d_cell + n_cells);
    g_launches += 2;
    if (cudaMemcpyAsync(cell.data(), g->d_cell, cell.size() * sizeof(int), cudaMemcpyDeviceToHost, stream) != cudaSuccess ||
        cudaStreamSynchronize(stream) != cudaSuccess)
      st = DGQ_ERR_CUDA;
  }
  for (int i = 0; i < n_cells && st == DGQ_OK; ++i) {
    float lo = 0.f, hi = 0.f;
    if (cell[i] != INT_MAX) {  // an empty cell keeps the range (0, 0)
      lo = ordered_to_float(cell[i]);
      hi = ordered_to_float(cell[n_cells + i]);
    }
    float s, inv_s;
    int Z;
    group_params(lo, hi, g->bits, s, inv_s, Z);
    const size_t o = (size_t)timestep * n_cells + i;
    g->scale[o] = s;
    g->inv_scale[o] = inv_s;
    g->zp[o] = Z;
  }
  if (st == DGQ_OK) {
    g->filled[timestep] = 1;
    st = groups_upload_tables(g, stream);
  }
  if (st != DGQ_OK) {
    if (fresh) {
      groups_free_device(g);
      delete g;
    }
    return st;
  }
  *inout = g;
  return DGQ_OK;
}

extern "C" dgq_status dgq_groups_from_host(int C, int P, int act_bits, int G, int R, int T,
                                           const int32_t* col_group, const int32_t* row_group, const float* scale,
                                           const int32_t* zp, dgq_groups** out) {
  using namespace dgq;
  if (!out || !col_group || !row_group || !scale || !zp) return DGQ_ERR_INVALID_ARG;
  if (C <= 0 || C > 8192 || P <= 0 || G < 1 || G > DGQ_MAX_GROUPS || R < 1 || R > DGQ_MAX_GROUPS || T < 1)
    return DGQ_ERR_INVALID_ARG;
  if (act_bits < 2 || act_bits > 8) return DGQ_ERR_INVALID_ARG;
  for (int c = 0; c < C; ++c)
    if (col_group[c] < 0 || col_group[c] >= G) return DGQ_ERR_INVALID_ARG;
  for (int p = 0; p < P; ++p)
    if (row_group[p] < 0 || row_group[p] >= R) return DGQ_ERR_INVALID_ARG;
  dgq_groups* g = new dgq_groups();
  g->C = C;
  g->P = P;
  g->bits = act_bits;
  g->G = G;
  g->R = R;
  g->T = T;
  g->dim = (G > 1 && R > 1) ? DGQ_DIM_BOTH : (R > 1 ? DGQ_DIM_PIXEL : DGQ_DIM_CHANNEL);
  g->col_group.assign(col_group, col_group + C);
  g->row_group.assign(row_group, row_group + P);
  const size_t tn = (size_t)T * R * G;
  g->scale.assign(scale, scale + tn);
  g->zp.assign(zp, zp + tn);
  g->inv_scale.resize(tn);
  for (size_t i = 0; i < tn; ++i) {
    if (!(g->scale[i] > 0.f)) {
      delete g;
      return DGQ_ERR_INVALID_ARG;
    }
    volatile float inv = 1.0f / g->scale[i];
    g->inv_scale[i] = inv;
  }
  g->filled.assign(T, 1);
  dgq_status st = groups_build_layout(g, nullptr);
  if (st == DGQ_OK) st = groups_upload_tables(g, nullptr);
  if (st != DGQ_OK) {
    groups_free_device(g);
    delete g;
    return st;
  }
  *out = g;
  return DGQ_OK;
}

extern "C" dgq_status dgq_groups_destroy(dgq_groups* g) {
  if (!g) return DGQ_OK;
  dgq::groups_free_device(g);
  delete g;
  return DGQ_OK;
}

extern "C" dgq_status dgq_groups_info(const dgq_groups* g, int* C, int* P, int* K_pad, int* G, int* R, int* T,
                                      int* dim, int* act_bits, double* D_channel, double* D_pixel) {
  if (!g) return DGQ_ERR_INVALID_ARG;
  if (C) *C = g->C;
  if (P) *P = g->P;
  if (K_pad) *K_pad = g->K_pad;
  if (G) *G = g->G;
  if (R) *R = g->R;
  if (T) *T = g->T;
  if (dim) *dim = g->dim;
  if (act_bits) *act_bits = g->bits;
  if (D_channel) *D_channel = g->D_channel;
  if (D_pixel) *D_pixel = g->D_pixel;
  return DGQ_OK;
}

extern "C" dgq_status dgq_groups_export(const dgq_groups* g, int32_t* perm, int32_t* col_group, int32_t* group_off,
                                        int32_t* row_group, float* scale, int32_t* zp) {
  if (!g) return DGQ_ERR_INVALID_ARG;
  if (perm) std::copy(g->perm.begin(), g->perm.end(), perm);
  if (col_group) std::copy(g->col_group.begin(), g->col_group.end(), col_group);
  if (group_off) std::copy(g->group_off.begin(), g->group_off.end(), group_off);
  if (row_group) std::copy(g->row_group.begin(), g->row_group.end(), row_group);
  if (scale) std::copy(g->scale.begin(), g->scale.end(), scale);
  if (zp) std::copy(g->zp.begin(), g->zp.end(), zp);
  return DGQ_OK;
}
