// Weight preparation: per-out-channel symmetric round-to-nearest codes, permuted and padded to the layer's
// group-contiguous code layout, int4 packed two per byte, plus the per-group column sums the de-quantizer needs.
//
// One kernel, one thread block per output row: the row's absolute maximum, its codes (kept in shared memory), the
// sums of every group and the padded row are one pass over the row's fp16 weights.  What a caller waits for is
// then the allocation, one launch and one small copy back (scales and the mask of residual groups); the
// host loops this replaces took 30 ms for 640 -> 5120.  The object keeps no host copy of the codes: an export
// reads them back out of the padded rows.
#pragma once

#include "groups.cuh"

struct dgq_weight {
  int N = 0, K = 0, C = 0, G = 0, w_bits = 8, is_conv = 0;
  int N_pad = 0;                 // N rounded up to a multiple of 256 (rows beyond N are zero)
  int Kt = 0;                    // length of the GEMM reduction in padded positions (multiple of 32)
  std::vector<int32_t> seg_end;  // [G] end of every group's segment, in 32-position atoms
  std::vector<int32_t> atoms;    // [G] atoms of every group (of one filter tap)
  std::vector<float> sw;         // host scales [N]
  std::vector<int2> chan;        // [C] reduction position of every channel's first tap, distance between its taps
  unsigned char* d_slab = nullptr;  // all device arrays below
  int8_t* d_w = nullptr;         // 8-bit: [N_pad][Kt] s8; 4-bit: [N_pad][Kt/2] packed
  float* d_sw = nullptr;         // [N_pad]; 4-bit: sw / 16 (the unpacked codes carry a factor 16)
  float* d_wsum = nullptr;       // [G][N_pad] column sums per group as fp32 (exact); 4-bit: x 16
  float* d_wres = nullptr;       // [G][N_pad] part of wsum the padding positions could not absorb
  int2* d_chan = nullptr;        // [C] copy of `chan`
  uint32_t res_mask = 0;         // bit g set: group g has a non-zero entry in d_wres
  int device = 0;                // device of the arrays above
};

namespace dgq {

constexpr int WP_THREADS = 256;

struct WeightArgs {
  const __half* W;       // [N][K], or null when the codes are given
  const int8_t* wq;      // [N][K] given codes
  const float* sw_in;    // [N] their scales
  int N, K, C, G, N_pad, Kt, K_pad, taps, qmax, four_bit;
  const int16_t* perm;   // [K_pad] channel of every padded position, -1 = padding
  int group_off[DGQ_MAX_GROUPS + 1];  // first padded position of every group
  int red_off[DGQ_MAX_GROUPS + 1];    // the same in the reduction, for one tap
  uint8_t* w;            // outputs, see dgq_weight
  float *sw, *wsum, *wres;
  float* sw_out;         // [N] scales as the caller sees them
  unsigned int* res_mask;
};

// Eight neighbouring reduction positions (always of one group) of one row: their codes, padding as 0.  The
// reduction is group-major, inside a group tap-major, then the group's padded positions.
__device__ __forceinline__ int weight_codes8(const WeightArgs& a, const int8_t* row, int pos, int (&c)[8], int& first_pad) {
  int g = 0;
  while (pos >= a.taps * a.red_off[g + 1]) ++g;
  const int len = a.red_off[g + 1] - a.red_off[g], local = pos - a.taps * a.red_off[g];
  const int tap = local / len, p0 = a.group_off[g] + local - tap * len;
  const int8_t* src = row + tap * a.C;
  const uint4 pv = __ldg(reinterpret_cast<const uint4*>(a.perm + p0));
  const int16_t* p = reinterpret_cast<const int16_t*>(&pv);
  first_pad = 8;
#pragma unroll
  for (int i = 7; i >= 0; --i) {
    c[i] = p[i] >= 0 ? src[p[i]] : 0;
    if (p[i] < 0) first_pad = i;  // padding follows a group's members
  }
  return g;
}

__global__ void __launch_bounds__(WP_THREADS) weight_rows_kernel(const __grid_constant__ WeightArgs a) {
  extern __shared__ int8_t row_s[];  // [K] codes of the row
  __shared__ float red[WP_THREADS / 32];
  __shared__ int sum_s[DGQ_MAX_GROUPS];
  const int o = blockIdx.x;
  const int row_bytes = a.four_bit ? a.Kt / 2 : a.Kt;
  uint8_t* out = a.w + (size_t)o * row_bytes;
  if (o >= a.N) {
    for (int i = threadIdx.x; i < row_bytes / 16; i += WP_THREADS) reinterpret_cast<uint4*>(out)[i] = make_uint4(0, 0, 0, 0);
    for (int g = threadIdx.x; g < a.G; g += WP_THREADS) a.wsum[(size_t)g * a.N_pad + o] = a.wres[(size_t)g * a.N_pad + o] = 0.f;
    if (threadIdx.x == 0) a.sw[o] = 0.f;
    return;
  }
  const float unit = a.four_bit ? 16.f : 1.f;
  if (threadIdx.x < a.G) sum_s[threadIdx.x] = 0;
  float s;
  if (a.W) {
    // fp32 sequence: sw = absmax / qmax, inv = 1 / sw, code = clamp(rint(w * inv), -qmax, qmax), 0 where that is NaN
    const __half* w = a.W + (size_t)o * a.K;
    const float qmax = (float)a.qmax;
    float amax = 0.f;
    for (int k = threadIdx.x; k < a.K; k += WP_THREADS) amax = fmaxf(amax, fabsf(__half2float(__ldg(w + k))));
#pragma unroll
    for (int d = 16; d > 0; d >>= 1) amax = fmaxf(amax, __shfl_xor_sync(0xffffffffu, amax, d));
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = amax;
    __syncthreads();
#pragma unroll
    for (int i = 0; i < WP_THREADS / 32; ++i) amax = fmaxf(amax, red[i]);
    s = amax > 0.f ? __fdiv_rn(amax, qmax) : 1.0f;
    const float inv = __fdiv_rn(1.0f, s);
    for (int k = threadIdx.x; k < a.K; k += WP_THREADS) {
      const float r = rintf(__fmul_rn(__half2float(__ldg(w + k)), inv));
      row_s[k] = r == r ? (int8_t)(int)fminf(fmaxf(r, -qmax), qmax) : (int8_t)0;
    }
  } else {
    s = __ldg(a.sw_in + o);
    for (int k = threadIdx.x; k < a.K; k += WP_THREADS) row_s[k] = __ldg(a.wq + (size_t)o * a.K + k);
  }
  if (threadIdx.x == 0) {
    a.sw[o] = __fdiv_rn(s, unit);
    a.sw_out[o] = s;
  }
  __syncthreads();
  int c[8], first_pad;
  for (int pos = threadIdx.x * 8; pos < a.Kt; pos += WP_THREADS * 8) {
    const int g = weight_codes8(a, row_s, pos, c, first_pad);
    if (first_pad > 0) atomicAdd(&sum_s[g], ((c[0] + c[1]) + (c[2] + c[3])) + ((c[4] + c[5]) + (c[6] + c[7])));
  }
  __syncthreads();
  // Linear layers: -sum of a group is spread over its padding positions (whose activation code is the zero-point
  // Z), so that acc + Z * (-sum) = acc - Z * wsum comes out of the integer product.  What does not fit in the
  // available positions stays in `wres` for the epilogue.  The conv's zero-centred codes have no zero-point term.
  for (int pos = threadIdx.x * 8; pos < a.Kt; pos += WP_THREADS * 8) {
    const int g = weight_codes8(a, row_s, pos, c, first_pad);
    if (a.taps == 1 && first_pad < 8) {
      // the padding starts somewhere in front of this word: count the positions it fills up to here
      int lo = a.group_off[g], hi = pos + first_pad;  // first padding position of the group lies in [lo, hi]
      while (lo < hi) {
        const int mid = (lo + hi) >> 1;
        if (__ldg(a.perm + mid) < 0) hi = mid;
        else lo = mid + 1;
      }
      const int neg = -sum_s[g], sign = neg < 0 ? -1 : 1;
#pragma unroll
      for (int i = 0; i < 8; ++i)
        if (i >= first_pad) c[i] = sign * min(a.qmax, max(0, sign * neg - (pos + i - lo) * a.qmax));
    }
    if (a.four_bit) {
      // Word of 8 positions: byte i holds code i in its low nibble and code 4 + i in its high nibble.  In the GEMM
      // (word << 4) & 0xF0F0F0F0 and word & 0xF0F0F0F0 are then bytes 0..3 and 4..7, each equal to 16 x the signed
      // code, with no per-byte sign extension.
      uint32_t v = 0;
#pragma unroll
      for (int i = 0; i < 4; ++i) v |= (uint32_t)((c[i] & 0xF) | ((c[4 + i] & 0xF) << 4)) << (8 * i);
      *reinterpret_cast<uint32_t*>(out + pos / 2) = v;
    } else {
      uint2 v = make_uint2(0, 0);
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        v.x |= (uint32_t)(c[i] & 0xFF) << (8 * i);
        v.y |= (uint32_t)(c[4 + i] & 0xFF) << (8 * i);
      }
      *reinterpret_cast<uint2*>(out + pos) = v;
    }
  }
  for (int g = threadIdx.x; g < a.G; g += WP_THREADS) {
    const int sum = sum_s[g];
    int members = 0, lo = a.group_off[g], hi = a.group_off[g + 1];
    const int end = hi;
    while (lo < hi) {
      const int mid = (lo + hi) >> 1;
      if (__ldg(a.perm + mid) < 0) hi = mid;
      else lo = mid + 1;
    }
    members = lo;
    const int room = (end - members) * a.qmax;
    const int left = sum < 0 ? min(0, sum + room) : max(0, sum - room);
    const int res = a.taps == 1 ? left : sum;
    a.wsum[(size_t)g * a.N_pad + o] = (float)sum * unit;
    a.wres[(size_t)g * a.N_pad + o] = (float)res * unit;
    if (res != 0 && a.taps == 1) atomicOr(a.res_mask, 1u << g);
  }
}

// Code of position `pos` of a padded row (see weight_rows_kernel for the order of 4-bit codes in a word).
__host__ __device__ __forceinline__ int8_t weight_code_at(const uint8_t* row, int pos, int four_bit) {
  if (!four_bit) return (int8_t)row[pos];
  const uint32_t b = row[pos / 8 * 4 + (pos & 3)];
  return (int8_t)((int)(((pos & 4) ? b >> 4 : b) << 28) >> 28);
}
// Codes in original channel order from the padded rows.
__global__ void weight_unpermute_kernel(const uint8_t* __restrict__ w, const int2* __restrict__ chan, int K, int C, int Kt,
                                        int four_bit, int8_t* __restrict__ out) {
  const uint8_t* row = w + (size_t)blockIdx.x * (four_bit ? Kt / 2 : Kt);
  for (int k = threadIdx.x; k < K; k += blockDim.x) {
    const int tap = k / C;
    const int2 ch = __ldg(chan + (k - tap * C));
    out[(size_t)blockIdx.x * K + k] = weight_code_at(row, ch.x + tap * ch.y, four_bit);
  }
}

// The codes of a weight in original channel order, in host memory.  Works on the weight's device whichever is current,
// on the library's own stream and outside the rules of a stream capture that the caller may have running (the arrays are
// complete since the build, so nothing has to be waited for).  Small weights, and those for which the device has no
// scratch memory left, are put in order on the host (2^9 codes 18 us, 2^11 codes 26 us; through a kernel 26 us and, up to
// 2^14 codes, no more than 29).
constexpr size_t WEIGHT_HOST_CODES = 1 << 11;
static dgq_status weight_codes_to_host(const dgq_weight* w, int8_t* wq) {
  DeviceScope on(w->device);
  DGQ_CUDA_OK(on.err);
  cudaStreamCaptureMode mode = cudaStreamCaptureModeRelaxed;
  DGQ_CUDA_OK(cudaThreadExchangeStreamCaptureMode(&mode));
  const size_t n = (size_t)w->N * w->K;
  const int four_bit = w->w_bits == 4;
  cudaStream_t stream = nullptr;
  cudaError_t e = own_stream(&stream);
  int8_t* d = nullptr;
  if (e != cudaSuccess) {
  } else if (n > WEIGHT_HOST_CODES && pool_alloc((void**)&d, n, stream, true) == cudaSuccess) {
    weight_unpermute_kernel<<<w->N, 256, 0, stream>>>((const uint8_t*)w->d_w, w->d_chan, w->K, w->C, w->Kt, four_bit, d);
    g_launches += 1;
    if ((e = cudaGetLastError()) == cudaSuccess) e = cudaMemcpyAsync(wq, d, n, cudaMemcpyDeviceToHost, stream);
    const cudaError_t done = cudaStreamSynchronize(stream);
    if (e == cudaSuccess) e = done;
    cudaFreeAsync(d, stream);
  } else {
    cudaGetLastError();  // (an allocation that failed)
    const size_t row_bytes = four_bit ? w->Kt / 2 : w->Kt;
    std::vector<uint8_t> rows(w->N * row_bytes);
    if ((e = cudaMemcpyAsync(rows.data(), w->d_w, rows.size(), cudaMemcpyDeviceToHost, stream)) == cudaSuccess)
      e = cudaStreamSynchronize(stream);
    for (int o = 0; o < w->N && e == cudaSuccess; ++o)
      for (int tap = 0, k = 0; k < w->K; ++tap)
        for (int c = 0; c < w->C; ++c, ++k)
          wq[(size_t)o * w->K + k] = weight_code_at(&rows[o * row_bytes], w->chan[c].x + tap * w->chan[c].y, four_bit);
  }
  cudaThreadExchangeStreamCaptureMode(&mode);
  return e == cudaSuccess ? DGQ_OK : DGQ_ERR_CUDA;
}

// Device arrays of a weight in one allocation, filled by weight_rows_kernel from fp16 weights `W` (device) or from
// codes `wq` and scales `sw` (host), whichever is given.
static dgq_status weight_build(const dgq_groups* g, const __half* W, const int8_t* wq, const float* sw, int N, int K, int w_bits,
                               const dgq_conv_desc* conv, dgq_weight** out, cudaStream_t stream) {
  const int taps = conv ? 9 : 1;
  if (conv && (conv->c != g->C || conv->n <= 0 || conv->h <= 0 || conv->w <= 0)) return DGQ_ERR_INVALID_ARG;
  if (K != taps * g->C) return DGQ_ERR_INVALID_ARG;
  if ((N % 8) != 0) return DGQ_ERR_UNSUPPORTED;
  WeightArgs a;
  std::memset(&a, 0, sizeof(a));
  a.qmax = (1 << (w_bits - 1)) - 1;
  if (wq)
    for (size_t i = 0; i < (size_t)N * K; ++i)
      if (wq[i] < -a.qmax || wq[i] > a.qmax) return DGQ_ERR_INVALID_ARG;
  // accumulator bound: |code| <= 255, |weight| <= 127 (4-bit: 7 * 16)
  if ((int64_t)taps * g->K_pad * 255 * 127 >= ((int64_t)1 << 31)) return DGQ_ERR_UNSUPPORTED;
  int dev = 0;
  DGQ_CUDA_OK(cudaGetDevice(&dev));
  // Layout tables and weights may lie on another device than the current one, where the object is made: those are
  // copied over first.
  bool w_remote = false;
  if (W) {
    cudaPointerAttributes at;
    DGQ_CUDA_OK(cudaPointerGetAttributes(&at, W));
    if (at.type == cudaMemoryTypeUnregistered) return DGQ_ERR_CUDA;
    w_remote = at.type == cudaMemoryTypeDevice && at.device != dev;
  }
  dgq_weight* w = new dgq_weight();
  w->device = dev;
  w->N = N;
  w->K = K;
  w->C = g->C;
  w->G = g->G;
  w->w_bits = w_bits;
  w->is_conv = conv ? 1 : 0;
  w->N_pad = (N + 255) / 256 * 256;
  // A linear layer's reduction is the padded code row.  A conv has no use for an atom that holds only padding
  // (zero-centred codes: it would add zeros), so its reduction leaves those out: 18 of 22 atoms per tap
  // remain for 320 channels in 16 groups.
  w->seg_end.resize(g->G);
  w->atoms.resize(g->G);
  for (int k = 0; k < g->G; ++k) {
    int members = 0;
    while (g->perm[g->group_off[k] + members] >= 0) ++members;  // every group ends in padding
    w->atoms[k] = conv ? std::max(1, (members + DGQ_K_ATOM - 1) / DGQ_K_ATOM) : (g->group_off[k + 1] - g->group_off[k]) / DGQ_K_ATOM;
    a.red_off[k + 1] = a.red_off[k] + w->atoms[k] * DGQ_K_ATOM;
    w->seg_end[k] = taps * a.red_off[k + 1] / DGQ_K_ATOM;
  }
  w->Kt = taps * a.red_off[g->G];

  size_t bytes = 0;
  auto part = [&](size_t n) {
    const size_t at = bytes;
    bytes += (n + 255) & ~size_t(255);
    return at;
  };
  const size_t w_bytes = (size_t)w->N_pad * w->Kt / (w_bits == 4 ? 2 : 1), per_group = (size_t)g->G * w->N_pad * sizeof(float);
  const size_t o_w = part(w_bytes), o_sw = part(w->N_pad * sizeof(float)), o_wsum = part(per_group), o_wres = part(per_group);
  const size_t o_chan = part(g->C * sizeof(int2)), o_back = part((size_t)(N + 1) * sizeof(float));  // scales, then the mask
  // for the duration of the call: given codes and scales or weights of another device, layout of another device
  const size_t slab_bytes = bytes;
  bytes = 0;
  const size_t o_in = part(wq ? (size_t)N * K : w_remote ? (size_t)N * K * sizeof(__half) : 0), o_in_sw = part(wq ? N * sizeof(float) : 0);
  const size_t o_perm = part(g->device != dev ? g->K_pad * sizeof(int16_t) : 0), temp_bytes = bytes;
  unsigned char* d_temp = nullptr;
  dgq_status st = DGQ_OK;
  auto ok = [&](cudaError_t e) {
    if (st == DGQ_OK && e != cudaSuccess) st = DGQ_ERR_CUDA;
    return st == DGQ_OK;
  };
  if (ok(pool_alloc((void**)&w->d_slab, slab_bytes, stream)) && (!temp_bytes || ok(pool_alloc((void**)&d_temp, temp_bytes, stream)))) {
    w->d_w = reinterpret_cast<int8_t*>(w->d_slab + o_w);
    w->d_sw = reinterpret_cast<float*>(w->d_slab + o_sw);
    w->d_wsum = reinterpret_cast<float*>(w->d_slab + o_wsum);
    w->d_wres = reinterpret_cast<float*>(w->d_slab + o_wres);
    w->d_chan = reinterpret_cast<int2*>(w->d_slab + o_chan);
    float* back = reinterpret_cast<float*>(w->d_slab + o_back);
    w->chan.resize(g->C);
    for (int k = 0; k < g->G; ++k)
      for (int p = g->group_off[k]; p < g->group_off[k + 1]; ++p)
        if (g->perm[p] >= 0)
          w->chan[g->perm[p]] = make_int2(taps * a.red_off[k] + p - g->group_off[k], a.red_off[k + 1] - a.red_off[k]);
    ok(cudaMemcpyAsync(w->d_chan, w->chan.data(), w->chan.size() * sizeof(int2), cudaMemcpyHostToDevice, stream));
    a.W = W;
    a.perm = g->d_perm;
    if (wq) {
      a.wq = reinterpret_cast<int8_t*>(d_temp + o_in);
      a.sw_in = reinterpret_cast<float*>(d_temp + o_in_sw);
      ok(cudaMemcpyAsync(d_temp + o_in, wq, (size_t)N * K, cudaMemcpyHostToDevice, stream));
      ok(cudaMemcpyAsync(d_temp + o_in_sw, sw, N * sizeof(float), cudaMemcpyHostToDevice, stream));
    } else if (w_remote) {
      a.W = reinterpret_cast<__half*>(d_temp + o_in);
      ok(cudaMemcpyAsync(d_temp + o_in, W, (size_t)N * K * sizeof(__half), cudaMemcpyDefault, stream));
    }
    if (g->device != dev) {
      a.perm = reinterpret_cast<int16_t*>(d_temp + o_perm);
      ok(cudaMemcpyAsync(d_temp + o_perm, g->d_perm, g->K_pad * sizeof(int16_t), cudaMemcpyDefault, stream));
    }
    ok(cudaMemsetAsync(back + N, 0, sizeof(float), stream));
    a.N = N;
    a.K = K;
    a.C = g->C;
    a.G = g->G;
    a.N_pad = w->N_pad;
    a.Kt = w->Kt;
    a.K_pad = g->K_pad;
    a.taps = taps;
    a.four_bit = w_bits == 4;
    std::copy(g->group_off.begin(), g->group_off.end(), a.group_off);
    a.w = reinterpret_cast<uint8_t*>(w->d_w);
    a.sw = w->d_sw;
    a.wsum = w->d_wsum;
    a.wres = w->d_wres;
    a.sw_out = back;
    a.res_mask = reinterpret_cast<unsigned int*>(back + N);
    if (K > 40 * 1024)
      ok(cudaFuncSetAttribute(weight_rows_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, 72 * 1024));
    std::vector<float> host(N + 1);
    if (st == DGQ_OK) {
      weight_rows_kernel<<<w->N_pad, WP_THREADS, (size_t)K, stream>>>(a);
      g_launches += 1;
      ok(cudaGetLastError());
      ok(cudaMemcpyAsync(host.data(), back, host.size() * sizeof(float), cudaMemcpyDeviceToHost, stream));
      ok(cudaStreamSynchronize(stream));
      std::memcpy(&w->res_mask, &host[N], sizeof(w->res_mask));
      host.resize(N);
      w->sw = std::move(host);
    }
  }
  if (d_temp) cudaFreeAsync(d_temp, stream);
  if (st != DGQ_OK) {
    pool_free(w->d_slab);
    delete w;
    return st;
  }
  *out = w;
  return DGQ_OK;
}

}  // namespace dgq

extern "C" dgq_status dgq_weight_from_codes(const dgq_groups* g, const int8_t* wq, const float* sw, int N, int K,
                                            int w_bits, const dgq_conv_desc* conv, dgq_weight** out) {
  if (!g || !wq || !sw || !out || N <= 0) return DGQ_ERR_INVALID_ARG;
  if (w_bits != 8 && w_bits != 4) return DGQ_ERR_INVALID_ARG;
  return dgq::weight_build(g, nullptr, wq, sw, N, K, w_bits, conv, out, nullptr);
}

extern "C" dgq_status dgq_weight_prepare(const dgq_groups* g, const void* W, int N, int K, int w_bits,
                                         const dgq_conv_desc* conv, dgq_weight** out, void* stream) {
  if (!g || !W || !out || N <= 0 || K <= 0) return DGQ_ERR_INVALID_ARG;
  if (w_bits != 8 && w_bits != 4) return DGQ_ERR_INVALID_ARG;
  return dgq::weight_build(g, (const __half*)W, nullptr, nullptr, N, K, w_bits, conv, out, (cudaStream_t)stream);
}

extern "C" dgq_status dgq_weight_destroy(dgq_weight* w) {
  if (!w) return DGQ_OK;
  dgq::pool_free(w->d_slab);
  delete w;
  return DGQ_OK;
}

extern "C" dgq_status dgq_weight_export(const dgq_weight* w, int8_t* wq, float* sw) {
  if (!w) return DGQ_ERR_INVALID_ARG;
  if (wq) {
    const dgq_status st = dgq::weight_codes_to_host(w, wq);
    if (st != DGQ_OK) return st;
  }
  if (sw) std::copy(w->sw.begin(), w->sw.end(), sw);
  return DGQ_OK;
}
