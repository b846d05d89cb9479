// Activation quantizer: Eq. 1 with the per-cell parameters of Eq. 6, fused with the channel
// permutation into the padded, group-contiguous code layout the GEMM reads.
//
// Rows are handled in pairs.  A thread block takes a batch of row pairs, loads them with 128-bit loads and
// leaves every pair interleaved in shared memory (one 32-bit word per channel: both rows' fp16 values), so that
// one 32-bit read fetches a channel of two rows.  A thread owns one 16-code chunk of one pair of the batch and the
// same chunk in every batch, so the 16 channels it gathers sit in registers as byte offsets (padding positions
// point at a word of NaN behind the row) and the values are read from shared memory once: range, parameters and codes
// work on registers.  The packed half-precision min / max and the packed fp32 arithmetic then serve both rows with
// one instruction.  Dynamic-token mode merges the ranges of a (row, group) cell with shared-memory atomics on
// order-preserving keys (a warp whose lanes all belong to one cell reduces first), every thread
// derives (s, 1/s, Z) of its two cells.
//
// Bound: about 430 (dynamic) or 300 (static) warp instructions per row of 512 codes (half of them two-cycle integer and conversion
// instructions) and the latency of one read-reduce-write chain for small matrices; the bytes (2 B read + 1 B written per
// element + 8 B per (token, group) in dynamic mode) would take a third of the time.  72 registers keep 28
// warps on an SM (4 to 60 bytes of a thread spill): at 80 an 8192-row matrix needs a second, nearly empty round of batches
// (5.5 against 5.1 us), at 64 the gathered values spill (5.9 us).  Blocks of 128 threads keep the barriers cheap (256: 5.8 us).
// Against one warp per two rows that scattered value by value into group order and read the chunks back twice, dynamic /
// static, inputs cold, 8 groups: 8192 x 320 6.4 -> 5.1 / 7.0 -> 3.8 us, 2048 x 5120 23.7 -> 15.7, 616 x 768 4.9 -> 3.1; 8192 x 1280 17.1 ->
// 17.1 / 13.6 -> 12.4, 32768 x 1280 54.7 -> 53.1 / 42.4 -> 36.4, 32768 x 2560 117 -> 112 / 80 -> 75.  It is the slower one for dynamic
// ranges of 960 and 1920 to 2048 channels at 8192 rows (14.5 -> 15.6, 24.3 -> 26.6, 25.9 -> 28.1) and of 1920 to 2048 beyond (32768 rows 83.6 ->
// 90.3, 88.7 -> 91.3): a pair fills its warps badly there and the barriers of a batch are waited for.
#pragma once

#include <type_traits>

#include "groups.cuh"

namespace dgq {

struct QuantArgs {
  const __half* X;
  uint8_t* Xq;
  int64_t M, ld;
  int C, K_pad, G, P, bits;
  int pairs;               // row pairs of a batch
  int pitch;               // 32-bit words of an interleaved row pair in shared memory
  const int16_t* perm;     // [K_pad] channel of every position, -1 = padding
  const uint8_t* chunk_group;  // [K_pad / 16]
  const int32_t* row_group;  // null if there is one row group
  const float* inv_scale;  // static: table row of the timestep [R][G]
  const int32_t* zp;
  float* dyn_scale;        // dynamic: outputs [M][G]
  int32_t* dyn_zp;
};

// Place of a channel in an interleaved pair.  Spread, four words are left out behind every 32: where neighbouring channels
// belong to one group (the whole layer, when it is grouped by pixel positions only) the lanes of a warp read words 16
// apart, which would lie in two banks; this way at most four lanes meet in one.
template <bool SPREAD>
__host__ __device__ inline int qa_word(int c) { return SPREAD ? c + (c >> 5) * 4 : c; }
// Words of the interleaved pair: the channels, a word of NaN for the padding, up to a multiple of four.
__host__ __device__ inline int qa_pitch(int C, bool spread) { return ((spread ? qa_word<true>(C) : C) + 1 + 3) & ~3; }
constexpr int QA_SMEM_MAX = 80 * 1024;  // three pairs of the widest layer that has three
// The row buffer and two sets of cell ranges.
__host__ inline size_t qa_smem_bytes(int pairs, int pitch, int G, bool dynamic) {
  const size_t cells = (size_t)pairs * 2 * G;
  return (size_t)pairs * pitch * 4 + (dynamic ? cells * 4 * 4 : 0);
}

// bits 0-3 of `m` spread to 0xFF bytes
__device__ __forceinline__ uint32_t nibble_to_byte_mask(uint32_t m) {
  return (((m & 0xFu) * 0x00204081u) & 0x01010101u) * 0xFFu;
}

// fp16 bits -> order-preserving integer and back
__device__ __forceinline__ int half_key(uint32_t h) {
  const int s = (int)(int16_t)h;
  return s ^ ((s >> 15) & 0x7FFF);
}
__device__ __forceinline__ float half_from_key(int k) {
  return __half2float(__ushort_as_half((uint16_t)(k ^ ((k >> 15) & 0x7FFF))));
}

// One 32-bit word of codes of four positions of a row: `y` holds x * (1/s) + 1.5 * 2^23 of the four.
// Eq. 1 without conversion instructions, bit-identical to quantize_code for |Z| <= 2^21: y carries rint(t) in its
// low mantissa bits (|t| < 2^22; a larger |t| ends at a clamp either way).  The lower clamp is taken on y (y >=
// 1.5 * 2^23 - Z means rint(t) + Z >= 0; NaN falls to the bound, hence to code 0, in fmaxf), then bits(y) -
// (0x4B400000 - Z) is the integer rint(t) + Z >= 0 and the upper clamp is the saturation of the packing
// instruction (8 bits) or an unsigned minimum.
template <bool CENTRED>
__device__ __forceinline__ uint32_t codes4(const float (&y)[4], float lowb, uint32_t off, uint32_t L, uint32_t sub) {
  uint32_t b[4];
#pragma unroll
  for (int i = 0; i < 4; ++i) b[i] = __float_as_uint(fmaxf(y[i], lowb)) - off;
  if (!CENTRED && L == 255u) {
    uint32_t hi, w;
    asm("cvt.pack.sat.u8.s32.b32 %0, %1, %2, %3;" : "=r"(hi) : "r"(b[3]), "r"(b[2]), "r"(0));
    asm("cvt.pack.sat.u8.s32.b32 %0, %1, %2, %3;" : "=r"(w) : "r"(b[1]), "r"(b[0]), "r"(hi));
    return w;
  }
#pragma unroll
  for (int i = 0; i < 4; ++i) b[i] = min(b[i], L) - (CENTRED ? sub : 0u);
  return __byte_perm(__byte_perm(b[0], b[1], 0x0040), __byte_perm(b[2], b[3], 0x0040), 0x5410);
}

// FAR: asks for the rows of the batch after the next one in L2.
template <bool DYNAMIC, bool CENTRED, bool WARP, bool FAR, bool SPREAD>
__global__ void __maxnreg__(72) quantize_act_kernel(const __grid_constant__ QuantArgs a) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int n_chunks = a.K_pad >> 4, n_cells = a.pairs * 2 * a.G;
  const int buf_bytes = a.pairs * a.pitch * 4;
  int* cell_lo = reinterpret_cast<int*>(smem_raw + buf_bytes);  // [2][n_cells]
  int* cell_hi = cell_lo + 2 * n_cells;
  const int tid = threadIdx.x, n_threads = blockDim.x;
  // Threads that share a row pair: all of the block, or (WARP) the warp that has the pair to itself.
  auto sync = [&]() {
    if (WARP) __syncwarp();
    else __syncthreads();
  };

  pdl_launch_dependents();
  // this thread's chunk: where its 16 values lie in an interleaved pair, its group, its padding positions
  const int my_pair = WARP ? tid >> 5 : tid / n_chunks, ch = WARP ? tid & 31 : tid - my_pair * n_chunks;
  const bool active = my_pair < a.pairs && ch < n_chunks;
  uint32_t off[16];  // shared-memory addresses
  uint32_t pm = 0;
  int g = 0;
  {
    const uint4* pp = reinterpret_cast<const uint4*>(a.perm) + (active ? ch : 0) * 2;
    const uint4 p0 = __ldg(pp), p1 = __ldg(pp + 1);
    const uint32_t pw[8] = {p0.x, p0.y, p0.z, p0.w, p1.x, p1.y, p1.z, p1.w};
    const uint32_t base = smem_u32(smem_raw) + (uint32_t)((active ? my_pair : 0) * a.pitch) * 4u;
#pragma unroll
    for (int i = 0; i < 16; ++i) {
      const int c = (int)(int16_t)(pw[i >> 1] >> (16 * (i & 1)));
      if (c < 0) pm |= 1u << i;
      off[i] = base + (uint32_t)qa_word<SPREAD>(c < 0 ? a.C : c) * 4u;
    }
    g = active ? __ldg(a.chunk_group + ch) : 0;
  }
  for (int i = tid; i < a.pairs; i += n_threads)
    *reinterpret_cast<uint32_t*>(smem_raw + ((size_t)i * a.pitch + qa_word<SPREAD>(a.C)) * 4) = 0x7FFF7FFFu;  // the word of NaN
  if (DYNAMIC)
    for (int i = tid; i < n_cells; i += n_threads) {
      cell_lo[i] = INT_MAX;
      cell_hi[i] = INT_MIN;
    }
  const int cell = my_pair * 2 * a.G + g;  // row 0 of the pair; row 1: + G
  const bool leads = active && (ch == 0 || __ldg(a.chunk_group + ch - 1) != g);  // the cell's first chunk
  bool one_cell = false;                   // every lane of the warp reduces into the same cell
  if (DYNAMIC) {
    const int first = __shfl_sync(0xffffffffu, cell, 0);
    one_cell = __all_sync(0xffffffffu, !active || cell == first);
  }
  // This thread's share of the row loads: at most two pieces of eight channels of a pair.  (With the requests to L2 there
  // are registers for one word, pair and piece, and the place in shared memory, which is then not worked out again.)
  const int vec = a.C >> 3;
  int lp[2], lv[2];
  bool lok[2];
  uint32_t place[2];
#pragma unroll
  for (int e = 0; e < 2; ++e) {
    const int task = tid + e * n_threads;
    lp[e] = WARP ? my_pair : task / vec;
    lv[e] = WARP ? (tid & 31) + 32 * e : task - lp[e] * vec;
    lok[e] = lp[e] < a.pairs && lv[e] < vec;
    if (FAR) {
      place[e] = (uint32_t)(lp[e] * a.pitch + qa_word<SPREAD>(lv[e] * 8)) * 4u;
      lp[e] = lok[e] ? lp[e] << 16 | lv[e] : -1;
    }
  }
  auto has = [&](int e) { return FAR ? lp[e] >= 0 : lok[e]; };
  auto pair_of = [&](int e) { return FAR ? lp[e] >> 16 : lp[e]; };
  auto piece_of = [&](int e) { return FAR ? lp[e] & 0xFFFF : lv[e]; };
  auto place_of = [&](int e) { return smem_raw + (FAR ? place[e] : (uint32_t)(lp[e] * a.pitch + qa_word<SPREAD>(lv[e] * 8)) * 4u); };
  float inv0 = 0.f, inv1 = 0.f;
  int z0 = 0, z1 = 0;
  if (!DYNAMIC && !a.row_group) {
    inv0 = inv1 = __ldg(a.inv_scale + g);
    z0 = z1 = __ldg(a.zp + g);
  }
  if (WARP) __syncthreads();  // the words of NaN and the cells are set
  pdl_wait();  // everything above reads only constants of the grouping; the rows may come from the previous kernel

  const int64_t rows_per_batch = 2 * (int64_t)a.pairs, step = rows_per_batch * gridDim.x;
  uint4 xa[2], xb[2];
  auto request = [&](int64_t row0) {
#pragma unroll
    for (int e = 0; e < 2; ++e) {
      const int64_t row = row0 + 2 * pair_of(e);
      if (has(e) && row < a.M) {
        const uint4* src = reinterpret_cast<const uint4*>(a.X + row * a.ld) + piece_of(e);
        xa[e] = __ldg(src);
        xb[e] = row + 1 < a.M ? __ldg(src + (a.ld >> 3)) : xa[e];
      }
    }
  };
  auto request_far = [&](int64_t row0) {  // one lane per 64 bytes of a row
#pragma unroll
    for (int e = 0; e < 2; ++e) {
      const int64_t row = row0 + 2 * pair_of(e);
      if (has(e) && row + 1 < a.M && (piece_of(e) & 3) == 0) {
        const uint4* src = reinterpret_cast<const uint4*>(a.X + row * a.ld) + piece_of(e);
        asm volatile("prefetch.global.L2 [%0];" ::"l"(src));
        asm volatile("prefetch.global.L2 [%0];" ::"l"(src + (a.ld >> 3)));
      }
    }
  };
  const int64_t first_row = (int64_t)blockIdx.x * rows_per_batch;
  if (first_row < a.M) request(first_row);
  int buf = 0;
  for (int64_t row0 = first_row; row0 < a.M; row0 += step, buf ^= 1) {
    // (dynamic: the barrier behind the ranges says so)
    if (!DYNAMIC && row0 != first_row) sync();  // every value of the last batch is in registers
#pragma unroll
    for (int e = 0; e < 2; ++e)
      if (has(e)) {
        uint4* dst = reinterpret_cast<uint4*>(place_of(e));
        dst[0] = make_uint4(__byte_perm(xa[e].x, xb[e].x, 0x5410), __byte_perm(xa[e].x, xb[e].x, 0x7632),
                            __byte_perm(xa[e].y, xb[e].y, 0x5410), __byte_perm(xa[e].y, xb[e].y, 0x7632));
        dst[1] = make_uint4(__byte_perm(xa[e].z, xb[e].z, 0x5410), __byte_perm(xa[e].z, xb[e].z, 0x7632),
                            __byte_perm(xa[e].w, xb[e].w, 0x5410), __byte_perm(xa[e].w, xb[e].w, 0x7632));
      }
    if (row0 + step < a.M) request(row0 + step);  // arrives while this batch is worked on
    if (FAR) request_far(row0 + 2 * step);
    sync();
    __half2 x[16];
#pragma unroll
    for (int i = 0; i < 16; ++i) {
      uint32_t v;
      asm volatile("ld.shared.b32 %0, [%1];" : "=r"(v) : "r"(off[i]));
      x[i] = *reinterpret_cast<const __half2*>(&v);
    }
    if (DYNAMIC) {
      __half2 lo = __hmin2(x[0], x[1]), hi = __hmax2(x[0], x[1]);  // NaN (padding, or a NaN input) never wins
#pragma unroll
      for (int i = 2; i < 16; ++i) {
        lo = __hmin2(lo, x[i]);
        hi = __hmax2(hi, x[i]);
      }
      const uint32_t lw = *reinterpret_cast<const uint32_t*>(&lo), hw = *reinterpret_cast<const uint32_t*>(&hi);
      int* c_lo = cell_lo + buf * n_cells;
      int* c_hi = cell_hi + buf * n_cells;
      int k[4] = {half_key(lw), half_key(lw >> 16), half_key(hw), half_key(hw >> 16)};
      const bool none0 = !active || (lw & 0x7FFFu) > 0x7C00u, none1 = !active || (lw & 0x7FFF0000u) > 0x7C000000u;
      if (none0) k[0] = INT_MAX, k[2] = INT_MIN;  // nothing but padding
      if (none1) k[1] = INT_MAX, k[3] = INT_MIN;
      if (one_cell) {
        k[0] = __reduce_min_sync(0xffffffffu, k[0]);
        k[1] = __reduce_min_sync(0xffffffffu, k[1]);
        k[2] = __reduce_max_sync(0xffffffffu, k[2]);
        k[3] = __reduce_max_sync(0xffffffffu, k[3]);
      }
      if (active && (!one_cell || (tid & 31) == 0)) {
        atomicMin(c_lo + cell, k[0]);
        atomicMin(c_lo + cell + a.G, k[1]);
        atomicMax(c_hi + cell, k[2]);
        atomicMax(c_hi + cell + a.G, k[3]);
      }
      sync();
      if (active) {
        // Every thread derives the parameters of its two cells itself: two more IEEE divisions per thread cost less
        // than a third barrier behind the few threads that would do it for all.
        float l0 = 0.f, h0 = 0.f, l1 = 0.f, h1 = 0.f, s0, s1;
        if (c_lo[cell] != INT_MAX) l0 = half_from_key(c_lo[cell]), h0 = half_from_key(c_hi[cell]);
        if (c_lo[cell + a.G] != INT_MAX) l1 = half_from_key(c_lo[cell + a.G]), h1 = half_from_key(c_hi[cell + a.G]);
        group_params(l0, h0, a.bits, s0, inv0, z0);
        group_params(l1, h1, a.bits, s1, inv1, z1);
        if (leads) {
          const int64_t o = (row0 + 2 * my_pair) * a.G + g;
          if (row0 + 2 * my_pair < a.M) {
            a.dyn_scale[o] = s0;
            a.dyn_zp[o] = z0;
          }
          if (row0 + 2 * my_pair + 1 < a.M) {
            a.dyn_scale[o + a.G] = s1;
            a.dyn_zp[o + a.G] = z1;
          }
          int* n_lo = cell_lo + (buf ^ 1) * n_cells + cell;  // for the next batch
          int* n_hi = cell_hi + (buf ^ 1) * n_cells + cell;
          n_lo[0] = n_lo[a.G] = INT_MAX;
          n_hi[0] = n_hi[a.G] = INT_MIN;
        }
      }
    }
    const int64_t row = row0 + 2 * my_pair;
    if (!active || row >= a.M) continue;
    const bool two = row + 1 < a.M;
    if (!DYNAMIC && a.row_group) {
      const int rg0 = __ldg(a.row_group + row % a.P) * a.G + g, rg1 = __ldg(a.row_group + (row + 1) % a.P) * a.G + g;
      inv0 = __ldg(a.inv_scale + rg0);
      z0 = __ldg(a.zp + rg0);
      inv1 = __ldg(a.inv_scale + rg1);
      z1 = __ldg(a.zp + rg1);
    }
    const uint32_t L = (1u << a.bits) - 1u;
    const uint32_t sub0 = CENTRED ? (uint32_t)z0 : 0u, sub1 = CENTRED ? (uint32_t)z1 : 0u;
    uint32_t w0[4], w1[4];
    if (abs(z0) <= (1 << 21) && abs(z1) <= (1 << 21)) {
      // product and sum rounded separately (x * (1/s) + (-0) is the rounded product, times one plus
      // 1.5 * 2^23 the rounded sum: an add in its place gets fused with the product), both rows per instruction
      const float MAGIC = 12582912.0f;
      const unsigned long long inv2 = pack_f32x2(inv0, inv1), magic2 = pack_f32x2(MAGIC, MAGIC);
      const unsigned long long nzero2 = pack_f32x2(-0.0f, -0.0f), one2 = pack_f32x2(1.0f, 1.0f);
      const float low0 = MAGIC - (float)z0, low1 = MAGIC - (float)z1;
      const uint32_t off0 = 0x4B400000u - (uint32_t)z0, off1 = 0x4B400000u - (uint32_t)z1;
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        float y0[4], y1[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          const float2 f = __half22float2(x[4 * q + i]);
          unpack_f32x2(fma_f32x2(fma_f32x2(pack_f32x2(f.x, f.y), inv2, nzero2), one2, magic2), y0[i], y1[i]);
        }
        w0[q] = codes4<CENTRED>(y0, low0, off0, L, sub0);
        w1[q] = codes4<CENTRED>(y1, low1, off1, L, sub1);
      }
    } else {
      const float Lf = (float)L, zf0 = (float)z0, zf1 = (float)z1;
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        w0[q] = w1[q] = 0;
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          const float2 f = __half22float2(x[4 * q + i]);
          w0[q] |= (((uint32_t)quantize_code(f.x, inv0, zf0, Lf) - sub0) & 0xFFu) << (8 * i);
          w1[q] |= (((uint32_t)quantize_code(f.y, inv1, zf1, Lf) - sub1) & 0xFFu) << (8 * i);
        }
      }
    }
    if (pm) {  // padding positions (NaN, so far code 0) carry the clamped zero-point (0 in the zero-centred layout)
      const uint32_t pad0 = (uint32_t)min(max(z0, 0), (int)L) * 0x01010101u, pad1 = (uint32_t)min(max(z1, 0), (int)L) * 0x01010101u;
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const uint32_t m = nibble_to_byte_mask(pm >> (4 * q));
        w0[q] = CENTRED ? w0[q] & ~m : w0[q] | (pad0 & m);
        w1[q] = CENTRED ? w1[q] & ~m : w1[q] | (pad1 & m);
      }
    }
    uint8_t* out = a.Xq + row * a.K_pad + ch * 16;
    *reinterpret_cast<uint4*>(out) = make_uint4(w0[0], w0[1], w0[2], w0[3]);
    if (two) *reinterpret_cast<uint4*>(out + a.K_pad) = make_uint4(w1[0], w1[1], w1[2], w1[3]);
  }
}

}  // namespace dgq

extern "C" dgq_status dgq_quantize_act(const dgq_groups* g, int timestep, int mode, int layout, const void* X,
                                       int64_t M, int64_t ld, void* Xq, float* dyn_scale, int32_t* dyn_zp,
                                       void* stream) {
  using namespace dgq;
  if (!g || !X || !Xq || M <= 0 || ld < g->C) return DGQ_ERR_INVALID_ARG;
  if (mode != DGQ_MODE_STATIC && mode != DGQ_MODE_DYNAMIC_TOKEN) return DGQ_ERR_INVALID_ARG;
  if (layout != DGQ_CODES_U8 && layout != DGQ_CODES_S8_CENTRED) return DGQ_ERR_INVALID_ARG;
  if (timestep < 0 || timestep >= g->T) return DGQ_ERR_INVALID_ARG;
  if (!aligned16(X) || !aligned16(Xq) || (ld % 8) != 0) return DGQ_ERR_ALIGNMENT;
  if ((g->C % 8) != 0) return DGQ_ERR_UNSUPPORTED;
  const int L = (1 << g->bits) - 1;
  const size_t trow = (size_t)timestep * g->R * g->G;
  if (mode == DGQ_MODE_STATIC) {
    if (!g->filled[timestep]) return DGQ_ERR_NOT_CALIBRATED;
    if (layout == DGQ_CODES_S8_CENTRED)
      for (int i = 0; i < g->R * g->G; ++i)
        if (g->zp[trow + i] > 128 || g->zp[trow + i] < L - 127) return DGQ_ERR_UNSUPPORTED;
  } else {
    if (!dyn_scale || !dyn_zp) return DGQ_ERR_INVALID_ARG;
    if (layout == DGQ_CODES_S8_CENTRED) return DGQ_ERR_UNSUPPORTED;
  }
  QuantArgs a;
  a.X = (const __half*)X;
  a.Xq = (uint8_t*)Xq;
  a.M = M;
  a.ld = ld;
  a.C = g->C;
  a.K_pad = g->K_pad;
  a.G = g->G;
  a.P = g->P;
  a.bits = g->bits;
  a.perm = g->d_perm;
  a.chunk_group = g->d_chunk_group;
  a.row_group = g->R > 1 ? g->d_row_group : nullptr;
  a.inv_scale = g->d_inv_scale + trow;
  a.zp = g->d_zp + trow;
  a.dyn_scale = dyn_scale;
  a.dyn_zp = dyn_zp;
  const bool dynamic = mode == DGQ_MODE_DYNAMIC_TOKEN;
  int n_sm = 0;
  DGQ_CUDA_OK(sm_count(&n_sm));
  // A block of about 128 threads, one per chunk of a batch (a single pair of a wide layer may need more), about 896
  // threads to an SM.  A matrix that would leave blocks without work gets smaller batches, down to one pair.
  const int n_chunks = g->K_pad / 16;
  const int64_t n_pairs = (M + 1) / 2;
  // Where the chunks of a pair nearly fill a warp, each warp has a pair to itself and the barriers of a batch are the
  // warp's own (32768 x 320 with 512 positions: 16.4 -> 15.4 us, static 11.5 -> 11.0).  Warp / block time, mean over 300 to 32768
  // rows: 32 chunks 0.98, 30 0.98, 28 0.99, 26 1.0, 24 1.0, 22 0.99, 20 1.02, 18 1.05, 16 1.16 (at 32768 rows 1.15 from 24 chunks down).
  const bool warp = n_chunks > 24 && n_chunks <= 32;
  const int per_pair = warp ? 32 : n_chunks;
  int pairs = std::max(1, 128 / per_pair);
  if (per_pair > 64) {
    // More chunks than half a block: 72 of them leave a quarter of three warps idle, three pairs fill 216 of 224 threads.  Of
    // one to three pairs the one with the most lanes at work, less 3 % for every warp that a barrier waits for, over all
    // rounds of the device (32768 x 960: 50.4 -> 46.8 us, x 1600: 73.9 -> 71.0, x 1920: 96.9 -> 92.2; x 1280 stays with one,
    // 56 against 61 us).
    double best = 0.;
    for (int p = 1; p <= 3; ++p) {
      const int warps = (p * per_pair + 31) / 32, blocks = 28 / warps;
      if (blocks == 0) break;
      const int64_t capacity = (int64_t)n_sm * blocks * p, rounds = (n_pairs + capacity - 1) / capacity;
      const double lanes = (double)(p * per_pair * blocks) * (33 - warps) * (double)n_pairs / (double)(rounds * capacity);
      if (lanes > best) best = lanes, pairs = p;
    }
  }
  int64_t slots = (int64_t)n_sm * std::max(1, 896 / (pairs * per_pair));
  if (n_pairs < slots * pairs) pairs = (int)std::max<int64_t>(1, (n_pairs + slots - 1) / slots);
  const int threads = (pairs * per_pair + 31) / 32 * 32;
  slots = (int64_t)n_sm * std::max(1, 896 / threads);
  // With many batches per block the rows of the batch after the next one are asked for in L2 as well (32768 x 2560: 125 ->
  // 115 us, 8192 x 3840: 46.0 -> 41.0, 8192 x 8000: 117 -> 101); with few the instructions cost more than that gives (8192 x 960,
  // three batches: 15.6 -> 16.1, 8192 x 1280, four: 17.2 -> 17.3, 32768 x 600, eight: 33.7 -> 34.3).
  const bool far = !warp && n_pairs > 8 * slots * pairs;
  // Where one group holds more than half of the layer (one group, static, 8192 x 2048: 29.1 -> 18.3 us, 32768 x 1280: 58.5 -> 35.5,
  // 8192 x 320: 5.3 -> 4.0 us; the instructions it costs take 1 to 2 % of a static pass over layers of several groups).
  int largest = 0;
  for (int k = 0; k < g->G; ++k) largest = std::max(largest, g->group_off[k + 1] - g->group_off[k]);
  const bool spread = 2 * largest > g->K_pad;
  a.pitch = qa_pitch(g->C, spread);
  a.pairs = pairs;
  const size_t smem = qa_smem_bytes(pairs, a.pitch, g->G, dynamic);
  static std::atomic<bool> attr_set[64];
  int dev = 0;
  DGQ_CUDA_OK(cudaGetDevice(&dev));
  if (dev >= 64 || !attr_set[dev].load()) {
    auto opt_in = [](auto f, auto s) {
      constexpr bool F = decltype(f)::value, S = decltype(s)::value;
      for (auto k : {quantize_act_kernel<true, false, false, F, S>, quantize_act_kernel<false, false, false, F, S>,
                     quantize_act_kernel<false, true, false, F, S>}) {
        const cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, QA_SMEM_MAX);
        if (e != cudaSuccess) return e;
      }
      return cudaSuccess;
    };
    const std::false_type no;
    const std::true_type yes;
    DGQ_CUDA_OK(opt_in(no, no));
    DGQ_CUDA_OK(opt_in(no, yes));
    DGQ_CUDA_OK(opt_in(yes, no));
    DGQ_CUDA_OK(opt_in(yes, yes));
    if (dev < 64) attr_set[dev].store(true);
  }
  const int grid = (int)std::min<int64_t>((n_pairs + pairs - 1) / pairs, slots);
  const bool centred = layout == DGQ_CODES_S8_CENTRED;
  auto pick = [&](auto w, auto f, auto s) {
    constexpr bool W = decltype(w)::value, F = decltype(f)::value, S = decltype(s)::value;
    return dynamic ? quantize_act_kernel<true, false, W, F, S>
                   : centred ? quantize_act_kernel<false, true, W, F, S> : quantize_act_kernel<false, false, W, F, S>;
  };
  auto pick_spread = [&](auto w, auto f) { return spread ? pick(w, f, std::true_type{}) : pick(w, f, std::false_type{}); };
  auto kernel = warp ? pick_spread(std::true_type{}, std::false_type{})
                     : far ? pick_spread(std::false_type{}, std::true_type{}) : pick_spread(std::false_type{}, std::false_type{});
  DGQ_CUDA_OK(launch_pdl(kernel, dim3(grid), dim3(threads), smem,
                         (cudaStream_t)stream, a));
  g_launches += 1;
  DGQ_CUDA_OK(cudaGetLastError());
  return DGQ_OK;
}
