// eco_params.cu -- whole agents' parameters: the founders' weights (Sec.
// 3.3: Kaiming-style initial weights, zero biases), the parameters a caller
// writes (both with their streamed BF16 / FP8 copy), and the parameters a
// caller reads.
//
// The logical order (the order of the Philox draws) holds a layer's weights
// by output row, the tiled block by input, so a layer is a transposition.
// A CTA takes one slot at a time and walks its layers in tiles of R output
// rows, all inputs of a row at once (an FP8 row's scale needs them all): the
// tile enters shared memory in logical order and leaves in physical order,
// 32 consecutive elements per warp store.  A Philox block gives four normals
// and each is used (drawing a block per element cost four times the Philox
// work), and the streamed copy is written from the tile instead of reading
// the masters back.
#include "eco_internal.cuh"
#include "eco_kernels.h"

#include <cuda_bf16.h>
#include <cuda_fp8.h>

namespace eco {

namespace {

constexpr int kParThreads = 512;
constexpr int kMaxRows = 32;

// Row stride of a tile of rows of nin inputs.  The tile is read four rows per
// lane, eight lanes to an input (32-row tiles), so rows four apart should
// differ by an odd multiple of 4 banks: rows of an odd length (every D of
// 3 k^2 + 4 or 8) stay packed, in logical order with the first Philox block's
// offset.  Rows of a multiple of 4 are padded by 2, an odd multiple of 8
// banks (two lanes per bank), and still take a block's normals as pairs.
__host__ __device__ inline bool tile_by4(int nin) { return (nin & 3) == 0; }
__host__ __device__ inline int tile_stride(int nin) { return tile_by4(nin) ? nin + 2 : nin; }

size_t tile_bytes(const Layout &L, int rows) {
  // k_params_in's row strides and k_params_out's
  const int nin[2] = {L.D, L.H};
  int widest = 0;
  for (int k = 0; k < 2; ++k) {
    const int a = tile_stride(nin[k]), b = nin[k] | 1;
    widest = a > widest ? a : widest;
    widest = b > widest ? b : widest;
  }
  return 4 * ((size_t)rows * widest + 8);
}

// Output rows per tile: whole 32-row tiles (128-byte stores) where they fit
// 100 KB, that is two CTAs per SM, else 16 or 8 (D up to 3,860).
int tile_rows(const Layout &L) {
  for (int r = kMaxRows; r > 8; r >>= 1)
    if (tile_bytes(L, r) <= 100 * 1024) return r;
  return 8;
}

__device__ __forceinline__ uint32_t fp8_code(float v) {
  return (uint32_t)__nv_cvt_float_to_fp8(v, __NV_SATFINITE, __NV_E4M3);
}

__device__ __forceinline__ float fp8_scale(float mx) {
  const float s = __fdiv_rn(mx, 448.0f);
  return s == 0.0f ? 1.0f : s;
}

// Philox4x32-10 of counter (c0, c1, 0, 0) under round keys made once (the
// same key serves a whole agent; the key schedule was a quarter of the
// generator's instructions).
struct PhiloxKeys {
  uint32_t k0[10], k1[10];
  __device__ __forceinline__ PhiloxKeys(uint32_t a, uint32_t b) {
#pragma unroll
    for (int i = 0; i < 10; ++i) {
      k0[i] = a + (uint32_t)i * 0x9E3779B9u;
      k1[i] = b + (uint32_t)i * 0xBB67AE85u;
    }
  }
  __device__ __forceinline__ U4 draw(uint32_t c0, uint32_t c1) const {
    uint32_t c2 = 0u, c3 = 0u;
#pragma unroll
    for (int i = 0; i < 10; ++i) {
      const uint32_t a0 = 0xD2511F53u * c0, h0 = __umulhi(0xD2511F53u, c0);
      const uint32_t a2 = 0xCD9E8D57u * c2, h2 = __umulhi(0xCD9E8D57u, c2);
      c0 = h2 ^ c1 ^ k0[i];
      c1 = a2;
      c2 = h0 ^ c3 ^ k1[i];
      c3 = a0;
    }
    return U4{c0, c1, c2, c3};
  }
};

// n / f correctly rounded, f = sqrt(fan-in) with its correctly rounded
// reciprocal r: one correction of the quotient n r (Markstein, "Computation
// of elementary functions on the IBM RISC System/6000 processor", 1990;
// Brisebarre, Muller and Raina, IEEE TC 53(8), 2004, on divisors known in
// advance).  Equal to the IEEE quotient for every significand of n and every
// fan-in the configuration allows, checked exhaustively; n is 0 or of normal
// magnitude, so no scaling is needed.
__device__ __forceinline__ float divide_by_known(float n, float f, float r) {
  const float q = n * r;
  return fmaf(fmaf(-q, f, n), r, q);
}

}  // namespace

// Parameters of slots [slot0, slot0 + n) into their blocks, with the streamed
// copy (BF16 elementwise RNE; FP8 per output row, scale = max|w| / 448,
// satfinite RNE codes; biases FP32).
//
// INIT, the founders' weights: weight p = N(0,1) * sqrt(gain / fan_in) from
// stream W_INIT at counter (local slot, p / 4), gain 1 for the plain (tanh)
// form and 2 for the paper (ReLU) form; biases and tau zero; every other slot
// all zero, with FP8 scales of 1.
// Bound by the arithmetic of the normals beside the writes: 65,536 slots of
// 371-64-64-9 BF16 are 11.2 GB, 1.7 ms at the copy rate, and the whole reset
// takes 3.8 ms (19.4 ms with a Philox block per element, the streamed copy
// from a second pass over the masters and one CTA per world placing the
// founders; 4.6 ms with the key schedule in every block, an IEEE division per
// weight and one row per lane); 683-128-128-9 FP8, 41.5 GB, 16.6 ms (231 ms,
// mostly FP8 rows read with a stride; 19 ms).  512 threads at 64 registers:
// 256 or 512 threads with 2 to 6 CTAs per SM lie within 5% in BF16, and up to
// 30% above in FP8.
//
// Otherwise: from `flat`, [n][P] in logical order, the caller's parameters
// on the device.
template <int PREC, bool INIT>
__global__ void __launch_bounds__(kParThreads, 2)
    k_params_in(Dev d, Layout L, int R, int rlog, int slot0, int n, const float *__restrict__ flat) {
  extern __shared__ __align__(16) float tile[];
  __shared__ uint32_t s_max[kMaxRows];
  __shared__ float s_scale[kMaxRows];
  const int D = L.D, H = L.H, A = L.A;
  const int tid = threadIdx.x, nt = kParThreads, lane = tid & 31, warp = tid >> 5, nw = nt >> 5;
  const int64_t mper = L.mstride / 4;
  // the scale of each fan-in (layout_fan_in), once per CTA: in the paper form
  // a factor, in the plain form (two fan-ins, D and H) a divisor
  auto scale_of = [&](int q) {
    const float fan = (float)layout_fan_in(L, q);
    return L.relu ? sqrtf(__fdiv_rn(2.0f, fan)) : sqrtf(fan);
  };
  const float f_vision = scale_of(0), f_internal = scale_of(L.patch * H), f_compass = scale_of((L.patch + 1) * H);
  const float f_hidden = scale_of(D * H);
  const float r_in = __frcp_rn(f_vision), r_hidden = __frcp_rn(f_hidden);
  for (int i = blockIdx.x; i < n; i += gridDim.x) {
    const int s = slot0 + i;
    const float *in = INIT ? nullptr : flat + (int64_t)i * L.P;
    const EnvDesc ed = d.env[d.env_of[s]];
    const uint32_t ls = (uint32_t)(s - ed.slot_off);
    float *m = d.master + (int64_t)s * mper;
    uint8_t *blk = d.wq + (int64_t)s * L.stride;
    if (INIT && (int)ls >= ed.init_alive) {  // an empty slot
      const uint4 z = make_uint4(0u, 0u, 0u, 0u);
      for (int k = tid; k < (int)(mper / 4); k += nt) reinterpret_cast<uint4 *>(m)[k] = z;
      if (PREC != PREC_FP32)
        for (int k = tid; k < (int)(L.stride / 16); k += nt) reinterpret_cast<uint4 *>(blk)[k] = z;
      if (PREC == PREC_FP8) {
        __syncthreads();
        for (int k = tid; k < H + L.L * H + A; k += nt) reinterpret_cast<float *>(blk + L.off_scale)[k] = 1.0f;
      }
      continue;
    }
    for (int layer = 0; layer <= L.L; ++layer) {
      const int nin = layer == 0 ? D : H;
      const int rs = tile_stride(nin);
      const bool by4 = tile_by4(nin);
      const int qbase = layer == 0 ? 0 : D * H + (layer - 1) * H * H;
      const int lrow0 = layer == 0 ? 0 : D * H + L.ns * H + (layer - 1) * (H * H + H);
      for (int o0 = 0; o0 < H; o0 += R) {
        // 1. the rows (INIT: their normals), in logical order
        const int lbase = lrow0 + o0 * nin, nel = R * nin;
        const int shift = INIT && !by4 ? lbase & 3 : 0;  // rows of a multiple of 4 start a block
        if (INIT) {
          const int b0 = lbase >> 2, b1 = (lbase + nel - 1) >> 2;
          const PhiloxKeys keys(ed.seed, S_W_INIT);
          for (int g = b0 + tid; g <= b1; g += nt) {
            float n4[4];
            normals4(keys.draw(ls, (uint32_t)g), n4);
            int at = 4 * (g - b0);
            if (by4) {
              at += (at / nin) * (rs - nin);
              *reinterpret_cast<float2 *>(tile + at) = make_float2(n4[0], n4[1]);
              *reinterpret_cast<float2 *>(tile + at + 2) = make_float2(n4[2], n4[3]);
            } else {
              *reinterpret_cast<float4 *>(tile + at) = make_float4(n4[0], n4[1], n4[2], n4[3]);
            }
          }
        } else {
          for (int rr = warp; rr < R; rr += nw)
            for (int j = lane; j < nin; j += 32) tile[rr * rs + j] = in[lbase + rr * nin + j];
        }
        if (PREC == PREC_FP8 && tid < R) s_max[tid] = 0u;
        __syncthreads();
        // 2. (INIT: scaled) to the master and the BF16 copy: a lane takes four
        // rows of one input
        const int wlog = rlog - 2, wd = lane & ((1 << wlog) - 1), per = 32 >> wlog;
        float *row = tile + shift + 4 * wd * rs;
        float mx[4] = {0.0f, 0.0f, 0.0f, 0.0f};
        for (int j = warp * per + (lane >> wlog); j < nin; j += nw * per) {
          float v[4];
#pragma unroll
          for (int k = 0; k < 4; ++k) v[k] = row[k * rs + j];
          if (INIT) {
            if (L.relu) {
              const float f = layer > 0 ? f_hidden : j < L.patch ? f_vision
                              : (j > L.patch && j < L.patch + 5) ? f_compass : f_internal;
#pragma unroll
              for (int k = 0; k < 4; ++k) v[k] *= f;
            } else {
              const float f = layer > 0 ? f_hidden : f_vision, r = layer > 0 ? r_hidden : r_in;
#pragma unroll
              for (int k = 0; k < 4; ++k) v[k] = divide_by_known(v[k], f, r);
            }
          }
          const int q = qbase + j * H + o0 + 4 * wd;
          *reinterpret_cast<float4 *>(m + q) = make_float4(v[0], v[1], v[2], v[3]);
          if (PREC == PREC_BF16) {
            const __nv_bfloat162 lo = __floats2bfloat162_rn(v[0], v[1]), hi = __floats2bfloat162_rn(v[2], v[3]);
            *reinterpret_cast<uint2 *>(reinterpret_cast<__nv_bfloat16 *>(blk) + q) =
                make_uint2(*reinterpret_cast<const uint32_t *>(&lo), *reinterpret_cast<const uint32_t *>(&hi));
          }
          if (PREC == PREC_FP8) {
#pragma unroll
            for (int k = 0; k < 4; ++k) {
              if (INIT) row[k * rs + j] = v[k];
              mx[k] = fmaxf(mx[k], fabsf(v[k]));
            }
          }
        }
        if (PREC == PREC_FP8) {
          // non-negative floats compare as their bits
#pragma unroll
          for (int k = 0; k < 4; ++k) atomicMax(&s_max[4 * wd + k], __float_as_uint(mx[k]));
          __syncthreads();
          if (tid < R) {
            const float sc = fp8_scale(__uint_as_float(s_max[tid]));
            s_scale[tid] = sc;
            reinterpret_cast<float *>(blk + L.off_scale)[(layer == 0 ? 0 : H + (layer - 1) * H) + o0 + tid] = sc;
          }
          __syncthreads();
          // 3. the codes, four rows per word
          const int words = R >> 2;
          for (int i = tid; i < nin * words; i += nt) {
            const int w = i & (words - 1), j = i >> (rlog - 2);
            uint32_t code = 0u;
#pragma unroll
            for (int k = 0; k < 4; ++k)
              code |= fp8_code(__fdiv_rn(tile[shift + (4 * w + k) * rs + j], s_scale[4 * w + k])) << (8 * k);
            *reinterpret_cast<uint32_t *>(blk + qbase + j * H + o0 + 4 * w) = code;
          }
        }
        __syncthreads();  // the tile is reused
      }
    }
    // the head (its physical order is the logical one): a warp per row
    const int q3 = D * H + L.L * H * H, out0 = D * H + L.ns * H + L.L * (H * H + H);
    for (int a = warp; a < A; a += nw) {
      float v[4] = {0.0f, 0.0f, 0.0f, 0.0f};
      if (lane < (H >> 2)) {
        if (INIT) {
          normals4(philox(ls, (uint32_t)((out0 + a * H) >> 2) + lane, 0u, 0u, ed.seed, S_W_INIT), v);
#pragma unroll
          for (int k = 0; k < 4; ++k) v[k] = L.relu ? v[k] * f_hidden : __fdiv_rn(v[k], f_hidden);
        } else {
#pragma unroll
          for (int k = 0; k < 4; ++k) v[k] = in[out0 + a * H + 4 * lane + k];
        }
        const int q = q3 + a * H + 4 * lane;
        *reinterpret_cast<float4 *>(m + q) = make_float4(v[0], v[1], v[2], v[3]);
        if (PREC == PREC_BF16)
#pragma unroll
          for (int k = 0; k < 4; ++k) reinterpret_cast<__nv_bfloat16 *>(blk)[q + k] = __float2bfloat16_rn(v[k]);
      }
      if (PREC == PREC_FP8) {
        float mx = fmaxf(fmaxf(fabsf(v[0]), fabsf(v[1])), fmaxf(fabsf(v[2]), fabsf(v[3])));
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xFFFFFFFFu, mx, off));
        const float sc = fp8_scale(mx);
        if (lane == 0) reinterpret_cast<float *>(blk + L.off_scale)[H + L.L * H + a] = sc;
        if (lane < (H >> 2)) {
          uint32_t code = 0u;
#pragma unroll
          for (int k = 0; k < 4; ++k) code |= fp8_code(__fdiv_rn(v[k], sc)) << (8 * k);
          *reinterpret_cast<uint32_t *>(blk + q3 + a * H + 4 * lane) = code;
        }
      }
    }
    // biases (and tau), and the block's padding
    for (int k = tid; k < (int)mper - L.nW; k += nt) {
      const float v = !INIT && k < L.nB ? in[layout_logical(L, L.nW + k)] : 0.0f;
      m[L.nW + k] = v;
      if (PREC != PREC_FP32 && k < L.nB) reinterpret_cast<float *>(blk + L.off_bias)[k] = v;
    }
  }
}

// The masters of slots [slot0, slot0 + n) to `flat`, [n][P] in logical
// order: the same tiles the other way, rows of an odd stride, so that 32
// lanes writing one input of 32 rows hit 32 banks.
__global__ void __launch_bounds__(kParThreads, 2)
    k_params_out(Dev d, Layout L, int R, int rlog, int slot0, int n, float *__restrict__ flat) {
  extern __shared__ __align__(16) float tile[];
  const int D = L.D, H = L.H;
  const int tid = threadIdx.x, nt = kParThreads, lane = tid & 31, warp = tid >> 5, nw = nt >> 5;
  const int64_t mper = L.mstride / 4;
  for (int i = blockIdx.x; i < n; i += gridDim.x) {
    const float *m = d.master + (int64_t)(slot0 + i) * mper;
    float *out = flat + (int64_t)i * L.P;
    for (int layer = 0; layer <= L.L; ++layer) {
      const int nin = layer == 0 ? D : H, rs = nin | 1;
      const int qbase = layer == 0 ? 0 : D * H + (layer - 1) * H * H;
      const int lrow0 = layer == 0 ? 0 : D * H + L.ns * H + (layer - 1) * (H * H + H);
      for (int o0 = 0; o0 < H; o0 += R) {
        const int rr = lane & (R - 1), sub = lane >> rlog, per = 32 >> rlog;
#pragma unroll 4
        for (int j = warp * per + sub; j < nin; j += nw * per) tile[rr * rs + j] = m[qbase + j * H + o0 + rr];
        __syncthreads();
        for (int r = warp; r < R; r += nw)
          for (int j = lane; j < nin; j += 32) out[lrow0 + (o0 + r) * nin + j] = tile[r * rs + j];
        __syncthreads();  // the tile is reused
      }
    }
    // the head, the biases and tau
    const int q3 = D * H + L.L * H * H;
    for (int q = q3 + tid; q < L.P; q += nt) out[layout_logical(L, q)] = m[q];
  }
}

// Launch of one of the tiled kernels over n slots: every CTA that fits.
template <class K, class F>
static cudaError_t launch_tiled(K *kernel, const Dev &d, const Layout &L, int slot0, int n, F flat, cudaStream_t s) {
  if (n <= 0) return cudaSuccess;
  const int rows = tile_rows(L);
  int rlog = 3;
  while ((1 << rlog) < rows) ++rlog;
  const size_t smem = tile_bytes(L, rows);
  cudaError_t e = allow_dynamic_smem((const void *)kernel, smem);
  if (e != cudaSuccess) return e;
  int dev = 0, sms = 0, per_sm = 0;
  if ((e = cudaGetDevice(&dev)) != cudaSuccess) return e;
  if ((e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess) return e;
  if ((e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, (const void *)kernel, kParThreads, smem)) !=
      cudaSuccess)
    return e;
  if (per_sm < 1) return cudaErrorInvalidConfiguration;
  kernel<<<n < sms * per_sm ? n : sms * per_sm, kParThreads, smem, s>>>(d, L, rows, rlog, slot0, n, flat);
  return cudaGetLastError();
}

template <bool INIT>
static cudaError_t params_in(const Dev &d, const Layout &L, const Rules &R, int slot0, int n, const float *flat,
                             cudaStream_t s) {
  if (R.precision == PREC_FP32) return launch_tiled(k_params_in<PREC_FP32, INIT>, d, L, slot0, n, flat, s);
  if (R.precision == PREC_BF16) return launch_tiled(k_params_in<PREC_BF16, INIT>, d, L, slot0, n, flat, s);
  return launch_tiled(k_params_in<PREC_FP8, INIT>, d, L, slot0, n, flat, s);
}

cudaError_t launch_init_params(const Dev &d, const Layout &L, const Rules &R, cudaStream_t s) {
  return params_in<true>(d, L, R, 0, d.total_slots, nullptr, s);
}

cudaError_t launch_params_in(const Dev &d, const Layout &L, const Rules &R, int slot0, int n, const float *flat,
                             cudaStream_t s) {
  return params_in<false>(d, L, R, slot0, n, flat, s);
}

cudaError_t launch_params_out(const Dev &d, const Layout &L, int slot0, int n, float *flat, cudaStream_t s) {
  return launch_tiled(k_params_out, d, L, slot0, n, flat, s);
}

}  // namespace eco
