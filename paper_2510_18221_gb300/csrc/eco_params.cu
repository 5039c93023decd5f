// eco_params.cu -- whole agents' parameters: the founders' weights (Sec.
// 3.3: Kaiming-style initial weights, zero biases) with their streamed
// BF16 / FP8 copy, and the re-derivation of the streamed copy from the FP32
// masters.
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

// Row stride of a tile of rows of nin inputs.  Rows whose length is a
// multiple of 4 are padded to an odd number of 16-byte units, so that 32
// lanes reading the same unit of their own rows as float4 hit every bank
// once per quarter-warp.  Other rows (every D of 3 k^2 + 4 or 8 is odd) stay
// packed, in logical order with the first Philox block's offset, and are
// read element by element, one bank per lane when nin is odd.
__host__ __device__ inline bool tile_by4(int nin) { return (nin & 3) == 0; }
__host__ __device__ inline int tile_stride(int nin) { return tile_by4(nin) && ((nin >> 2) & 1) == 0 ? nin + 4 : nin; }

size_t tile_bytes(const Layout &L, int rows) {
  const int a = tile_stride(L.D), b = tile_stride(L.H);
  return 4 * ((size_t)rows * (a > b ? a : b) + 8);
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

}  // namespace

// Founders' weights: weight p = N(0,1) * sqrt(gain / fan_in) from stream
// W_INIT at counter (local slot, p / 4), gain 1 for the plain (tanh) form and
// 2 for the paper (ReLU) form; biases and tau zero; every other slot all
// zero, with FP8 scales of 1.  PREC: the streamed copy derived with them
// (BF16 elementwise RNE; FP8 per output row, scale = max|w| / 448, satfinite
// RNE codes).
//
// Bound by the arithmetic of the normals beside the writes: 65,536 slots of
// 371-64-64-9 BF16 are 11.2 GB, 1.7 ms at the copy rate, and the whole reset
// takes 4.6 ms (19.4 ms with a Philox block per element, the streamed copy
// from a second pass over the masters and one CTA per world placing the
// founders); 683-128-128-9 FP8, 41.5 GB, 19 ms (231 ms, mostly FP8 rows read
// with a stride).  512 threads at 64 registers: 256 or 512 threads with 2 to
// 6 CTAs per SM lie within 5% in BF16, and up to 30% above in FP8.
template <int PREC>
__global__ void __launch_bounds__(kParThreads, 2) k_init_params(Dev d, Layout L, int R, int rlog) {
  extern __shared__ __align__(16) float tile[];
  __shared__ uint32_t s_max[kMaxRows];
  __shared__ float s_scale[kMaxRows];
  const int D = L.D, H = L.H, A = L.A;
  const int tid = threadIdx.x, nt = kParThreads, lane = tid & 31, warp = tid >> 5, nw = nt >> 5;
  const int64_t mper = L.mstride / 4;
  // the scale of each fan-in (layout_fan_in), once per CTA: a factor in the
  // paper form, a divisor in the plain form
  auto scale_of = [&](int q) {
    const float fan = (float)layout_fan_in(L, q);
    return L.relu ? sqrtf(__fdiv_rn(2.0f, fan)) : sqrtf(fan);
  };
  const float f_vision = scale_of(0), f_internal = scale_of(L.patch * H), f_compass = scale_of((L.patch + 1) * H);
  const float f_hidden = scale_of(D * H);
  for (int s = blockIdx.x; s < d.total_slots; s += gridDim.x) {
    const EnvDesc ed = d.env[d.env_of[s]];
    const uint32_t ls = (uint32_t)(s - ed.slot_off);
    float *m = d.master + (int64_t)s * mper;
    uint8_t *blk = d.wq + (int64_t)s * L.stride;
    if ((int)ls >= ed.init_alive) {  // an empty slot
      const uint4 z = make_uint4(0u, 0u, 0u, 0u);
      for (int i = tid; i < (int)(mper / 4); i += nt) reinterpret_cast<uint4 *>(m)[i] = z;
      if (PREC != PREC_FP32)
        for (int i = tid; i < (int)(L.stride / 16); i += nt) reinterpret_cast<uint4 *>(blk)[i] = z;
      if (PREC == PREC_FP8) {
        __syncthreads();
        for (int i = tid; i < H + L.L * H + A; i += nt) reinterpret_cast<float *>(blk + L.off_scale)[i] = 1.0f;
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
        // 1. the rows' normals, in logical order
        const int lbase = lrow0 + o0 * nin, nel = R * nin;
        const int b0 = lbase >> 2, b1 = (lbase + nel - 1) >> 2;
        const int shift = by4 ? 0 : lbase & 3;  // rows of a multiple of 4 start a block
        for (int g = b0 + tid; g <= b1; g += nt) {
          float n4[4];
          normals4(philox(ls, (uint32_t)g, 0u, 0u, ed.seed, S_W_INIT), n4);
          int at = 4 * (g - b0);
          if (by4) {
            const int rr = at / nin;
            at += rr * (rs - nin);
          }
          *reinterpret_cast<float4 *>(tile + at) = make_float4(n4[0], n4[1], n4[2], n4[3]);
        }
        if (PREC == PREC_FP8 && tid < R) s_max[tid] = 0u;
        __syncthreads();
        // 2. scaled, to the master (and the BF16 copy): lane = row
        const int rr = lane & (R - 1), sub = lane >> rlog, per = 32 >> rlog;
        float *row = tile + shift + rr * rs;
        float mx = 0.0f;
        auto put = [&](int j, float n) -> float {
          const int q = qbase + j * H + o0 + rr;
          const float f = layer > 0 ? f_hidden : j < L.patch ? f_vision
                          : (j > L.patch && j < L.patch + 5) ? f_compass : f_internal;
          const float v = L.relu ? n * f : __fdiv_rn(n, f);
          m[q] = v;
          if (PREC == PREC_BF16) reinterpret_cast<__nv_bfloat16 *>(blk)[q] = __float2bfloat16_rn(v);
          if (PREC == PREC_FP8) mx = fmaxf(mx, fabsf(v));
          return v;
        };
        if (by4) {
          for (int c = warp * per + sub; c < (nin >> 2); c += nw * per) {
            float4 v = *reinterpret_cast<const float4 *>(row + 4 * c);
            v.x = put(4 * c, v.x);
            v.y = put(4 * c + 1, v.y);
            v.z = put(4 * c + 2, v.z);
            v.w = put(4 * c + 3, v.w);
            if (PREC == PREC_FP8) *reinterpret_cast<float4 *>(row + 4 * c) = v;
          }
        } else {
          for (int j = warp * per + sub; j < nin; j += nw * per) {
            const float v = put(j, row[j]);
            if (PREC == PREC_FP8) row[j] = v;
          }
        }
        if (PREC == PREC_FP8) {
          // non-negative floats compare as their bits
          atomicMax(&s_max[rr], __float_as_uint(mx));
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
        normals4(philox(ls, (uint32_t)((out0 + a * H) >> 2) + lane, 0u, 0u, ed.seed, S_W_INIT), v);
#pragma unroll
        for (int k = 0; k < 4; ++k) v[k] = L.relu ? v[k] * f_hidden : __fdiv_rn(v[k], f_hidden);
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
    for (int q = L.nW + tid; q < (int)mper; q += nt) m[q] = 0.0f;
    if (PREC != PREC_FP32)
      for (int k = tid; k < L.nB; k += nt) reinterpret_cast<float *>(blk + L.off_bias)[k] = 0.0f;
  }
}

// Streamed copy of slots [slot0, slot0 + n) from their masters: BF16
// elementwise (RNE), FP8 per output row, biases FP32.
__global__ void k_requant_bf16(Dev d, Layout L, int slot0, int n) {
  const int nW = L.nW;
  const int per = L.nW + L.nB;
  const int64_t total = (int64_t)n * per;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < total;
       i += (int64_t)gridDim.x * blockDim.x) {
    const int s = slot0 + (int)(i / per);
    const int q = (int)(i % per);
    const float *m = d.master + (int64_t)s * (L.mstride / 4);
    uint8_t *blk = d.wq + (int64_t)s * L.stride;
    if (q < nW) {
      reinterpret_cast<__nv_bfloat16 *>(blk)[q] = __float2bfloat16_rn(m[q]);
    } else {
      reinterpret_cast<float *>(blk + L.off_bias)[q - nW] = m[L.moff_bias / 4 + (q - nW)];
    }
  }
}

__global__ void k_requant_fp8(Dev d, Layout L, int slot0, int n) {
  const int H = L.H, rows = H + L.L * H + L.A;
  const int lane = threadIdx.x & 31;
  // biases (and tau) are copied unchanged
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < (int64_t)n * L.nB;
       i += (int64_t)gridDim.x * blockDim.x) {
    const int s = slot0 + (int)(i / L.nB), k = (int)(i % L.nB);
    reinterpret_cast<float *>(d.wq + (int64_t)s * L.stride + L.off_bias)[k] =
        d.master[(int64_t)s * (L.mstride / 4) + L.moff_bias / 4 + k];
  }
  const int64_t warps = (int64_t)n * rows;
  for (int64_t w = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; w < warps;
       w += ((int64_t)gridDim.x * blockDim.x) >> 5) {
    const int s = slot0 + (int)(w / rows);
    const int row = (int)(w % rows);
    const float *m = d.master + (int64_t)s * (L.mstride / 4);
    uint8_t *blk = d.wq + (int64_t)s * L.stride;
    int base, stride, cnt;
    if (row < H) {  // W_in row o: elements (j, o), j < D
      base = row; stride = H; cnt = L.D;
    } else if (row < H + L.L * H) {  // hidden layer l, row o
      const int l = (row - H) / H, o = (row - H) - l * H;
      base = L.D * H + l * H * H + o; stride = H; cnt = H;
    } else {  // head row a
      base = L.D * H + L.L * H * H + (row - H - L.L * H) * H; stride = 1; cnt = H;
    }
    float mx = 0.0f;
    for (int j = lane; j < cnt; j += 32) mx = fmaxf(mx, fabsf(m[base + j * stride]));
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xFFFFFFFFu, mx, off));
    const float sc = fp8_scale(mx);
    for (int j = lane; j < cnt; j += 32) {
      const int idx = base + j * stride;
      blk[idx] = (uint8_t)fp8_code(__fdiv_rn(m[idx], sc));
    }
    if (lane == 0) reinterpret_cast<float *>(blk + L.off_scale)[row] = sc;
  }
}

cudaError_t launch_requant(const Dev &d, const Layout &L, const Rules &R, int slot0, int n,
                           cudaStream_t s) {
  if (R.precision == PREC_FP32 || n <= 0) return cudaSuccess;
  if (R.precision == PREC_BF16) {
    const long long work = (long long)n * (L.nW + L.nB);
    k_requant_bf16<<<grid_for(work, 256, 152 * 32), 256, 0, s>>>(d, L, slot0, n);
  } else {
    const long long work = (long long)n * (L.H + L.L * L.H + L.A) * 32;
    k_requant_fp8<<<grid_for(work, 256, 152 * 32), 256, 0, s>>>(d, L, slot0, n);
  }
  return cudaGetLastError();
}

// Launch of one of the tiled kernels: `rows` rows of shared memory, every
// CTA that fits.
template <class K, class... Args>
static cudaError_t launch_tiled(K *kernel, const Layout &L, int rows, int slots, cudaStream_t s, Args... args) {
  const size_t smem = tile_bytes(L, rows);
  cudaError_t e = cudaFuncSetAttribute((const void *)kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  int dev = 0, sms = 0, per_sm = 0;
  if ((e = cudaGetDevice(&dev)) != cudaSuccess) return e;
  if ((e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess) return e;
  if ((e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, (const void *)kernel, kParThreads, smem)) !=
      cudaSuccess)
    return e;
  if (per_sm < 1) return cudaErrorInvalidConfiguration;
  kernel<<<grid_for((long long)slots * kParThreads, kParThreads, sms * per_sm), kParThreads, smem, s>>>(args...);
  return cudaGetLastError();
}

static int log2_of(int v) {
  int k = 0;
  while ((1 << k) < v) ++k;
  return k;
}

cudaError_t launch_init_params(const Dev &d, const Layout &L, const Rules &R, cudaStream_t s) {
  const int rows = tile_rows(L), rlog = log2_of(rows);
  if (R.precision == PREC_FP32) return launch_tiled(k_init_params<PREC_FP32>, L, rows, d.total_slots, s, d, L, rows, rlog);
  if (R.precision == PREC_BF16) return launch_tiled(k_init_params<PREC_BF16>, L, rows, d.total_slots, s, d, L, rows, rlog);
  return launch_tiled(k_init_params<PREC_FP8>, L, rows, d.total_slots, s, d, L, rows, rlog);
}

}  // namespace eco
