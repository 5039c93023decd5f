// eco_init.cu -- reset of every environment (Sec. 3.2: grid world with
// randomly distributed resources and a founding population), the recount
// of the statistics after a state write, and the state in the form its
// readers get.  The founders' weights are drawn in
// eco_params.cu.
//
// Founders: the K non-wall cells with the smallest 64-bit keys
// (PLACE draw << 32 | local cell) -- all keys are distinct -- found by a
// radix select on the draw's two 16-bit digits (a histogram pass over the
// cells per digit, the first one inside the pass that fills the cells), a
// rank among the cells that share the last founder's draw, then a two-pass
// tiled scan that numbers the founders in ascending cell order.
#include "eco_internal.cuh"
#include "eco_kernels.h"

namespace eco {

__device__ __forceinline__ unsigned long long place_key(const EnvDesc &ed, int local_cell) {
  const U4 r = philox((uint32_t)(local_cell >> 2), 0u, 0u, 0u, ed.seed, S_PLACE);
  return ((unsigned long long)word_of(r, local_cell & 3) << 32) | (unsigned long long)(uint32_t)local_cell;
}

// Walls, food, empty occupancy, cleared claims (paper rules: a food cell
// holds one bite, e_food energy), the per-slot agent fields (founders get
// alive / facing / energy here; their cells come from the placement below)
// and the first digit's placement histogram.
//
// Bound by the writes, 53 bytes per cell: four cells per thread share each
// Philox block and go out as 16-byte stores.  The counts of food, water and
// biomass are summed here, per CTA, into the step's (zeroed) records, and
// k_place_find<0> turns them into the initial statistics.
__device__ __forceinline__ int env_of_slot(const EnvDesc *env, int n_envs, int slot) {
  int lo = 0, hi = n_envs - 1;
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (env[mid].slot_off <= slot)
      lo = mid;
    else
      hi = mid - 1;
  }
  return lo;
}

__global__ void __launch_bounds__(256) k_reset_world(Dev d, Rules R) {
  const int g0 = blockIdx.x * blockDim.x + threadIdx.x, gs = gridDim.x * blockDim.x;
  const bool terrain = R.rules == RULES_TERRAIN;
  long long sum[3] = {0, 0, 0};  // food, water, biomass of environment e
  int e = -1;
  EnvDesc ed = d.env[0];
  const int stat[3] = {ST_FOOD_TOTAL, ST_WATER_CELLS, ST_BIO_CELLS};
  auto flush = [&]() {
    for (int k = 0; k < 3; ++k)
      if (e >= 0 && sum[k])
        atomicAdd((unsigned long long *)&d.stats_step[e * N_ST + stat[k]], (unsigned long long)sum[k]);
    sum[0] = sum[1] = sum[2] = 0;
  };
  for (int g = g0; g < (d.total_cells >> 2); g += gs) {
    const int c0 = g << 2;
    if (e < 0 || (e + 1 < d.n_envs && d.env[e + 1].cell_off <= c0)) {
      flush();
      e = env_of_cell(d.env, d.n_envs, c0);
      ed = d.env[e];
    }
    const uint32_t blk = (uint32_t)((c0 - ed.cell_off) >> 2);
    const U4 rw = philox(blk, 0u, 0u, 0u, ed.seed, S_WALL);
    const U4 rf = philox(blk, 0u, 0u, 0u, ed.seed, S_FOOD_INIT);
    const U4 rp = philox(blk, 0u, 0u, 0u, ed.seed, S_PLACE);
    U4 rb = {0u, 0u, 0u, 0u};
    int4 rk = make_int4(0, 0, 0, 0);
    if (terrain) {
      rb = philox(blk, 0u, 0u, 0u, ed.seed, S_BIOMASS);
      rk = reinterpret_cast<const int4 *>(d.rock)[g];
    }
    const int rkv[4] = {rk.x, rk.y, rk.z, rk.w};
    uint8_t cf[4];
    int res[4], water[4], bio[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const bool wall = word_of(rw, k) < R.thr_wall;
      const bool food = !wall && word_of(rf, k) < R.thr_food;
      cf[k] = (uint8_t)((wall ? CELL_WALL : 0u) | (food ? CELL_FOOD : 0u));
      res[k] = (R.rules != RULES_SIMPLE && food) ? R.e_food : 0;
      // terrain rules: water fills the cells whose rock lies below sea level;
      // a Bernoulli(biomass_density) site (stream BIOMASS) holds b_site
      water[k] = (terrain && !wall && rkv[k] < R.sea_level) ? R.sea_level - rkv[k] : 0;
      bio[k] = (terrain && !wall && word_of(rb, k) < R.thr_bio) ? R.b_site : 0;
      sum[0] += food ? 1 : 0;
      sum[1] += water[k];
      sum[2] += bio[k];
      if (!wall && ed.init_alive > 0) atomicAdd(&d.hist[(size_t)e * 65536 + (word_of(rp, k) >> 16)], 1u);
    }
    const uint4 z = make_uint4(0u, 0u, 0u, 0u);
    reinterpret_cast<uchar4 *>(d.cellf)[g] = make_uchar4(cf[0], cf[1], cf[2], cf[3]);
    reinterpret_cast<int4 *>(d.res)[g] = make_int4(res[0], res[1], res[2], res[3]);
    reinterpret_cast<int4 *>(d.occ)[g] = make_int4(-1, -1, -1, -1);
    reinterpret_cast<int4 *>(d.water)[g] = make_int4(water[0], water[1], water[2], water[3]);
    reinterpret_cast<int4 *>(d.bio)[g] = make_int4(bio[0], bio[1], bio[2], bio[3]);
    reinterpret_cast<uint4 *>(d.photo)[g] = z;
    reinterpret_cast<uint4 *>(d.flow)[g] = z;
    reinterpret_cast<uint4 *>(d.cnt_move)[g] = z;
#pragma unroll
    for (int k = 0; k < 2; ++k) {
      reinterpret_cast<uint4 *>(d.claim_move)[2 * g + k] = z;
      reinterpret_cast<uint4 *>(d.claim_birth)[2 * g + k] = z;
      reinterpret_cast<uint4 *>(d.att_cell)[2 * g + k] = z;
    }
  }
  // one addition per CTA and count when its threads ended in one environment
  __shared__ int s_e;
  __shared__ unsigned long long s_sum[3];
  if (threadIdx.x == 0) s_e = e;
  if (threadIdx.x < 3) s_sum[threadIdx.x] = 0ull;
  __syncthreads();
  if (__syncthreads_and(e == s_e || e < 0)) {
    for (int k = 0; k < 3; ++k) {
      long long v = sum[k];
#pragma unroll
      for (int off = 16; off > 0; off >>= 1) v += __shfl_xor_sync(0xFFFFFFFFu, v, off);
      if ((threadIdx.x & 31) == 0 && v) atomicAdd(&s_sum[k], (unsigned long long)v);
    }
    __syncthreads();
    if (threadIdx.x < 3 && s_e >= 0 && s_sum[threadIdx.x])
      atomicAdd((unsigned long long *)&d.stats_step[s_e * N_ST + stat[threadIdx.x]], s_sum[threadIdx.x]);
  } else {
    flush();
  }

  for (int s = g0; s < d.total_slots; s += gs) {
    const int es = env_of_slot(d.env, d.n_envs, s);
    const EnvDesc eds = d.env[es];
    const int ls = s - eds.slot_off;
    const bool founder = ls < eds.init_alive;
    d.env_of[s] = (uint16_t)es;
    d.alive[s] = founder ? 1 : 0;
    d.pos[s] = 0;
    uint8_t f = 0;
    if (founder) {
      const U4 r = philox((uint32_t)(ls >> 2), 0u, 0u, 0u, eds.seed, S_FACING_INIT);
      f = (uint8_t)(word_of(r, ls & 3) >> 30);
    }
    d.facing[s] = f;
    d.energy[s] = founder ? R.e_init : 0;
    d.parent[s] = -1;
    d.birth[s] = -1;
    d.act[s] = 0;
    d.tgt[s] = -1;
    d.gain[s] = 0;
    d.hp[s] = (founder && R.rules != RULES_SIMPLE) ? R.hp_max : 0;
    d.a_water[s] = (founder && terrain) ? R.w_init : 0;
    d.a_bio[s] = (founder && terrain) ? R.b_body : 0;
    d.age[s] = 0;
    // colour trait (Sec. 3.3): three uniforms of COLOUR at counter (slot, 0, 0, 0)
    float4 col = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
    if (founder) {
      const U4 r = philox((uint32_t)ls, 0u, 0u, 0u, eds.seed, S_COLOUR);
      col = make_float4(uniform01(r.x), uniform01(r.y), uniform01(r.z), 0.0f);
    }
    d.colour[s] = col;
  }
}

// Sum of a 64-bit value over the CTA (every thread gets the total).
__device__ long long block_sum_ll(long long v, unsigned long long *acc) {
  if (threadIdx.x == 0) *acc = 0ull;
  __syncthreads();
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) v += __shfl_xor_sync(0xFFFFFFFFu, v, off);
  if ((threadIdx.x & 31) == 0) atomicAdd(acc, (unsigned long long)v);
  __syncthreads();
  const long long total = (long long)*acc;
  __syncthreads();
  return total;
}

// Second digit: histogram of the draw's low half among the non-wall cells
// whose high half is the digit found first.
__global__ void __launch_bounds__(256) k_place_hist(Dev d) {
  const int gs = gridDim.x * blockDim.x;
  for (int g = blockIdx.x * blockDim.x + threadIdx.x; g < (d.total_cells >> 2); g += gs) {
    const int c0 = g << 2;
    const int e = env_of_cell(d.env, d.n_envs, c0);
    const EnvDesc ed = d.env[e];
    if (ed.init_alive == 0) continue;
    const uint32_t hi = (uint32_t)d.place_key[e];
    const uchar4 cf = reinterpret_cast<const uchar4 *>(d.cellf)[g];
    const uint8_t cfv[4] = {cf.x, cf.y, cf.z, cf.w};
    const U4 r = philox((uint32_t)((c0 - ed.cell_off) >> 2), 0u, 0u, 0u, ed.seed, S_PLACE);
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const uint32_t w = word_of(r, k);
      if ((w >> 16) == hi && !(cfv[k] & CELL_WALL)) atomicAdd(&d.hist[(size_t)e * 65536 + (w & 0xFFFFu)], 1u);
    }
  }
}

// Initial statistics of environment e from the sums k_reset_world left in
// the step's record: alive = K, food count, energy = K * e_init, step 0;
// paper rules: energy on cells = food count * e_food; terrain rules: water
// and biomass on cells and carried (K * w_init, K * b_body).  Block-level.
__device__ void init_stats(const Dev &d, const Rules &R, int e) {
  const EnvDesc ed = d.env[e];
  const bool terrain = R.rules == RULES_TERRAIN;
  long long *st = d.stats_step + e * N_ST;
  const long long total = st[ST_FOOD_TOTAL], wt = st[ST_WATER_CELLS], bt = st[ST_BIO_CELLS];
  __syncthreads();
  for (int k = threadIdx.x; k < N_ST; k += blockDim.x) {
    long long v = 0;
    if (k == ST_ALIVE) v = ed.init_alive;
    else if (k == ST_FOOD_TOTAL) v = total;
    else if (k == ST_ENERGY_TOTAL) v = (long long)ed.init_alive * R.e_init;
    else if (k == ST_RES_TOTAL && R.rules != RULES_SIMPLE) v = total * R.e_food;
    else if (k == ST_WATER_CELLS && terrain) v = wt;
    else if (k == ST_BIO_CELLS && terrain) v = bt;
    else if (k == ST_WATER_AGENTS && terrain) v = (long long)ed.init_alive * R.w_init;
    else if (k == ST_BIO_AGENTS && terrain) v = (long long)ed.init_alive * R.b_body;
    d.stats_total[e * N_ST + k] = v;
    d.stats_last[e * N_ST + k] = v;
    st[k] = 0;
  }
}

// One CTA per environment: the bin of `remaining`-th smallest digit; the
// histogram is cleared behind the search.  Each warp reads 2,048
// consecutive bins, 512 bytes at a time (one thread per 64 bins, whose
// 256-byte strides left every load uncoalesced, took 69 us per digit).
// A missing bin (fewer than K non-wall cells) sets the status word.
// DIGIT 0: place_key = the digit, place_remaining = the rank inside the bin,
// and the initial statistics.  DIGIT 1: place_key = the last founder's key;
// when more cells share its draw than are needed, the CTA walks the
// environment's cells in order to the one that fills the rank.
template <int DIGIT>
__global__ void __launch_bounds__(1024) k_place_find(Dev d, Rules R) {
  __shared__ int sh[33];
  __shared__ int found_bin, found_before, found_cnt;
  const int e = blockIdx.x;
  const EnvDesc ed = d.env[e];
  if (DIGIT == 0) init_stats(d, R, e);
  if (ed.init_alive == 0) return;
  const int remaining = DIGIT == 0 ? ed.init_alive : d.place_remaining[e];
  uint4 *h = reinterpret_cast<uint4 *>(d.hist + (size_t)e * 65536);
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  if (threadIdx.x == 0) found_bin = -1;
  uint4 v[16];
  int cnt = 0;
#pragma unroll
  for (int i = 0; i < 16; ++i) {
    v[i] = h[warp * 512 + i * 32 + lane];
    cnt += (int)(v[i].x + v[i].y + v[i].z + v[i].w);
  }
#pragma unroll
  for (int i = 0; i < 16; ++i) h[warp * 512 + i * 32 + lane] = make_uint4(0u, 0u, 0u, 0u);
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) cnt += __shfl_xor_sync(0xFFFFFFFFu, cnt, off);
  if (lane == 0) sh[warp] = cnt;
  __syncthreads();
  int before = 0;
  for (int w = 0; w < warp; ++w) before += sh[w];
  if (before < remaining && before + cnt >= remaining) {  // this warp's bins hold it
    int run = before;
#pragma unroll
    for (int i = 0; i < 16; ++i) {
      const uint32_t w4[4] = {v[i].x, v[i].y, v[i].z, v[i].w};
      const int own = (int)(v[i].x + v[i].y + v[i].z + v[i].w);
      int incl = own;
#pragma unroll
      for (int off = 1; off < 32; off <<= 1) {
        const int o = __shfl_up_sync(0xFFFFFFFFu, incl, off);
        if (lane >= off) incl += o;
      }
      int at = run + incl - own;
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        if (at < remaining && at + (int)w4[k] >= remaining) {  // one lane, one bin
          found_bin = 4 * (warp * 512 + i * 32 + lane) + k;
          found_before = at;
          found_cnt = (int)w4[k];
        }
        at += (int)w4[k];
      }
      run += __shfl_sync(0xFFFFFFFFu, incl, 31);
    }
  }
  __syncthreads();
  if (found_bin < 0) {
    if (threadIdx.x == 0) {
      atomicOr(&d.counters[CNT_STATUS], 1);
      d.place_key[e] = DIGIT == 0 ? 0ull : ~0ull;
      d.place_remaining[e] = remaining;
    }
    return;
  }
  const int rest = remaining - found_before;
  if (DIGIT == 0) {
    if (threadIdx.x == 0) {
      d.place_key[e] = (unsigned long long)found_bin;
      d.place_remaining[e] = rest;
    }
    return;
  }
  const uint32_t draw = (uint32_t)(d.place_key[e] << 16) | (uint32_t)found_bin;
  __syncthreads();  // the key is read by every thread before it is replaced
  if (rest == found_cnt) {
    if (threadIdx.x == 0) d.place_key[e] = ((unsigned long long)draw << 32) | 0xFFFFFFFFull;
    return;
  }
  const int n = ed.side * ed.side;
  int seen = 0;
  for (int base = 0; base < n && seen < rest; base += (int)blockDim.x) {
    const int c = base + (int)threadIdx.x;
    const bool hit = c < n && !(d.cellf[ed.cell_off + c] & CELL_WALL) && (uint32_t)(place_key(ed, c) >> 32) == draw;
    int total;
    const int at = seen + block_exclusive_scan(hit ? 1 : 0, &total, sh);
    if (hit && at == rest - 1) d.place_key[e] = ((unsigned long long)draw << 32) | (unsigned long long)(uint32_t)c;
    seen += total;
  }
}

// Founders are the non-wall cells with key <= the last founder's, numbered
// in ascending cell order.  Tiles of kPlaceTile cells, 16 consecutive cells
// per thread; the first pass counts each tile, the second adds up the tiles
// before it and writes, so that a large world's cells spread over the chip.
constexpr int kPlaceTile = 4096;

__device__ __forceinline__ uint32_t founder_mask(const Dev &d, const EnvDesc &ed, unsigned long long thr, int c0) {
  uint32_t mask = 0u;
  const int n = ed.side * ed.side;
  for (int k = 0; k < 16 && c0 + k < n; k += 4) {
    const uchar4 cf = *reinterpret_cast<const uchar4 *>(d.cellf + ed.cell_off + c0 + k);
    const uint8_t cfv[4] = {cf.x, cf.y, cf.z, cf.w};
    const U4 r = philox((uint32_t)((c0 + k) >> 2), 0u, 0u, 0u, ed.seed, S_PLACE);
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const unsigned long long key =
          ((unsigned long long)word_of(r, q) << 32) | (unsigned long long)(uint32_t)(c0 + k + q);
      if (!(cfv[q] & CELL_WALL) && key <= thr) mask |= 1u << (k + q);
    }
  }
  return mask;
}

template <bool WRITE>
__global__ void __launch_bounds__(kPlaceTile / 16) k_place_number(Dev d) {
  __shared__ int sh[33];
  const int tile = blockIdx.x;
  int lo = 0, hi = d.n_envs - 1;  // the tile's environment
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (d.env[mid].ctile_off <= tile) lo = mid;
    else hi = mid - 1;
  }
  const int e = lo;
  const EnvDesc ed = d.env[e];
  if (ed.init_alive == 0) return;
  const unsigned long long thr = d.place_key[e];
  const int c0 = (tile - ed.ctile_off) * kPlaceTile + (int)threadIdx.x * 16;
  uint32_t mask = founder_mask(d, ed, thr, c0);
  int total;
  if (!WRITE) {
    block_exclusive_scan(__popc(mask), &total, sh);
    if (threadIdx.x == 0) d.place_tiles[tile] = total;
    return;
  }
  int before = 0, base;
  for (int k = ed.ctile_off + (int)threadIdx.x; k < tile; k += blockDim.x) before += d.place_tiles[k];
  block_exclusive_scan(before, &base, sh);
  int at = base + block_exclusive_scan(__popc(mask), &total, sh);
  while (mask) {
    const int k = __ffs(mask) - 1;
    mask &= mask - 1;
    // the guard only matters when the select failed (status already set)
    if (at < ed.init_alive) {
      const int slot = ed.slot_off + at, gc = ed.cell_off + c0 + k;
      d.pos[slot] = c0 + k;
      d.occ[gc] = slot;
      d.cellf[gc] |= (uint8_t)CELL_AGENT;
    }
    ++at;
  }
  const int n = ed.side * ed.side;
  if (threadIdx.x == 0 && (tile - ed.ctile_off + 1) * kPlaceTile >= n && base + total != ed.init_alive)
    atomicOr(&d.counters[CNT_STATUS], 2);
}

int place_tiles(int side) { return (side * side + kPlaceTile - 1) / kPlaceTile; }

__global__ void k_init_static(Dev d) {
  for (int s = blockIdx.x * blockDim.x + threadIdx.x; s < d.total_slots; s += gridDim.x * blockDim.x) {
    int e = 0;
    while (e + 1 < d.n_envs && d.env[e + 1].slot_off <= s) ++e;
    d.env_of[s] = (uint16_t)e;
  }
  for (int c = blockIdx.x * blockDim.x + threadIdx.x; c < d.total_cells; c += gridDim.x * blockDim.x)
    d.occ[c] = -1;
}

// One CTA per environment: alive count, food count, energy sum (and, under
// the paper rules, the energy lying on cells) of the current state become
// the "now" statistics; the step counter is copied.
__global__ void __launch_bounds__(1024) k_recount(Dev d, Rules R) {
  __shared__ unsigned long long acc;
  const int e = blockIdx.x;
  const EnvDesc ed = d.env[e];
  const int n = ed.side * ed.side;
  long long food = 0, alive = 0, energy = 0, res = 0, wc = 0, bc = 0, wa = 0, ba = 0;
  for (int c = threadIdx.x; c < n; c += blockDim.x) {
    food += (d.cellf[ed.cell_off + c] & CELL_FOOD) ? 1 : 0;
    res += d.res[ed.cell_off + c];
    wc += d.water[ed.cell_off + c];
    bc += d.bio[ed.cell_off + c];
  }
  for (int s = threadIdx.x; s < ed.n_slots; s += blockDim.x) {
    const int g = ed.slot_off + s;
    if (d.alive[g]) {
      ++alive;
      energy += d.energy[g];
      wa += d.a_water[g];
      ba += d.a_bio[g];
    }
  }
  const bool terrain = R.rules == RULES_TERRAIN;
  const long long wct = block_sum_ll(wc, &acc), bct = block_sum_ll(bc, &acc);
  const long long wat = block_sum_ll(wa, &acc), bat = block_sum_ll(ba, &acc);
  const long long ft = block_sum_ll(food, &acc);
  const long long at = block_sum_ll(alive, &acc);
  const long long et = block_sum_ll(energy, &acc);
  const long long rt = block_sum_ll(res, &acc);
  if (threadIdx.x == 0) {
    const long long t = d.step[0];
    long long *tot = d.stats_total + e * N_ST, *last = d.stats_last + e * N_ST;
    tot[ST_ALIVE] = last[ST_ALIVE] = at;
    tot[ST_FOOD_TOTAL] = last[ST_FOOD_TOTAL] = ft;
    tot[ST_ENERGY_TOTAL] = last[ST_ENERGY_TOTAL] = et;
    tot[ST_RES_TOTAL] = last[ST_RES_TOTAL] = R.rules != RULES_SIMPLE ? rt : 0;
    tot[ST_WATER_CELLS] = last[ST_WATER_CELLS] = terrain ? wct : 0;
    tot[ST_BIO_CELLS] = last[ST_BIO_CELLS] = terrain ? bct : 0;
    tot[ST_WATER_AGENTS] = last[ST_WATER_AGENTS] = terrain ? wat : 0;
    tot[ST_BIO_AGENTS] = last[ST_BIO_AGENTS] = terrain ? bat : 0;
    tot[ST_STEP] = last[ST_STEP] = t;
  }
}

__global__ void __launch_bounds__(256) k_pack(PackList list, uint8_t *base) {
  const int k = blockIdx.y;
  const uint8_t *src = reinterpret_cast<const uint8_t *>(list.src[k]);
  uint8_t *dst = base + list.at[k];
  const uint32_t n = list.bytes[k], i0 = blockIdx.x * blockDim.x + threadIdx.x, step = gridDim.x * blockDim.x;
  // slot arrays of bytes may start at any address; words where they allow it
  if ((((uintptr_t)src | n) & 3u) == 0u)
    for (uint32_t i = i0; i < n / 4; i += step)
      reinterpret_cast<uint32_t *>(dst)[i] = reinterpret_cast<const uint32_t *>(src)[i];
  else
    for (uint32_t i = i0; i < n; i += step) dst[i] = src[i];
}

cudaError_t launch_pack(const PackList &list, uint8_t *base, cudaStream_t s) {
  if (list.n == 0) return cudaSuccess;
  k_pack<<<dim3(8, list.n), 256, 0, s>>>(list, base);
  return cudaGetLastError();
}

__global__ void __launch_bounds__(256) k_state_out(Dev d, int env, int c0, int nc, int s0, int ns, uint8_t *cells,
                                                   uint8_t *slots) {
  const EnvDesc ed = d.env[env];
  const int g0 = blockIdx.x * blockDim.x + threadIdx.x, gs = gridDim.x * blockDim.x;
  int32_t *occ = reinterpret_cast<int32_t *>(cells);
  uint8_t *food = cells + 4 * (size_t)nc, *wall = cells + 5 * (size_t)nc;
  for (int g = g0; g < nc / 4; g += gs) {  // sides are even: whole groups of four
    const int c = ed.cell_off + c0 + 4 * g;
    const uchar4 cf = *reinterpret_cast<const uchar4 *>(d.cellf + c);
    int4 o = *reinterpret_cast<const int4 *>(d.occ + c);
    o.x = o.x < 0 ? -1 : o.x - ed.slot_off;
    o.y = o.y < 0 ? -1 : o.y - ed.slot_off;
    o.z = o.z < 0 ? -1 : o.z - ed.slot_off;
    o.w = o.w < 0 ? -1 : o.w - ed.slot_off;
    occ[4 * g] = o.x, occ[4 * g + 1] = o.y, occ[4 * g + 2] = o.z, occ[4 * g + 3] = o.w;
    const uint8_t v[4] = {cf.x, cf.y, cf.z, cf.w};
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      food[4 * g + k] = (v[k] & CELL_FOOD) ? 1 : 0;
      wall[4 * g + k] = (v[k] & CELL_WALL) ? 1 : 0;
    }
  }
  int32_t *x = reinterpret_cast<int32_t *>(slots), *y = x + ns;
  float *rgb = reinterpret_cast<float *>(y + ns);
  for (int i = g0; i < ns; i += gs) {
    const int s = ed.slot_off + s0 + i, p = d.pos[s];
    x[i] = p % ed.side;
    y[i] = p / ed.side;
    const float4 c = d.colour[s];
    rgb[3 * i] = c.x, rgb[3 * i + 1] = c.y, rgb[3 * i + 2] = c.z;
  }
}

cudaError_t launch_state_out(const Dev &d, int env, int c0, int nc, int s0, int ns, uint8_t *cells, uint8_t *slots,
                             cudaStream_t s) {
  const int work = nc / 4 > ns ? nc / 4 : ns;
  k_state_out<<<grid_for(work, 256, 1024), 256, 0, s>>>(d, env, c0, nc, s0, ns, cells, slots);
  return cudaGetLastError();
}

cudaError_t launch_init_static(const Dev &d, const EnvGrid &g, cudaStream_t s) {
  const long long n = d.total_slots > d.total_cells ? d.total_slots : d.total_cells;
  k_init_static<<<grid_for(n, 256, g.sms * 16), 256, 0, s>>>(d);
  return cudaGetLastError();
}

cudaError_t launch_recount(const Dev &d, const Rules &R, cudaStream_t s) {
  k_recount<<<d.n_envs, 1024, 0, s>>>(d, R);
  return cudaGetLastError();
}

cudaError_t launch_reset(const Dev &d, const Layout &L, const Rules &R, const EnvGrid &g,
                         cudaStream_t s) {
  cudaError_t err;
  const int T = 256;
  const int cb = grid_for(d.total_cells / 4 > d.total_slots ? d.total_cells / 4 : d.total_slots, T, g.sms * 8);
  if ((err = cudaMemsetAsync(d.counters, 0, sizeof(int32_t) * CNT_N, s)) != cudaSuccess) return err;
  if ((err = cudaMemsetAsync(d.step, 0, sizeof(long long), s)) != cudaSuccess) return err;
  if ((err = cudaMemsetAsync(d.stats_step, 0, sizeof(long long) * N_ST * (size_t)d.n_envs, s)) != cudaSuccess)
    return err;
  if ((err = cudaMemsetAsync(d.birth_contenders, 0, sizeof(int32_t) * (size_t)d.n_envs, s)) != cudaSuccess)
    return err;
  if ((err = cudaMemsetAsync(d.hist, 0, sizeof(uint32_t) * 65536 * (size_t)d.n_envs, s)) != cudaSuccess)
    return err;
  k_reset_world<<<cb, T, 0, s>>>(d, R);
  k_place_find<0><<<d.n_envs, 1024, 0, s>>>(d, R);
  k_place_hist<<<grid_for(d.total_cells / 4, T, g.sms * 8), T, 0, s>>>(d);
  k_place_find<1><<<d.n_envs, 1024, 0, s>>>(d, R);
  k_place_number<false><<<d.place_tile_count, kPlaceTile / 16, 0, s>>>(d);
  k_place_number<true><<<d.place_tile_count, kPlaceTile / 16, 0, s>>>(d);
  if ((err = cudaGetLastError()) != cudaSuccess) return err;
  return launch_init_params(d, L, R, s);
}

}  // namespace eco
