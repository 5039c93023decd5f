// eco_kernels.h -- host-side launchers of the library's kernels (internal).
#pragma once

#include <cuda_runtime.h>

#include "eco_internal.cuh"

namespace eco {

// Policy phase (eco_policy.cu).
struct PolicyLaunch {
  void *fn;
  int threads, blocks;
  size_t smem;
  int xs_floats;
};
int policy_variant_count();
const char *policy_variant_name(int k);
// Variants that stream only the W_in rows of nonzero inputs (opt-in: the
// autotuner chooses among them only when asked to, policy_variant = -1).
bool policy_variant_sparse(int k);
typedef void (*PolicyFn)(Dev, Layout, Rules, int, int);
// Floats of one warp's shared-memory slice: observation (xs_floats, a
// multiple of 4), hidden activation (H), logits (16) and, for the sparse
// variants, the list of nonzero inputs (xs_floats shorts, rounded up to whole
// 16-byte units).  Every part is a multiple of 4 floats, so each warp's
// slice and the float4 reads of its activations stay 16-byte aligned.
__host__ __device__ inline int policy_warp_floats(int xs_floats, int H, bool sparse) {
  return xs_floats + H + 16 + (sparse ? ((xs_floats / 2 + 3) & ~3) : 0);
}
// Kernel instance of variant k for a hidden width (one translation unit per
// precision: eco_policy_fp32.cu, eco_policy_bf16.cu, eco_policy_fp8.cu).
PolicyFn policy_pick_fp32(int H, int variant);
PolicyFn policy_pick_bf16(int H, int variant);
PolicyFn policy_pick_fp8(int H, int variant);
cudaError_t policy_prepare(const Layout &L, const Rules &R, int variant, PolicyLaunch *pl);
// apply_moves: also apply facing / turns and file move claims (the step);
// false leaves the world state untouched (timing, parity of the policy).
cudaError_t policy_launch(const PolicyLaunch &pl, const Dev &d, const Layout &L, const Rules &R,
                          cudaStream_t s, bool apply_moves);

// Environment phases (eco_env.cu).
struct EnvGrid {
  int sms;                // SM count
  int slot_blocks;        // blocks of 256 threads for per-agent phases
  int cell_blocks;        // blocks of 256 threads for per-cell phases
  int birth_blocks;       // CTAs of the mutation kernel
  int persistent_blocks;  // co-resident CTAs of the persistent form (0: unavailable)
  int use_persistent;     // run the environment phases as one persistent kernel
  int cluster;            // the persistent form's CTAs are one thread-block cluster
};
__host__ __device__ int compact_tiles(int total_slots);

// Let `kernel` be launched with `bytes` of dynamic shared memory.  The limit
// belongs to the function on the device, not to a handle, so it is only ever
// raised: a handle of a smaller shape leaves a larger one's launches their
// room.  Safe from several host threads.
cudaError_t allow_dynamic_smem(const void *kernel, size_t bytes);

// Alive list of the current state (ascending slots) and its count.
cudaError_t launch_compact(const Dev &d, cudaStream_t s);
// Shared-memory attributes and the persistent form's grid size.
cudaError_t env_prepare(const Layout &L, EnvGrid *g);
// A small batch: one cluster of a few CTAs in place of one CTA per SM.
void env_use_small_grid(const Layout &L, EnvGrid *g);
cudaError_t launch_env_phases(const Dev &d, const Layout &L, const Rules &R, const EnvGrid &g,
                              cudaStream_t s);

// Reset (eco_init.cu).
cudaError_t launch_reset(const Dev &d, const Layout &L, const Rules &R, const EnvGrid &g,
                         cudaStream_t s);
// Static per-slot tables (environment of every slot) at create.
cudaError_t launch_init_static(const Dev &d, const EnvGrid &g, cudaStream_t s);
// Recompute the "now" statistics (alive, food, energy, step) from the state.
cudaError_t launch_recount(const Dev &d, const Rules &R, cudaStream_t s);
// State I/O (eco_init.cu).  Pieces of device memory, packed one behind the
// other at `base`.
constexpr int kPackMost = 16;
struct PackList {
  int n;
  const void *src[kPackMost];
  uint32_t at[kPackMost], bytes[kPackMost];  // at: a multiple of 8
};
cudaError_t launch_pack(const PackList &list, uint8_t *base, cudaStream_t s);
// Cells [c0, c0 + nc) (c0 a multiple of 4) of environment env to `cells`: the
// env-local occupants (i32), then food, then wall (u8); slots [s0, s0 + ns) to
// `slots`: x, then y (i32), then RGB (3 f32).
cudaError_t launch_state_out(const Dev &d, int env, int c0, int nc, int s0, int ns, uint8_t *cells, uint8_t *slots,
                             cudaStream_t s);

// Placement tiles of a world of side L (reset).
int place_tiles(int side);

// Parameters (eco_params.cu).  Founders' weights and the streamed copy of
// every slot; n slots from global slot slot0 out of or into `flat`, device
// memory [n][P] in logical order (params_in also derives the streamed copy).
cudaError_t launch_init_params(const Dev &d, const Layout &L, const Rules &R, cudaStream_t s);
cudaError_t launch_params_in(const Dev &d, const Layout &L, const Rules &R, int slot0, int n, const float *flat,
                             cudaStream_t s);
cudaError_t launch_params_out(const Dev &d, const Layout &L, int slot0, int n, float *flat, cudaStream_t s);

}  // namespace eco
