// rmp_internal.h -- types shared by the library's host code and kernels (not part of the
// public ABI).  Layouts in HBM:
//   * occupancy brick: one 8^3 voxel block = 512 bits = 64 bytes = 16 uint32 words; bit
//     b = lx + 8 ly + 64 lz lives in word b >> 5, bit b & 31 (a TSDF voxel is occupied iff
//     its value is <= 0; a dense voxel iff it is nonzero).
//   * box field: for every voxel of an occupied block and each of the 8 octants of ray
//     directions one byte, 0 if the voxel is occupied, else 64 | ex | ey << 2 | ez << 4: the
//     2^ex x 2^ey x 2^ez voxels from it on in that octant are free.  4 KB per occupied block,
//     by slot: octant o (bit a set: axis a climbs) at 512 o, voxels in reflected order (an
//     axis the octant descends counts from 7 down).
//   * grid layout (dense maps, and hashed maps whose block bounding box is moderate): the
//     bricks of every block in the bounding box, x fastest (all-zero where free), plus 8
//     planes (octants) of one word per block: 2^31 | slot of an occupied block, else the log2
//     extents in blocks of the free box from it on (2 bits per axis).  The march crosses a
//     whole free box of blocks or voxels in one exact step.
//   * hash layout (fallback for very large extents): power-of-two array of 16-byte entries
//     {key, slot, box}; key packs the block coordinates (21 bits each, offset by 2^20); empty
//     entries hold ~0; linear probing from a Fibonacci (multiply-shift) hash, load factor
//     <= 1/4; blocks without occupied voxels keep their key with slot -1; box: the block's
//     slot in the box field.
#pragma once

#include <cstdint>
#include <cuda_runtime.h>

#include "rmp.h"

namespace rmp {

constexpr int kBrickWords = 16;
constexpr unsigned long long kEmptyKey = ~0ull;
constexpr int kKeyBias = 1 << 20;
constexpr int kMaxGrid = 4096;          // CTAs of one evaluation (grid-stride beyond)
constexpr int kWsHeaderBytes = 1024;
constexpr int kMaxRangeVoxels = 16384;  // keeps every DDA crossing numerator below 2^31

struct HashEntry {
  unsigned long long key;
  uint32_t slot;
  uint32_t box;
};

constexpr int kLayoutGrid = 0;
constexpr int kLayoutHash = 1;
constexpr uint64_t kBoxBytes = 4096;                  // box field of one occupied block
// Largest box field (8 M occupied blocks); a map beyond it, or one whose field does not fit (see
// box_field_fits), is marched voxel by voxel inside occupied blocks
constexpr uint64_t kMaxBoxFieldBytes = 32ull << 30;
constexpr int kCellDistCap = 4;                       // cell free distances are capped here
constexpr uint64_t kMaxCellBytes = 256ull << 20;      // cell distances given up to this size
constexpr uint64_t kMaxGridBricks = 1ull << 26;       // grid layout up to 4 GiB of bricks

struct DevMap {
  int kind;                 // RMP_MAP_DENSE_U8 (rays exit at the grid) / RMP_MAP_HASHED_TSDF
  int layout;               // kLayoutGrid / kLayoutHash
  int hash_shift;           // 64 - log2(capacity)
  uint32_t cap_mask;
  float vs_f;               // RN32(voxel size)
  double vs;
  double origin[3];         // dense only (hashed maps are world-anchored)
  int dims[3];              // dense voxels per axis
  int gmin[3];              // grid: block coordinates of the grid's first brick
  int gdim[3];              // grid: bricks per axis
  const uint4* bricks;      // grid: brick (x + gdim0 (y + gdim1 z)); hash: by slot
  const uint32_t* top;      // grid: 8 planes of one word per brick (see above)
  const uint32_t* cells;    // the box field's bytes (null: march occupied blocks voxel by voxel)
  const HashEntry* table;   // hash layout only
};

// One state as the kernels use it: the position quantised (2^-16 voxels) and in FP32, the
// velocity as an FP32 pair.
struct CtaState {
  long long P[3];
  float v[3];     // RN32(xdot)
  float vl[3];    // RN32(xdot - v)
  float xf[3];    // RN32(x) (scans)
  int bad[3];     // the axis's position is not finite or beyond 2^22 voxels
};

// Constants of one evaluation derived on the host from rmp_params_t.
struct EvalConsts {
  float eta_rep, inv_nu_rep, eta_damp, inv_nu_damp, eps, c, r_up, inv_r;
  float r_hi, r_lo;         // r = r_hi + r_lo (FP32 pair)
  float quiet_v2;           // |xdot|^2 below which inactive or far hits add exact zeros
  float min_up, max_dn;     // scans: d >= min_range <=> d >= min_up; d <= max <=> d <= max_dn
  long long R_fx;           // llrint(max_range / vs * 2^16)
  uint32_t n_rays, halton_offset;
  uint32_t perm_M, perm_Q, perm_R;   // coherent ray order (see ray_of_slot)
  uint32_t lg_segs;                  // each ray is marched as 2^lg_segs segments
  int w_mode, reduce_mode;
  double c64;                        // soft-normalisation c (FP64, attractor)
  double att_alpha, att_beta;        // attractor gain and damping (combined evaluations)
  int att_mean;                      // combined: ray sums divided by the ray count first
  uint32_t seg_threads;              // batches: threads of the persistent launch (segments)
  uint32_t sms;                      // batches and rollouts: SMs of the device
  CtaState cs0;                      // the state carried in the launch itself, read when the
                                     // kernel's state pointer is null (synchronous calls)
};

// Closed-loop rollout of point robots (per robot, device-resident).
struct RolloutDev {
  double seg_start[3], prev_seg[3];
  double path_length, smooth_sum;
  uint32_t status, steps, smooth_n, have_prev;
};

struct RolloutConsts {
  double dt, goal_tol, inv_rays;            // inv_rays: 1 / n_rays, exact for powers of two
  uint32_t max_steps, seg_steps, n_rays, pad;
};

// What the control step after an evaluation works on (rollouts): the robots' records, states and
// ray counts; `running` (nullable) counts the robots that go on.
struct RolloutArgs {
  RolloutConsts rc;
  RolloutDev* rs;           // null: no control step
  double* states;
  const double* goals;
  uint32_t* n_rays;
  uint32_t* running;
};

// Workspace of one single-state evaluation: a header, then one partial slot per CTA.  A
// slot is empty when every byte is 0xFF; CTA i > 0 fills slot i, CTA 0 waits for the
// slots, reads them and empties them again (see grid_finish).
struct WsHeader {
  unsigned int poisoned;    // nonzero after a timed-out finish: re-initialise the workspace
  unsigned int pad[kWsHeaderBytes / 4 - 1];
};

struct CtaPartial {         // 80 bytes per CTA
  double v[9];              // sum A (6), sum A f (3)
  unsigned int n_hits, n_active;
};

inline size_t workspace_bytes() {
  return kWsHeaderBytes + sizeof(CtaPartial) * (size_t)kMaxGrid;
}

// Header zero, partial slots empty: the state every evaluation leaves a workspace in.
inline cudaError_t workspace_reset(void* ws, cudaStream_t s) {
  cudaError_t e = cudaMemsetAsync(ws, 0, kWsHeaderBytes, s);
  if (e == cudaSuccess)
    e = cudaMemsetAsync((char*)ws + kWsHeaderBytes, 0xFF, workspace_bytes() - kWsHeaderBytes, s);
  return e;
}

inline size_t align256(size_t x) { return (x + 255) & ~(size_t)255; }

// ------------------------------------------------------------------ batched evaluation
// A state's rays are summed in partials of 32 / S rays (S a function of its ray count and the
// launch shape), kBatchGroup consecutive ones a group (the warp that completes a group sums it),
// and the last group of a state sums the groups and resolves.  Work is another cut of the same
// rays: chunks of 32 threads (32 / s rays, s <= S segments marched per ray, s from the whole
// batch's load) that the warps of a persistent grid take from a counter; a chunk stores S / s
// partials.  s therefore changes no bit of a result.
constexpr uint32_t kBatchGroup = 32;
constexpr uint32_t kMaxBatchStates = 1u << 16;
constexpr uint32_t kMaxBatchSegs = 4;        // workspace is sized for up to 4 segments per ray

struct BatchState {         // 80 bytes, written by the prep kernel
  long long P[3];           // quantised position (2^-16 voxels)
  float v[3], vl[3];        // velocity as an FP32 pair
  uint32_t n_rays, work0, part0, group0;   // first work chunk, partial and group
  uint32_t perm_M, perm_Q;  // direction cells (the remainder n_rays - perm_Q perm_M is derived)
  uint32_t lg_segs;         // log2 S | log2 s << 8
  int status;               // RMP_OK or RMP_ERR_INVALID_ARG
};

struct BatchHeader {        // 128 bytes
  uint32_t next_chunk;      // work counter of the persistent grid
  uint32_t total_chunks;    // work chunks
  uint32_t n_states;
  uint32_t pad[29];
};

// States and robots evaluated by one CTA each have their partials in shared memory.
constexpr uint32_t kStateRays = 4096, kStateGroups = kStateRays * kMaxBatchSegs / (32 * 32);
// Batches with a CTA per state (see raycast_state_kernel): where a CTA's 32 warps hold a state's
// rays, and up to 16 states an SM (of the smallest CTAs), beyond which the packed chunks of the
// persistent grid gain as much as the set-up costs (us on 152 SMs, CTA per state / packed: 128
// states of 16 to 256 rays 13.5 / 25, 17.8 / 30; 304 of 1024 43 / 77; 1216 of 32 to 1024 71 / 74;
// 2432 of 64 to 256 73 / 82; 5000 of 64 to 256 142 / 137; above 1024 rays 64 states of 512 to 4096
// 55 / 34).
inline bool state_per_cta(uint32_t n_states, uint32_t max_rays, uint32_t sms) {
  return max_rays <= 1024 && n_states <= 16 * sms;
}
// Rollouts with a CTA per robot for all its steps (see rollout_kernel): up to 1024 rays, or as many
// as its shared memory holds where two robots an SM take them all; more rays of few robots are
// spread over all SMs instead, robots of many rays packed (us a step with its share of the call,
// CTA per robot / evaluated together: 8 robots of 1024 rays 23 / 34, of 4096 70 / 37; 32 of 2048
// 40 / 45; 128 of 1024 38 / 68, of 4096 77 / 121; 304 of 4096 186 / 207, 608 361 / 347; 1216 of
// 256 175 / 227, of 1024 258 / 318).  Few-ray robots have no upper bound: 16 steps of 65536 robots
// take 11.7 ms with 16 rays each and 25.7 with 64, 4096 robots of 1024 6.6 (set-up and evaluation
// launched per step, before: 197, 245 and 63).
inline bool rollout_resident(uint32_t n_robots, uint32_t n_rays, uint32_t sms) {
  return n_rays <= 1024 ||
         (n_rays <= kStateRays && n_rays <= 64 * n_robots && n_robots <= 2 * sms);
}

struct BatchLayout {
  size_t states, sticket, gticket, cparts, gparts, total;
  uint64_t chunks_per_state, groups_per_state;
};

inline BatchLayout batch_layout(uint32_t n_states, uint32_t max_rays) {
  BatchLayout L;
  L.chunks_per_state = ((uint64_t)max_rays * kMaxBatchSegs + 31) / 32;
  L.groups_per_state = (L.chunks_per_state + kBatchGroup - 1) / kBatchGroup;
  const uint64_t n = n_states;
  L.states = align256(sizeof(BatchHeader));
  L.sticket = align256(L.states + sizeof(BatchState) * n);
  L.gticket = align256(L.sticket + 4 * n);
  L.cparts = align256(L.gticket + 4 * n * L.groups_per_state);
  L.gparts = align256(L.cparts + sizeof(CtaPartial) * n * L.chunks_per_state);
  L.total = align256(L.gparts + sizeof(CtaPartial) * n * L.groups_per_state);
  return L;
}

#ifdef __CUDACC__
__host__ __device__
#endif
inline unsigned long long pack_key(int bx, int by, int bz) {
  return (unsigned long long)(uint32_t)(bx + kKeyBias) |
         ((unsigned long long)(uint32_t)(by + kKeyBias) << 21) |
         ((unsigned long long)(uint32_t)(bz + kKeyBias) << 42);
}

// ESDF policy constants (FP64) of one evaluation.
struct EsdfConsts {
  double eta_rep, nu_rep, eta_damp, nu_damp, r, c, eps;
  double alpha, beta;       // attractor (with goals)
  int w_mode;
  uint32_t sms;             // SMs of the device
};

// Launchers (rmp_kernels.cu).  All enqueue on `stream` and return cudaGetLastError().
int raycast_occupancy(const DevMap& m, int reduce_mode, int block);   // CTAs per SM
cudaError_t launch_raycast(const DevMap& m, const EvalConsts& k, const double* state_dev,
                           void* ws, rmp_result_t* out_dev, rmp_ray_hit_t* hits,
                           float* per_ray, int block, int grid, cudaStream_t stream);

int ctx_device(const rmp_ctx* ctx);                                  // CUDA device of a context
int batch_occupancy(const DevMap& m, int reduce_mode, int block);     // CTAs per SM
// Prep kernel + persistent batch kernel; n_rays_dev / states_dev on the device.  With
// goals_dev (3 doubles per state) each state's rays are combined with its attractor, and with
// step.rs each robot then takes its control step (see rollout_step).
cudaError_t launch_batch(const DevMap& m, const EvalConsts& k, const double* states_dev,
                         const uint32_t* n_rays_dev, uint32_t n_states, uint32_t max_rays,
                         void* ws, rmp_result_t* out_dev, rmp_ray_hit_t* hits, float* per_ray,
                         int block, int grid, cudaStream_t stream,
                         const double* goals_dev = nullptr,
                         const RolloutArgs& step = RolloutArgs());
// L2 read-bandwidth probe (see rmp_probe_l2_read): grid CTAs of 512 threads.
cudaError_t launch_probe_l2(const uint4* buf, size_t n16, uint32_t passes, int grid,
                            uint64_t* checksum, cudaStream_t stream);
// The ESDF policy for n states (see rmp_esdf_eval_async).  prims32: two float4 per primitive,
// centre and kind (1 sphere, 0 box), size and the sum of the six magnitudes (rounded up).
cudaError_t launch_esdf_eval(const rmp_primitive_t* prims, const float4* prims32,
                             uint32_t n_prims, const EsdfConsts& k, const double* states,
                             const double* goals, uint32_t n_states, rmp_result_t* out,
                             double* query, cudaStream_t stream);
// Up to `steps` control steps of the rollouts, a CTA per robot (see rollout_resident).
cudaError_t launch_rollout(const DevMap& m, const EvalConsts& k, const RolloutArgs& g, uint32_t n,
                           uint32_t steps, cudaStream_t stream);
// Up to `steps` control steps with the ESDF policy; `running` counts the robots that still run.
cudaError_t launch_esdf_rollout(const rmp_primitive_t* prims, const float4* prims32,
                                uint32_t n_prims, const EsdfConsts& k, const DevMap& m,
                                const RolloutArgs& g, uint32_t n, uint32_t steps,
                                rmp_result_t* res, uint32_t* running, cudaStream_t stream);
cudaError_t launch_scan(const float* pts, const EvalConsts& k, const double* state_dev,
                        void* ws, rmp_result_t* out_dev, float* per_ray, int block, int grid,
                        cudaStream_t stream);
cudaError_t launch_dense_bricks(const uint8_t* occ, const int dims[3], const int nb[3],
                                uint32_t* bricks, cudaStream_t stream);
// Slots of the occupied blocks (see block_slots_kernel; *count zeroed by the caller), then the
// box field: level 1 (grid layout, m.gdim) into `top`, level 0 into `field` (null: none; room
// for `cap` slots).
cudaError_t launch_block_slots(const uint32_t* bricks, uint32_t n, const int32_t* keys,
                               const DevMap& m, HashEntry* table, uint32_t* slot_of,
                               uint32_t* list, uint32_t* count, cudaStream_t stream);
cudaError_t launch_box_field(const DevMap& m, const uint32_t* bricks, const int32_t* keys,
                             const uint32_t* slot_of, const uint32_t* list, const uint32_t* count,
                             uint32_t cap, uint8_t* field, uint32_t* top, int sm_count,
                             cudaStream_t stream);
// Free distance of every 2^3 cell of the occupied bricks of a grid (8 words per brick,
// see rmp_map_cell_distances).
cudaError_t launch_cell_dist(const uint32_t* bricks, const DevMap& m, uint32_t* cells,
                             cudaStream_t stream);
// info: 8 words, see key_bbox_kernel (word 0 is launch_hash_build's err).
cudaError_t launch_key_bbox(const int32_t* keys, const uint32_t* bricks, uint32_t n_blocks,
                            int* info, cudaStream_t stream);
cudaError_t launch_grid_scatter(const int32_t* keys, const uint32_t* bricks, uint32_t n_blocks,
                                const DevMap& m, uint32_t* grid_bricks, cudaStream_t stream);
cudaError_t launch_tsdf_bricks(const float* tsdf, uint32_t n_blocks, uint32_t* bricks,
                               cudaStream_t stream);
cudaError_t launch_hash_build(const int32_t* keys, uint32_t n_blocks, const uint32_t* bricks,
                              HashEntry* table, uint32_t cap_mask, int hash_shift,
                              unsigned int* err, cudaStream_t stream);

}  // namespace rmp
