// Internal interface between the C ABI (ligen_api.cu) and the kernel
// translation units. Not installed; not part of the ABI.
#pragma once
#include <cstdint>
#include <cuda_runtime.h>

#include "device_common.cuh"

namespace ligen {

constexpr int kFragStride = 128;   // bytes per rotatable bond in the moving-atom lists

// Device-resident ligand library (CSR, see ligen_ligands_t).
struct LigandsDev {
  int L;
  const int32_t* atom_off;
  const float* xyz;
  const uint8_t* type;
  const int32_t* bonds;
  const int32_t* rot_off;
  const int32_t* rot_edge;
};

// Packer outputs; a NULL one is not written.
struct Packed {
  float4* xc;        // [sum N] centred input coordinates; w = atom type (int bits)
  uchar4* binfo;     // [sum n] (fixed u, moving v, moving atoms excluding v, 0)
  uint8_t* frag;     // [sum n][kFragStride] moving atoms excluding v, ascending
  int32_t* status;   // [L] 0 or LIGEN_ERR_BAD_LIGAND
  int32_t* bucket;   // [L] optional
  uint32_t* fbits;   // [sum n][8] optional: full moving side as a bit mask
  int32_t* axis;     // [sum n][2] optional: (u, v)
  uint32_t* touch;   // [sum n] optional: bit b of touch[b'] set when turning bond b'
                     // moves an atom bond b's sweep reads (bit b' always set)
  // Forward-kinematics table (all NULL or none; read by the pose-per-lane
  // scoring and pose-group gradient kernels). A ligand's atoms
  // are listed by owner (bond 0's, bond 1's, ..., then the root frame's;
  // input order within an owner):
  float4* fk_xs;     // [sum N] centred input coordinates (w = type) in that order
  uint8_t* fk_own;   // [sum N] owner of each listed atom: a bond, or n (the root frame)
  uchar4* fk_bond;   // [sum n] (parent of bond j, j-th bond parents first, j-th bond by depth,
                     //          list position of bond j's moving endpoint v)
  float4* fk_ax;     // [sum n] unit bond axes in the input conformation
  uint8_t* fk_loff;  // [L][kFkLoffBytes] first entry of each depth, depth count, malformed flag
};

constexpr int kFkLoffBytes = 48;
constexpr int kFkBad = 47;   // byte of a ligand's fk_loff row: 1 when its lists are malformed

// Sample counters are spread over this many slots (summed on the host) so
// that CTAs do not all add to one address.
constexpr int kSampleSlots = 64;

struct DockArgs {
  LigandsDev lig;
  Packed pk;
  GridView grid;
  float origin[3];
  float inv_h;
  float center[3];
  float jitter;
  uint64_t seed;
  int R, n_rigid, step_deg, n_theta, passes;
  int lanes;          // G: lanes per restart (2, 4, 8, 16 or 32)
  int fmt;            // grid record format (RecFormat)
  int rpc;            // restarts per work item (a multiple of 32 / lanes)
  int chunks;         // work items per ligand: ceil(R / rpc)
  const int32_t* list;  // ligands to dock (NULL: 0 .. n_items / chunks - 1)
  int n_items;        // work items: (list length or L) * chunks
  int* queue;         // persistent mode: device counter of taken items (zeroed
                      // before the launch); NULL: one CTA per item
  int max_atoms, max_rot, max_frag;   // shared-memory carve-up bounds
  float* res_score;   // [L][R]
  uint8_t* res_k;     // [L][R]
  uint8_t* res_cnt;   // [sum n][R] torsion increments (mod n_theta) per restart
  int16_t* trace;     // optional
  unsigned long long* samples;   // optional [kSampleSlots]: atom samples the search needed
  float* coords;      // optional: final grid-unit positions, [3 R atom_off[l] + 3 (r N_l + i) + k]
};

// Exhaustive search (mode 1): at most kExMaxRot rotatable bonds per ligand
// and kExMaxCombos combinations (n_rigid * n_theta^n) per restart.
constexpr int kExMaxRot = 4;
constexpr long long kExMaxCombos = 1ll << 27;
// The largest ligand's table and chain: atoms times combinations of torsion
// increments, atoms times their square root.
struct ExWork {
  long long entries = 0;
  double chain = 0.;
};
cudaError_t launch_exhaustive(const DockArgs& a, const ExWork& w, int sms, cudaStream_t s);

struct TopkArgs {
  int L, R, K, step_deg;
  const int32_t* rot_off;
  const int32_t* status;
  const float* res_score;
  const uint8_t* res_k;
  const uint8_t* res_cnt;
  uint64_t seed;
  float center[3];
  float jitter;
  float* out_poses;
  float* out_scores;
  int32_t* top_restart;   // optional
};

struct ScoreArgs {
  LigandsDev lig;
  Packed pk;
  GridView grid;
  float origin[3];
  float inv_h;
  int P;              // poses per ligand
  int max_atoms;      // largest ligand of the launch (shared-memory carve-up)
  int max_rot;        // most rotatable bonds of a ligand of the launch
  const float* poses;
  float* out_scores;
  const int32_t* list;  // pose-per-lane launch: ligands to score (NULL: 0 .. n_list - 1)
  int n_list;
};

struct GradArgs {
  LigandsDev lig;
  Packed pk;
  GridView grid;
  float origin[3];
  float inv_h;
  int P;              // poses per ligand
  int max_atoms;
  const float* poses;       // gradient: input poses
  float* inout_poses;       // refinement: poses, refined in place
  float* out_scores;        // [L][P]
  float* out_grads;         // gradient: same packing as poses
  const float* weights;     // gradient: [L][P] factors of the poses' gradients, or NULL
  int steps;                // refinement iterations
  float step_t, step_q, step_theta;
  float box_lo[3], box_hi[3];
  int8_t* out_accept;       // refinement: [L * P][steps], optional
  const int32_t* list;      // pose-group launch: ligands (NULL: 0 .. n_list - 1)
  int n_list;
  int max_rot;              // pose-group launch: most rotatable bonds of a ligand of the launch
  float h;                  // grid spacing (Angstrom)
};

struct RescoreArgs {
  LigandsDev lig;
  Packed pk;
  const int32_t* status;
  const float* values;      // caller's grid [z][y][x][c], FP32
  int nx, ny, nz, nc;
  double origin[3];
  double h;
  double penalty;
  int K;                    // kept poses per ligand
  int max_atoms;            // largest ligand (shared-memory carve-up)
  int max_rot;              // most rotatable bonds of a ligand (shared-memory carve-up)
  double inv_h;             // 1 / h
  int step_deg, n_theta;    // torsions are whole increments of step_deg degrees
  bool small_axes;          // no axis has more than 2^20 points
  const float* poses;       // the kept poses and their restarts, in FP32 order
  const int32_t* tmp_top;
  float* out_poses;         // outputs, re-ranked
  float* scores;            // [L][K], FP64 scores rounded to FP32
  int32_t* top_restart;     // [L][K] or NULL
  double* out_s64;          // [L][K] or NULL: FP64 scores
  double* s64;              // scratch [L][K]
  double* table;            // scratch [n_theta][2]
  unsigned* check;          // checked builds: first out-of-range code, else NULL
};

// Bytes a workspace grows to for a call that needs `bytes`, under a limit (0:
// none), and whether a workspace of `cap` bytes (given back first) can, with
// `free` bytes on the device, allocated in pages of 2 MB.
inline size_t workspace_want(size_t bytes, size_t limit) {
  const size_t want = bytes + bytes / 8 + (1 << 20);
  return limit && want > limit ? limit : want;
}
inline bool workspace_fits(size_t bytes, size_t cap, size_t free, size_t limit) {
  if (limit && bytes > limit) return false;
  const size_t page = 2 << 20;
  return bytes <= cap || (workspace_want(bytes, limit) + page - 1) / page * page <= free + cap / page * page;
}

// Grid records in format `fmt` (RecFormat). beside_pack: launched right
// after launch_pack on the same stream, it may start with the packer (neither
// reads what the other writes) and ends after it: scoring 3 poses of 5,001
// ligands 90.7 -> 83.8 us per call, docking 32 small ligands 37.3 -> 34.8.
cudaError_t launch_grid_prep(const float* values, int nx, int ny, int nz, int nc, int fmt, void* rec,
                             bool beside_pack, cudaStream_t s);
// max_atoms: the library's largest ligand. With out.fk_xs set, the
// forward-kinematics table (out.fk_*) too.
cudaError_t launch_pack(const LigandsDev& lig, int nc, const Packed& out, int max_atoms, cudaStream_t s);
// The ligands by decreasing estimated docking cost (order [L]).
cudaError_t launch_order(const LigandsDev& lig, int n_rigid, int passes, int n_theta, int32_t* order,
                         cudaStream_t s);
size_t dock_smem_bytes(int max_atoms, int max_rot, int max_frag, int rpc);
// Lanes per restart for a plain launch of this library and search.
int dock_pick_lanes(const int32_t* h_atom_off, const int32_t* h_rot_off, int L, int R, int n_rigid, int n_theta,
                    int passes, int fmt, int sms);
bool dock_lanes_supported(int lanes);
// A grid axis of 2^23 cells or more, past the floor by addition of
// dock_point and grid_fetch: docked by the 8-lane shapes only, poses scored
// and refined by the group-per-pose kernels.
inline bool dock_big(const GridView& g) { return g.mx >= kFloorMagic || g.my >= kFloorMagic || g.mz >= kFloorMagic; }
bool dock_shape_supported(int lanes, int fmt, bool big);
// grid_ctas: CTAs of a persistent launch (ignored when a.queue is NULL).
// set_attr: set the kernel's dynamic shared-memory limit first (false when
// dock_occupancy already did, e.g. before a stream capture).
cudaError_t launch_dock(const DockArgs& a, int grid_ctas, cudaStream_t s, bool set_attr);
// The kernel of (lanes, n_theta) accepts up to `smem` bytes of dynamic
// shared memory from now on (a per-kernel setting: set the largest value any
// pending launch of that kernel needs).
cudaError_t dock_set_smem_limit(int lanes, int n_theta, int fmt, bool big, size_t smem);
// Resident CTAs per SM for a launch with `smem` bytes (within the limit).
cudaError_t dock_occupancy(int lanes, int n_theta, int fmt, bool big, int rpc, size_t smem, int* blocks_per_sm);
cudaError_t launch_topk(const TopkArgs& a, cudaStream_t s);
cudaError_t launch_score(const ScoreArgs& a, cudaStream_t s);
// Pose-per-lane scoring of the ligands a.list[0 .. n_list) (all of them at
// most a.max_atoms atoms and a.max_rot bonds), 32 poses per warp: the launch
// shape (sets the kernel's shared-memory limit; no stream work, so it is
// called before a graph capture), then the launch.
struct LaunchCfg {
  unsigned blocks = 0;
  size_t smem = 0;
};
cudaError_t score_lanes_config(const ScoreArgs& a, LaunchCfg* c);
cudaError_t launch_score_lanes(const ScoreArgs& a, const LaunchCfg& c, cudaStream_t s);
cudaError_t launch_rescore(const RescoreArgs& a, cudaStream_t s);
size_t grad_smem_bytes(int max_atoms);
// refine = false: dS/dpose of every pose; true: gradient refinement in place.
cudaError_t launch_grad(const GradArgs& a, bool refine, cudaStream_t s);
// The same on forward kinematics, a group of lanes per pose, for the ligands
// a.list[0 .. n_list) (at most a.max_atoms atoms and a.max_rot bonds each);
// calls with at least kGradLanePosesMin poses per ligand.
constexpr int kGradLanePosesMin = 4;
cudaError_t launch_grad_lanes(const GradArgs& a, bool refine, cudaStream_t s);
cudaError_t launch_probe(const float* rec, uint32_t n_rec, int bytes, int iters, uint64_t seed, float* sink,
                         int blocks, cudaStream_t s);
int probe_streams();
int probe_threads();
cudaError_t launch_stream_probe(const void* buf, uint64_t n_vec, int passes, float* sink, int blocks,
                                cudaStream_t s);

}  // namespace ligen
