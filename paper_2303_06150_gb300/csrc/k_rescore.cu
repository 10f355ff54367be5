// FP64 re-score of kept poses and re-ranking: FP64 arithmetic on the GPU is
// spent only on the K kept poses of each ligand, where near-ties between
// FP32 scores decide the ranking.
//
// Everything is recomputed in FP64 from the caller's FP32 inputs: the input
// centroid, the pose's atom positions, and the trilinear value from the
// eight FP32 node values of the caller's [z][y][x][c] grid. The positions
// follow the pose definition (torsions bond by bond in index order, each
// about its current axis; then R(q/|q|) and t) as forward kinematics in
// FP64, equal in exact arithmetic: bond b's transform is its parent's
// composed with the rotation by theta_b about b's input-frame axis through
// its moving endpoint v, and an atom's position is its owner's transform of
// its centred input coordinates (owners, parents and the bond order from
// fk_stage, as in the scoring kernels).
//
// Mapping. GB300 issues FP64 at a small fraction of its FP32 rate (one warp
// instruction in 64 cycles per scheduler, however few lanes are active), so
// the FP64 instruction count decides the time. A warp holds kRsPoses poses of
// one ligand, a group of kRsLanes lanes per pose:
//   * the bond axes and pivots once per warp, one lane per bond;
//   * torsions are whole increments, so their sines and cosines come from a
//     table of the call's increments (rescore_table_kernel);
//   * every (pose, bond) rotation matrix in one pass over the warp's lanes;
//   * row r of a bond's transform needs row r of its parent's only: lanes 0-2
//     of a group carry one row each through the bonds, parents first;
//   * transforms map to grid units, so an atom costs one 3x4 product;
//   * box test, cell and floor by integer operations on the coordinate's
//     bits, and node values widened by shifting theirs: conversions and
//     comparisons would run on the FP64 pipe.
// 27 FP64 instructions an atom (53 with conversions, comparisons and world
// coordinates). Measured on GB300, the kernel for the 180,000 kept poses of
// 6,000 screening ligands: 1,371 us before these last five points, 957 us after.
// Earlier versions, re-score stage of 600,000 poses: a warp per pose 28 ms,
// torsions atom by atom 8.5, forward kinematics with 4 poses per warp 6.5,
// with 8 poses per warp 5.1.
// Re-ranking: one warp per ligand orders its K poses by FP64 score
// (descending; ties by the restart that produced them) and rewrites poses,
// scores and restart ids in that order.
#include <cmath>

#include "../../include/ligen.h"
#include "internal.h"
#include "fk_pose.cuh"

namespace ligen {
namespace {

constexpr int kResWarps = 4;
// lanes per pose: the warp's per-pose FP64 passes (root, sines and cosines,
// transforms by depth) serve 32 / kRsLanes poses. Measured on GB300, the
// re-score stage of a screening step: 8 lanes 6.6 ms, 4 lanes 5.2 ms,
// 2 lanes 5.6 ms.
constexpr int kRsLanes = 4;
constexpr int kRsPoses = 32 / kRsLanes;            // poses per warp (one ligand)
constexpr unsigned kFull = 0xffffffffu;

__device__ __forceinline__ double warp_sum_d(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(kFull, v, o);
  return v;
}

__device__ __forceinline__ double group_sum_d(double v) {
#pragma unroll
  for (int o = kRsLanes / 2; o > 0; o >>= 1) v += __shfl_xor_sync(kFull, v, o);
  return v;
}

// A float as a double by moving its bits (sign, exponent rebiased, mantissa):
// exact for zeros and normal values; the rest takes the conversion.
__device__ __forceinline__ double widen(float v) {
  const unsigned b = __float_as_uint(v), a = b & 0x7fffffffu;
  if (a - 1u >= 0x007fffffu && a < 0x7f800000u)   // zero or a normal value
    return __hiloint2double((int)((b & 0x80000000u) | (a ? (a >> 3) + 0x38000000u : 0u)), (int)(b << 29));
  return (double)v;
}

// The cell and fraction of coordinate u on an axis of n points; false outside
// 0 <= u <= n - 1. The bits of a double order like an integer's, and its
// floor is the mantissa cut at the exponent. Axes of up to 2^20 points.
__device__ __forceinline__ bool cell64(double u, int n, double last, int* i, double* f) {
  const long long b = __double_as_longlong(u);
  if ((unsigned long long)b > (unsigned long long)__double_as_longlong(last) && u != 0.0) return false;
  const int hi = (int)(b >> 32) & 0x7fffffff, drop = 20 - ((hi >> 20) - 1023);   // fraction bits of the high word
  int c = ((hi & 0xfffff) | 0x100000) >> min(drop, 31);
  double fl = __hiloint2double(drop > 20 ? 0 : hi & ~((1 << max(drop, 0)) - 1), 0);
  if (c > n - 2) {   // the upper face: the last cell at f = 1
    c = n - 2;
    fl = last - 1.0;
  }
  *i = c;
  *f = u - fl;
  return true;
}

__device__ __forceinline__ bool cell64_any(double u, int n, double last, int* i, double* f) {
  if (!(u >= 0.0 && u <= last)) return false;
  *i = min(__double2int_rd(u), n - 2);
  *f = u - *i;
  return true;
}

// FP64 trilinear value of channel c at grid point (u0, u1, u2): 7
// interpolations (x, then y, then z) of the 8 FP32 node values widened to
// FP64. Outside the box: the penalty.
__device__ __forceinline__ double trilinear64(const RescoreArgs& a, double u0, double u1, double u2, int c) {
  int i0, i1, i2;
  double f0, f1, f2;
  if (a.small_axes) {   // uniform
    if (!cell64(u0, a.nx, (double)(a.nx - 1), &i0, &f0) || !cell64(u1, a.ny, (double)(a.ny - 1), &i1, &f1) ||
        !cell64(u2, a.nz, (double)(a.nz - 1), &i2, &f2))
      return a.penalty;
  } else {
    if (!cell64_any(u0, a.nx, (double)(a.nx - 1), &i0, &f0) || !cell64_any(u1, a.ny, (double)(a.ny - 1), &i1, &f1) ||
        !cell64_any(u2, a.nz, (double)(a.nz - 1), &i2, &f2))
      return a.penalty;
  }
  const size_t sx = (size_t)a.nc, sy = sx * a.nx, sz = sy * a.ny;
  const size_t base = ((size_t)i2 * a.ny + i1) * a.nx + i0;
  if (!lg_check(a.check, c >= 0 && c < a.nc && base + (size_t)a.nx * a.ny + a.nx + 1 < (size_t)a.nx * a.ny * a.nz,
                kChkRescoreNode))
    return a.penalty;
  const float* v = a.values + base * sx + c;
  const float v000 = v[0], v100 = v[sx], v010 = v[sy], v110 = v[sy + sx];
  const float v001 = v[sz], v101 = v[sz + sx], v011 = v[sz + sy], v111 = v[sz + sy + sx];
  const double c000 = widen(v000), c010 = widen(v010), c001 = widen(v001), c011 = widen(v011);
  const double e00 = fma(f0, widen(v100) - c000, c000), e10 = fma(f0, widen(v110) - c010, c010);
  const double e01 = fma(f0, widen(v101) - c001, c001), e11 = fma(f0, widen(v111) - c011, c011);
  const double e0 = fma(f1, e10 - e00, e00), e1 = fma(f1, e11 - e01, e01);
  return fma(f2, e1 - e0, e0);
}

// Sine and cosine of every torsion increment, in its pose's FP32 radians
// (the values topk writes), in FP64: table[2 j], table[2 j + 1].
__global__ void rescore_table_kernel(int n_theta, int step_deg, double* table) {
  const int j = blockIdx.x * blockDim.x + threadIdx.x;
  if (j < n_theta) sincos((double)torsion_radians(j, step_deg), &table[2 * j], &table[2 * j + 1]);
}

// Shared memory of one warp: the staged ligand (fk_stage), then per bond
// its unit axis and pivot v in the input frame (FP64, 6 each), then the
// transforms of the warp's poses (FP64, 12 each) [slot][pose][12], the
// centred input coordinates (FP64, 3 per atom).
__host__ __device__ inline size_t rs_warp_bytes(int acap, int ncap, unsigned char* base, FkLigand* S, double** B,
                                                double** T, double** Y) {
  const size_t lb = fk_ligand_carve(acap, ncap, base, S, true);   // a multiple of 16
  const size_t bb = (size_t)ncap * 6 * sizeof(double);
  const size_t tb = (size_t)(ncap + 1) * kRsPoses * 12 * sizeof(double);
  const size_t yb = ((size_t)acap * 3 * sizeof(double) + 15) & ~(size_t)15;
  if (base) {
    *B = reinterpret_cast<double*>(base + lb);
    *T = reinterpret_cast<double*>(base + lb + bb);
    *Y = reinterpret_cast<double*>(base + lb + bb + tb);
  }
  return lb + bb + tb + yb;
}

__global__ void __launch_bounds__(32 * kResWarps) rescore_kernel(const RescoreArgs a) {
  extern __shared__ __align__(16) unsigned char rs_smem[];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int grp = lane / kRsLanes, sub = lane % kRsLanes;
  const int acap = a.max_atoms, ncap = a.max_rot;
  FkLigand S;
  double *B, *T, *Y;
  const size_t per = rs_warp_bytes(acap, ncap, nullptr, nullptr, nullptr, nullptr, nullptr);
  rs_warp_bytes(acap, ncap, rs_smem + (size_t)w * per, &S, &B, &T, &Y);
  const int wpl = (a.K + kRsPoses - 1) / kRsPoses;   // warps per ligand
  const size_t gw = (size_t)blockIdx.x * kResWarps + w;
  if (gw >= (size_t)a.lig.L * wpl) return;   // uniform over the warp
  const int l = (int)(gw / wpl);
  const int p0 = (int)(gw % wpl) * kRsPoses + grp;
  const bool own = p0 < a.K;
  const int p = own ? p0 : a.K - 1;          // spare groups shadow the last pose
  const size_t gp = (size_t)l * a.K + p;
  const int a0 = a.lig.atom_off[l];
  const int N = a.lig.atom_off[l + 1] - a0;
  const int r0 = a.lig.rot_off[l];
  const int n = a.lig.rot_off[l + 1] - r0;
  bool ok = a.status[l] == 0 && lg_check(a.check, N <= acap && n <= ncap, kChkItemShape);   // uniform
  if (ok) ok = lg_check(a.check, fk_stage(a.pk, a0, N, r0, n, S, lane), kChkAtomIndex);
  if (!ok) {
    if (own && sub == 0) a.s64[gp] = -INFINITY;
    return;
  }
  // FP64 centroid of the input coordinates
  double c0[3] = {0.0, 0.0, 0.0};
  for (int i = lane; i < N; i += 32)
    for (int k = 0; k < 3; ++k) c0[k] += (double)a.lig.xyz[3 * (a0 + i) + k];
  for (int k = 0; k < 3; ++k) c0[k] = warp_sum_d(c0[k]);
  {   // one division for the three components
    const double q = (lane == 0 ? c0[0] : lane == 1 ? c0[1] : c0[2]) / N;
    for (int k = 0; k < 3; ++k) c0[k] = __shfl_sync(kFull, q, k);
  }
  for (int i = lane; i < N; i += 32)   // centred coordinates, once for the warp's poses
    for (int k = 0; k < 3; ++k) Y[3 * i + k] = (double)a.lig.xyz[3 * (a0 + i) + k] - c0[k];
  // per bond, once for the warp's poses: unit axis u -> v and pivot v in the
  // input frame (fk_stage checked both ends against N)
  for (int b = lane; b < n; b += 32) {
    const uchar4 bi = S.sb[b];
    double pu[3], pv[3];
    for (int k = 0; k < 3; ++k) {
      pu[k] = (double)a.lig.xyz[3 * (a0 + bi.x) + k] - c0[k];
      pv[k] = (double)a.lig.xyz[3 * (a0 + bi.y) + k] - c0[k];
    }
    const double kx = pv[0] - pu[0], ky = pv[1] - pu[1], kz = pv[2] - pu[2];
    const double inv = rsqrt(kx * kx + ky * ky + kz * kz);
    double* bb = B + 6 * b;
    bb[0] = kx * inv; bb[1] = ky * inv; bb[2] = kz * inv;
    bb[3] = pv[0]; bb[4] = pv[1]; bb[5] = pv[2];
  }
  // the pose's transforms (input frame -> grid units): the root R(q/|q|) / h
  // and (t - origin) / h, then bond by bond, parents first: bond b's is its
  // parent's composed with the rotation by theta_b about b's axis through v
  const float* pose = a.poses + (size_t)a.K * (7 * (size_t)l + r0) + (size_t)p * (7 + n);
  const size_t stride = (size_t)kRsPoses * 12;
  double* Tg = T + 12 * grp;
  __syncwarp();   // axes and coordinates
  // every (pose, bond) rotation c I + s [k]x + (1 - c) k k^T, right-handed
  // about k, parked in the slot that its transform takes later
  for (int b = sub; b < n; b += kRsLanes) {
    const int jt = torsion_increment(pose[7 + b], a.step_deg, a.n_theta);
    const double sn = __ldg(a.table + 2 * jt), cs = __ldg(a.table + 2 * jt + 1);
    const double* bb = B + 6 * b;
    const double kx = bb[0], ky = bb[1], kz = bb[2];
    const double tc = 1.0 - cs, tx = tc * kx, ty = tc * ky, tz = tc * kz;
    const double sx = sn * kx, sy = sn * ky, sz = sn * kz;
    double* Rb = Tg + (size_t)b * stride;
    Rb[0] = fma(tx, kx, cs); Rb[1] = fma(tx, ky, -sz); Rb[2] = fma(tx, kz, sy);
    Rb[3] = fma(tx, ky, sz); Rb[4] = fma(ty, ky, cs);  Rb[5] = fma(ty, kz, -sx);
    Rb[6] = fma(tx, kz, -sy); Rb[7] = fma(ty, kz, sx); Rb[8] = fma(tz, kz, cs);
  }
  const double inv_h = a.inv_h;
  const int r = sub < 3 ? sub : 2;   // the row this lane carries (the spare lane repeats the last)
  {
    const double qi = rsqrt((double)pose[3] * pose[3] + (double)pose[4] * pose[4] + (double)pose[5] * pose[5] +
                            (double)pose[6] * pose[6]);
    const double qw = pose[3] * qi, qv[3] = {pose[4] * qi, pose[5] * qi, pose[6] * qi};
    // row r of R: column c = r: 1 - 2 (y^2 + z^2) of the other two; else 2 (v_r v_c +- w v_k)
    const int c1 = r == 2 ? 0 : r + 1, c2 = r == 0 ? 2 : r - 1;
    const double vr = r == 0 ? qv[0] : r == 1 ? qv[1] : qv[2];
    const double v1 = c1 == 0 ? qv[0] : c1 == 1 ? qv[1] : qv[2], v2 = c2 == 0 ? qv[0] : c2 == 1 ? qv[1] : qv[2];
    double* Tr = Tg + (size_t)n * stride + 4 * r;
    if (sub < 3) {
      const double o = r == 0 ? a.origin[0] : r == 1 ? a.origin[1] : a.origin[2];
      Tr[r] = (1.0 - 2.0 * (v1 * v1 + v2 * v2)) * inv_h;
      Tr[c1] = 2.0 * (vr * v1 - qw * v2) * inv_h;
      Tr[c2] = 2.0 * (vr * v2 + qw * v1) * inv_h;
      Tr[3] = ((double)pose[r] - o) * inv_h;
    }
  }
  __syncwarp();   // rotations
  for (int k = 0; k < n; ++k) {
    const int b = S.ord[k];
    const double* P = Tg + (size_t)S.par[b] * stride + 4 * r;   // written by this lane
    double* Tb = Tg + (size_t)b * stride;
    const double* bb = B + 6 * b;
    const double p0r = P[0], p1r = P[1], p2r = P[2], p3r = P[3];
    const double m0 = p0r * Tb[0] + p1r * Tb[3] + p2r * Tb[6];
    const double m1 = p0r * Tb[1] + p1r * Tb[4] + p2r * Tb[7];
    const double m2 = p0r * Tb[2] + p1r * Tb[5] + p2r * Tb[8];
    // v keeps its place: o_b = T_p(v) - M_b v
    const double tp = p0r * bb[3] + p1r * bb[4] + p2r * bb[5] + p3r;
    const double ob = tp - (m0 * bb[3] + m1 * bb[4] + m2 * bb[5]);
    __syncwarp();   // the rotation is read by all three rows before any is written
    if (sub < 3) {
      Tb[4 * r] = m0;
      Tb[4 * r + 1] = m1;
      Tb[4 * r + 2] = m2;
      Tb[4 * r + 3] = ob;
    }
    __syncwarp();
  }
  // the group's lanes split the atoms: owner's transform, FP64 trilinear value
  double Sg = 0.0;
  for (int i = sub; i < N; i += kRsLanes) {
    const double* M = Tg + (size_t)S.own[i] * stride;
    const double* y = Y + 3 * i;
    double u[3];
    for (int e = 0; e < 3; ++e) u[e] = M[4 * e] * y[0] + M[4 * e + 1] * y[1] + M[4 * e + 2] * y[2] + M[4 * e + 3];
    Sg -= trilinear64(a, u[0], u[1], u[2], a.lig.type[a0 + i]);
  }
  Sg = group_sum_d(Sg);
  if (own && sub == 0) a.s64[gp] = Sg;
}

// Re-rank the K poses of each ligand by FP64 score; ties go to the lower
// restart. Up to 32 poses: a lane per pose counts the poses before its own
// (6,000 ligands x 30 poses: 189 us with a round per rank that read the
// scores from memory, 42 us). More: a round per rank.
__global__ void __launch_bounds__(32 * kResWarps) rerank_kernel(const RescoreArgs a) {
  const int lane = threadIdx.x & 31;
  const int l = blockIdx.x * kResWarps + (threadIdx.x >> 5);
  if (l >= a.lig.L) return;
  const int r0 = a.lig.rot_off[l];
  const int n = a.lig.rot_off[l + 1] - r0;
  const int plen = 7 + n;
  const size_t base = (size_t)a.K * (7 * (size_t)l + r0);
  const double* s = a.s64 + (size_t)l * a.K;
  if (a.K <= 32) {   // uniform
    const bool have = lane < a.K;
    const double raw = have ? s[lane] : -INFINITY;
    const double v = isnan(raw) ? -INFINITY : raw;
    const int key = have ? a.tmp_top[(size_t)l * a.K + lane] : 0;
    int rank = 0;
    for (int p = 0; p < a.K; ++p) {
      const double ov = __shfl_sync(kFull, v, p);
      const int ok = __shfl_sync(kFull, key, p);
      rank += ov > v || (ov == v && (ok < key || (ok == key && p < lane)));
    }
    if (have) {
      const size_t o = (size_t)l * a.K + rank;
      a.scores[o] = (float)v;
      if (a.out_s64) a.out_s64[o] = v;
      if (a.top_restart) a.top_restart[o] = key;
    }
#pragma unroll 4
    for (int p = 0; p < a.K; ++p) {
      const int to = __shfl_sync(kFull, rank, p);
      for (int e = lane; e < plen; e += 32)
        a.out_poses[base + (size_t)to * plen + e] = a.poses[base + (size_t)p * plen + e];
    }
    return;
  }
  double last_s = INFINITY;
  int last_key = -1;
  for (int rank = 0; rank < a.K; ++rank) {
    double bs = -INFINITY;
    int bkey = 0x7fffffff, bp = 0;
    for (int p = lane; p < a.K; p += 32) {
      const double v = isnan(s[p]) ? -INFINITY : s[p];
      const int key = a.tmp_top[(size_t)l * a.K + p];
      const bool after = (v < last_s) || (v == last_s && key > last_key);
      if (after && (v > bs || (v == bs && key < bkey))) { bs = v; bkey = key; bp = p; }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      const double os = __shfl_xor_sync(kFull, bs, o);
      const int ok = __shfl_xor_sync(kFull, bkey, o);
      const int op = __shfl_xor_sync(kFull, bp, o);
      if (os > bs || (os == bs && ok < bkey)) { bs = os; bkey = ok; bp = op; }
    }
    last_s = bs;
    last_key = bkey;
    for (int e = lane; e < plen; e += 32)
      a.out_poses[base + (size_t)rank * plen + e] = a.poses[base + (size_t)bp * plen + e];
    if (lane == 0) {
      a.scores[(size_t)l * a.K + rank] = (float)bs;
      if (a.out_s64) a.out_s64[(size_t)l * a.K + rank] = bs;
      if (a.top_restart) a.top_restart[(size_t)l * a.K + rank] = a.tmp_top[(size_t)l * a.K + bp];
    }
  }
}

}  // namespace

cudaError_t launch_rescore(const RescoreArgs& a, cudaStream_t s) {
  const size_t total = (size_t)a.lig.L * a.K;
  if (total == 0) return cudaSuccess;
  const size_t smem =
      (size_t)kResWarps * rs_warp_bytes(a.max_atoms, a.max_rot, nullptr, nullptr, nullptr, nullptr, nullptr);
  if (smem > 48 * 1024) {
    cudaError_t e = cudaFuncSetAttribute(rescore_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
  }
  rescore_table_kernel<<<(a.n_theta + 127) / 128, 128, 0, s>>>(a.n_theta, a.step_deg, a.table);
  const size_t warps = (size_t)a.lig.L * ((a.K + kRsPoses - 1) / kRsPoses);
  rescore_kernel<<<(unsigned)((warps + kResWarps - 1) / kResWarps), 32 * kResWarps, smem, s>>>(a);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  rerank_kernel<<<(unsigned)((a.lig.L + kResWarps - 1) / kResWarps), 32 * kResWarps, 0, s>>>(a);
  return cudaGetLastError();
}

}  // namespace ligen
