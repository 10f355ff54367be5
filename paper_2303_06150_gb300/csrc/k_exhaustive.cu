// Exhaustive search (mode 1, small ligands): for every restart, every
// combination of a cube rotation k and torsion increments (j_0 .. j_{n-1})
// is scored and the best kept, ties going to the combination that comes
// first in lexicographic order of (k, j_0, .., j_{n-1}). It is the brute
// force the greedy search is an approximation of: per restart, greedy <=
// exhaustive. The result is written in the greedy kernel's per-restart
// format (score, k, increments), so top-K, pose compaction and the FP64
// re-score follow unchanged.
//
// An atom's position in a combination depends on k and on the increments of
// the bonds that move it, not on the others: a bond that moves another
// bond's axis moves that bond's whole list. So an atom moved by m of the n
// bonds has n_theta^m energies per rotation, not n_theta^n, and they are
// sampled once into a table in shared memory; a combination then costs one
// table read and one subtraction per atom, in atom order, which gives the
// same bits as rebuilding and sampling every atom of every combination.
// Atoms go into the table by ascending m while kExTable entries hold them;
// the ones that do not fit (many increments, deeply nested bonds) are
// rebuilt per combination.
//
// A cluster of 1, 2, 4 or 8 CTAs takes one (ligand, restart), the rotations
// split over its CTAs, and joins its winners through distributed shared
// memory: without the split a call of a few hundred restarts leaves the
// chip to the few ligands with the most bonds, with it every CTA more stages
// the ligand and lays out the table again. launch_exhaustive has the rule.
// Measured on GB300, 97 ligands of 8-20 atoms and 0-3 bonds, 8 restarts, 30
// degree steps, whole call: 2,780 us with every combination rebuilt by one
// CTA per (ligand, restart), 173-273 us this way by the seed's library (269
// where eight CTAs for every call take 280).
#include <cooperative_groups.h>

#include "../../include/ligen.h"
#include "internal.h"

namespace ligen {
namespace {

constexpr int kExThreads = 128;
constexpr int kExCluster = 8;     // CTAs per (ligand, restart), at most: the portable maximum
constexpr int kExTable = 6144;    // table entries: 24 KB
constexpr int kExSmall = 1024;    // table entries of the build for little work
constexpr int kExVec = 4;         // combinations a thread sums side by side
constexpr uint16_t kExDirect = 0xffffu;

// q / d for q < 2^27 by multiplication: m = ceil(2^40 / d) is off by less
// than d / 2^40 relative to 1 / d, q * d < 2^40, and the product fits 64 bits
// because q < n_rigid * d^4 and q < 2^27.
struct ExDiv {
  unsigned d;
  unsigned long long m;
  explicit ExDiv(unsigned dd) : d(dd), m(((1ull << 40) + dd - 1) / dd) {}
  __device__ unsigned operator()(unsigned q) const { return d == 1 ? q : (unsigned)((q * m) >> 40); }
};

// A launch: CTAs per (ligand, restart), table entries per CTA, atoms of the
// largest ligand rounded up to 16.
struct ExLaunch {
  int cluster, table, acap;
  ExDiv by_nt;
};

// Shared memory for ligands of at most acap atoms (a multiple of 16), the
// table behind them.
struct ExLigand {
  float4* sx;
  uint2* stride;     // table strides of bonds 0..3, 16 bits each
  uint16_t* base;    // first table entry, or kExDirect
  uint8_t* mask;     // bonds that move the atom
  uint8_t* slot;     // tabled atoms by first entry
  float* tab;
  int (*axis)[2];    // [kExMaxRot]
  int n_slots, entries;
};
__host__ __device__ inline size_t ex_smem_bytes(int acap, int table) { return 28 * (size_t)acap + 4 * (size_t)table; }

// Bond b's axis after the earlier bonds of `use` with increments j: moving
// end pv, unit direction kd, and the turn's cosine and sine.
__device__ __forceinline__ void ex_axes(const ExLigand& S, unsigned use, int n, const int (&j)[kExMaxRot], int step_deg,
                                        float (&pv)[kExMaxRot][3], float (&kd)[kExMaxRot][3], float (&cs)[kExMaxRot],
                                        float (&sn)[kExMaxRot]) {
#pragma unroll
  for (int b = 0; b < kExMaxRot; ++b) {
    if (b >= n) break;
    if (!(use >> b & 1u)) continue;
    const int iu = S.axis[b][0], iv = S.axis[b][1];
    float pu[3] = {S.sx[iu].x, S.sx[iu].y, S.sx[iu].z};
    float pw[3] = {S.sx[iv].x, S.sx[iv].y, S.sx[iv].z};
#pragma unroll
    for (int e = 0; e < kExMaxRot; ++e) {
      if (e >= b) break;
      if (!(use >> e & 1u)) continue;
      if (S.mask[iu] >> e & 1u) rodrigues_apply(pu, pv[e], kd[e], cs[e], sn[e]);
      if (S.mask[iv] >> e & 1u) rodrigues_apply(pw, pv[e], kd[e], cs[e], sn[e]);
    }
    const float d0 = pw[0] - pu[0], d1 = pw[1] - pu[1], d2 = pw[2] - pu[2];
    const float inv = rsqrtf(d0 * d0 + d1 * d1 + d2 * d2);
    kd[b][0] = d0 * inv; kd[b][1] = d1 * inv; kd[b][2] = d2 * inv;
    pv[b][0] = pw[0]; pv[b][1] = pw[1]; pv[b][2] = pw[2];
    torsion_cs(j[b], step_deg, &cs[b], &sn[b]);
  }
}

// Energy of atom i, turned by the bonds of its mask, under the rotation and
// scaling Mk and the offset o.
template <int FMT>
__device__ __forceinline__ float ex_energy(const DockArgs& a, const ExLigand& S, int i, int n, const float* Mk,
                                           const float* o, const float (&pv)[kExMaxRot][3],
                                           const float (&kd)[kExMaxRot][3], const float (&cs)[kExMaxRot],
                                           const float (&sn)[kExMaxRot]) {
  const float4 X = S.sx[i];
  float y[3] = {X.x, X.y, X.z};
#pragma unroll
  for (int b = 0; b < kExMaxRot; ++b) {
    if (b >= n) break;
    if (S.mask[i] >> b & 1u) rodrigues_apply(y, pv[b], kd[b], cs[b], sn[b]);
  }
  const float ux = fmaf(Mk[0], y[0], fmaf(Mk[1], y[1], fmaf(Mk[2], y[2], o[0])));
  const float uy = fmaf(Mk[3], y[0], fmaf(Mk[4], y[1], fmaf(Mk[5], y[2], o[1])));
  const float uz = fmaf(Mk[6], y[0], fmaf(Mk[7], y[1], fmaf(Mk[8], y[2], o[2])));
  return grid_sample_fmt<FMT>(a.grid, ux, uy, uz, __float_as_int(X.w));
}

// Best of `total` combinations that start at combination c0 of the search
// (whole rotations; the table holds them), all atoms tabled. NB >= n.
template <int NB>
__device__ __forceinline__ void ex_sum(const ExLigand& S, int N, int n, const ExDiv& by_nt,
                                       unsigned total, long long c0, float& best, long long& bestc) {
  for (unsigned t = threadIdx.x; t < total; t += kExThreads * kExVec) {
    unsigned off[kExVec];
    unsigned j[kExVec][NB];
    float acc[kExVec];
#pragma unroll
    for (int v = 0; v < kExVec; ++v) {
      unsigned q = min(t + v * kExThreads, total - 1);
#pragma unroll
      for (int b = NB - 1; b >= 0; --b) {
        j[v][b] = 0u;
        if (b < n) {
          const unsigned up = by_nt(q);
          j[v][b] = q - up * by_nt.d;
          q = up;
        }
      }
      off[v] = q * S.entries;
      acc[v] = 0.f;
    }
    for (int i = 0; i < N; ++i) {
      const uint2 s = S.stride[i];
      const unsigned base = S.base[i];
#pragma unroll
      for (int v = 0; v < kExVec; ++v) {
        unsigned at = base + off[v] + j[v][0] * (s.x & 0xffffu);
        if constexpr (NB > 1) at += j[v][1] * (s.x >> 16);
        if constexpr (NB > 2) at += j[v][2] * (s.y & 0xffffu);
        if constexpr (NB > 3) at += j[v][3] * (s.y >> 16);
        acc[v] -= S.tab[at];
      }
    }
#pragma unroll
    for (int v = 0; v < kExVec; ++v)   // t ascends per thread: ties keep the first
      if (t + v * kExThreads < total && acc[v] > best) {
        best = acc[v];
        bestc = c0 + t + v * kExThreads;
      }
  }
}

// MINB: resident CTAs asked of the register allocator: 1 (155 registers, three
// CTAs per SM), or 8 (64, spilling) for launches of little work, whose time is
// what every CTA does before and after it.
template <int FMT, int MINB>
__global__ void __launch_bounds__(kExThreads, MINB) exhaustive_kernel(const DockArgs a, const ExLaunch x, unsigned first) {
  namespace cg = cooperative_groups;
  extern __shared__ __align__(16) unsigned char ex_smem[];
  __shared__ int s_axis[kExMaxRot][2];
  __shared__ int s_table[2];   // tabled atoms, entries
  __shared__ float red_s[kExThreads / 32];
  __shared__ long long red_c[kExThreads / 32];
  __shared__ float cta_s;
  __shared__ long long cta_c;

  ExLigand S;
  S.sx = reinterpret_cast<float4*>(ex_smem);
  S.stride = reinterpret_cast<uint2*>(S.sx + x.acap);
  S.tab = reinterpret_cast<float*>(S.stride + x.acap);
  S.base = reinterpret_cast<uint16_t*>(S.tab + x.table);
  S.mask = reinterpret_cast<uint8_t*>(S.base + x.acap);
  S.slot = S.mask + x.acap;
  S.axis = s_axis;
  const unsigned item = first + blockIdx.x / (unsigned)x.cluster;   // < 2^31 (checked on the host)
  const int rank = (int)(blockIdx.x % (unsigned)x.cluster);
  const int l = (int)(item / (unsigned)a.R), r = (int)(item % (unsigned)a.R);
  if (a.pk.status[l] != 0) return;   // uniform over the cluster
  const int tid = threadIdx.x;
  const int a0 = a.lig.atom_off[l];
  const int N = a.lig.atom_off[l + 1] - a0;
  const int r0 = a.lig.rot_off[l];
  const int n = a.lig.rot_off[l + 1] - r0;   // <= kExMaxRot (checked on the host)
  if (!lg_check(a.grid.check, N <= x.acap && n <= kExMaxRot, kChkItemShape)) return;   // uniform

  for (int i = tid; i < N; i += kExThreads) {
    S.sx[i] = a.pk.xc[a0 + i];
    S.mask[i] = 0;
  }
  __syncthreads();
  for (int b = 0; b < n; ++b) {   // one bond after another: a list names an atom once
    const uchar4 bi = a.pk.binfo[r0 + b];
    if (tid == 0) {
      S.axis[b][0] = bi.x;
      S.axis[b][1] = bi.y;
      lg_check(a.grid.check, bi.x < N && bi.y < N, kChkAtomIndex);
    }
    for (int t = tid; t < bi.z; t += kExThreads) {
      const int i = a.pk.frag[(size_t)(r0 + b) * kFragStride + t];
      if (!lg_check(a.grid.check, i < N, kChkAtomIndex)) continue;
      S.mask[i] |= (uint8_t)(1u << b);
    }
    __syncthreads();
  }
  // table layout for one rotation: atoms by ascending count of bonds, then by index
  const unsigned nt = x.by_nt.d;
  if (tid < 32) {
    unsigned used = 0, slots = 0, size = 1;   // entries of an atom moved by m bonds; past the table: any larger value
    for (int m = 0; m <= n; ++m) {
      const unsigned room = size <= (unsigned)x.table ? (x.table - used) / size : 0u;
      unsigned seen = 0;
      for (int w = 0; w < N; w += 32) {
        const int i = w + tid;
        const bool in = i < N && __popc(S.mask[i < N ? i : 0]) == m;
        const unsigned all = __ballot_sync(0xffffffffu, in);
        const unsigned at = seen + __popc(all & ((1u << tid) - 1u));
        if (in) {
          const bool tabled = at < room;
          unsigned st[kExMaxRot] = {0u, 0u, 0u, 0u};
          if (tabled) {
            unsigned s = 1u;
            for (int b = n - 1; b >= 0; --b)
              if (S.mask[i] >> b & 1u) { st[b] = s; s *= nt; }
            S.slot[slots + at] = (uint8_t)i;
          }
          S.stride[i] = make_uint2(st[0] | st[1] << 16, st[2] | st[3] << 16);
          S.base[i] = tabled ? (uint16_t)(used + at * size) : kExDirect;
        }
        seen += __popc(all);
      }
      const unsigned kept = min(seen, room);
      used += kept * size;
      slots += kept;
      size = min(size * nt, (unsigned)kExTable + 1u);
    }
    if (tid == 0) {
      s_table[0] = (int)slots;
      s_table[1] = (int)used;
    }
  }
  __syncthreads();
  S.n_slots = s_table[0];
  S.entries = s_table[1];

  // restart orientation and translation, as in the greedy kernel
  float u[6];
#pragma unroll
  for (int k = 0; k < 6; ++k) u[k] = restart_uniform(a.seed, (uint32_t)l, (uint32_t)r, (uint32_t)k);
  const Quat qr = qnormalize(shoemake(u[0], u[1], u[2]));
  float Rm[9], M[9];
  qmat(qr, Rm);
#pragma unroll
  for (int i = 0; i < 9; ++i) M[i] = Rm[i] * a.inv_h;
  float o[3];
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    const float t = a.center[k] + (2.0f * u[3 + k] - 1.0f) * a.jitter;
    o[k] = (t - a.origin[k]) * a.inv_h;
  }

  const ExDiv& by_nt = x.by_nt;
  unsigned per_k = 1;   // <= 2^27 (checked on the host)
  for (int b = 0; b < n; ++b) per_k *= nt;
  const int k_lo = a.n_rigid * rank / x.cluster, k_hi = a.n_rigid * (rank + 1) / x.cluster;
  const int batch = S.entries ? max(1, x.table / S.entries) : k_hi - k_lo;   // rotations tabled together
  float best = -INFINITY;
  long long bestc = 0x7fffffffffffffffll;
  for (int k0 = k_lo; k0 < k_hi; k0 += batch) {
    const int nk = min(batch, k_hi - k0);
    for (int e = tid; e < nk * S.entries; e += kExThreads) {
      const int kk = e / S.entries;
      unsigned q = (unsigned)(e - kk * S.entries);
      int lo = 0, hi = S.n_slots - 1;   // last slot that starts at or before q
      while (lo < hi) {
        const int mid = (lo + hi + 1) / 2;
        if (S.base[S.slot[mid]] <= q) lo = mid; else hi = mid - 1;
      }
      const int i = S.slot[lo];
      const unsigned mask = S.mask[i];
      q -= S.base[i];
      int j[kExMaxRot];
#pragma unroll
      for (int b = kExMaxRot - 1; b >= 0; --b) {
        j[b] = 0;
        if (mask >> b & 1u) {
          const unsigned up = by_nt(q);
          j[b] = (int)(q - up * nt);
          q = up;
        }
      }
      float pv[kExMaxRot][3], kd[kExMaxRot][3], cs[kExMaxRot], sn[kExMaxRot];
      ex_axes(S, mask, n, j, a.step_deg, pv, kd, cs, sn);
      float G[9], Mk[9];
      cube_mat(k0 + kk, G);
      mat3mul(M, G, Mk);
      S.tab[e] = ex_energy<FMT>(a, S, i, n, Mk, o, pv, kd, cs, sn);
    }
    __syncthreads();
    const unsigned total = per_k * (unsigned)nk;
    const long long c0 = (long long)k0 * per_k;
    if (S.n_slots == N) {
      if (n <= 1) ex_sum<1>(S, N, n, by_nt, total, c0, best, bestc);
      else if (n == 2) ex_sum<2>(S, N, n, by_nt, total, c0, best, bestc);
      else if (n == 3) ex_sum<3>(S, N, n, by_nt, total, c0, best, bestc);
      else ex_sum<4>(S, N, n, by_nt, total, c0, best, bestc);
    } else {
      for (unsigned t = tid; t < total; t += kExThreads) {
        unsigned q = t;
        int j[kExMaxRot];
#pragma unroll
        for (int b = kExMaxRot - 1; b >= 0; --b) {
          j[b] = 0;
          if (b < n) {
            const unsigned up = by_nt(q);
            j[b] = (int)(q - up * nt);
            q = up;
          }
        }
        float pv[kExMaxRot][3], kd[kExMaxRot][3], cs[kExMaxRot], sn[kExMaxRot];
        ex_axes(S, 0xfu, n, j, a.step_deg, pv, kd, cs, sn);
        float G[9], Mk[9];
        cube_mat(k0 + (int)q, G);
        mat3mul(M, G, Mk);
        float acc = 0.f;
        for (int i = 0; i < N; ++i) {
          if (S.base[i] != kExDirect) {   // uniform
            const uint2 s = S.stride[i];
            acc -= S.tab[S.base[i] + q * S.entries + j[0] * (s.x & 0xffffu) + j[1] * (s.x >> 16) +
                       j[2] * (s.y & 0xffffu) + j[3] * (s.y >> 16)];
          } else {
            acc -= ex_energy<FMT>(a, S, i, n, Mk, o, pv, kd, cs, sn);
          }
        }
        if (acc > best) { best = acc; bestc = c0 + t; }   // t ascends per thread: ties keep the first
      }
    }
    __syncthreads();
  }
  // argmax: higher score, then lower combination index
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) {
    const float os = __shfl_xor_sync(0xffffffffu, best, off);
    const long long oc = __shfl_xor_sync(0xffffffffu, bestc, off);
    if (os > best || (os == best && oc < bestc)) { best = os; bestc = oc; }
  }
  if ((tid & 31) == 0) { red_s[tid >> 5] = best; red_c[tid >> 5] = bestc; }
  __syncthreads();
  if (tid == 0) {
    for (int w = 1; w < kExThreads / 32; ++w)
      if (red_s[w] > best || (red_s[w] == best && red_c[w] < bestc)) { best = red_s[w]; bestc = red_c[w]; }
    cta_s = best;
    cta_c = bestc;
  }
  cg::cluster_group cluster = cg::this_cluster();
  if (x.cluster > 1) cluster.sync();
  if (rank == 0 && tid == 0) {
    for (int c = 1; c < x.cluster; ++c) {
      const float os = *cluster.map_shared_rank(&cta_s, c);
      const long long oc = *cluster.map_shared_rank(&cta_c, c);
      if (os > best || (os == best && oc < bestc)) { best = os; bestc = oc; }
    }
    const long long total = (long long)per_k * a.n_rigid;
    if (bestc >= total) bestc = 0;   // only if every score is NaN; keeps the indices in range
    const size_t lr = (size_t)l * a.R + r;
    if (a.samples) atomicAdd(&a.samples[item % kSampleSlots], (unsigned long long)(total * N));
    a.res_score[lr] = best;
    long long rem = bestc;
    uint8_t* cnt = a.res_cnt + (size_t)r0 * a.R + (size_t)r * n;
    for (int b = n - 1; b >= 0; --b) { cnt[b] = (uint8_t)(rem % nt); rem /= nt; }
    a.res_k[lr] = (uint8_t)rem;
  }
  if (x.cluster > 1) cluster.sync();   // the other CTAs' winners stay readable until here
}

}  // namespace

// The CTAs of a (ligand, restart) and the build. Each of items * C CTAs costs
// about 5.6 us of a slot (3 per SM) before and after its work, so C of them
// lengthen the launch by a C; the chain of the largest ligand's rotations
// shortens it to b / C, at about 14 ns per rotation, atom and square root of
// its combinations (an atom's table entries lie between 1 and all
// combinations; the geometric mean). The C with the smallest sum is taken,
// no more than there are rotations; where all rotations fit kExSmall entries
// the chain is short whatever C. One CTA takes the small build while all
// rotations fit kExTable entries: its time is then its fixed work, of which the
// small build runs eight CTAs to the other's three (two bonds at 180 degrees,
// 5,000 x 16: 1,243 rebuilt, 1,887 and 1,268 us with the large and the small
// build; one bond at 90 degrees 1,090, 1,624 and 1,016). Measured on GB300,
// whole calls (us; 1,000,
// 100, 50 or 5,000 ligands of 8-20 atoms, restarts, 30 degree steps, 24
// rotations), * the one chosen; "rebuilt" is one CTA per (ligand, restart)
// with every combination rebuilt:
//                        rebuilt   C = 1     2       4       8     small build
//   0 bonds   5,000 x 16     844    1,053   2,041   3,902   8,567     591*
//   0-1       5,000 x 16   1,644    1,363   2,534   4,680   9,806     984*
//   2         1,000 x 16   4,469      854*  1,078   1,564   2,705     846
//   2         1,000 x 1      425      268     151*    141     199     473
//   3         50 x 16      4,035      255     243     254*    331     312
//   0-3       100 x 1      2,651      236     132      85      64*    404
cudaError_t launch_exhaustive(const DockArgs& a, const ExWork& w, int sms, cudaStream_t s) {
  const long long items = (long long)a.lig.L * a.R;
  const double per_cta = 5.6 * (double)items / (3. * sms), chain = 0.014 * a.n_rigid * w.chain;
  int C = 1;
  if (w.entries * a.n_rigid > kExSmall)
    for (int c = 2; c <= kExCluster && c <= a.n_rigid; c *= 2)
      if (per_cta * c + chain / c < per_cta * C + chain / C) C = c;
  const bool small = C == 1 && w.entries <= kExSmall && w.entries * a.n_rigid <= kExTable;
  const auto kernel = small ? a.fmt == kRecF32   ? exhaustive_kernel<kRecF32, 8>
                              : a.fmt == kRecF16 ? exhaustive_kernel<kRecF16, 8>
                                                 : exhaustive_kernel<kRecBF16, 8>
                      : a.fmt == kRecF32   ? exhaustive_kernel<kRecF32, 1>
                        : a.fmt == kRecF16 ? exhaustive_kernel<kRecF16, 1>
                                           : exhaustive_kernel<kRecBF16, 1>;
  const ExLaunch x{C, small ? kExSmall : kExTable, (a.max_atoms + 15) / 16 * 16, ExDiv((unsigned)a.n_theta)};
  const long long most = (1ll << 31) / C - 1;   // grid limit
  for (long long first = 0; first < items; first += most) {
    const long long here = items - first < most ? items - first : most;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3((unsigned)(here * C));
    cfg.blockDim = dim3(kExThreads);
    cfg.dynamicSmemBytes = ex_smem_bytes(x.acap, x.table);   // <= 32 KB
    cfg.stream = s;
    cudaLaunchAttribute at{};
    at.id = cudaLaunchAttributeClusterDimension;
    at.val.clusterDim.x = (unsigned)C;
    at.val.clusterDim.y = at.val.clusterDim.z = 1;
    cfg.attrs = &at;
    cfg.numAttrs = C > 1 ? 1 : 0;
    const cudaError_t e = cudaLaunchKernelEx(&cfg, kernel, a, x, (unsigned)first);
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

}  // namespace ligen
