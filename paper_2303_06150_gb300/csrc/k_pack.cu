// Ligand packer: one warp per ligand.
//
// Converts the CSR library into what the other kernels stage: centred
// coordinates (float4, type in w), and for every rotatable bond its axis
// (fixed endpoint u, moving endpoint v), the list of moving atoms and the
// touch mask; on request also the forward-kinematics table (see Packed).
// Cutting rotatable bond (a, b) splits the tree in two; the moving side is
// the smaller part, and on a tie the part without atom 0.
// Invalid ligands (not a tree, ids or types out of range, too large) get
// status LIGEN_ERR_BAD_LIGAND; nothing traps.
//
// What bounds it is the latency of one ligand's dependent steps, so none of
// them is serial over atoms. The tree is walked from atom 0 level by level,
// every lane holding its edges in registers; an atom takes its parent's path
// mask (bit b: rotatable bond b lies between the atom and atom 0) with the
// edge's own bonds ORed in. Bond b's far side is then the ballot of bit b
// over the atoms, and lane b keeps its bond's masks in registers: sizes,
// sides, lists and touch masks are popcounts and shuffles. N - 1 edges that
// reach every atom are a tree, so the walk is the validity check too.
// Measured on GB300 against one lane walking the tree depth first with
// per-atom loops, and the table in a kernel of its own (kernel time): 20,000
// screening ligands 133 -> 45 us, with the table 126 + 57 -> 54 us; five
// ligands 33 -> 13 us. ligen_pack_ligands on 50,000 bimodal ligands (45
// atoms, 8 bonds on average) 490 -> 84 us per call, the host's size checks
// included.
#include "../../include/ligen.h"
#include "internal.h"

namespace ligen {
namespace {

constexpr int kPackWarps = 4;
constexpr unsigned kFull = 0xffffffffu;

// One warp's shared memory, for ligands of at most acap atoms.
struct PackMem {
  float4* xc;        // [acap] centred coordinates (only with the table)
  uint32_t* path;    // [acap] rotatable bonds between the atom and atom 0
  uint32_t* emask;   // [acap] rotatable bonds of each edge
  uint32_t* start;   // [LIGEN_MAX_ROT + 1] next list position of each owner
  uint16_t* edge;    // [acap] endpoints of each edge (a | b << 8)
  uint8_t* seen;     // [acap]
  uint8_t* own;      // [acap] owner of each atom
  uint8_t* pos;      // [acap] list position of each atom
  uint8_t* ord;      // [LIGEN_MAX_ROT]
  uint8_t* lord;     // [LIGEN_MAX_ROT]
};

__host__ __device__ inline size_t pack_carve(int acap, bool table, unsigned char* base, PackMem* S) {
  const size_t a16 = (size_t)(acap + 15) / 16 * 16;
  size_t o = 0;
  const size_t oxc = o;    o += table ? a16 * 16 : 0;
  const size_t opath = o;  o += a16 * 4;
  const size_t omask = o;  o += a16 * 4;
  const size_t ostart = o; o += 144;
  const size_t oedge = o;  o += a16 * 2;
  const size_t oseen = o;  o += a16;
  const size_t oown = o;   o += a16;
  const size_t opos = o;   o += a16;
  const size_t oord = o;   o += LIGEN_MAX_ROT;
  const size_t olord = o;  o += LIGEN_MAX_ROT;
  if (S) {
    S->xc = (float4*)(base + oxc);
    S->path = (uint32_t*)(base + opath);
    S->emask = (uint32_t*)(base + omask);
    S->start = (uint32_t*)(base + ostart);
    S->edge = (uint16_t*)(base + oedge);
    S->seen = base + oseen;
    S->own = base + oown;
    S->pos = base + opos;
    S->ord = base + oord;
    S->lord = base + olord;
  }
  return o;
}

__device__ __forceinline__ int rot_class(int n) {
  const int edges[11] = {0, 1, 2, 3, 4, 6, 8, 12, 16, 24, 32};
  int c = 10;
#pragma unroll
  for (int k = 10; k >= 0; --k)
    if (n <= edges[k]) c = k;
  return c;
}

__device__ __forceinline__ int atom_class(int N) {
  return N <= 32 ? 0 : N <= 64 ? 1 : N <= 128 ? 2 : 3;
}

// The forward-kinematics table of a valid ligand (Packed::fk_*). Lane b
// holds bond b: moving atoms `moved` without v (cnt of them) and moving end
// v; every lane holds atoms lane, lane + 32, ... `key[w]`: the owner of the
// lane's w-th atom in its low 6 bits (n: the root frame).
template <int W>
__device__ __forceinline__ void pack_table(const Packed& out, const PackMem& S, int l, int a0, int N, int r0, int n,
                                           int lane, int u, int v, int cnt, const unsigned (&key)[W]) {
  const bool bond = lane < n;
#pragma unroll
  for (int w = 0; w < W; ++w)
    if (32 * w + lane < N) S.own[32 * w + lane] = (uint8_t)(key[w] & 63u);
  S.start[lane] = 0u;
  if (lane == 0) S.start[LIGEN_MAX_ROT] = 0u;
  __syncwarp();
#pragma unroll
  for (int w = 0; w < W; ++w)
    if (32 * w + lane < N) atomicAdd(&S.start[key[w] & 63u], 1u);
  // a bond's parent owns its moving end; larger lists first, then by depth
  const int par = bond ? S.own[v] : n;
  int rank = 0;
  for (int b = 0; b < n; ++b) {
    const int mb = __shfl_sync(kFull, cnt, b);
    rank += (mb > cnt) || (mb == cnt && b < lane);
  }
  int depth = 0, p = par;
  for (int i = 0; i < n; ++i) {
    const int up = __shfl_sync(kFull, par, p & 31);
    if (!__any_sync(kFull, bond && p < n)) break;
    if (bond && p < n) { ++depth; p = up; }
  }
  const int depths = n ? __reduce_max_sync(kFull, bond ? depth : 0) + 1 : 0;
  int lpos = 0, below = 0;   // entries before this bond by depth; bonds less deep than `lane`
  for (int b = 0; b < n; ++b) {
    const int db = __shfl_sync(kFull, depth, b), rb = __shfl_sync(kFull, rank, b);
    lpos += db < depth || (db == depth && rb < rank);
    below += db < lane;
  }
  if (bond) {
    S.ord[rank] = (uint8_t)lane;
    S.lord[lpos] = (uint8_t)lane;
  }
  __syncwarp();
  // list positions: owners' ranges in bond order, the root's last, atoms ascending inside each
  const unsigned c = bond ? S.start[lane] : 0u;
  unsigned before = c;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const unsigned t = __shfl_up_sync(kFull, before, o);
    if (lane >= o) before += t;
  }
  const unsigned owned = __shfl_sync(kFull, before, 31);
  __syncwarp();
  if (bond) S.start[lane] = before - c;
  if (lane == 0) S.start[n] = owned;
  __syncwarp();
#pragma unroll
  for (int w = 0; w < W; ++w) {
    if (32 * w >= N) break;   // uniform
    const int i = 32 * w + lane;
    const unsigned o = i < N ? (key[w] & 63u) : 64u + lane;
    const unsigned same = __match_any_sync(kFull, o);
    unsigned at = 0u;
    if (i < N) at = S.start[o] + __popc(same & ((1u << lane) - 1u));
    __syncwarp();
    if (i < N) {
      if ((same >> lane) == 1u) S.start[o] = at + 1u;   // the owner's last atom of this word
      S.pos[i] = (uint8_t)at;
      out.fk_xs[a0 + at] = S.xc[i];
      out.fk_own[a0 + at] = (uint8_t)o;
    }
    __syncwarp();
  }
  if (bond) {
    const float4 xv = S.xc[v], xu = S.xc[u];
    float kx = xv.x - xu.x, ky = xv.y - xu.y, kz = xv.z - xu.z;
    const float kn = rsqrtf(kx * kx + ky * ky + kz * kz);
    out.fk_ax[r0 + lane] = make_float4(kx * kn, ky * kn, kz * kn, 0.f);
    out.fk_bond[r0 + lane] = make_uchar4((uint8_t)par, S.ord[lane], S.lord[lane], S.pos[v]);
  }
  uint8_t* row = out.fk_loff + (size_t)l * kFkLoffBytes;
  row[lane] = lane <= depths ? (uint8_t)below : 0;
  if (lane + 32 < kFkLoffBytes) row[lane + 32] = lane == 0 ? (uint8_t)depths : 0;   // LIGEN_MAX_ROT: the depths
}

// W: words of 32 atoms of the launch's largest ligand.
template <int W>
__global__ void __launch_bounds__(32 * kPackWarps) pack_kernel(const LigandsDev lig, int nc, const Packed out,
                                                               int acap) {
  static_assert(LIGEN_MAX_ROT == 32, "one lane per rotatable bond");
  extern __shared__ __align__(16) unsigned char pack_smem[];
  asm volatile("griddepcontrol.launch_dependents;");   // the grid records (launch_grid_prep) need nothing of this
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int l = blockIdx.x * kPackWarps + warp;
  if (l >= lig.L) return;
  const bool table = out.fk_xs != nullptr;
  PackMem S;
  pack_carve(acap, table, pack_smem + (size_t)warp * pack_carve(acap, table, nullptr, nullptr), &S);
  const int a0 = lig.atom_off[l];
  const int N = lig.atom_off[l + 1] - a0;
  const int e0 = a0 - l;
  const int r0 = lig.rot_off[l];
  const int n = lig.rot_off[l + 1] - r0;

  bool bad = (N < 1) | (N > acap) | (n < 0) | (n > LIGEN_MAX_ROT);
  int myedge = -1;   // edge of this lane's rotatable bond
  if (!bad) {        // uniform
    // every input read at once
    float x[W], y[W], z[W];
    int ty[W], ea[W], eb[W];
#pragma unroll
    for (int w = 0; w < W; ++w) {
      const int i = 32 * w + lane;
      x[w] = y[w] = z[w] = 0.f;
      ty[w] = ea[w] = eb[w] = 0;
      if (32 * w >= N) continue;   // uniform
      if (i < N) {
        x[w] = lig.xyz[3 * (a0 + i)];
        y[w] = lig.xyz[3 * (a0 + i) + 1];
        z[w] = lig.xyz[3 * (a0 + i) + 2];
        ty[w] = lig.type[a0 + i];
      }
      if (i < N - 1) {
        ea[w] = lig.bonds[2 * (e0 + i)];
        eb[w] = lig.bonds[2 * (e0 + i) + 1];
      }
    }
    if (lane < n) {
      myedge = lig.rot_edge[r0 + lane];
      bad |= (myedge < 0) | (myedge >= N - 1);
    }
    float sx = 0.f, sy = 0.f, sz = 0.f;
#pragma unroll
    for (int w = 0; w < W; ++w) {
      const int i = 32 * w + lane;
      if (i < N) {
        sx += x[w];
        sy += y[w];
        sz += z[w];
        bad |= ty[w] >= nc;
        S.path[i] = 0u;
        S.emask[i] = 0u;
        S.seen[i] = i == 0;
      }
      if (i < N - 1) {
        bad |= (ea[w] < 0) | (ea[w] >= N) | (eb[w] < 0) | (eb[w] >= N);
        S.edge[i] = (uint16_t)((ea[w] & 0xff) | (eb[w] & 0xff) << 8);
      }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      sx += __shfl_xor_sync(kFull, sx, o);
      sy += __shfl_xor_sync(kFull, sy, o);
      sz += __shfl_xor_sync(kFull, sz, o);
    }
    const float inv = 1.0f / (float)N;
    // rounded products: never contracted into the subtractions below, so the
    // centred coordinates do not depend on W
    sx = __fmul_rn(sx, inv); sy = __fmul_rn(sy, inv); sz = __fmul_rn(sz, inv);
#pragma unroll
    for (int w = 0; w < W; ++w) {
      const int i = 32 * w + lane;
      if (i < N) {
        float4 v;
        v.x = x[w] - sx;
        v.y = y[w] - sy;
        v.z = z[w] - sz;
        v.w = __int_as_float(ty[w]);
        if (out.xc) out.xc[a0 + i] = v;
        if (table) S.xc[i] = v;
      }
    }
  }
  bad = __any_sync(kFull, bad);
  __syncwarp();

  if (!bad) {
    // The walk from atom 0; an edge is used when exactly one end was seen.
    // Edges and their bonds are in registers and a round's reads
    // unconditional, so a round is two shared-memory latencies whatever W
    // (with the reads behind each edge's own test a round was eight).
    if (lane < n) atomicOr(&S.emask[myedge], 1u << lane);
    __syncwarp();
    unsigned edge[W], bonds[W];
    unsigned left = 0u;   // this lane's unused edges, bit w
#pragma unroll
    for (int w = 0; w < W; ++w) {
      edge[w] = bonds[w] = 0u;   // no edge: atom 0 to itself, never used
      if (32 * w + lane < N - 1) {
        edge[w] = S.edge[32 * w + lane];
        bonds[w] = S.emask[32 * w + lane];
        left |= 1u << w;
      }
    }
    while (true) {   // every round with progress uses an edge: at most N - 1 rounds
      unsigned use = 0u, child_b = 0u;
#pragma unroll
      for (int w = 0; w < W; ++w) {
        const unsigned sa = S.seen[edge[w] & 0xffu], sb = S.seen[edge[w] >> 8];
        use |= (sa ^ sb) << w;
        child_b |= sa << w;
      }
      use &= left;
      if (!__any_sync(kFull, use != 0u)) break;
      unsigned path[W];
#pragma unroll
      for (int w = 0; w < W; ++w)
        path[w] = S.path[child_b >> w & 1u ? edge[w] & 0xffu : edge[w] >> 8] | bonds[w];
#pragma unroll
      for (int w = 0; w < W; ++w)
        if (use >> w & 1u) {
          const unsigned ch = child_b >> w & 1u ? edge[w] >> 8 : edge[w] & 0xffu;
          S.path[ch] = path[w];
          S.seen[ch] = 1;
        }
      left &= ~use;
      __syncwarp();
    }
    bool missing = false;
#pragma unroll
    for (int w = 0; w < W; ++w) {
      const int i = 32 * w + lane;
      if (i < N) missing |= S.seen[i] == 0;
    }
    bad = __any_sync(kFull, missing);   // N - 1 edges that do not reach every atom: not a tree
  }

  if (!bad) {
    const int words = (N + 31) >> 5;
    // lane b: the atoms beyond bond b, as seen from atom 0
    unsigned word[W];
#pragma unroll
    for (int w = 0; w < W; ++w) {
      word[w] = 0u;
      if (w < words) {
        const int i = 32 * w + lane;
        const unsigned pm = i < N ? S.path[i] : 0u;
        for (int b = 0; b < n; ++b) {
          const unsigned in = __ballot_sync(kFull, pm >> b & 1u);
          if (lane == b) word[w] = in;
        }
      }
    }
    int u = 0, v = 0, cnt = 0;
    unsigned moved[W], reads[W];   // the atoms a turn moves (moving side without v) and a sweep reads (moving side, u)
    if (lane < n) {
      const unsigned e = S.edge[myedge];
      const int pa = e & 0xffu, pb = e >> 8;
      int sz = 0;
      bool far_b = false;
#pragma unroll
      for (int w = 0; w < W; ++w) {
        sz += __popc(word[w]);
        if (w == pb >> 5) far_b = word[w] >> (pb & 31) & 1u;
      }
      const int child = far_b ? pb : pa, par = far_b ? pa : pb;
      const bool child_moves = 2 * sz <= N;   // smaller side; tie: side without atom 0
      v = child_moves ? child : par;
      u = child_moves ? par : child;
#pragma unroll
      for (int w = 0; w < W; ++w) {
        const int have = N - 32 * w;
        const unsigned all = have >= 32 ? 0xffffffffu : have > 0 ? (1u << have) - 1u : 0u;
        if (!child_moves) word[w] = ~word[w] & all;
      }
    }
#pragma unroll
    for (int w = 0; w < W; ++w) {
      moved[w] = w == v >> 5 ? word[w] & ~(1u << (v & 31)) : word[w];
      reads[w] = lane < n && w == u >> 5 ? word[w] | 1u << (u & 31) : word[w];
      cnt += __popc(moved[w]);
    }
    if (lane < n) {
      const int gb = r0 + lane;
      if (out.binfo) out.binfo[gb] = make_uchar4((uint8_t)u, (uint8_t)v, (uint8_t)cnt, 0);
      if (out.axis) { out.axis[2 * gb] = u; out.axis[2 * gb + 1] = v; }
      if (out.fbits) {
        uint32_t* fb = out.fbits + (size_t)gb * 8;
        if ((reinterpret_cast<uintptr_t>(out.fbits) & 15) == 0) {   // the caller's buffer: any 4-byte alignment
          uint4 lo = make_uint4(word[0], 0u, 0u, 0u), hi = make_uint4(0u, 0u, 0u, 0u);
          if constexpr (W > 1) lo.y = word[1];
          if constexpr (W > 2) { lo.z = word[2]; lo.w = word[3]; }
          if constexpr (W > 4) hi = make_uint4(word[4], word[5], word[6], word[7]);
          reinterpret_cast<uint4*>(fb)[0] = lo;
          reinterpret_cast<uint4*>(fb)[1] = hi;
        } else {
#pragma unroll
          for (int w = 0; w < 8; ++w) fb[w] = w < W ? word[w < W ? w : 0] : 0u;
        }
      }
    }
    // moving-atom lists, owners (the shortest list holding the atom, the
    // first of equal ones) and touch masks, bond by bond
    const bool lists = out.frag || out.touch || table;   // masks and axes alone need none of this
    unsigned key[W], touch = 1u << lane;
#pragma unroll
    for (int w = 0; w < W; ++w) key[w] = 0xffffffc0u | n;
    for (int b = 0; lists && b < n; ++b) {
      const unsigned mb = __shfl_sync(kFull, cnt, b);
      uint8_t* list = out.frag ? out.frag + (size_t)(r0 + b) * kFragStride : nullptr;
      unsigned hit = 0u;
#pragma unroll
      for (int w = 0; w < W; ++w) {
        if (w >= words) break;   // uniform
        const unsigned m = __shfl_sync(kFull, moved[w], b);
        hit |= moved[w] & __shfl_sync(kFull, reads[w], b);
        if (m >> lane & 1u) {
          key[w] = min(key[w], mb << 6 | b);
          if (list) list[__popc(m & ((1u << lane) - 1u))] = (uint8_t)(32 * w + lane);
        }
        if (list) list += __popc(m);
      }
      if (hit) touch |= 1u << b;
    }
    // touch[b'] bit b: turning bond b' moves an atom that bond b's sweep reads
    // (its moving side, v included, or its fixed endpoint u). Turning b'
    // moves its moving side except v_b', which lies on its own axis.
    if (out.touch && lane < n) out.touch[r0 + lane] = touch;
    if (table) pack_table<W>(out, S, l, a0, N, r0, n, lane, u, v, cnt, key);
  } else {
    for (int b = lane; b < n && b < LIGEN_MAX_ROT; b += 32) {
      const int gb = r0 + b;
      if (out.binfo) out.binfo[gb] = make_uchar4(0, 0, 0, 0);
      if (out.fbits)
        for (int w = 0; w < 8; ++w) out.fbits[(size_t)gb * 8 + w] = 0u;
      if (out.axis) { out.axis[2 * gb] = -1; out.axis[2 * gb + 1] = -1; }
      if (out.touch) out.touch[gb] = 0u;
    }
    if (table) {   // nothing of the ligand is read: only the flag
      uint8_t* row = out.fk_loff + (size_t)l * kFkLoffBytes;
      row[lane] = 0;
      if (lane + 32 < kFkLoffBytes) row[lane + 32] = lane + 32 == kFkBad ? 1 : 0;
    }
  }
  if (lane == 0) {
    if (out.status) out.status[l] = bad ? LIGEN_ERR_BAD_LIGAND : 0;
    if (out.bucket) out.bucket[l] = atom_class(N) * 11 + rot_class(n);
  }
}

// Ligands by decreasing estimated docking cost (the cost of plan_groups):
// one CTA, a counting sort over the cost's exponent and three mantissa bits,
// so ligands within 1/8 of each other come in any order.
constexpr int kOrderThreads = 1024;
constexpr int kOrderBins = 512;

__global__ void __launch_bounds__(kOrderThreads) order_kernel(const LigandsDev lig, int n_rigid, int passes,
                                                              int n_theta, int32_t* order) {
  __shared__ int start[kOrderBins];
  __shared__ int warp_sum[kOrderBins / 32];
  const int tid = threadIdx.x;
  auto bin = [&](int l) {
    const int N = lig.atom_off[l + 1] - lig.atom_off[l], n = lig.rot_off[l + 1] - lig.rot_off[l];
    const float c = 4.f * N * n_rigid + (float)passes * n * n_theta * (N + 4);
    const int b = (int)(__float_as_uint(c) >> 20) - (127 << 3);   // c >= 1: 8 bins per power of two
    return kOrderBins - 1 - min(max(b, 0), kOrderBins - 1);
  };
  if (tid < kOrderBins) start[tid] = 0;
  __syncthreads();
  for (int l = tid; l < lig.L; l += kOrderThreads) atomicAdd(&start[bin(l)], 1);
  __syncthreads();
  int v = 0, sum = 0;   // exclusive prefix sums
  if (tid < kOrderBins) {
    v = sum = start[tid];
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int t = __shfl_up_sync(kFull, sum, o);
      if ((tid & 31) >= o) sum += t;
    }
    if ((tid & 31) == 31) warp_sum[tid >> 5] = sum;
  }
  __syncthreads();
  if (tid < kOrderBins) {
    for (int w = 0; w < tid >> 5; ++w) sum += warp_sum[w];
    start[tid] = sum - v;
  }
  __syncthreads();
  for (int l = tid; l < lig.L; l += kOrderThreads) order[atomicAdd(&start[bin(l)], 1)] = l;
}

}  // namespace

cudaError_t launch_order(const LigandsDev& lig, int n_rigid, int passes, int n_theta, int32_t* order,
                         cudaStream_t s) {
  order_kernel<<<1, kOrderThreads, 0, s>>>(lig, n_rigid, passes, n_theta, order);
  return cudaGetLastError();
}

cudaError_t launch_pack(const LigandsDev& lig, int nc, const Packed& out, int max_atoms, cudaStream_t s) {
  if (lig.L == 0) return cudaSuccess;
  const int blocks = (lig.L + kPackWarps - 1) / kPackWarps;
  const size_t smem = kPackWarps * pack_carve(max_atoms, out.fk_xs != nullptr, nullptr, nullptr);   // <= 33 KB
  const int words = (max_atoms + 31) / 32;
  const auto kernel = words <= 1 ? pack_kernel<1> : words <= 2 ? pack_kernel<2> : words <= 4 ? pack_kernel<4> : pack_kernel<8>;
  kernel<<<blocks, 32 * kPackWarps, smem, s>>>(lig, nc, out, max_atoms);
  return cudaGetLastError();
}

}  // namespace ligen
