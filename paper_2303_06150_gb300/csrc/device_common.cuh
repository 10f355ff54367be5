// Device building blocks shared by the docking kernels: the restart random
// stream, quaternion algebra, the cube rotation table and the grid sampler.
#pragma once
#include <cmath>
#include <cstdint>
#include <cuda_bf16.h>
#include <cuda_fp16.h>
#include <cuda_runtime.h>

namespace ligen {

// ------------------------------------------------------------------ RNG --
// SplitMix64 (Steele, Lea, Flood 2014): first output of a generator whose
// state is x.
__host__ __device__ __forceinline__ uint64_t splitmix64(uint64_t x) {
  uint64_t z = x + 0x9E3779B97F4A7C15ull;
  z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
  z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
  return z ^ (z >> 31);
}

// Uniform k of restart r of ligand l: 24 high bits of
// SplitMix64(seed ^ ((l * 2^32 + r) * 8 + k)) scaled by 2^-24; exact in FP32.
__device__ __forceinline__ float restart_uniform(uint64_t seed, uint32_t lig, uint32_t r, uint32_t k) {
  uint64_t c = ((((uint64_t)lig << 32) + (uint64_t)r) << 3) + k;
  return (float)(uint32_t)(splitmix64(seed ^ c) >> 40) * (1.0f / 16777216.0f);
}

// ------------------------------------------------------------ rotations --
struct Quat {
  float w, x, y, z;
};

__device__ __forceinline__ Quat qmul(Quat a, Quat b) {
  return {a.w * b.w - a.x * b.x - a.y * b.y - a.z * b.z,
          a.w * b.x + a.x * b.w + a.y * b.z - a.z * b.y,
          a.w * b.y - a.x * b.z + a.y * b.w + a.z * b.x,
          a.w * b.z + a.x * b.y - a.y * b.x + a.z * b.w};
}

__device__ __forceinline__ Quat qnormalize(Quat q) {
  float s = rsqrtf(q.w * q.w + q.x * q.x + q.y * q.y + q.z * q.z);
  return {q.w * s, q.x * s, q.y * s, q.z * s};
}

// Row-major rotation matrix of a unit quaternion.
__device__ __forceinline__ void qmat(Quat q, float* m) {
  float w = q.w, x = q.x, y = q.y, z = q.z;
  m[0] = 1.f - 2.f * (y * y + z * z); m[1] = 2.f * (x * y - w * z);       m[2] = 2.f * (x * z + w * y);
  m[3] = 2.f * (x * y + w * z);       m[4] = 1.f - 2.f * (x * x + z * z); m[5] = 2.f * (y * z - w * x);
  m[6] = 2.f * (x * z - w * y);       m[7] = 2.f * (y * z + w * x);       m[8] = 1.f - 2.f * (x * x + y * y);
}

// Shoemake (1992) uniform rotation from three uniforms:
// (sqrt(u0) cos 2pi u2, sqrt(1-u0) sin 2pi u1, sqrt(1-u0) cos 2pi u1, sqrt(u0) sin 2pi u2).
__device__ __forceinline__ Quat shoemake(float u0, float u1, float u2) {
  float r1 = sqrtf(1.0f - u0), r2 = sqrtf(u0);
  float s1, c1, s2, c2;
  sincospif(2.0f * u1, &s1, &c1);
  sincospif(2.0f * u2, &s2, &c2);
  return {r2 * c2, r1 * s1, r1 * c1, r2 * s2};
}

// The 24 proper rotations of the cube as unit quaternions (w, x, y, z):
//  0 identity; 1-3 half turns about x, y, z; 4-9 quarter turns +x, -x, +y,
//  -y, +z, -z; 10-17 third turns (120 deg) about the body diagonal
//  (sx, sy, sz) with m = k - 10 and s = -1 where bit 2 (x), 1 (y), 0 (z) of m
//  is set; 18-23 half turns about the face diagonals (1,1,0), (1,-1,0),
//  (0,1,1), (0,1,-1), (1,0,1), (1,0,-1).
#define LIGEN_H_ 0.5f
#define LIGEN_S_ 0.70710678118654752f
static __constant__ float kCubeQuat[24][4] = {
    {1, 0, 0, 0},
    {0, 1, 0, 0}, {0, 0, 1, 0}, {0, 0, 0, 1},
    {LIGEN_S_, LIGEN_S_, 0, 0}, {LIGEN_S_, -LIGEN_S_, 0, 0},
    {LIGEN_S_, 0, LIGEN_S_, 0}, {LIGEN_S_, 0, -LIGEN_S_, 0},
    {LIGEN_S_, 0, 0, LIGEN_S_}, {LIGEN_S_, 0, 0, -LIGEN_S_},
    {LIGEN_H_, LIGEN_H_, LIGEN_H_, LIGEN_H_}, {LIGEN_H_, LIGEN_H_, LIGEN_H_, -LIGEN_H_},
    {LIGEN_H_, LIGEN_H_, -LIGEN_H_, LIGEN_H_}, {LIGEN_H_, LIGEN_H_, -LIGEN_H_, -LIGEN_H_},
    {LIGEN_H_, -LIGEN_H_, LIGEN_H_, LIGEN_H_}, {LIGEN_H_, -LIGEN_H_, LIGEN_H_, -LIGEN_H_},
    {LIGEN_H_, -LIGEN_H_, -LIGEN_H_, LIGEN_H_}, {LIGEN_H_, -LIGEN_H_, -LIGEN_H_, -LIGEN_H_},
    {0, LIGEN_S_, LIGEN_S_, 0}, {0, LIGEN_S_, -LIGEN_S_, 0},
    {0, 0, LIGEN_S_, LIGEN_S_}, {0, 0, LIGEN_S_, -LIGEN_S_},
    {0, LIGEN_S_, 0, LIGEN_S_}, {0, LIGEN_S_, 0, -LIGEN_S_},
};
#undef LIGEN_H_
#undef LIGEN_S_

__device__ __forceinline__ Quat cube_quat(int k) {
  return {kCubeQuat[k][0], kCubeQuat[k][1], kCubeQuat[k][2], kCubeQuat[k][3]};
}

// Matrix of cube rotation k, exact: its entries are 0 or +-1, so the FP32
// matrix of the (rounded) quaternion is rounded to the nearest integer.
__device__ __forceinline__ void cube_mat(int k, float* g) {
  float m[9];
  qmat(cube_quat(k), m);
#pragma unroll
  for (int i = 0; i < 9; ++i) g[i] = rintf(m[i]);
}

// c = a * b for row-major 3x3 matrices.
__device__ __forceinline__ void mat3mul(const float* a, const float* b, float* c) {
#pragma unroll
  for (int r = 0; r < 3; ++r)
#pragma unroll
    for (int col = 0; col < 3; ++col)
      c[3 * r + col] = a[3 * r] * b[col] + a[3 * r + 1] * b[3 + col] + a[3 * r + 2] * b[6 + col];
}

// Torsion increment j of a step of `step_deg` degrees: (cos, sin) of
// j * step_deg degrees. Every kernel uses this one definition, so the
// rotation applied after a decision is the one that was scored.
__device__ __forceinline__ void torsion_cs(int j, int step_deg, float* c, float* s) {
  sincospif((float)(j * step_deg) * (1.0f / 180.0f), s, c);
}

// The angle of torsion increment j as poses hold it: radians in [-pi, pi).
__device__ __forceinline__ float torsion_radians(int j, int step_deg) {
  int deg = (j * step_deg) % 360;
  if (deg >= 180) deg -= 360;
  return (float)deg * 0.017453292519943295f;
}

// The increment of an angle written by torsion_radians.
__device__ __forceinline__ int torsion_increment(float radians, int step_deg, int n_theta) {
  const int j = __float2int_rn(radians * 57.29577951308232f / (float)step_deg);
  return j < 0 ? j + n_theta : j;
}

// Rotation of point x by the angle with cosine c and sine s about the line
// through v with unit direction k (right-handed): the component along k
// stays, the perpendicular part turns. Same arithmetic as the docking
// kernel's sweep.
__device__ __forceinline__ void rodrigues_apply(float* x, const float* v, const float* k, float c, float s) {
  const float dx = x[0] - v[0], dy = x[1] - v[1], dz = x[2] - v[2];
  const float kd = k[0] * dx + k[1] * dy + k[2] * dz;
  const float px = fmaf(k[0], kd, v[0]), py = fmaf(k[1], kd, v[1]), pz = fmaf(k[2], kd, v[2]);
  const float ex = fmaf(-k[0], kd, dx), ey = fmaf(-k[1], kd, dy), ez = fmaf(-k[2], kd, dz);
  const float qx = k[1] * dz - k[2] * dy, qy = k[2] * dx - k[0] * dz, qz = k[0] * dy - k[1] * dx;
  x[0] = fmaf(ex, c, fmaf(qx, s, px));
  x[1] = fmaf(ey, c, fmaf(qy, s, py));
  x[2] = fmaf(ez, c, fmaf(qz, s, pz));
}

// --------------------------------------------------------------- sampler --
// The grid is stored per cell and channel as the 8 coefficients of its
// trilinear polynomial, E(f) = a0 + ax fx + ay fy + az fz + axy fx fy +
// axz fx fz + ayz fy fz + axyz fx fy fz with f the position inside the cell.
// One 32-byte record per (cell, channel) makes one sample one aligned 32-byte
// load (one L2 sector) instead of eight scattered corner loads.
//
// Records are channel-major, [c][iz][iy][ix][8]. With the channel innermost
// instead, all lanes sampling atoms of one type would hit the same 32-byte
// position inside their 128-byte lines: measured on GB300, such 256-bit
// gathers run at two thirds of the rate of gathers at mixed positions (the
// L1 data banks serve one position per cycle). Channel-major puts the
// position at ix mod 4, which varies from lane to lane.
struct GridView {
  const float* coef;   // records at rec_index, 256-byte aligned
  int cx, cy, cz;      // record cells per axis (rec_cells of the format)
  int nc;
  float mx, my, mz;    // points - 1 per axis: upper box bound in grid units (axis_bounds)
  // operands of the docking kernel's sampler (DockPoint)
  float lx, ly, lz;    // the floats below mx, my, mz
  unsigned hx, hy, hz; // bits of mx, my, mz
  unsigned cells;      // cx cy cz, modulo 2^32
  unsigned bias;       // the bits of 2^23 times (cy cx + cx + 1), modulo 2^32
  float penalty;
  size_t n_rec;        // records in the buffer (checked builds compare with it)
  unsigned* check;     // checked builds: first out-of-range code, else NULL
  // points - 2: the last cell of FP32 records (axis_bounds). Last, because the
  // docking kernel reads the fields above as pairs from the constant bank:
  // with these three after mz, 20,000 screening ligands took 1.1% longer, 8 of
  // 256 atoms on 32 lanes 11%.
  float kx, ky, kz;
};

// The upper box bound and the last cell of an axis of n points as floats,
// rounded towards zero: past 2^24 points the nearest float can lie beyond the
// last point, and a coordinate there would be given a cell past the records.
inline void axis_bounds(int n, float* top, float* last_cell) {
  auto below = [](int v) {
    const float f = (float)v;
    return (double)f > (double)v ? std::nextafterf(f, 0.f) : f;
  };
  *top = below(n - 1);
  *last_cell = below(n - 2);
}

// Checked builds (compiled with -DLIGEN_CHECKED=1): every data-dependent
// index is compared with its bound before use; a violation stores its code
// in *check (the first one wins) and the access is skipped, so the kernel
// carries on without touching memory out of range. Other builds compile the
// checks away.
#ifndef LIGEN_CHECKED
#define LIGEN_CHECKED 0
#endif
enum CheckCode : unsigned {
  kChkGridRecord = 1,   // grid record index or channel out of range
  kChkRescoreNode = 2,  // FP64 re-score: lattice node out of range
  kChkItemShape = 3,    // a ligand larger than the launch's shared-memory carve-up
  kChkAtomIndex = 4,    // a bond endpoint or moving-atom index >= the ligand's atoms
};
__device__ __forceinline__ bool lg_check(unsigned* check, bool ok, unsigned code) {
  if constexpr (LIGEN_CHECKED) {
    if (!ok && check) atomicCAS(check, 0u, code);
    return ok;
  }
  return true;
}

// Index (in records) of the record of channel c, cell (ix, iy, iz); the
// grid preparation writes records at the same indices. A channel of 16-bit
// records can hold more than 2^31 cells: an accepted grid has at most 2e9
// cells times channels, the records' padding (rec_cells) multiplies a thin
// grid's by up to 8.
__host__ __device__ __forceinline__ size_t rec_index(int cx, int cy, int cz, int c, int ix, int iy, int iz) {
  return (size_t)c * cz * cy * cx + ((size_t)iz * cy + iy) * cx + ix;
}
// The same for coefficient records, which have no padding: a channel's at
// most 2e9 cells are counted in 32 bits.
__host__ __device__ __forceinline__ size_t rec_index_f32(int cx, int cy, int cz, int c, int ix, int iy, int iz) {
  return (size_t)c * cz * cy * cx + (unsigned)((iz * cy + iy) * cx + ix);
}
// Records to allocate for a grid of cx * cy * cz cells and nc channels.
__host__ __device__ __forceinline__ size_t rec_count(int cx, int cy, int cz, int nc) {
  return (size_t)cx * cy * cz * nc;
}

// Packed FP32 pairs (sm_100 family: fma.rn.f32x2, sub.rn.f32x2): one
// instruction for two independent operations, each element rounded exactly
// as the scalar operation, so results are bit-identical to scalar code.
__device__ __forceinline__ unsigned long long pk2(float lo, float hi) {
  unsigned long long r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
  return r;
}
__device__ __forceinline__ float2 upk2(unsigned long long v) {
  float2 r;
  asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(v));
  return r;
}
__device__ __forceinline__ float2 fma2(float2 a, float2 b, float2 c) {   // a * b + c
  unsigned long long d;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(pk2(a.x, a.y)), "l"(pk2(b.x, b.y)), "l"(pk2(c.x, c.y)));
  return upk2(d);
}
__device__ __forceinline__ float2 sub2(float2 a, float2 b) {   // a - b
  unsigned long long d;
  asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(pk2(a.x, a.y)), "l"(pk2(b.x, b.y)));
  return upk2(d);
}

__device__ __forceinline__ float2 add2_rz(float2 a, float2 b) {   // a + b, rounded towards zero
  unsigned long long d;
  asm("add.rz.f32x2 %0, %1, %2;" : "=l"(d) : "l"(pk2(a.x, a.y)), "l"(pk2(b.x, b.y)));
  return upk2(d);
}

// 256-bit read-only load (sm_100+): one 32-byte record in one instruction,
// not volatile (no side effect, so the compiler may batch it), and without
// allocating the line in L1 (L1::no_allocate): the samplers' 32-byte
// records are rarely read twice from L1 (~3% hits), and not allocating them
// keeps L1 for the kernels' other data. Measured on
// GB300 (8,000 screening ligands): FP32 docking 18.97 -> 18.35 ms, gradient
// refinement of their top 16 poses 9.27 -> 8.52 ms. The same hint on the
// 16-byte records made FP16 docking 1.2% slower, so they keep the default.
__device__ __forceinline__ void ld_global_v8_na(const float* p, float (&v)[8]) {
  asm("ld.global.nc.L1::no_allocate.v8.f32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
               : "=f"(v[0]), "=f"(v[1]), "=f"(v[2]), "=f"(v[3]), "=f"(v[4]), "=f"(v[5]), "=f"(v[6]),
                 "=f"(v[7])
               : "l"(p));
}

// Energy of channel `c` at grid-unit position u (u = (x - origin) / spacing).
// Inside iff 0 <= u <= n - 1 on every axis; cell i = min(floor(u), n - 2),
// f = u - i. Outside: the penalty.
__device__ __forceinline__ float grid_sample(const GridView& g, float ux, float uy, float uz, int c) {
  bool inb = (ux >= 0.f) & (ux <= g.mx) & (uy >= 0.f) & (uy <= g.my) & (uz >= 0.f) & (uz <= g.mz);
  float e = g.penalty;
  if (inb) {
    float fx = fminf(floorf(ux), g.kx);
    float fy = fminf(floorf(uy), g.ky);
    float fz = fminf(floorf(uz), g.kz);
    int ix = (int)fx, iy = (int)fy, iz = (int)fz;
    float dx = ux - fx, dy = uy - fy, dz = uz - fz;
    const size_t ri = rec_index_f32(g.cx, g.cy, g.cz, c, ix, iy, iz);
    if (!lg_check(g.check, c >= 0 && c < g.nc && ri < g.n_rec, kChkGridRecord)) return g.penalty;
    const float* rec = g.coef + ri * 8;
    float a[8];
    ld_global_v8_na(rec, a);
    float t1 = fmaf(dz, a[7], a[4]);
    float t2 = fmaf(dy, t1, a[1]);
    t2 = fmaf(dz, a[5], t2);
    float t3 = fmaf(dz, a[6], a[2]);
    e = fmaf(dz, a[3], a[0]);
    e = fmaf(dy, t3, e);
    e = fmaf(dx, t2, e);
  }
  return e;
}

// Grid record formats of the docking kernel.
//   kRecF32:  32-byte records, the 8 FP32 coefficients of the cell's
//             trilinear polynomial (one 256-bit load, 7 FMA);
//   kRecF16, kRecBF16: 16-byte records, the 8 corner values of the cell in
//             FP16 or BF16 (one 128-bit load, FP32 interpolation).
// Records are channel-major in every format.
enum RecFormat { kRecF32 = 0, kRecF16 = 1, kRecBF16 = 2 };

__host__ __device__ constexpr int rec_bytes(int fmt) { return fmt == kRecF32 ? 32 : 16; }

// Extra record layers past the lattice's last node, 16-bit formats.
constexpr int kRecPad16 = 0;

// Cells per axis of the record grid of a lattice with n points per axis.
// FP32 coefficient records cover its n - 1 cells; the sampler clamps the
// cell index so that a point on an upper face (u = n - 1) uses the last cell
// at f = 1. The 16-bit corner records add one layer on each upper face (its
// corners repeat the face's node values, plus kRecPad16 spare layers), so
// their sampler needs no clamp: a point on an upper face samples that layer
// at f = 0 and gets the node value exactly. Measured on GB300: the padded,
// clamp-free FP16 sampler is 2.5% faster; the same padding made FP32 records
// 5.7% slower, so FP32 keeps n - 1 cells.
__host__ __device__ constexpr int rec_cells(int n, int fmt) { return fmt == kRecF32 ? n - 1 : n + kRecPad16; }

template <int FMT>
__device__ __forceinline__ float2 unpack2(unsigned int w) {
  if constexpr (FMT == kRecF16) {
    __half2 h = *reinterpret_cast<__half2*>(&w);
    return __half22float2(h);
  } else {
    __nv_bfloat162 h = *reinterpret_cast<__nv_bfloat162*>(&w);
    return __bfloat1622float2(h);
  }
}

// Trilinear value of a 16-bit record at (dx, dy, dz) inside its cell: 7
// lerps v0 + d (v1 - v0), x-lerps and y-lerps in packed pairs (measured:
// 1.5% faster FP16 docking; the FP32 sampler lost 1% the same way).
template <int FMT>
__device__ __forceinline__ float lerp16(uint4 v, float dx, float dy, float dz) {
  const float2 a = unpack2<FMT>(v.x), b = unpack2<FMT>(v.y);   // (c000, c100), (c010, c110)
  const float2 d = unpack2<FMT>(v.z), f = unpack2<FMT>(v.w);   // (c001, c101), (c011, c111)
  const float2 dxx = make_float2(dx, dx);
  const float2 p0 = make_float2(a.x, b.x), q0 = make_float2(a.y, b.y);   // (c000, c010), (c100, c110)
  const float2 p1 = make_float2(d.x, f.x), q1 = make_float2(d.y, f.y);   // (c001, c011), (c101, c111)
  const float2 x0 = fma2(dxx, sub2(q0, p0), p0);                         // (x00, x10)
  const float2 x1 = fma2(dxx, sub2(q1, p1), p1);                         // (x01, x11)
  const float2 lo = make_float2(x0.x, x1.x), hi = make_float2(x0.y, x1.y);
  const float2 y = fma2(make_float2(dy, dy), sub2(hi, lo), lo);          // (y0, y1)
  return fmaf(dz, y.y - y.x, y.x);
}

// grid_sample for any record format (see RecFormat).
template <int FMT>
__device__ __forceinline__ float grid_sample_fmt(const GridView& g, float ux, float uy, float uz, int c) {
  if constexpr (FMT == kRecF32) {
    return grid_sample(g, ux, uy, uz, c);
  } else {
    bool inb = (ux >= 0.f) & (ux <= g.mx) & (uy >= 0.f) & (uy <= g.my) & (uz >= 0.f) & (uz <= g.mz);
    float e = g.penalty;
    if (inb) {
      float fx = floorf(ux);   // <= n - 1: the padding layer holds the upper faces
      float fy = floorf(uy);
      float fz = floorf(uz);
      int ix = (int)fx, iy = (int)fy, iz = (int)fz;
      float dx = ux - fx, dy = uy - fy, dz = uz - fz;
      const size_t ri = rec_index(g.cx, g.cy, g.cz, c, ix, iy, iz);
      if (!lg_check(g.check, c >= 0 && c < g.nc && ri < g.n_rec, kChkGridRecord)) return g.penalty;
      const uint4* rec = reinterpret_cast<const uint4*>(g.coef) + ri;
      const uint4 v = __ldg(rec);
      e = lerp16<FMT>(v, dx, dy, dz);
    }
    return e;
  }
}

// The docking kernel's sampler, in steps, so that two samples share their
// packed instructions (positions, cells and fractions of a pair). Same values
// as grid_sample_fmt, bit for bit.
//
//   floor     u + 2^23 rounded towards zero has floor(u) in its low mantissa
//             bits (0 <= u < 2^23) and gives it back as a float by
//             subtracting 2^23: two full-rate additions instead of a
//             round-down and a conversion;
//   clamp     coefficient records end below the upper faces (rec_cells): the
//             coordinate is cut to the float below n - 1 before its floor, so
//             a point on a face takes the last cell at f = 1;
//   inside    the bits of a float order like unsigned integers, negative ones
//             and NaN above every coordinate of the box: one comparison per
//             axis. A coordinate of -0 would count as outside; positions here
//             are sums that start from t - origin, which is never -0;
//   record    32-bit index arithmetic (no axis has 2^23 cells here, so a
//             channel has fewer than 2^32, padding included) on the
//             unreduced bits, their constant part subtracted once
//             (GridView::bias). Bounds, bias and cell counts are
//             constant-bank operands: none takes a register.
//
// Measured on GB300 against floorf, conversions, six comparisons and a clamp
// per scalar sample (docking kernel, 12,000 screening / 3,000 bimodal
// ligands): FP32 26.28 -> 23.12 / 11.93 -> 9.66 ms (2,000 screening ligands:
// 3.67 -> 2.44 G warp instructions, 4.69 -> 3.88 ms, 303 G samples/s of the
// 308 G/s gather ceiling), FP16 26.25 -> 25.28 / 11.76 -> 11.23 ms.
constexpr float kFloorMagic = 8388608.f;   // 2^23

struct DockPoint {   // a position, its cell as unreduced bits, its fractions
  float ux, uy, uz;
  unsigned bx, by, bz;
  float dx, dy, dz;
};

template <int FMT>
__device__ __forceinline__ DockPoint dock_point(const GridView& g, float ux, float uy, float uz) {
  constexpr bool kClamp = FMT == kRecF32;
  const float tx = __fadd_rz(kClamp ? fminf(ux, g.lx) : ux, kFloorMagic);
  const float ty = __fadd_rz(kClamp ? fminf(uy, g.ly) : uy, kFloorMagic);
  const float tz = __fadd_rz(kClamp ? fminf(uz, g.lz) : uz, kFloorMagic);
  return {ux, uy, uz, __float_as_uint(tx), __float_as_uint(ty), __float_as_uint(tz),
          ux - (tx - kFloorMagic), uy - (ty - kFloorMagic), uz - (tz - kFloorMagic)};
}

// Two points at once, FP32 records.
__device__ __forceinline__ void dock_points2(const GridView& g, float2 x, float2 y, float2 z, DockPoint& p,
                                             DockPoint& q) {
  const float2 m = make_float2(kFloorMagic, kFloorMagic);
  const float2 tx = add2_rz(make_float2(fminf(x.x, g.lx), fminf(x.y, g.lx)), m);
  const float2 ty = add2_rz(make_float2(fminf(y.x, g.ly), fminf(y.y, g.ly)), m);
  const float2 tz = add2_rz(make_float2(fminf(z.x, g.lz), fminf(z.y, g.lz)), m);
  const float2 dx = sub2(x, sub2(tx, m)), dy = sub2(y, sub2(ty, m)), dz = sub2(z, sub2(tz, m));
  p = {x.x, y.x, z.x, __float_as_uint(tx.x), __float_as_uint(ty.x), __float_as_uint(tz.x), dx.x, dy.x, dz.x};
  q = {x.y, y.y, z.y, __float_as_uint(tx.y), __float_as_uint(ty.y), __float_as_uint(tz.y), dx.y, dy.y, dz.y};
}

__device__ __forceinline__ bool dock_in(const GridView& g, const DockPoint& p) {
  return (__float_as_uint(p.ux) <= g.hx) & (__float_as_uint(p.uy) <= g.hy) & (__float_as_uint(p.uz) <= g.hz);
}

// Channel c's records: for coefficient records (at most 2^31 of them) an
// index offset, for 16-bit ones (padded, possibly more) an address.
template <int FMT>
struct DockChannel {
  unsigned off;
  const unsigned char* base;
  __device__ __forceinline__ DockChannel(const GridView& g, int c) {
    if constexpr (FMT == kRecF32) {
      off = (unsigned)c * g.cells - g.bias;
      base = nullptr;
    } else {
      off = 0u;   // the bias is subtracted as a constant operand
      base = reinterpret_cast<const unsigned char*>(g.coef) + (size_t)c * g.cz * g.cy * g.cx * 16;
    }
  }
};

// Energy at a point; with GUARD any point (the first record is loaded for one
// outside the box, without a branch), else one for which dock_in holds.
template <int FMT, bool GUARD = false>
__device__ __forceinline__ float dock_energy(const GridView& g, const DockChannel<FMT>& ch, const DockPoint& p, int c) {
  const bool in = !GUARD || dock_in(g, p);
  const unsigned cell = (p.bz * g.cy + p.by) * g.cx + p.bx;
  if constexpr (FMT == kRecF32) {
    const unsigned ri = in ? cell + ch.off : 0u;
    if (!lg_check(g.check, c >= 0 && c < g.nc && ri < g.n_rec, kChkGridRecord)) return g.penalty;
    float a[8];
    ld_global_v8_na(g.coef + (size_t)ri * 8, a);
    const float t1 = fmaf(p.dz, a[7], a[4]);
    float t2 = fmaf(p.dy, t1, a[1]);
    t2 = fmaf(p.dz, a[5], t2);
    const float t3 = fmaf(p.dz, a[6], a[2]);
    float e = fmaf(p.dz, a[3], a[0]);
    e = fmaf(p.dy, t3, e);
    e = fmaf(p.dx, t2, e);
    return in ? e : g.penalty;
  } else {
    const unsigned ri = in ? cell - g.bias : 0u;
    if (!lg_check(g.check, c >= 0 && c < g.nc && (size_t)c * g.cz * g.cy * g.cx + ri < g.n_rec, kChkGridRecord))
      return g.penalty;
    const float e = lerp16<FMT>(__ldg(reinterpret_cast<const uint4*>(ch.base) + ri), p.dx, p.dy, p.dz);
    return in ? e : g.penalty;
  }
}

// Value and gradient (per grid unit) of channel `c` at grid-unit position u:
// the derivative of the cell's trilinear polynomial, zero outside the box.
__device__ __forceinline__ float grid_sample_grad(const GridView& g, float ux, float uy, float uz, int c,
                                                  float* gx, float* gy, float* gz) {
  bool inb = (ux >= 0.f) & (ux <= g.mx) & (uy >= 0.f) & (uy <= g.my) & (uz >= 0.f) & (uz <= g.mz);
  float e = g.penalty;
  *gx = *gy = *gz = 0.f;
  if (inb) {
    float fx = fminf(floorf(ux), g.kx);
    float fy = fminf(floorf(uy), g.ky);
    float fz = fminf(floorf(uz), g.kz);
    int ix = (int)fx, iy = (int)fy, iz = (int)fz;
    float dx = ux - fx, dy = uy - fy, dz = uz - fz;
    const size_t ri = rec_index_f32(g.cx, g.cy, g.cz, c, ix, iy, iz);
    if (!lg_check(g.check, c >= 0 && c < g.nc && ri < g.n_rec, kChkGridRecord)) return g.penalty;
    const float* rec = g.coef + ri * 8;
    float a[8];
    ld_global_v8_na(rec, a);
    float t1 = fmaf(dz, a[7], a[4]);
    float t2 = fmaf(dy, t1, a[1]);
    t2 = fmaf(dz, a[5], t2);
    float t3 = fmaf(dz, a[6], a[2]);
    e = fmaf(dz, a[3], a[0]);
    e = fmaf(dy, t3, e);
    e = fmaf(dx, t2, e);
    *gx = t2;                                              // ax + axy fy + axz fz + axyz fy fz
    *gy = fmaf(dx, t1, t3);                                // ay + axy fx + ayz fz + axyz fx fz
    *gz = fmaf(dx, fmaf(dy, a[7], a[5]), fmaf(dy, a[6], a[3]));  // az + axz fx + ayz fy + axyz fx fy
  }
  return e;
}

// A coefficient record fetched ahead of its use: the scoring and gradient
// kernels issue the loads of several atoms before they use any. Same cell,
// fractions and box test as grid_sample; a point outside loads the first
// record. Adding +0 first makes a coordinate of -0 (poses are given, so it
// can occur) compare as inside.
struct FetchedRecord {
  float a[8];
  float dx, dy, dz;
  bool in;
};

__device__ __forceinline__ FetchedRecord grid_fetch(const GridView& g, float ux, float uy, float uz, int c) {
  FetchedRecord r;
  ux += 0.f; uy += 0.f; uz += 0.f;
  const DockPoint p = dock_point<kRecF32>(g, ux, uy, uz);
  r.dx = p.dx; r.dy = p.dy; r.dz = p.dz;
  r.in = dock_in(g, p);
  const unsigned ri = r.in ? (p.bz * g.cy + p.by) * g.cx + p.bx + DockChannel<kRecF32>(g, c).off : 0u;
  if (!lg_check(g.check, c >= 0 && c < g.nc && ri < g.n_rec, kChkGridRecord)) {
    r.in = false;
    return r;
  }
  ld_global_v8_na(g.coef + (size_t)ri * 8, r.a);
  return r;
}

__device__ __forceinline__ float fetched_value(const GridView& g, const FetchedRecord& r) {
  const float t1 = fmaf(r.dz, r.a[7], r.a[4]);
  float t2 = fmaf(r.dy, t1, r.a[1]);
  t2 = fmaf(r.dz, r.a[5], t2);
  const float t3 = fmaf(r.dz, r.a[6], r.a[2]);
  float e = fmaf(r.dz, r.a[3], r.a[0]);
  e = fmaf(r.dy, t3, e);
  e = fmaf(r.dx, t2, e);
  return r.in ? e : g.penalty;
}

// The value, and the gradient per grid unit (zero outside).
__device__ __forceinline__ float fetched_grad(const GridView& g, const FetchedRecord& r, float* gx, float* gy,
                                              float* gz) {
  const float t1 = fmaf(r.dz, r.a[7], r.a[4]);
  float t2 = fmaf(r.dy, t1, r.a[1]);
  t2 = fmaf(r.dz, r.a[5], t2);
  const float t3 = fmaf(r.dz, r.a[6], r.a[2]);
  float e = fmaf(r.dz, r.a[3], r.a[0]);
  e = fmaf(r.dy, t3, e);
  e = fmaf(r.dx, t2, e);
  const float hy = fmaf(r.dx, t1, t3);
  const float hz = fmaf(r.dx, fmaf(r.dy, r.a[7], r.a[5]), fmaf(r.dy, r.a[6], r.a[3]));
  *gx = r.in ? t2 : 0.f;   // ax + axy fy + axz fz + axyz fy fz
  *gy = r.in ? hy : 0.f;   // ay + axy fx + ayz fz + axyz fx fz
  *gz = r.in ? hz : 0.f;   // az + axz fx + ayz fy + axyz fx fy
  return r.in ? e : g.penalty;
}

}  // namespace ligen
