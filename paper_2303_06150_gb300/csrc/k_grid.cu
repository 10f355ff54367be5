// Grid preparation: node values [z][y][x][c] -> per-(cell, channel) records
// of the 8 coefficients of the cell's trilinear polynomial (or its 8 corner
// values in 16 bits), at rec_index (channel-major, see GridView).
//
// The bound is the write of the records (96^3 x 8 nodes: 219 MB in FP32
// against 28 MB read). A thread owns one (x, y, channel) column of cells and
// marches along z, so a cell's lower corners are the registers of the cell
// below and every step costs four loads (consecutive threads: consecutive
// channels, then x, then y; whole lines, and no idle threads however short a
// row is), twelve additions and one store of the whole record; indices are
// divided out once per thread. Measured on GB300, 96^3 x 8: FP32 63 -> 40.5 us
// (6.1 TB/s), FP16 66 -> 35 us, against one thread per record with 64-bit
// divisions and eight loads each. With a block's threads inside one row, a
// call with a 2 x 1500 x 1500 x 1 grid took 179 us, now 23. A plane that
// fits a block several times over gives the spare threads the marches above it
// (2 x 2 x 4000001 x 1, whole call: 242 us without, 50), two cells each where
// it is narrower than a warp (with 12, 78 us: a warp's stores lie 384 bytes
// apart).
#include "internal.h"

namespace ligen {
namespace {

constexpr int kPrepThreads = 128;
// Cells a thread marches through, at most: each march loads one plane of
// nodes more than it has cells. Small grids march less far, down to 2 cells,
// to make kPrepBlocks blocks (16 per SM): 40^3 x 4 with 12 cells is 312
// blocks and takes 9 us, with 2 cells 1,560 blocks.
constexpr int kPrepMarch = 12;
constexpr int kPrepBlocks = 2432;

__device__ __forceinline__ void st_global_v8(float* p, const float (&v)[8]) {
  asm volatile("st.global.v8.f32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8};" ::"l"(p), "f"(v[0]), "f"(v[1]), "f"(v[2]),
               "f"(v[3]), "f"(v[4]), "f"(v[5]), "f"(v[6]), "f"(v[7])
               : "memory");
}

template <int FMT>
__device__ __forceinline__ unsigned pack16(float a, float b) {   // rounded to nearest
  if constexpr (FMT == kRecF16) {
    const __half2 h = __floats2half2_rn(a, b);
    return *reinterpret_cast<const unsigned*>(&h);
  } else {
    const __nv_bfloat162 h = __floats2bfloat162_rn(a, b);
    return *reinterpret_cast<const unsigned*>(&h);
  }
}

// Block: (tile of the plane's (x, y, channel) columns, march), or with THIN
// `per` marches of a plane that fits a block `per` times over. 16-bit record
// grids have rec_cells(n) = n cells per axis: corners past the last node
// repeat it (the padding layers of the clamp-free sampler).
template <int FMT, bool THIN>
__global__ void __launch_bounds__(kPrepThreads) grid_prep_kernel(const float* __restrict__ v, int nx, int ny, int nz,
                                                                 int nc, unsigned tiles, int march, int per,
                                                                 void* __restrict__ out) {
  const int cx = rec_cells(nx, FMT), cy = rec_cells(ny, FMT), cz = rec_cells(nz, FMT);
  const unsigned tile = blockIdx.x % tiles;
  unsigned t = tile * kPrepThreads + threadIdx.x;   // < 2^32 (check_grid)
  const unsigned row = (unsigned)cx * nc;
  int m = (int)(blockIdx.x / tiles);   // march
  if constexpr (THIN) {
    const unsigned sub = t / (row * cy);
    if (sub >= (unsigned)per) return;
    t -= sub * (row * cy);
    m = m * per + (int)sub;
    if (m >= (cz + march - 1) / march) return;
  }
  const int z0 = m * march;
  const int iy = (int)(t / row);
  if (iy >= cy) return;
  const int ix = (int)(t % row / nc), c = (int)(t % row % nc);
  const int z1 = min(z0 + march, cz);
  const int x1 = FMT == kRecF32 ? ix + 1 : min(ix + 1, nx - 1), y1 = FMT == kRecF32 ? iy + 1 : min(iy + 1, ny - 1);
  const size_t plane = (size_t)nx * ny * nc;
  // node (x, y) of plane z: z * plane + one of these
  const size_t o00 = ((size_t)iy * nx + ix) * nc + c, o10 = ((size_t)iy * nx + x1) * nc + c;
  const size_t o01 = ((size_t)y1 * nx + ix) * nc + c, o11 = ((size_t)y1 * nx + x1) * nc + c;
  const float* p = v + (size_t)z0 * plane;
  float c000 = p[o00], c100 = p[o10], c010 = p[o01], c110 = p[o11];
  size_t r = rec_index(cx, cy, cz, c, ix, iy, z0);
  const size_t step = (size_t)cy * cx;
#pragma unroll 4
  for (int iz = z0; iz < z1; ++iz, r += step) {
    if (FMT == kRecF32 || iz + 1 < nz) p += plane;   // past the last node: repeat it
    const float c001 = p[o00], c101 = p[o10], c011 = p[o01], c111 = p[o11];
    if constexpr (FMT == kRecF32) {
      // FP32 differences of differences: each coefficient takes at most three
      // roundings at the grid values' magnitude. (The same sums in FP64 ran on
      // the chip's narrow FP64 pipe: 0.37 ms for a 96^3 x 8 grid against
      // 0.07 ms, measured on GB300.)
      const float dx00 = c100 - c000, dx10 = c110 - c010, dx01 = c101 - c001, dx11 = c111 - c011;
      const float ay = c010 - c000, axy = dx10 - dx00;
      const float rec[8] = {c000, dx00, ay, c001 - c000,           // a0, ax, ay, az
                            axy, dx01 - dx00, (c011 - c001) - ay,  // axy, axz, ayz
                            (dx11 - dx01) - axy};                  // axyz
      st_global_v8(static_cast<float*>(out) + r * 8, rec);
    } else {
      // c000, c100, c010, c110, c001, c101, c011, c111
      static_cast<uint4*>(out)[r] = make_uint4(pack16<FMT>(c000, c100), pack16<FMT>(c010, c110),
                                               pack16<FMT>(c001, c101), pack16<FMT>(c011, c111));
    }
    c000 = c001; c100 = c101; c010 = c011; c110 = c111;
  }
  // beside_pack: what follows this kernel in the stream also follows the packer
  asm volatile("griddepcontrol.wait;" ::: "memory");
}

template <int FMT>
cudaError_t launch_prep(const float* values, int nx, int ny, int nz, int nc, void* rec, bool beside_pack,
                        cudaStream_t s) {
  const size_t cx = rec_cells(nx, FMT), cy = rec_cells(ny, FMT), cz = rec_cells(nz, FMT);
  const size_t columns = cx * cy * nc;
  const size_t tiles = (columns + kPrepThreads - 1) / kPrepThreads;
  const size_t per = columns < kPrepThreads ? kPrepThreads / columns : 1;
  const size_t full = tiles * cz / kPrepBlocks;
  const size_t march = full < 2 || columns < 32 ? 2 : full < kPrepMarch ? full : kPrepMarch;
  const size_t marches = (cz + march - 1) / march;
  const size_t blocks = tiles * ((marches + per - 1) / per);
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3((unsigned)blocks);
  cfg.blockDim = dim3(kPrepThreads);
  cfg.stream = s;
  cudaLaunchAttribute at{};
  at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at.val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = &at;
  cfg.numAttrs = beside_pack ? 1 : 0;
  return cudaLaunchKernelEx(&cfg, per > 1 ? grid_prep_kernel<FMT, true> : grid_prep_kernel<FMT, false>, values, nx, ny,
                            nz, nc, (unsigned)tiles, (int)march, (int)per, rec);
}

}  // namespace

cudaError_t launch_grid_prep(const float* values, int nx, int ny, int nz, int nc, int fmt, void* rec,
                             bool beside_pack, cudaStream_t s) {
  return fmt == kRecF32   ? launch_prep<kRecF32>(values, nx, ny, nz, nc, rec, beside_pack, s)
         : fmt == kRecF16 ? launch_prep<kRecF16>(values, nx, ny, nz, nc, rec, beside_pack, s)
                          : launch_prep<kRecBF16>(values, nx, ny, nz, nc, rec, beside_pack, s);
}

}  // namespace ligen
