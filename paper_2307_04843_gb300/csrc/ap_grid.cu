// ap_grid.cu -- packed copies of the static grid field.
//
// The six component arrays of the grid (Sec. 2.1, E2/B2) are re-laid out in
// one of two forms:
//   AP_PACK_NODES: one 32-byte record per node (Ex, Ey, Ez, Bx, By, Bz, 0, 0),
//     so that the refetch of a particle's cell reads 8 sectors instead of 24
//     (6 arrays x 4 rows of 2 adjacent nodes); the values are unchanged.
//   AP_PACK_CELLS: one 192-byte record per cell holding, per component, the
//     coefficients of the trilinear interpolant in the monomial basis
//       F(w) = a0 + a1 wx + a2 wy + a3 wz + a4 wx wy + a5 wy wz + a6 wx wz + a7 wx wy wz,
//     a0 = c000, a1 = c100 - c000, ..., a7 = the alternating sum of the 8
//     corners (cijk = corner i along x, j along y, k along z), computed in
//     double and rounded once; the refetch is one contiguous record and the
//     evaluation 7 FMA per component.  The components are interleaved in
//     pairs so that packed (f32x2) FMA evaluate two components at once.
#include <cuda_runtime.h>

#include "ap_internal.h"

namespace {

__global__ void pack_nodes_kernel(const float *__restrict__ f0, const float *__restrict__ f1,
                                  const float *__restrict__ f2, const float *__restrict__ f3,
                                  const float *__restrict__ f4, const float *__restrict__ f5,
                                  float4 *__restrict__ out, long long nodes) {
  const long long stride = (long long)gridDim.x * blockDim.x;
  for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < nodes; i += stride) {
    out[2 * i] = make_float4(f0[i], f1[i], f2[i], f3[i]);
    out[2 * i + 1] = make_float4(f4[i], f5[i], 0.0f, 0.0f);
  }
}

struct CompPtrs {
  const float *f[6];
};

// x - y as hi + lo exactly (Knuth's TwoSum of x and -y)
struct Diff {
  float hi, lo;
};
__device__ __forceinline__ Diff two_diff(float x, float y) {
  const float s = __fsub_rn(x, y);
  const float b = __fsub_rn(s, x);
  return {s, __fsub_rn(__fsub_rn(x, __fsub_rn(s, b)), __fadd_rn(y, b))};
}
// (p - q) as a float-float sum, and rounded to one float
__device__ __forceinline__ Diff diff(Diff p, Diff q) {
  Diff d = two_diff(p.hi, q.hi);
  d.lo = __fadd_rn(d.lo, __fsub_rn(p.lo, q.lo));
  return d;
}
__device__ __forceinline__ float diff_rn(Diff p, Diff q) {
  const Diff d = diff(p, q);
  return __fadd_rn(d.hi, d.lo);
}

// The eight coefficients of one component from its corners c[i + 2 j + 4 k].
// The differences of differences are formed in float-float arithmetic: the
// first differences exactly, the second and third to 2^-48 of the first (not of
// the result), which drops bits only where corners of three magnitudes meet: the
// low parts are multiples of the smallest corner's last place, and their sums
// fit a float otherwise (cells that cancel to their last bits are tested against
// exact differences).  Forming them from exact parts throughout took 23 % longer,
// only where one cancels below 2^-16 8 %.  In double each difference would run
// on the FP64 pipe, which together with the conversions is what bounded the
// whole copy (see pack_cells_kernel).  A corner that is not finite, or one so
// large that a float difference overflows, shows up in a5, a6 or a7 (between
// them they take in every difference): then the coefficients come from the
// plain double differences.
__device__ __forceinline__ void cell_coeffs(const float c[8], float a[8]) {
  const Diff x00 = two_diff(c[1], c[0]), x10 = two_diff(c[3], c[2]);
  const Diff x01 = two_diff(c[5], c[4]), x11 = two_diff(c[7], c[6]);
  const Diff y0 = two_diff(c[2], c[0]), y1 = two_diff(c[6], c[4]);
  a[0] = c[0];
  a[1] = x00.hi;
  a[2] = y0.hi;
  a[3] = __fsub_rn(c[4], c[0]);
  const Diff xy0 = diff(x10, x00), xy1 = diff(x11, x01);
  a[4] = __fadd_rn(xy0.hi, xy0.lo);
  a[5] = diff_rn(y1, y0);
  a[6] = diff_rn(x01, x00);
  a[7] = diff_rn(xy1, xy0);
  if (!(fabsf(a[5]) + fabsf(a[6]) + fabsf(a[7]) <= 3.402823466e38f)) {
    double d[8];
    for (int k = 0; k < 8; ++k) d[k] = (double)c[k];
    a[1] = (float)(d[1] - d[0]);
    a[2] = (float)(d[2] - d[0]);
    a[3] = (float)(d[4] - d[0]);
    a[4] = (float)((d[3] - d[1]) - (d[2] - d[0]));
    a[5] = (float)((d[6] - d[2]) - (d[4] - d[0]));
    a[6] = (float)((d[5] - d[1]) - (d[4] - d[0]));
    a[7] = (float)(((d[7] - d[3]) - (d[5] - d[1])) - ((d[6] - d[2]) - (d[4] - d[0])));
  }
}

// Record = 12 float4 with the components interleaved in pairs (Ex, Ey),
// (Ez, Bx), (By, Bz): float 16 p + 2 k + h is coefficient a_k of component
// 2 p + h.  Bound by the writes: 192 bytes per cell against 24 read.  A warp
// takes 32 consecutive cells, lane l computing cell l, and turns its 6 KB of
// records around in shared memory (slot k of cell l at [k][l], one float4 of
// padding per row, so both directions are free of bank conflicts up to the
// wrap from one record to the next), so that every store is 512 contiguous
// bytes.  Measured at 256^3 (3.59 GB): 6.88 ms with
// double differences and 4-byte stores 8 bytes apart, 0.69 ms so (5.19 TB/s).
constexpr int kPackWarps = 8;
constexpr int kPackRow = 33;  // float4 per slot row

__global__ void __launch_bounds__(32 * kPackWarps)
    pack_cells_kernel(const __grid_constant__ CompPtrs src, int nx, int ny, int nz, float4 *__restrict__ out) {
  extern __shared__ __align__(16) float4 s_rec[];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  float4 *rec = s_rec + warp * (12 * kPackRow);
  const unsigned cx = nx - 1, cy = ny - 1;
  const unsigned cells = cx * cy * (unsigned)(nz - 1);  // fewer than the nodes, so below 2^31
  const int sy = nx, sz = nx * ny;
  const unsigned n_warps = gridDim.x * kPackWarps;
  const unsigned groups = (cells + 31u) / 32u;
  for (unsigned g = blockIdx.x * kPackWarps + warp; g < groups; g += n_warps) {
    const unsigned first = 32u * g;
    const unsigned n = cells - first < 32u ? cells - first : 32u;
    const unsigned c = first + (lane < (int)n ? lane : (int)n - 1);  // spare lanes repeat the last cell
    const unsigned iz = c / (cx * cy);
    const unsigned r = c - iz * cx * cy;
    const unsigned iy = r / cx;
    const int b = (int)(iz * (unsigned)sz + iy * (unsigned)sy + (r - iy * cx));
#pragma unroll
    for (int p = 0; p < 3; ++p) {
      float a[2][8];
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const float *__restrict__ f = src.f[2 * p + h] + b;
        const float v[8] = {__ldg(f),      __ldg(f + 1),      __ldg(f + sy),      __ldg(f + sy + 1),
                            __ldg(f + sz), __ldg(f + sz + 1), __ldg(f + sz + sy), __ldg(f + sz + sy + 1)};
        cell_coeffs(v, a[h]);
      }
#pragma unroll
      for (int j = 0; j < 4; ++j)
        rec[(4 * p + j) * kPackRow + lane] = make_float4(a[0][2 * j], a[1][2 * j], a[0][2 * j + 1], a[1][2 * j + 1]);
    }
    __syncwarp();
    float4 *dst = out + 12ull * first;
#pragma unroll
    for (int m = 0; m < 12; ++m) {
      const unsigned o = lane + 32 * m;
      if (o < 12u * n) dst[o] = rec[(o % 12u) * kPackRow + o / 12u];
    }
    __syncwarp();
  }
}

bool grid_shape_ok(const ap_grid *g) {
  return g && g->nx >= 2 && g->ny >= 2 && g->nz >= 2 &&
         (double)g->nx * g->ny * g->nz <= 2147483647.0 &&
         (g->packed_layout == AP_PACK_NODES || g->packed_layout == AP_PACK_CELLS);
}

}  // namespace

extern "C" {

size_t ap_grid_packed_bytes(const ap_grid *g) {
  if (!grid_shape_ok(g)) return 0;
  if (g->packed_layout == AP_PACK_CELLS)
    return (size_t)(g->nx - 1) * (g->ny - 1) * (g->nz - 1) * 48 * sizeof(float);
  return (size_t)g->nx * g->ny * g->nz * 8 * sizeof(float);
}

int ap_grid_pack(const ap_grid *g, float *packed, void *stream) {
  if (!grid_shape_ok(g) || !packed) return AP_ERR_ARG;
  for (int c = 0; c < 6; ++c) {
    if (!g->f[c]) return AP_ERR_ARG;
    if (reinterpret_cast<uintptr_t>(g->f[c]) & 3u) return AP_ERR_ALIGN;
  }
  if (reinterpret_cast<uintptr_t>(packed) & 15u) return AP_ERR_ALIGN;
  int dev = 0, sms = 1;
  if (cudaGetDevice(&dev) != cudaSuccess ||
      cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
    return AP_ERR_CUDA;
  const int block = 256;
  const long long cap = (long long)sms * 8;
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  if (g->packed_layout == AP_PACK_CELLS) {
    const long long cells = (long long)(g->nx - 1) * (g->ny - 1) * (g->nz - 1);
    const long long want = (cells + block - 1) / block;
    CompPtrs src;
    for (int c = 0; c < 6; ++c) src.f[c] = g->f[c];
    // shared memory lets four blocks of eight warps stay resident
    const size_t smem = sizeof(float4) * 12 * kPackRow * kPackWarps;
    if (apt::allow_smem(reinterpret_cast<const void *>(pack_cells_kernel), smem) != AP_OK) return AP_ERR_CUDA;
    const long long resident = (long long)sms * 4;
    pack_cells_kernel<<<(int)(want < resident ? want : resident), 32 * kPackWarps, smem, s>>>(
        src, g->nx, g->ny, g->nz, reinterpret_cast<float4 *>(packed));
  } else {
    const long long nodes = (long long)g->nx * g->ny * g->nz;
    const long long want = (nodes + block - 1) / block;
    pack_nodes_kernel<<<(int)(want < cap ? want : cap), block, 0, s>>>(
        g->f[0], g->f[1], g->f[2], g->f[3], g->f[4], g->f[5], reinterpret_cast<float4 *>(packed), nodes);
  }
  return cudaGetLastError() == cudaSuccess ? AP_OK : AP_ERR_CUDA;
}

}  // extern "C"
