// ap_lines.cuh -- what the register-resident float lines share (vacuum Yee
// lines, plasma lines, the split line of Sec. 4).
//
// One block per line.  Thread t owns two runs of C consecutive nodes,
// [t C, t C + C) and [H + t C, H + t C + C) with H = C times the block, held in
// the two halves of packed (f32x2) values: every update of a node of the first
// run is issued together with the same update of the second, with no shuffling
// between them.  The updates are additions, subtractions and products of one
// rounding each, so half the instructions is what packing saves; the scalar
// form issued 23.5 instructions per node-step of the plasma line at 93 % of the
// issue slots.  Only the values at run boundaries move, through shared memory:
// slot t for the first run, slot block + t for the second, so the last thread's
// right neighbour in the first run is simply the next slot.
#pragma once

#include "ap_step.cuh"

namespace apt {

// A packed product that stays apart from the sum it feeds: the assembler fuses
// a packed multiplication whose only uses are sums with each of them (see
// ap_pair.cuh), while the lines have to reproduce a plain loop of separately
// rounded operations bit for bit.  a b + (-0) is the rounded
// product, signs of zeros included, in one operation that nothing can be fused
// into; the -0 comes as a kernel argument, so that it is not known to be one.
struct LineMul {
  F2 nzero;
  __device__ __forceinline__ explicit LineMul(float nz) : nzero(nz) {}
  __device__ __forceinline__ F2 operator()(F2 a, F2 b) const { return rfma(a, b, nzero); }
};
__device__ __forceinline__ F2 ladd(F2 a, F2 b) { return a + b; }
__device__ __forceinline__ F2 lsub(F2 a, F2 b) { return a - b; }

// The run boundaries of a block: each half of a value goes to its own slot.
// Neighbours past the ends read as zero; what they would feed is a node whose
// value is kept (below).
struct LineEdge {
  float *s;  // [2 block]
  __device__ __forceinline__ void put(F2 v) const {
    s[threadIdx.x] = v.x;
    s[blockDim.x + threadIdx.x] = v.y;
  }
  __device__ __forceinline__ F2 next() const {  // of each run's last node
    const int t = threadIdx.x, bd = blockDim.x;
    return F2(s[t + 1], t + 1 < bd ? s[bd + t + 1] : 0.0f);
  }
  __device__ __forceinline__ F2 prev() const {  // of each run's first node
    const int t = threadIdx.x, bd = blockDim.x;
    return F2(t > 0 ? s[t - 1] : 0.0f, s[bd + t - 1]);
  }
};

// E_0 and B_{nz-1} never change: E_0 belongs to thread 0, and the thread that
// owns node nz - 1 puts B back after each update (the test is uniform for
// every other warp).  Nodes past nz - 1 start from zeros, take on whatever the
// updates give (B_{nz-1} and, on the split line, J1 reach them) and are not
// stored; they feed nothing but the B that is put back.
struct LineEnds {
  int ix, iy;      // index of node nz - 1 in this thread's first, second run, or -1
  float keep;      // B_{nz-1}
  bool warp_has;   // whether a thread of this warp owns it
  template <int C>
  __device__ __forceinline__ void init(int nz, const F2 (&b)[C]) {
    const int t = threadIdx.x, H = C * blockDim.x, k = nz - 1;
    ix = k >= t * C && k < t * C + C ? k - t * C : -1;
    iy = k >= H + t * C && k < H + t * C + C ? k - H - t * C : -1;
    keep = 0.0f;
#pragma unroll
    for (int i = 0; i < C; ++i) {
      if (i == ix) keep = b[i].x;
      if (i == iy) keep = b[i].y;
    }
    warp_has = __any_sync(0xffffffffu, ix >= 0 || iy >= 0);
  }
  template <int C>
  __device__ __forceinline__ void restore(F2 (&b)[C]) const {
    if (warp_has) {
#pragma unroll
      for (int i = 0; i < C; ++i) {
        if (i == ix) b[i].x = keep;
        if (i == iy) b[i].y = keep;
      }
    }
  }
};

template <int C>
__device__ __forceinline__ void line_load(F2 (&v)[C], const float *g, int nz) {
  const int t = threadIdx.x, H = C * blockDim.x;
#pragma unroll
  for (int i = 0; i < C; ++i) {
    const int k = t * C + i;
    v[i] = F2(k < nz ? g[k] : 0.0f, H + k < nz ? g[H + k] : 0.0f);
  }
}
template <int C>
__device__ __forceinline__ void line_store(const F2 (&v)[C], float *g, int nz) {
  const int t = threadIdx.x, H = C * blockDim.x;
#pragma unroll
  for (int i = 0; i < C; ++i) {
    const int k = t * C + i;
    if (k < nz) g[k] = v[i].x;
    if (H + k < nz) g[H + k] = v[i].y;
  }
}

// B half step: b_k -= h (e_{k+1} - e_k), en the node after the run
template <int C>
__device__ __forceinline__ void line_b_step(F2 (&b)[C], const F2 (&e)[C], F2 en, F2 h, const LineMul &lmul) {
#pragma unroll
  for (int i = 0; i < C; ++i) {
    const F2 enx = i + 1 < C ? e[i + 1 < C ? i + 1 : i] : en;
    b[i] = lsub(b[i], lmul(h, lsub(enx, e[i])));
  }
}

// threads of a line's block: two runs of C nodes each, whole warps
template <int C>
inline int line_block(int nz) { return ((nz + 2 * C - 1) / (2 * C) + 31) / 32 * 32; }

}  // namespace apt
