// collect.cuh -- the push's flux accumulators turned into J_PIC: shared by the
// stand-alone collection (particles.cu) and the field kernels that carry it
// along (fields.cu).
#pragma once
#include "hff_common.cuh"

namespace hff {

// The accumulators (see deposit in particles.cu) are added to J_PIC (face
// areas, node volumes and dt applied) and cleared for the next push, at the
// end of the push stage.
// FP32: a warp owns 32 columns of cell records and walks kCollectRows rows
// upward; each record is read (and, if anything was deposited, cleared) once,
// by one lane, the parts of neighbouring cells that meet at a location are
// summed by a shuffle along theta and in registers along r, and added to J
// with one coalesced reduction per location (two at the borders of a warp's
// area).  HBM-bound on large grids: 32 B read per cell, plus 32 B and the J
// traffic where particles are.
// FP64: the three arrays, element by element.
// In a whole step the collection shares a launch with grid work that does not
// touch J (Faraday's first half step, or the fused update's halo snapshot):
// a launch of its own costs about 3 us of a small step.
constexpr int kCollectThreads = 128;
constexpr int kCollectRows = 16;

template <typename R> __host__ __device__ inline int collect_blocks_x(const Params<R> &p) {
  return (p.nt + 1 + (sizeof(R) == 8 ? 1 : 0) + kCollectThreads - 1) / kCollectThreads;
}
template <typename R> __host__ __device__ inline int collect_blocks_y(const Params<R> &p) {
  return (p.nr + 1 + (sizeof(R) == 8 ? 1 : 0) + kCollectRows - 1) / kCollectRows;
}

__device__ __forceinline__ void add_j(const Params<float> &p, int which, int i, int j, float v) {
  if (v == 0.f) return;
  const int nr = p.nr, nt = p.nt, n1 = nt + 1;
  if (which == 0) { if (i < nr && j <= nt) atomicAdd(&p.f.jr[ix(i, j, n1)], v * p.t.dep_r[i] * p.t.inv_dch[j]); }
  else if (which == 1) { if (i <= nr && j < nt) atomicAdd(&p.f.jt[ix(i, j, nt)], v * p.t.dep_t[i] * p.t.inv_sh[j]); }
  else if (i <= nr && j <= nt) atomicAdd(&p.f.jp[ix(i, j, n1)], v * p.t.dep_p[i] * p.t.inv_dch[j]);
}
__device__ __forceinline__ void collect_block(const Params<float> &p, int bx, int by) {
  const int n1 = p.nt + 1, lane = threadIdx.x & 31;
  const int j = bx * kCollectThreads + (int)threadIdx.x, i0 = by * kCollectRows;
  const int i1 = min(i0 + kCollectRows, p.nr + 1);
  float tb = 0.f, c0 = 0.f, c1 = 0.f;   // J_th and J_ph parts for the row above
  for (int i = i0; i < i1; ++i) {
    float4 a = make_float4(0.f, 0.f, 0.f, 0.f), c = a;
    if (j < n1) {
      float4 *rec = reinterpret_cast<float4 *>(p.jacc + 8 * ix(i, j, n1));
      a = rec[0];
      c = rec[1];
      const float4 z = make_float4(0.f, 0.f, 0.f, 0.f);
      if (a.x != 0.f || a.y != 0.f || a.z != 0.f || a.w != 0.f) rec[0] = z;
      if (c.x != 0.f || c.y != 0.f || c.z != 0.f || c.w != 0.f) rec[1] = z;
    }
    const float right = c.y + c1;   // J_ph at (i, j + 1) from this column's cells
    const float ra = __shfl_up_sync(0xffffffffu, a.y, 1), rc = __shfl_up_sync(0xffffffffu, right, 1);
    add_j(p, 0, i, j, a.x + (lane ? ra : 0.f));
    add_j(p, 1, i, j, a.z + tb);
    add_j(p, 2, i, j, c.x + c0 + (lane ? rc : 0.f));
    if (lane == 31) { add_j(p, 0, i, j + 1, a.y); add_j(p, 2, i, j + 1, right); }
    tb = a.w; c0 = c.z; c1 = c.w;
  }
  const float rc = __shfl_up_sync(0xffffffffu, c1, 1);
  add_j(p, 1, i1, j, tb);
  add_j(p, 2, i1, j, c0 + (lane ? rc : 0.f));
  if (lane == 31) add_j(p, 2, i1, j + 1, c1);
}
__device__ __forceinline__ void collect_block(const Params<double> &p, int bx, int by) {
  const int nr = p.nr, nt = p.nt, n1 = nt + 1, ld = nt + 2;
  const int j = bx * kCollectThreads + (int)threadIdx.x, i0 = by * kCollectRows, i1 = min(i0 + kCollectRows, nr + 2);
  if (j >= ld) return;
  const int64_t nn = (int64_t)(nr + 2) * ld;
  for (int i = i0; i < i1; ++i) {
    double *q = p.jacc + ix(i, j, ld);
    const double r = q[0], t = q[nn], f = q[2 * nn];
    if (r != 0.0) { q[0] = 0.0; if (i < nr && j <= nt) p.f.jr[ix(i, j, n1)] += r * p.t.dep_r[i] * p.t.inv_dch[j]; }
    if (t != 0.0) { q[nn] = 0.0; if (i <= nr && j < nt) p.f.jt[ix(i, j, nt)] += t * p.t.dep_t[i] * p.t.inv_sh[j]; }
    if (f != 0.0) {
      q[2 * nn] = 0.0;
      if (i <= nr && j <= nt) p.f.jp[ix(i, j, n1)] += f * p.t.dep_p[i] * p.t.inv_dch[j];
    }
  }
}

}  // namespace hff
