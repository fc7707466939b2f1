// collect.cuh -- the push's flux accumulators turned into J_PIC: shared by the
// stand-alone collection (particles.cu) and the field kernels that carry it
// along (fields.cu).
#pragma once
#include "hff_common.cuh"

namespace hff {

// The accumulators (see deposit in particles.cu) are added to J_PIC (face
// areas, node volumes and dt applied) and cleared for the next push, at the
// end of the push stage.
// FP32: a warp owns 32 columns of cell records and kCollectRows rows, which it
// reads first and then walks upward (a chain of rows, each loaded behind the
// last one's stores, was the longest piece of a small step: with 16 rows a
// step took 52.2 us on 96 x 80, 156 on 500 x 380 and 204 on 256 x 128 in FP64;
// now 42.4, 143 and 187; 4 rows 43.5, 144, 190; large grids the same within
// 0.3%); each record is read (and, if anything was deposited, cleared) once,
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
constexpr int kCollectRows = 2;

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
  const float4 z = make_float4(0.f, 0.f, 0.f, 0.f);
  float tb = 0.f, c0 = 0.f, c1 = 0.f;   // J_th and J_ph parts for the row above
  float4 a[kCollectRows], c[kCollectRows];
#pragma unroll
  for (int k = 0; k < kCollectRows; ++k) {
    a[k] = c[k] = z;
    if (i0 + k < i1 && j < n1) {
      const float4 *rec = reinterpret_cast<const float4 *>(p.jacc + 8 * ix(i0 + k, j, n1));
      a[k] = rec[0];
      c[k] = rec[1];
    }
  }
#pragma unroll
  for (int k = 0; k < kCollectRows; ++k) {
    const int i = i0 + k;
    if (i >= i1) break;
    float4 *rec = reinterpret_cast<float4 *>(p.jacc + 8 * ix(i, j, n1));   // zero past the row: not cleared
    if (a[k].x != 0.f || a[k].y != 0.f || a[k].z != 0.f || a[k].w != 0.f) rec[0] = z;
    if (c[k].x != 0.f || c[k].y != 0.f || c[k].z != 0.f || c[k].w != 0.f) rec[1] = z;
    const float right = c[k].y + c1;   // J_ph at (i, j + 1) from this column's cells
    const float ra = __shfl_up_sync(0xffffffffu, a[k].y, 1), rc = __shfl_up_sync(0xffffffffu, right, 1);
    add_j(p, 0, i, j, a[k].x + (lane ? ra : 0.f));
    add_j(p, 1, i, j, a[k].z + tb);
    add_j(p, 2, i, j, c[k].x + c0 + (lane ? rc : 0.f));
    if (lane == 31) { add_j(p, 0, i, j + 1, a[k].y); add_j(p, 2, i, j + 1, right); }
    tb = a[k].w; c0 = c[k].z; c1 = c[k].w;
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
  double v[kCollectRows][3];
#pragma unroll
  for (int k = 0; k < kCollectRows; ++k) {
    const double *q = p.jacc + ix(min(i0 + k, i1 - 1), j, ld);
    v[k][0] = q[0]; v[k][1] = q[nn]; v[k][2] = q[2 * nn];
  }
#pragma unroll
  for (int k = 0; k < kCollectRows; ++k) {
    const int i = i0 + k;
    if (i >= i1) break;
    double *q = p.jacc + ix(i, j, ld);
    const double r = v[k][0], t = v[k][1], f = v[k][2];
    if (r != 0.0) { q[0] = 0.0; if (i < nr && j <= nt) p.f.jr[ix(i, j, n1)] += r * p.t.dep_r[i] * p.t.inv_dch[j]; }
    if (t != 0.0) { q[nn] = 0.0; if (i <= nr && j < nt) p.f.jt[ix(i, j, nt)] += t * p.t.dep_t[i] * p.t.inv_sh[j]; }
    if (f != 0.0) {
      q[2 * nn] = 0.0;
      if (i <= nr && j <= nt) p.f.jp[ix(i, j, n1)] += f * p.t.dep_p[i] * p.t.inv_dch[j];
    }
  }
}

}  // namespace hff
