// sort.cu -- stable sort of the species' particles by tile key with
// compaction of removed particles, and the (species, tile, chunk) work list
// of the tiled push.
//
// Key = tile index (cells grouped in tile_r x tile_t blocks, row-major over
// tiles); removed particles get the key ntiles and sort last, and so does a
// cell index outside the grid (never produced by the push; only a caller's
// input can hold one), which is also reported through a flag word.  The sort is an
// LSD radix sort over 8-bit digits of (key, index) pairs.  Each pass: per-block
// digit histograms (kSortBlock elements per block), one exclusive scan over the
// digit-major histogram matrix, and a stable scatter in which every element's
// rank inside its block comes from warp match masks, so equal keys keep their
// order (the result equals a stable sort by key).  The particle payload moves
// once, in a final gather.
//
// All species of an instance are sorted by the same launches (blockIdx.y), and
// the passes run over the slots in use: the slot count lives on the device, so
// (to stay capturable in a CUDA graph) the grids cover the capacity and the
// blocks past the count leave at once.
#include <algorithm>
#include <mutex>

#include "../../include/hff.h"
#include "hff_common.cuh"

namespace hff {


// the divisions by nt, tile_r and tile_t by multiplication (FastDiv): three
// run-time integer divisions would cost several times the rest.  The first
// histogram computes the key of every slot and leaves it for the scatter
// (computed twice, the keys were 55 of 300 us per 2.5e7 slots each time).
__device__ __forceinline__ uint32_t tile_key(int cell, int nt, const FastDiv &dnt, const FastDiv &dtr,
                                             const FastDiv &dtt, int ntt, uint32_t ncells, uint32_t dead) {
  if ((uint32_t)cell >= ncells) return dead;   // negative cells too: nr * nt fits 31 bits
  const uint32_t i = fastdiv(dnt, (uint32_t)cell), j = (uint32_t)cell - i * (uint32_t)nt;
  return fastdiv(dtr, i) * (uint32_t)ntt + fastdiv(dtt, j);
}

// one species of a sort
struct SortOne {
  const int32_t *cell;      // first pass: keys are computed from the cells
  uint32_t *keys[2], *idx[2];  // passes alternate between the two
  uint32_t *order;          // the last pass leaves the sorted order here
  uint32_t *hist, *part;
  const long long *n;       // slots to sort (device)
};
struct SortArgs {
  SortOne s[kMaxSpecies];
  uint32_t ncells;          // nr * nt: larger cell indices are invalid input
  unsigned *bad;            // flag word: bad_bit is or-ed in for an invalid cell
  unsigned bad_bit;
  int pass, passes, nt, ntt;
  FastDiv dnt, dtr, dtt;    // divisions by nt, tile_r, tile_t
  uint32_t dead;
};

// blocks of the radix passes over n slots
__host__ __device__ __forceinline__ int64_t sort_blocks(int64_t n) { return (n + kSortBlock - 1) / kSortBlock; }

constexpr int kSortWarps = kSortThreads / 32;
__global__ void __launch_bounds__(kSortThreads) k_hist(const __grid_constant__ SortArgs a) {
  const SortOne &o = a.s[blockIdx.y];
  const int64_t n = *o.n, nb = sort_blocks(n), base = (int64_t)blockIdx.x * kSortBlock;
  if (base >= n) return;
  __shared__ uint32_t h[256];
  h[threadIdx.x] = 0;
  __syncthreads();
  const int lane = threadIdx.x & 31;
  const int64_t first = base + (threadIdx.x >> 5) * (kSortBlock / kSortWarps) + lane;
  bool bad = false;
  uint32_t d[kSortItems];
#pragma unroll
  for (int r = 0; r < kSortItems; ++r) {
    const int64_t e = first + 32 * r;
    d[r] = 256u;
    if (e < n) {
      if (a.pass == 0) {
        const int c = o.cell[e];
        bad = bad || (c >= 0 && (uint32_t)c >= a.ncells);
        d[r] = tile_key(c, a.nt, a.dnt, a.dtr, a.dtt, a.ntt, a.ncells, a.dead);
        o.keys[1][e] = d[r];
      } else {
        d[r] = o.keys[(a.pass + 1) & 1][e];
      }
      d[r] = (d[r] >> (8 * a.pass)) & 255u;
    }
  }
  // particles in nearly sorted order: a warp of equal digits counts them in a
  // register and adds once per change of digit
  uint32_t run = 256u, len = 0;
#pragma unroll
  for (int r = 0; r < kSortItems; ++r) {
    const uint32_t d0 = __shfl_sync(0xffffffffu, d[r], 0);
    if (__all_sync(0xffffffffu, d[r] == d0)) {
      if (d0 != run) {
        if (lane == 0 && run < 256u) atomicAdd(&h[run], len);
        run = d0;
        len = 0;
      }
      len += 32u;
    } else if (d[r] < 256u) {
      atomicAdd(&h[d[r]], 1u);
    }
  }
  if (lane == 0 && run < 256u) atomicAdd(&h[run], len);
  if (__any_sync(0xffffffffu, bad) && (threadIdx.x & 31) == 0) atomicOr(a.bad, a.bad_bit);
  __syncthreads();
  o.hist[(int64_t)threadIdx.x * nb + blockIdx.x] = h[threadIdx.x];
}

// exclusive scan of the histogram matrix in place: block sums, scan of the
// sums, apply (the first two are left out where one block covers it)
__global__ void __launch_bounds__(1024) k_scan_sums(const __grid_constant__ SortArgs a) {
  const SortOne &o = a.s[blockIdx.y];
  const int64_t n = 256 * sort_blocks(*o.n), base = (int64_t)blockIdx.x * kScanBlock;
  if (base >= n) return;
  const uint32_t *x = o.hist;
  __shared__ uint32_t w[32];
  uint32_t s = 0;
  for (int k = threadIdx.x; k < kScanBlock; k += 1024) {
    const int64_t e = base + k;
    if (e < n) s += x[e];
  }
  for (int d = 16; d > 0; d >>= 1) s += __shfl_down_sync(0xffffffffu, s, d);
  if ((threadIdx.x & 31) == 0) w[threadIdx.x >> 5] = s;
  __syncthreads();
  if (threadIdx.x < 32) {
    uint32_t v = w[threadIdx.x];
    for (int d = 16; d > 0; d >>= 1) v += __shfl_down_sync(0xffffffffu, v, d);
    if (threadIdx.x == 0) o.part[blockIdx.x] = v;
  }
}

__device__ __forceinline__ uint32_t block_excl_scan(uint32_t v, uint32_t *w, uint32_t &total) {
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = blockDim.x >> 5;
  uint32_t x = v;
  for (int o = 1; o < 32; o <<= 1) {
    const uint32_t y = __shfl_up_sync(0xffffffffu, x, o);
    if (lane >= o) x += y;
  }
  if (lane == 31) w[wid] = x;
  __syncthreads();
  if (threadIdx.x < 32) {
    uint32_t t = (threadIdx.x < nw) ? w[threadIdx.x] : 0u;
    uint32_t z = t;
    for (int o = 1; o < 32; o <<= 1) {
      const uint32_t y = __shfl_up_sync(0xffffffffu, z, o);
      if (threadIdx.x >= o) z += y;
    }
    w[threadIdx.x] = z - t;  // exclusive warp offsets
    if (threadIdx.x == 31) w[32] = z;
  }
  __syncthreads();
  const uint32_t r = w[wid] + x - v;
  total = w[32];
  __syncthreads();
  return r;
}

__global__ void __launch_bounds__(1024) k_scan_parts(const __grid_constant__ SortArgs a) {
  const SortOne &o = a.s[blockIdx.y];
  const int64_t m = (256 * sort_blocks(*o.n) + kScanBlock - 1) / kScanBlock;
  uint32_t *part = o.part;
  __shared__ uint32_t w[33];
  __shared__ uint32_t carry;
  if (threadIdx.x == 0) carry = 0;
  __syncthreads();
  for (int64_t seg = 0; seg < m; seg += 1024) {
    const int64_t k = seg + threadIdx.x;
    const uint32_t v = (k < m) ? part[k] : 0u;
    uint32_t tot;
    const uint32_t ex = block_excl_scan(v, w, tot);
    if (k < m) part[k] = carry + ex;
    __syncthreads();
    if (threadIdx.x == 0) carry += tot;
    __syncthreads();
  }
}

__global__ void __launch_bounds__(1024) k_scan_apply(const __grid_constant__ SortArgs a, int parts) {
  const SortOne &o = a.s[blockIdx.y];
  const int64_t n = 256 * sort_blocks(*o.n), base = (int64_t)blockIdx.x * kScanBlock;
  if (base >= n) return;
  uint32_t *x = o.hist;
  __shared__ uint32_t w[33];
  __shared__ uint32_t carry;
  if (threadIdx.x == 0) carry = parts > 1 ? o.part[blockIdx.x] : 0u;
  __syncthreads();
  for (int seg = 0; seg < kScanBlock; seg += 1024) {
    const int64_t e = base + seg + threadIdx.x;
    const uint32_t v = (e < n) ? x[e] : 0u;
    uint32_t tot;
    const uint32_t ex = block_excl_scan(v, w, tot);
    if (e < n) x[e] = carry + ex;
    __syncthreads();
    if (threadIdx.x == 0) carry += tot;
    __syncthreads();
  }
}

// Stable scatter.  A block's elements are ordered warp by warp (each warp a
// contiguous piece, walked 32 at a time); an element's rank among those of its
// digit is its warp's count so far plus its place in the match mask.  The
// block's elements are put in digit order in shared memory and written from
// there, so that the writes of a digit are contiguous: written straight from
// the ranks, elements in random order (a load) go out four bytes at a time.
// Bound by its memory traffic (16 B an element and pass) and the ranking's
// shared-memory latency.
struct ScatterSmem {
  uint32_t key[kSortBlock], val[kSortBlock];   // in digit order
  uint32_t cnt[kSortWarps][256];               // per warp: counts, then offsets within the digit
  uint32_t start[256];                         // first place of a digit in the block
  uint32_t base[256];                          // its global place minus start
  uint32_t w[33];
};
template <bool kFirst>   // in the first pass an element's value is its place
__global__ void __launch_bounds__(kSortThreads, 5) k_scatter(const __grid_constant__ SortArgs a) {
  const SortOne &o = a.s[blockIdx.y];
  const int64_t n = *o.n, nb = sort_blocks(n), base = (int64_t)blockIdx.x * kSortBlock;
  if (base >= n) return;
  extern __shared__ __align__(16) unsigned char sort_smem[];
  static_assert(sizeof(ScatterSmem) <= 48 * 1024, "what every kernel may have");
  ScatterSmem &m = *reinterpret_cast<ScatterSmem *>(sort_smem);
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, tid = threadIdx.x, shift = 8 * a.pass;
  for (int w = 0; w < kSortWarps; ++w) m.cnt[w][tid] = 0;
  __syncthreads();
  const unsigned below = (1u << lane) - 1u;
  const int64_t first = base + wid * (kSortBlock / kSortWarps) + lane;
  uint32_t key[kSortItems], val[kFirst ? 1 : kSortItems], rank[kSortItems / 2];   // ranks in pairs of 16 bits
#pragma unroll
  for (int r = 0; r < kSortItems; ++r) {
    const int64_t e = first + 32 * r;
    key[r] = 0xffffffffu;
    if (e < n) {
      key[r] = o.keys[(a.pass + 1) & 1][e];
    }
    if constexpr (!kFirst) val[r] = e < n ? o.idx[(a.pass + 1) & 1][e] : 0u;
  }
  // a warp of equal digits (particles in nearly sorted order) keeps its count
  // in a register until the digit changes
  uint32_t run = 256u, len = 0;
#pragma unroll
  for (int r = 0; r < kSortItems; ++r) {
    const uint32_t d = first + 32 * r < n ? (key[r] >> shift) & 255u : 256u;
    const uint32_t d0 = __shfl_sync(0xffffffffu, d, 0);
    uint32_t rk;
    if (__all_sync(0xffffffffu, d == d0)) {
      if (d0 != run) {
        if (lane == 0 && run < 256u) m.cnt[wid][run] = len;
        __syncwarp();
        run = d0;
        len = d0 < 256u ? m.cnt[wid][d0] : 0u;
      }
      rk = len + lane;
      len += 32u;
    } else {
      if (lane == 0 && run < 256u) m.cnt[wid][run] = len;
      __syncwarp();
      run = 256u;
      const unsigned peers = __match_any_sync(0xffffffffu, d);
      const uint32_t before = d < 256u ? m.cnt[wid][d] : 0u;
      __syncwarp();
      if (d < 256u && (peers & below) == 0) m.cnt[wid][d] = before + __popc(peers);
      __syncwarp();
      rk = before + __popc(peers & below);
    }
    rank[r / 2] = (r & 1) ? rank[r / 2] | (rk << 16) : rk;
  }
  if (lane == 0 && run < 256u) m.cnt[wid][run] = len;
  __syncthreads();
  {  // thread t owns digit t: offsets over the warps, places in the block, and the global place
    uint32_t sum = 0;
    for (int w = 0; w < kSortWarps; ++w) {
      const uint32_t c = m.cnt[w][tid];
      m.cnt[w][tid] = sum;
      sum += c;
    }
    uint32_t tot;
    const uint32_t st = block_excl_scan(sum, m.w, tot);
    m.start[tid] = st;
    m.base[tid] = o.hist[(int64_t)tid * nb + blockIdx.x] - st;
  }
  __syncthreads();
#pragma unroll
  for (int r = 0; r < kSortItems; ++r)
    if (first + 32 * r < n) {
      const uint32_t d = (key[r] >> shift) & 255u, at = m.start[d] + m.cnt[wid][d] + ((rank[r / 2] >> (16 * (r & 1))) & 0xffffu);
      m.key[at] = key[r];
      m.val[at] = kFirst ? (uint32_t)(first + 32 * r) : val[kFirst ? 0 : r];
    }
  __syncthreads();
  const int total = (int)min((int64_t)kSortBlock, n - base);
  uint32_t *keys_out = o.keys[a.pass & 1], *idx_out = a.pass == a.passes - 1 ? o.order : o.idx[a.pass & 1];
  for (int k = tid; k < total; k += kSortThreads) {
    const uint32_t q = m.key[k], at = m.base[(q >> shift) & 255u] + k;
    keys_out[at] = q;
    idx_out[at] = m.val[k];
  }
}

// the slots to sort, and the counts of a species without removed particles
__global__ void k_sort_begin(long long *n_sort, long long *count, long long *count_sorted, int s0, int ns, long long n) {
  const int s = threadIdx.x;
  if (s >= ns) return;
  const long long v = n >= 0 ? n : count[s0 + s];
  n_sort[s0 + s] = v;
  count[s0 + s] = v;
  count_sorted[s0 + s] = v;
}

// One pass over the sorted keys: the live count (the first removed particle's
// place) and the tile bounds.  Four keys per thread (one 16-byte load; the
// keys buffers are 256-byte aligned), plus the neighbours of the group.
__global__ void __launch_bounds__(256) k_finish(const __grid_constant__ SortArgs a, long long *count,
                                                long long *count_sorted, int s0, int *bounds, int ntiles) {
  const SortOne &o = a.s[blockIdx.y];
  const int species = s0 + blockIdx.y;
  const int64_t n = *o.n, groups = (n + 3) / 4;
  const uint32_t *keys = o.keys[(a.passes + 1) & 1], dead = a.dead;
  int *start = bounds + (int64_t)2 * species * (ntiles + 1), *end = start + ntiles + 1;
  for (int64_t g = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; g < groups; g += (int64_t)gridDim.x * blockDim.x) {
    const int64_t q0 = 4 * g;
    uint32_t k[6];  // k[0] = key before the group, k[5] = key after it
    if (q0 + 3 < n) {
      const uint4 v = *reinterpret_cast<const uint4 *>(keys + q0);
      k[1] = v.x; k[2] = v.y; k[3] = v.z; k[4] = v.w;
    } else {
      for (int e = 0; e < 4; ++e) k[1 + e] = (q0 + e < n) ? keys[q0 + e] : dead;
    }
    k[0] = q0 > 0 ? keys[q0 - 1] : dead;
    k[5] = q0 + 4 < n ? keys[q0 + 4] : dead;
    for (int e = 0; e < 4; ++e) {
      const int64_t q = q0 + e;
      if (q >= n) break;
      const uint32_t c = k[1 + e];
      if (c == dead) {
        if (q == 0 || k[e] != dead) { count[species] = q; count_sorted[species] = q; }
        break;
      }
      if (q == 0 || k[e] != c) start[c] = (int)q;
      if (q == n - 1 || k[2 + e] != c) end[c] = (int)(q + 1);
    }
  }
}

// the payload gather of one species: slots below the (already compacted) count
constexpr int kGatherItems = 4;
template <typename R>
__global__ void __launch_bounds__(256) k_gather_live(Species<R> src, Species<R> dst, const uint32_t *idx,
                                                     const long long *count, int species) {
  // kGatherItems particles at a time: their index loads, then their seven
  // words each, are in flight together
  const int64_t n = count[species], step = (int64_t)gridDim.x * blockDim.x * kGatherItems;
  const R *const in[6] = {src.xo, src.yo, src.ur, src.ut, src.up, src.w};
  R *const out[6] = {dst.xo, dst.yo, dst.ur, dst.ut, dst.up, dst.w};
  for (int64_t q0 = blockIdx.x * (int64_t)blockDim.x * kGatherItems + threadIdx.x; q0 < n; q0 += step) {
    uint32_t k[kGatherItems];
    int c[kGatherItems];
    R v[6][kGatherItems];
#pragma unroll
    for (int i = 0; i < kGatherItems; ++i) {
      const int64_t q = q0 + i * (int64_t)blockDim.x;
      k[i] = q < n ? idx[q] : 0u;
    }
#pragma unroll
    for (int i = 0; i < kGatherItems; ++i) {
      c[i] = src.cell[k[i]];
#pragma unroll
      for (int a = 0; a < 6; ++a) v[a][i] = in[a][k[i]];
    }
#pragma unroll
    for (int i = 0; i < kGatherItems; ++i) {
      const int64_t q = q0 + i * (int64_t)blockDim.x;
      if (q >= n) break;
      dst.cell[q] = c[i];
#pragma unroll
      for (int a = 0; a < 6; ++a) out[a][q] = v[a][i];
    }
  }
}

// Gather in arbitrary order (a load) through records: seven words of a
// particle from seven places are seven 32-byte sectors, so they are first
// packed (read and written in order) into one aligned record of 32 (FP32) or
// 64 bytes, which the gather then reads whole.
template <typename R> struct alignas(16) Record { uint32_t w[sizeof(R) == 4 ? 8 : 16]; };
template <typename R>
__device__ __forceinline__ void put_word(Record<R> &rec, int k, R v) {
  if constexpr (sizeof(R) == 4) {
    rec.w[1 + k] = __float_as_uint(v);
  } else {
    rec.w[2 + 2 * k] = (uint32_t)__double2loint(v);
    rec.w[3 + 2 * k] = (uint32_t)__double2hiint(v);
  }
}
template <typename R>
__device__ __forceinline__ R get_word(const Record<R> &rec, int k) {
  if constexpr (sizeof(R) == 4) return __uint_as_float(rec.w[1 + k]);
  else return __hiloint2double((int)rec.w[3 + 2 * k], (int)rec.w[2 + 2 * k]);
}
template <typename R>
__global__ void __launch_bounds__(256) k_pack(Species<R> src, Record<R> *rec, int64_t n) {
  for (int64_t q = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; q < n; q += (int64_t)gridDim.x * blockDim.x) {
    Record<R> r{};
    r.w[0] = (uint32_t)src.cell[q];
    put_word<R>(r, 0, src.xo[q]); put_word<R>(r, 1, src.yo[q]);
    put_word<R>(r, 2, src.ur[q]); put_word<R>(r, 3, src.ut[q]); put_word<R>(r, 4, src.up[q]);
    put_word<R>(r, 5, src.w[q]);
    uint4 *d = reinterpret_cast<uint4 *>(rec + q);
    const uint4 *s = reinterpret_cast<const uint4 *>(&r);
#pragma unroll
    for (int k = 0; k < (int)(sizeof(r) / 16); ++k) d[k] = s[k];
  }
}
template <typename R>
__global__ void __launch_bounds__(256) k_unpack(const Record<R> *rec, Species<R> dst, const uint32_t *idx,
                                                const long long *count, int species) {
  constexpr int kItems = sizeof(R) == 4 ? 4 : 2;   // records in flight per thread
  const int64_t n = count[species], step = (int64_t)gridDim.x * blockDim.x * kItems;
  for (int64_t q0 = blockIdx.x * (int64_t)blockDim.x * kItems + threadIdx.x; q0 < n; q0 += step) {
    uint32_t k[kItems];
    Record<R> r[kItems];
#pragma unroll
    for (int i = 0; i < kItems; ++i) {
      const int64_t q = q0 + i * (int64_t)blockDim.x;
      k[i] = q < n ? idx[q] : 0u;
    }
#pragma unroll
    for (int i = 0; i < kItems; ++i) {
      const uint4 *s = reinterpret_cast<const uint4 *>(rec + k[i]);
      uint4 *d = reinterpret_cast<uint4 *>(&r[i]);
#pragma unroll
      for (int j = 0; j < (int)(sizeof(Record<R>) / 16); ++j) d[j] = s[j];
    }
#pragma unroll
    for (int i = 0; i < kItems; ++i) {
      const int64_t q = q0 + i * (int64_t)blockDim.x;
      if (q >= n) break;
      dst.cell[q] = (int32_t)r[i].w[0];
      dst.xo[q] = get_word<R>(r[i], 0); dst.yo[q] = get_word<R>(r[i], 1);
      dst.ur[q] = get_word<R>(r[i], 2); dst.ut[q] = get_word<R>(r[i], 3); dst.up[q] = get_word<R>(r[i], 4);
      dst.w[q] = get_word<R>(r[i], 5);
    }
  }
}

// Is a species in the state a sort leaves (no removed or appended particles,
// keys ascending)?  Its tile bounds are taken afresh on the way; *unsettled is
// set if not, and its bounds then mean nothing: every run of a tile's particles
// writes the same two entries.
__global__ void __launch_bounds__(kSortThreads) k_settled(const int32_t *cell, const long long *count,
                                                          const long long *count_sorted, int species,
                                                          const __grid_constant__ SortArgs a, int *bounds, int ntiles,
                                                          int *unsettled) {
  const int64_t n = count[species];
  int *start = bounds + (int64_t)2 * species * (ntiles + 1), *end = start + ntiles + 1;
  bool bad = count_sorted[species] != n;
  auto key = [&](int64_t q) {
    return q >= 0 && q < n ? tile_key(cell[q], a.nt, a.dnt, a.dtr, a.dtt, a.ntt, a.ncells, a.dead) : a.dead;
  };
  const int lane = threadIdx.x & 31;
  for (int64_t base = blockIdx.x * (int64_t)kSortBlock; base < n; base += (int64_t)gridDim.x * kSortBlock) {
    const int64_t first = base + (threadIdx.x >> 5) * (kSortBlock / kSortWarps) + lane;
    uint32_t k[kSortItems + 2];   // this lane's keys; before and after the warp's piece (lanes 31 and 0)
    k[0] = lane == 31 ? key(first - 32) : 0u;
    k[kSortItems + 1] = lane == 0 ? key(first + 32 * kSortItems) : 0u;
#pragma unroll
    for (int r = 0; r < kSortItems; ++r) k[r + 1] = key(first + 32 * r);
#pragma unroll
    for (int r = 1; r <= kSortItems; ++r) {
      const uint32_t up = __shfl_up_sync(0xffffffffu, k[r], 1), down = __shfl_down_sync(0xffffffffu, k[r], 1);
      const uint32_t last = __shfl_sync(0xffffffffu, k[r - 1], 31), next = __shfl_sync(0xffffffffu, k[r + 1], 0);
      const uint32_t before = lane ? up : last, after = lane < 31 ? down : next;
      const int64_t q = first + 32 * (r - 1);
      if (q >= n) continue;
      if (k[r] == a.dead || after < k[r]) { bad = true; continue; }
      if (k[r] != before) start[k[r]] = (int)q;
      if (k[r] != after) end[k[r]] = (int)(q + 1);
    }
  }
  if (__any_sync(0xffffffffu, bad) && lane == 0) *unsettled = 1;
}

// ceil(count/chunk) items per non-empty tile, species after species.  The sum
// is bounded (by the length that the list was given) for the bounds of sorted
// particles only: after a load beside an unsettled species there are none yet,
// the list is left empty, and the sort that follows makes it.
__global__ void __launch_bounds__(1024) k_worklist(const int *bounds, int ntiles, int n_species, int chunk, int4 *items,
                                                   int *n_items, int max_items, unsigned *status, const int *unsettled) {
  if (unsettled && *unsettled) {
    if (threadIdx.x == 0) *n_items = 0;
    return;
  }
  __shared__ uint32_t w[33];
  __shared__ uint32_t carry;
  if (threadIdx.x == 0) carry = 0u;
  __syncthreads();
  for (int species = 0; species < n_species; ++species) {
    const int *start = bounds + (int64_t)2 * species * (ntiles + 1), *end = start + ntiles + 1;
    for (int seg = 0; seg < ntiles; seg += 1024) {
      const int k = seg + threadIdx.x;
      int cnt = 0;
      if (k < ntiles) cnt = end[k] - start[k];
      const uint32_t ni = cnt > 0 ? (uint32_t)((cnt + chunk - 1) / chunk) : 0u;
      int64_t total = 0;   // of the tile, all species
      for (int t = 0; t < n_species && ni; ++t)
        total += bounds[(int64_t)(2 * t + 1) * (ntiles + 1) + k] - bounds[(int64_t)2 * t * (ntiles + 1) + k];
      const int word = species + kItemTotal * (int)min(total, (int64_t)kItemTotalMax);
      uint32_t tot;
      const uint32_t ex = block_excl_scan(ni, w, tot);
      for (uint32_t c = 0; c < ni; ++c) {
        const uint32_t slot = carry + ex + c;
        if (slot < (uint32_t)max_items) {
          const int s0 = start[k] + (int)c * chunk;
          const int len = min(chunk, end[k] - s0);
          items[slot] = make_int4(word, k, s0, len);
        } else {
          atomicOr(status, kStWorklist);
        }
      }
      __syncthreads();
      if (threadIdx.x == 0) carry += tot;
      __syncthreads();
    }
  }
  if (threadIdx.x == 0) *n_items = (int)min(carry, (uint32_t)max_items);
}

static int bits_for(uint32_t v) {
  int b = 0;
  while ((1ull << b) <= v) ++b;
  return b;
}

// the radix passes over species 0 .. ns-1 of a (grids for `cap` slots)
static void radix_passes(SortArgs &a, int ns, int64_t cap, cudaStream_t st) {
  const int nb = (int)std::max<int64_t>(1, (cap + kSortBlock - 1) / kSortBlock);
  const int parts = (int)(((int64_t)nb * 256 + kScanBlock - 1) / kScanBlock);
  a.passes = (bits_for(a.dead) + 7) / 8;
  for (a.pass = 0; a.pass < a.passes; ++a.pass) {
    k_hist<<<dim3(nb, ns), kSortThreads, 0, st>>>(a);
    if (parts > 1) {
      k_scan_sums<<<dim3(parts, ns), 1024, 0, st>>>(a);
      k_scan_parts<<<dim3(1, ns), 1024, 0, st>>>(a);
    }
    k_scan_apply<<<dim3(parts, ns), 1024, 0, st>>>(a, parts);
    if (a.pass == 0) k_scatter<true><<<dim3(nb, ns), kSortThreads, sizeof(ScatterSmem), st>>>(a);
    else k_scatter<false><<<dim3(nb, ns), kSortThreads, sizeof(ScatterSmem), st>>>(a);
  }
}

template <typename R>
static SortArgs sort_args(const Params<R> &p, const SortScratch &ss, int s0, int ns) {
  SortArgs a{};
  for (int k = 0; k < ns; ++k) {
    const int s = s0 + k;
    SortOne &o = a.s[k];
    o.cell = p.sp[s].cell;
    o.order = const_cast<uint32_t *>(p.sidx[s]);
    for (int b = 0; b < 2; ++b) {
      o.keys[b] = ss.keys + (2 * s + b) * ss.stride;
      o.idx[b] = ss.idx + (2 * s + b) * ss.stride;
    }
    o.hist = ss.hist + s * ss.hist_stride;
    o.part = ss.part + s * ss.part_stride;
    o.n = ss.n_sort + s;
  }
  a.ncells = (uint32_t)((int64_t)p.nr * p.nt);
  a.bad = p.status;
  a.bad_bit = kStBadCell;
  a.nt = p.nt; a.ntt = p.ntt;
  a.dnt = make_fastdiv((uint32_t)p.nt); a.dtr = make_fastdiv((uint32_t)p.tile_r); a.dtt = make_fastdiv((uint32_t)p.tile_t);
  a.dead = (uint32_t)ss.ntiles;
  return a;
}

template <typename R>
void launch_sort(const Params<R> &p, const SortScratch &ss, cudaStream_t st) {
  const int ns = p.n_species;
  SortArgs a = sort_args(p, ss, 0, ns);
  k_sort_begin<<<1, 32, 0, st>>>(ss.n_sort, p.count, p.count_sorted, 0, ns, -1);
  cudaMemsetAsync(ss.bounds, 0, sizeof(int) * 2 * ns * (ss.ntiles + 1), st);
  radix_passes(a, ns, ss.cap, st);
  k_finish<<<dim3((unsigned)std::max<int64_t>(1, std::min<int64_t>(1216, (ss.cap + 1023) / 1024)), ns), 256, 0, st>>>(
      a, p.count, p.count_sorted, 0, ss.bounds, ss.ntiles);
}

template <typename R>
void launch_load_sorted(const Params<R> &p, int s, const Species<R> &src, int64_t n, void *records, const SortScratch &ss,
                        int *unsettled, cudaStream_t st) {
  SortArgs a = sort_args(p, ss, s, 1);
  a.s[0].cell = src.cell;
  k_sort_begin<<<1, 32, 0, st>>>(ss.n_sort, p.count, p.count_sorted, s, 1, (long long)n);
  cudaMemsetAsync(ss.bounds, 0, sizeof(int) * 2 * p.n_species * (ss.ntiles + 1), st);
  cudaMemsetAsync(unsettled, 0, sizeof(int), st);
  const unsigned grid = (unsigned)std::max<int64_t>(1, std::min<int64_t>(2432, (n + 255) / 256));
  if (n > 0) {
    if (records) k_pack<R><<<grid, 256, 0, st>>>(src, static_cast<Record<R> *>(records), n);
    radix_passes(a, 1, n, st);
    k_finish<<<dim3((unsigned)std::min<int64_t>(1216, (n + 1023) / 1024), 1), 256, 0, st>>>(
        a, p.count, p.count_sorted, s, ss.bounds, ss.ntiles);
    if (records) k_unpack<R><<<grid, 256, 0, st>>>(static_cast<const Record<R> *>(records), p.sp[s], p.sidx[s], p.count, s);
    else k_gather_live<R><<<grid, 256, 0, st>>>(src, p.sp[s], p.sidx[s], p.count, s);
  }
  for (int t = 0; t < p.n_species; ++t)
    if (t != s) k_settled<<<(unsigned)std::max<int64_t>(1, std::min<int64_t>(1216, sort_blocks(ss.cap))), kSortThreads, 0, st>>>(p.sp[t].cell, p.count, p.count_sorted, t, a, ss.bounds, ss.ntiles, unsettled);
}
template <typename R> size_t load_record_bytes() { return sizeof(Record<R>); }

// Loaded particles of a configuration without sorting: a cell index at or
// past nr * nt is invalid input; the particle is removed (cell = -1) and
// kStBadCell latched.
__global__ void k_check_cells(int32_t *cell, int64_t n, int64_t ncells, unsigned *status) {
  bool bad = false;
  for (int64_t q = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; q < n; q += (int64_t)gridDim.x * blockDim.x)
    if (cell[q] >= ncells) { cell[q] = -1; bad = true; }
  if (bad) atomicOr(status, kStBadCell);
}

void launch_check_cells(int32_t *cell, int64_t n, int64_t ncells, unsigned *status, cudaStream_t st) {
  if (n > 0) k_check_cells<<<(unsigned)std::min<int64_t>((n + 255) / 256, 4096), 256, 0, st>>>(cell, n, ncells, status);
}

template <typename R>
void launch_materialize(const Params<R> &p, int s, cudaStream_t st) {
  k_gather_live<R><<<1216, 256, 0, st>>>(p.src[s], p.sp[s], p.sidx[s], p.count, s);
}

template <typename R>
void launch_worklist(const Params<R> &p, const SortScratch &ss, const WorkList &wl, const int *unsettled, cudaStream_t st) {
  k_worklist<<<1, 1024, 0, st>>>(ss.bounds, ss.ntiles, p.n_species, wl.chunk, wl.items, wl.n_items, wl.max_items, p.status, unsettled);
}

#define HFF_INST(R)                                                                                   \
  template void launch_sort<R>(const Params<R> &, const SortScratch &, cudaStream_t);                  \
  template void launch_load_sorted<R>(const Params<R> &, int, const Species<R> &, int64_t, void *, const SortScratch &, \
                                      int *, cudaStream_t);                                            \
  template size_t load_record_bytes<R>();                                                              \
  template void launch_materialize<R>(const Params<R> &, int, cudaStream_t);                           \
  template void launch_worklist<R>(const Params<R> &, const SortScratch &, const WorkList &, const int *, cudaStream_t);
HFF_INST(float)
HFF_INST(double)
#undef HFF_INST

// ------------------------------------------------- allocation-free variant
// hff_tile_order_noalloc runs the same radix passes with its scratch in a
// fixed device array instead of memory passed in or allocated, for callers
// that may not allocate device memory at all.  The paper has no counterpart.
namespace noalloc {

constexpr int64_t kMaxN = HFF_NOALLOC_MAX_PARTICLES;
constexpr int64_t kMaxBlocks = (kMaxN + kSortBlock - 1) / kSortBlock;
constexpr int64_t kMaxHist = kMaxBlocks * 256;
constexpr int64_t kMaxParts = (kMaxHist + kScanBlock - 1) / kScanBlock;
// keys (2) | idx (2) | histogram | block sums | live count, invalid-cell flag,
// slot count (64 bits)
constexpr int64_t kPartWords = (kMaxParts + 63) & ~int64_t(63);
constexpr int64_t kWords = 4 * kMaxN + kMaxHist + kPartWords + 64;

// One copy per device, alive until the process exits; shared by every call.
static __device__ __align__(256) uint32_t g_scratch[kWords];

constexpr int kMaxDevices = 64;
std::mutex g_mu;
uint32_t *g_addr[kMaxDevices] = {};

// live count and invalid-cell flag: written afresh at the start of every call
__global__ void k_live_init(uint32_t *live, uint32_t n) {
  live[0] = n;
  live[1] = 0u;
  *reinterpret_cast<long long *>(live + 2) = (long long)n;
}

// first slot holding a removed particle (keys are sorted, removed ones last)
__global__ void k_live_count(const uint32_t *keys, int64_t n, uint32_t dead, uint32_t *live) {
  for (int64_t q = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; q < n; q += (int64_t)gridDim.x * blockDim.x)
    if (keys[q] == dead && (q == 0 || keys[q - 1] != dead)) *live = (uint32_t)q;
}

}  // namespace noalloc
}  // namespace hff

thread_local const char *hff_noalloc_err = "";

extern "C" const char *hff_noalloc_last_error(void) { return hff_noalloc_err; }

extern "C" int hff_tile_order_noalloc(const int32_t *cell, int64_t n, int32_t nr, int32_t nt, int32_t tile_r,
                                      int32_t tile_t, uint32_t *order, int64_t *n_live, void *stream) {
  using namespace hff;
  using namespace hff::noalloc;
  // an error left by earlier, unrelated work would otherwise be reported
  // (and cleared) by the check after this call's launches
  (void)cudaGetLastError();
  if (n < 0 || nr < 1 || nt < 1 || tile_r < 1 || tile_t < 1 || !n_live || (n > 0 && (!cell || !order))) {
    hff_noalloc_err = "hff_tile_order_noalloc: invalid argument";
    return HFF_ERR_ARG;
  }
  if (n > kMaxN) {
    hff_noalloc_err = "hff_tile_order_noalloc: n exceeds HFF_NOALLOC_MAX_PARTICLES";
    return HFF_ERR_CAPACITY;
  }
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices) {
    hff_noalloc_err = "hff_tile_order_noalloc: no usable current device";
    return HFF_ERR_CUDA;
  }
  uint32_t *base = nullptr;
  {
    // first call on this device: resolve the device address of the array
    // (host code only sees a stand-in symbol; the device address differs)
    std::lock_guard<std::mutex> lock(g_mu);
    if (!g_addr[dev]) {
      void *ptr = nullptr;
      if (cudaGetSymbolAddress(&ptr, g_scratch) != cudaSuccess || !ptr) {
        hff_noalloc_err = "hff_tile_order_noalloc: cudaGetSymbolAddress failed";
        return HFF_ERR_CUDA;
      }
      g_addr[dev] = static_cast<uint32_t *>(ptr);
    }
    base = g_addr[dev];
  }
  cudaStream_t st = (cudaStream_t)stream;
  const int ntt = (nt + tile_t - 1) / tile_t;
  const int64_t ntiles = (int64_t)((nr + tile_r - 1) / tile_r) * ntt;
  if (ntiles >= 0x7fffffffLL) {
    hff_noalloc_err = "hff_tile_order_noalloc: too many tiles";
    return HFF_ERR_ARG;
  }
  uint32_t *hist = base + 4 * kMaxN, *part = hist + kMaxHist, *live = part + kPartWords;
  const uint32_t dead = (uint32_t)ntiles;
  if (n == 0) {
    *n_live = 0;
    hff_noalloc_err = "";
    return HFF_OK;
  }
  SortArgs a{};
  SortOne &o = a.s[0];
  o.cell = cell;
  o.keys[0] = base; o.keys[1] = base + kMaxN;
  o.idx[0] = base + 2 * kMaxN; o.idx[1] = base + 3 * kMaxN;
  o.order = order;
  o.hist = hist; o.part = part;
  o.n = reinterpret_cast<const long long *>(live + 2);
  a.ncells = (uint32_t)std::min<int64_t>((int64_t)nr * nt, 0x7fffffff);
  a.bad = live + 1;
  a.bad_bit = 1u;
  a.nt = nt; a.ntt = ntt;
  a.dnt = make_fastdiv((uint32_t)nt); a.dtr = make_fastdiv((uint32_t)tile_r); a.dtt = make_fastdiv((uint32_t)tile_t);
  a.dead = dead;
  k_live_init<<<1, 1, 0, st>>>(live, (uint32_t)n);
  radix_passes(a, 1, n, st);
  // the live count and the flag were written at the start of this call
  // (previous contents of the shared array are never read)
  k_live_count<<<(int)((n + 255) / 256), 256, 0, st>>>(o.keys[(a.passes + 1) & 1], n, dead, live);
  uint32_t h_live[2] = {0u, 0u};
  if (cudaMemcpyAsync(h_live, live, 2 * sizeof(uint32_t), cudaMemcpyDeviceToHost, st) != cudaSuccess ||
      cudaStreamSynchronize(st) != cudaSuccess || cudaGetLastError() != cudaSuccess) {
    hff_noalloc_err = "hff_tile_order_noalloc: a CUDA call failed";
    return HFF_ERR_CUDA;
  }
  if (h_live[1]) {
    hff_noalloc_err = "hff_tile_order_noalloc: a cell index is at or past nr * nt (ordered as removed)";
    return HFF_ERR_ARG;
  }
  *n_live = (int64_t)h_live[0];
  hff_noalloc_err = "";
  return HFF_OK;
}
