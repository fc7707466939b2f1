// fields.cu -- grid kernels of the hybrid step: flux function (Eq. 27),
// force-free perpendicular current (Eq. 24, first term), Yee advance in
// Stokes form (Eqs. 18-19) with the blended current (Eq. 28), the E
// renormalisation (Eqs. 25-26), the corotating star and the absorber.
//
// Mapping: theta is the fastest index of every array, so a warp walks 32
// consecutive theta points of one r row (coalesced); blockIdx.y is the row.
// All these kernels are HBM-bound stencils: each reads its inputs once per
// step through L1/L2 (neighbour reuse hits cache) and writes its outputs once.
//
// B is held as the static initial field B_0 plus the perturbation dB, and
// the Yee update advances dB only, with curl B_0 added as a source computed
// once in FP64.  In FP32 the rounding of B then scales with |dB| instead of
// |B|: near the star of a fine grid the rounding of a stored |B| ~ 1, divided
// by a cell of 1e-3 r*, would otherwise enter E every step through the curl.
#include <algorithm>
#include <type_traits>

#include "collect.cuh"
#include "hff_common.cuh"

namespace hff {

constexpr int kRowThreads = 128;

// ------------------------------------------------------------ Psi (Eq. 27)
// Psi(i, 0) = 0, Psi(i, j+1) = Psi(i, j) + B_r(i, j+1/2) r_i^2 dcp_j, an
// inclusive prefix along theta.  One block per r row: the row is staged
// through shared memory (coalesced in and out), each thread sums a
// contiguous chunk serially, one block-wide scan of the chunk totals gives
// the offsets, and the prefix is rounded to the working precision.  The
// staged row is padded by one word every 32 (element j at j + j/32), so that
// the threads of a warp, each walking its own contiguous chunk, hit distinct
// banks.
//
// Accumulation: FP64 for FP64 instances.  For FP32 instances every term is
// formed exactly as a float pair (B_r = B_0 + dB by two-sum, times the FP64
// face factor held as a float pair, the product by fma) and summed in a
// compensated pair (the rounding error of every addition carried in a second
// float); the prefix leaves the kernel as a normalised pair, about 48
// significant bits, at FP32 instead of FP64 throughput.
constexpr int kPsiThreads = 256;
__host__ __device__ __forceinline__ int psi_pad(int j) { return j + (j >> 5); }

struct Acc64 {
  using Term = double;
  double v;
  __device__ __forceinline__ void add(double x) { v += x; }
  __device__ __forceinline__ void add(const Acc64 &o) { v += o.v; }
  __device__ __forceinline__ Acc64 neg() const { return {-v}; }
  __device__ __forceinline__ Acc64 shfl_up(int o) const { return {__shfl_up_sync(0xffffffffu, v, o)}; }
  __device__ __forceinline__ double times(double r2) const { return r2 * v; }
  static __device__ __forceinline__ double term(const Params<double> &p, double b0, double db, int j) {
    return (b0 + db) * p.t.dcp[j];
  }
  static __device__ __forceinline__ double zero() { return 0.0; }
};
struct Acc32x2 {
  using Term = float2;
  float hi, lo;
  __device__ __forceinline__ void add(float x) {
    const float2 s = two_sum(hi, x);
    hi = s.x;
    lo += s.y;
  }
  __device__ __forceinline__ void add(float2 t) {
    add(t.x);
    lo += t.y;
  }
  __device__ __forceinline__ void add(const Acc32x2 &o) {
    add(o.hi);
    lo += o.lo;
  }
  __device__ __forceinline__ Acc32x2 neg() const { return {-hi, -lo}; }
  __device__ __forceinline__ Acc32x2 shfl_up(int o) const {
    return {__shfl_up_sync(0xffffffffu, hi, o), __shfl_up_sync(0xffffffffu, lo, o)};
  }
  // (hi + lo) (r2h + r2l) as a normalised pair (r2 split on the host side of
  // the loop)
  __device__ __forceinline__ float2 times2(float r2h, float r2l) const {
    const float ph = hi * r2h;
    const float pe = fmaf(hi, r2h, -ph) + fmaf(hi, r2l, lo * r2h);
    const float h = ph + pe;
    return make_float2(h, pe - (h - ph));
  }
  // (b0 + db) * dcp_j: the sum exactly by two-sum, the product by fma
  static __device__ __forceinline__ float2 term(const Params<float> &p, float b0, float db, int j) {
    const float2 b = two_sum(b0, db), d = p.t.dcp2[j];
    const float ph = b.x * d.x;
    return make_float2(ph, fmaf(b.x, d.x, -ph) + fmaf(b.x, d.y, b.y * d.x));
  }
  static __device__ __forceinline__ float2 zero() { return make_float2(0.f, 0.f); }
};
template <typename R> struct PsiAccOf { using T = Acc64; };
template <> struct PsiAccOf<float> { using T = Acc32x2; };

template <typename A>
__device__ __forceinline__ typename PsiOf<double>::T psi_out(const A &a, double r2) { return a.times(r2); }
__device__ __forceinline__ float2 psi_out(const Acc32x2 &a, double r2) {
  const float r2h = (float)r2, r2l = (float)(r2 - (double)r2h);
  return a.times2(r2h, r2l);
}

template <typename R>
__global__ void __launch_bounds__(kPsiThreads) k_psi(Params<R> p) {
  using A = typename PsiAccOf<R>::T;
  using T = typename A::Term;
  using P = typename PsiOf<R>::T;
  extern __shared__ __align__(16) unsigned char psmem[];
  T *row = reinterpret_cast<T *>(psmem);  // nt + 1 terms
  __shared__ A warp_tot[kPsiThreads / 32];
  const int i = blockIdx.x, nt = p.nt, tid = threadIdx.x;
  const R *br = p.f.br + (int64_t)i * nt;
  const R *br0 = p.f.br0 + (int64_t)i * nt;
  for (int j = tid; j < nt; j += kPsiThreads) row[psi_pad(j)] = A::term(p, br0[j], br[j], j);
  __syncthreads();
  const int chunk = (nt + kPsiThreads - 1) / kPsiThreads;
  const int j0 = min(tid * chunk, nt), j1 = min(j0 + chunk, nt);
  A acc{};
  for (int j = j0; j < j1; ++j) acc.add(row[psi_pad(j)]);
  // exclusive scan of the chunk totals over the block
  const int lane = tid & 31, wid = tid >> 5;
  A x = acc;
  for (int o = 1; o < 32; o <<= 1) {
    const A y = x.shfl_up(o);
    if (lane >= o) x.add(y);
  }
  if (lane == 31) warp_tot[wid] = x;
  __syncthreads();
  A run = x;
  run.add(acc.neg());
  for (int w = 0; w < wid; ++w) run.add(warp_tot[w]);
  const double r2 = p.t.r2n[i];
  // rewrite the chunk in place with the prefix (inclusive, shifted by one;
  // a term and a Psi value have the same type), then store the row coalesced
  static_assert(sizeof(T) == sizeof(P), "term and Psi share the staged row");
  for (int j = j0; j < j1; ++j) {
    run.add(row[psi_pad(j)]);
    row[psi_pad(j)] = psi_out(run, r2);  // becomes Psi(i, j+1)
  }
  __syncthreads();
  P *psi = p.f.psi + (int64_t)i * (nt + 1);
  for (int j = tid; j <= nt; j += kPsiThreads) psi[j] = (j == 0) ? P{} : row[psi_pad(j - 1)];
}

// ----------------------------------------------------------- collocation
// Arithmetic means of the staggered neighbours at node (i, j) (Sect. 3);
// interior rows only; transverse components vanish on the axis.
template <typename R>
__device__ __forceinline__ void collocate(const Params<R> &p, int i, int j, R e[3], R b[3]) {
  const int nt = p.nt, n1 = nt + 1;
  const bool axis = (j == 0 || j == nt);
  const Fields<R> &f = p.f;
  e[0] = R(0.5) * (f.er[ix(i - 1, j, n1)] + f.er[ix(i, j, n1)]);
  e[1] = axis ? R(0) : R(0.5) * (f.et[ix(i, j - 1, nt)] + f.et[ix(i, j, nt)]);
  e[2] = axis ? R(0) : f.ep[ix(i, j, n1)];
  auto br = [&](int a, int c) { const int64_t k = ix(a, c, nt); return f.br0[k] + f.br[k]; };
  auto bt = [&](int a, int c) { const int64_t k = ix(a, c, n1); return f.bt0[k] + f.bt[k]; };
  auto bp = [&](int a, int c) { const int64_t k = ix(a, c, nt); return f.bp0[k] + f.bp[k]; };
  b[0] = (j == 0) ? br(i, 0) : (j == nt) ? br(i, nt - 1) : R(0.5) * (br(i, j - 1) + br(i, j));
  b[1] = axis ? R(0) : R(0.5) * (bt(i - 1, j) + bt(i, j));
  b[2] = axis ? R(0) : R(0.25) * (bp(i - 1, j - 1) + bp(i - 1, j) + bp(i, j - 1) + bp(i, j));
}

template <typename R> __device__ __forceinline__ R b2min();
template <> __device__ __forceinline__ float b2min<float>() { return 1e-30f; }
template <> __device__ __forceinline__ double b2min<double>() { return 1e-30; }

// ----------------------------------------------------------- node pass A
// rho = div E / 4 pi over the node dual cell and J_perp = c rho E x B / B^2
// (first term of Eq. 24) from E^n, B^n; plus the per-cell pure force-free
// flag f(Psi_cell) >= 1 used to remove particles (Eq. 29: no particles).
template <typename R>
__global__ void __launch_bounds__(kRowThreads) k_node_a(Params<R> p) {
  const int i = blockIdx.y, j = blockIdx.x * blockDim.x + threadIdx.x;
  const int nr = p.nr, nt = p.nt, n1 = nt + 1;
  if (j > nt) return;
  const Fields<R> &f = p.f;
  if (i < nr && j < nt) f.ffcell[ix(i, j, nt)] = ff_cell(p, i, j) ? 1 : 0;
  R jx = 0, jy = 0, jz = 0;
  if (i >= 1 && i < nr) {
    R e[3], b[3];
    collocate(p, i, j, e, b);
    R div = p.t.rho_a[i] * (p.t.rh2[i] * f.er[ix(i, j, n1)] - p.t.rh2[i - 1] * f.er[ix(i - 1, j, n1)]);
    R dt = 0;
    if (j < nt) dt += p.t.sh[j] * f.et[ix(i, j, nt)];
    if (j > 0) dt -= p.t.sh[j - 1] * f.et[ix(i, j - 1, nt)];
    const R rho = div + p.t.rho_b[i] * dt * p.t.inv_dch[j];
    const R b2 = b[0] * b[0] + b[1] * b[1] + b[2] * b[2];
    if (b2 > b2min<R>()) {
      const R s = rho / b2;
      jx = s * (e[1] * b[2] - e[2] * b[1]);
      jy = s * (e[2] * b[0] - e[0] * b[2]);
      jz = s * (e[0] * b[1] - e[1] * b[0]);
    }
  }
  f.jpr[ix(i, j, n1)] = jx;
  f.jpt[ix(i, j, n1)] = jy;
  f.jpp[ix(i, j, n1)] = jz;
}

// ---------------------------------------------------------------- Faraday
// Eq. 18 over the exact primary faces, dB -= h dt curl E; optionally the
// absorber B -= sigma (B - B_0), i.e. dB -= sigma dB, afterwards.  Blocks
// past the rows collect the push's current, if the launch has any.
static_assert(kRowThreads == kCollectThreads, "k_faraday's collecting blocks");
template <typename R>
__global__ void __launch_bounds__(kRowThreads) k_faraday(const __grid_constant__ Params<R> p, R hdt, bool absorb) {
  const int nr = p.nr, nt = p.nt, n1 = nt + 1;
  if (blockIdx.y > nr) {
    collect_block(p, blockIdx.x, blockIdx.y - (nr + 1));
    return;
  }
  const int i = blockIdx.y, j = blockIdx.x * blockDim.x + threadIdx.x;
  if (j > nt) return;
  const Fields<R> &f = p.f;
  const Tables<R> &t = p.t;
  if (j < nt) {  // B_r(i, j+1/2), i = 0..nr
    const R c = t.inv_rn[i] * (t.sn[j + 1] * f.ep[ix(i, j + 1, n1)] - t.sn[j] * f.ep[ix(i, j, n1)]) *
                t.inv_dcp[j];
    R v = f.br[ix(i, j, nt)] - hdt * c;
    if (absorb) { const R sg = t.sig_n[i]; if (sg > R(0)) v -= sg * v; }
    f.br[ix(i, j, nt)] = v;
  }
  if (i < nr) {
    // B_th(i+1/2, j): zero on the axis
    R v = R(0);
    if (j > 0 && j < nt) {
      v = f.bt[ix(i, j, n1)] +
          hdt * t.c_b2[i] * (t.rn[i + 1] * f.ep[ix(i + 1, j, n1)] - t.rn[i] * f.ep[ix(i, j, n1)]);
      if (absorb) { const R sg = t.sig_h[i]; if (sg > R(0)) v -= sg * v; }
    }
    f.bt[ix(i, j, n1)] = v;
    if (j < nt) {  // B_ph(i+1/2, j+1/2)
      const R c = t.c_b2[i] * (t.rn[i + 1] * f.et[ix(i + 1, j, nt)] - t.rn[i] * f.et[ix(i, j, nt)]) -
                  t.c_bp2[i] * (f.er[ix(i, j + 1, n1)] - f.er[ix(i, j, n1)]);
      R w = f.bp[ix(i, j, nt)] - hdt * c;
      if (absorb) { const R sg = t.sig_h[i]; if (sg > R(0)) w -= sg * w; }
      f.bp[ix(i, j, nt)] = w;
    }
  }
}

// mean of a node quantity over the two nodes of a radial edge (interior
// nodes only: rows 0 and nr carry the boundary conditions)
template <typename R>
__device__ __forceinline__ R edge_r_mean(const R *a, int i, int j, int nr, int n1) {
  const bool lo = i >= 1, hi = i + 1 <= nr - 1;
  R v = R(0);
  if (lo) v += a[ix(i, j, n1)];
  if (hi) v += a[ix(i + 1, j, n1)];
  return (lo && hi) ? R(0.5) * v : v;
}

// ---------------------------------------------------------------- Ampere
// Eq. 19 over the exact dual faces, curl B = curl dB + curl B_0, with
// J = (1 - f) J_PIC + f J_FFE (Eq. 28);
// then the corotating star (tangential E fixed, Sect. 4), the conducting
// outer wall, E_ph = 0 on the axis, the absorber on E, and J_PIC cleared.
template <typename R>
__global__ void __launch_bounds__(kRowThreads) k_ampere(Params<R> p) {
  const int i = blockIdx.y, j = blockIdx.x * blockDim.x + threadIdx.x;
  const int nr = p.nr, nt = p.nt, n1 = nt + 1;
  if (j > nt) return;
  const Fields<R> &f = p.f;
  const Tables<R> &t = p.t;
  const R dt = p.dt, fp = R(4.0 * kPi) * p.dt;
  if (i < nr) {  // E_r(i+1/2, j)
    R c = R(0);
    if (j < nt) c += t.sh[j] * f.bp[ix(i, j, nt)];
    if (j > 0) c -= t.sh[j - 1] * f.bp[ix(i, j - 1, nt)];
    c *= t.inv_rh[i] * t.inv_dch[j];
    const R fb = blend_redge(p, i, j);
    const int64_t k = ix(i, j, n1);
    const R jt = (R(1) - fb) * f.jr[k] + fb * edge_r_mean(f.jpr, i, j, nr, n1);
    f.er[k] = (f.er[k] + dt * (c + f.sr[k]) - fp * jt) * (R(1) - t.sig_h[i]);
    f.jr[k] = R(0);
  }
  if (j < nt) {  // E_th(i, j+1/2)
    const int64_t k = ix(i, j, nt);
    R v;
    if (i == 0) {
      v = -p.omega * t.rn[0] * t.sh[j] * (f.br0[ix(0, j, nt)] + f.br[ix(0, j, nt)]);
    } else if (i == nr) {
      v = R(0);
    } else {
      const R c = -t.c_e2[i] * (t.rh[i] * f.bp[ix(i, j, nt)] - t.rh[i - 1] * f.bp[ix(i - 1, j, nt)]);
      const R fb = blend_tedge(p, i, j);
      const R jt = (R(1) - fb) * f.jt[k] + fb * R(0.5) * (f.jpt[ix(i, j, n1)] + f.jpt[ix(i, j + 1, n1)]);
      v = (f.et[k] + dt * (c + f.st[k]) - fp * jt) * (R(1) - t.sig_n[i]);
    }
    f.et[k] = v;
    f.jt[k] = R(0);
  }
  {  // E_ph(i, j)
    const int64_t k = ix(i, j, n1);
    R v = R(0);
    if (i >= 1 && i < nr && j >= 1 && j < nt) {
      const R c = t.c_e2[i] * (t.rh[i] * f.bt[ix(i, j, n1)] - t.rh[i - 1] * f.bt[ix(i - 1, j, n1)]) -
                  t.c_ep2[i] * (f.br[ix(i, j, nt)] - f.br[ix(i, j - 1, nt)]);
      const R fb = blend_node(p, i, j);
      const R jt = (R(1) - fb) * f.jp[k] + fb * f.jpp[k];
      v = (f.ep[k] + dt * (c + f.sp[k]) - fp * jt) * (R(1) - t.sig_n[i]);
    }
    f.ep[k] = v;
    f.jp[k] = R(0);
  }
}

// ----------------------------------------------------------- node pass B
// Renormalisation at interior nodes from E^{n+1} and B^{n+1/2}:
// E' = E - (E.B) B/B^2 (Eq. 25), E'' = sqrt(B^2/E'^2) E' if E'^2 > B^2 (Eq. 26).
// Stores Delta E = E'' - E, or E'' itself when the corrected field returns to
// the edges (ff_interp_e = 1; 0 and 2 return the corrections, see
// k_correct).  With the optional fourth-difference filter it also
// stores sigma/16 D4 E_r (along r) at the E_r edge (i+1/2, j) and sigma/16
// D4 E_th (along theta) at the E_th edge (i, j+1/2), from the same
// uncorrected E, in the J_PIC arrays: those are zero between Ampere's law and
// the next deposit, and the correction reads and clears them.
template <typename R>
__global__ void __launch_bounds__(kRowThreads) k_node_b(Params<R> p) {
  const int i = blockIdx.y, j = blockIdx.x * blockDim.x + threadIdx.x;
  const int nr = p.nr, nt = p.nt, n1 = nt + 1;
  if (j > nt) return;
  if (p.ff_sigma16 != R(0)) {
    const Fields<R> &f = p.f;
    if (i >= 2 && i <= nr - 3) {
      const R d4 = f.er[ix(i - 2, j, n1)] - R(4) * f.er[ix(i - 1, j, n1)] + R(6) * f.er[ix(i, j, n1)] -
                   R(4) * f.er[ix(i + 1, j, n1)] + f.er[ix(i + 2, j, n1)];
      f.jr[ix(i, j, n1)] = p.ff_sigma16 * d4;
    }
    if (i >= 1 && i <= nr - 1 && j >= 2 && j <= nt - 3) {
      const R d4 = f.et[ix(i, j - 2, nt)] - R(4) * f.et[ix(i, j - 1, nt)] + R(6) * f.et[ix(i, j, nt)] -
                   R(4) * f.et[ix(i, j + 1, nt)] + f.et[ix(i, j + 2, nt)];
      f.jt[ix(i, j, nt)] = p.ff_sigma16 * d4;
    }
  }
  R d0 = 0, d1 = 0, d2 = 0;
  bool clamped = false;
  if (i >= 1 && i < nr) {
    R e[3], b[3];
    collocate(p, i, j, e, b);
    // the stellar-row return needs row 1's collocated E_r before any edge
    // moves: kept in the (zero) J_PIC slot of the radial edge (0, j)
    if (i == 1 && p.ff_interp_e == 2) p.f.jr[ix(0, j, n1)] = e[0];
    const R b2 = b[0] * b[0] + b[1] * b[1] + b[2] * b[2];
    if (b2 > b2min<R>()) {
      const R s = (e[0] * b[0] + e[1] * b[1] + e[2] * b[2]) / b2;
      const R x = e[0] - s * b[0], y = e[1] - s * b[1], z = e[2] - s * b[2];
      const R e2 = x * x + y * y + z * z;
      const R sc = (e2 > b2) ? sqrt(b2 / e2) : R(1);
      d0 = sc * x - e[0];
      d1 = sc * y - e[1];
      d2 = sc * z - e[2];
      clamped = e2 > b2;
    }
    if (p.ff_interp_e == 1) { d0 += e[0]; d1 += e[1]; d2 += e[2]; }
  }
  // running count of Eq. 26 activations (failure detection: a force-free
  // region that keeps needing the clamp is going unstable)
  const unsigned act = __activemask(), m = __ballot_sync(act, clamped);
  if (m && (threadIdx.x & 31) == (unsigned)(__ffs(act) - 1)) atomicAdd(p.clamps, (unsigned long long)__popc(m));
  p.f.der[ix(i, j, n1)] = d0;
  p.f.det[ix(i, j, n1)] = d1;
  p.f.dep[ix(i, j, n1)] = d2;
}

// Delta E interpolated back to the staggered mesh by arithmetic means and
// applied with the blend weight f (Sect. 3, Eqs. 29-31); or, with
// ff_interp_e = 1, the corrected node field itself: E <- E + f (<E''> - E);
// with ff_interp_e = 2, Delta E everywhere except the radial edges at the
// star, which take E''(1) (their only interior node).
// The optional filter term (node pass B, in the J_PIC arrays) is subtracted
// with the same weight and its slot cleared for the next deposit.
template <typename R>
__global__ void __launch_bounds__(kRowThreads) k_correct(Params<R> p) {
  const int i = blockIdx.y, j = blockIdx.x * blockDim.x + threadIdx.x;
  const int nr = p.nr, nt = p.nt, n1 = nt + 1;
  if (j > nt) return;
  const Fields<R> &f = p.f;
  const bool lit = p.ff_interp_e == 1;
  const bool filt = p.ff_sigma16 != R(0);
  if (i < nr) {
    const int64_t k = ix(i, j, n1);
    const R fb = blend_redge(p, i, j);
    // ff_interp_e = 2: the radial edge at the star (one interior node, row 1)
    // takes the corrected node field E''(1) = Delta E(1) + collocated E(1)
    const bool star = p.ff_interp_e == 2 && i == 0 && nr > 1;
    R g = R(0), e1 = R(0);
    if (star) { e1 = f.jr[k]; f.jr[k] = R(0); }
    else if (filt) { g = f.jr[k]; f.jr[k] = R(0); }
    if (fb != R(0)) {
      const R m = edge_r_mean(f.der, i, j, nr, n1) - g + e1;
      f.er[k] += fb * ((lit || star) ? m - f.er[k] : m);
    }
  }
  if (i >= 1 && i < nr) {
    if (j < nt) {
      const int64_t k = ix(i, j, nt);
      const R fb = blend_tedge(p, i, j);
      R g = R(0);
      if (filt) { g = f.jt[k]; f.jt[k] = R(0); }
      if (fb != R(0)) {
        const R m = R(0.5) * (f.det[ix(i, j, n1)] + f.det[ix(i, j + 1, n1)]) - g;
        f.et[k] += fb * (lit ? m - f.et[k] : m);
      }
    }
    if (j >= 1 && j < nt) {
      const R fb = blend_node(p, i, j);
      if (fb != R(0)) {
        const int64_t k = ix(i, j, n1);
        const R m = f.dep[k];
        f.ep[k] += fb * (lit ? m - f.ep[k] : m);
      }
    }
  }
}

// ------------------------------------------------------- fused field update
// The field update between the push and the injection -- J_perp at the
// nodes from E^n, B^n (first term of Eq. 24), Faraday's first half step
// (Eq. 18), Ampere's law with the blended current (Eqs. 19, 28) and the
// boundaries, the renormalisation at the nodes (Eqs. 25-26), the return to
// the edges with the blend weights, and Faraday's second half step with the
// absorber -- as one pass.  A warp owns a strip of theta columns, one per
// lane, with a halo recomputed on each side, and a segment of rows (with
// kFuseWarm rows of warm-up below it), and walks the rows upward.  Everything
// a column has in flight sits in registers, and what the stencils need of the
// columns beside it comes by shuffles (16 a row), so warps neither share
// memory nor wait for each other at every row.  Row step k does
//   F1  B^{n+1/2} at node row k (B_r) and half row k-1 (B_th, B_ph), and
//       J_perp at node row k;
//   A   E^{n+1} at half row k-1 (E_r) and node row k-1 (E_th, E_ph), with the
//       blend weights f kept for C;
//   N   Delta E (or E'') at node row k-2;
//   C   the corrected E at half row k-3 and node row k-3;
//   F2  dB^{n+1} at node row k-3 (B_r) and half row k-4 (B_th, B_ph);
// after issuing the copies of row k+2.
// E^n and dB^n are read once and every output written once; the arithmetic is
// that of k_node_a, k_faraday, k_ampere, k_node_b and k_correct, location by
// location.  F2 needs the corrected E at columns c, c+1; C Delta E at c, c+1
// (and with the theta filter the uncorrected E at c-2 .. c+2); N and A one
// column to the left, F1 and J_perp one more on either side: two columns of
// halo on each side, three with the filter, and likewise three or four rows
// of warm-up.
//
// Bound by issue and dependent-instruction latency (640 instructions per warp
// and row at 4 warps per scheduler, 60% of the issue slots; DRAM at 45%): FP32
// 0.16 ms at 2048^2 and 0.57 at 4096^2 (0.19 and 0.68 where many nodes are
// mixed or clamped), FP64 1.78 ms at 2048^2 (FP64 pipe).
// With the rows in shared-memory rings of a 128-thread block, four barriers a
// row and 1,050 instructions, it took 0.24, 0.81 (0.25, 0.85) and 1.96 ms.  10 warps a
// block at 96 registers: the same at 2048^2, 0.64 ms at 4096^2; blocks of 4 or
// 5 warps: 0.18 - 0.19 and 0.72 - 0.76 ms, for their snapshot columns.
//
// The update is in place.  Within a block, whose warps own neighbouring
// strips, a barrier every four rows keeps them close enough that the neighbours'
// copies of a row r are complete (at step r) before its owner overwrites it
// (from step r+3).  A block's outer halo columns and its warm-up / trailing rows belong
// to other blocks, which overwrite them during the same launch; those are read
// from a snapshot of them taken just before (k_fuse_prepare).  J_PIC is only
// read, and the caller clears it after the launch.
constexpr int kFuseHalo = 3;          // snapshot columns on each side of a block boundary
constexpr int kFuseWarm = 4;          // rows recomputed below a segment
constexpr int kFuseTrail = 4;         // rows above a segment the pipeline reads (up to i_e + 3)
constexpr int kFuseMaxRows = 384;     // rows of a segment
constexpr int kFuseArrays = 6;        // E_r E_th E_ph dB_r dB_th dB_ph
// FP32: 8 warps a block, two blocks per SM at 128 registers; FP64 4 warps
__host__ __device__ constexpr int fuse_warps(size_t real) { return real == 4 ? 8 : 4; }
__host__ __device__ constexpr int fuse_halo(bool filt) { return filt ? 3 : 2; }
// theta columns a block owns
__host__ __device__ constexpr int fuse_cols(size_t real, bool filt) {
  return fuse_warps(real) * (32 - 2 * fuse_halo(filt));
}
// radial tables of a row, staged in shared memory for the whole segment
enum FuseTab { TB_RN, TB_INV_RN, TB_C_E2, TB_C_EP2, TB_SIG_N, TB_RHO_A, TB_RHO_B, TB_RH, TB_INV_RH, TB_C_B2,
               TB_C_BP2, TB_SIG_H, TB_RH2, TB_COUNT };
constexpr int kTabN = 16;
static_assert(TB_COUNT <= kTabN, "table row");
// rows of the table of a segment: from five below it (k - 4 of the first
// step) to its last step
__host__ __device__ constexpr int fuse_tab_rows(int seg_rows) { return seg_rows + kFuseWarm + kFuseTrail + 8; }

// Geometry of a launch: strips of `cols` owned columns, segments of seg_rows
// owned rows.  Snapshot of E^n and dB^n (six arrays, every array addressed as
// (nr+1) x (nt+1)): for every strip boundary b = 1 .. strips-1 the 2 kFuseHalo
// columns around column b cols over all rows, and for every segment boundary
// b = 1 .. segs-1 the rows from b seg_rows - kFuseWarm to b seg_rows +
// kFuseTrail - 1 over all columns.
struct FuseGeom {
  int strips, segs, seg_rows;
};
__host__ __device__ inline FuseGeom fuse_geom(int nr, int nt, int seg_rows, int cols) {
  FuseGeom g;
  g.strips = (nt + 1 + cols - 1) / cols;
  g.seg_rows = seg_rows;
  g.segs = (nr + 1 + seg_rows - 1) / seg_rows;
  return g;
}
__host__ __device__ inline int64_t fuse_snap_cols(int nr, int strips) {
  return (int64_t)(strips > 1 ? strips - 1 : 0) * kFuseArrays * (nr + 1) * (2 * kFuseHalo);
}
__host__ __device__ inline int64_t fuse_snap_rows(int nt, int segs) {
  return (int64_t)(segs > 1 ? segs - 1 : 0) * kFuseArrays * (kFuseWarm + kFuseTrail) * (nt + 1);
}

template <typename R>
__device__ __forceinline__ const R *fuse_array(const Params<R> &p, int a, int &ld, int &rows, int &cols) {
  const int nr = p.nr, nt = p.nt;
  switch (a) {
    case 0: ld = nt + 1; rows = nr; cols = nt + 1; return p.f.er;
    case 1: ld = nt; rows = nr + 1; cols = nt; return p.f.et;
    case 2: ld = nt + 1; rows = nr + 1; cols = nt + 1; return p.f.ep;
    case 3: ld = nt; rows = nr + 1; cols = nt; return p.f.br;
    case 4: ld = nt + 1; rows = nr; cols = nt + 1; return p.f.bt;
    default: ld = nt; rows = nr; cols = nt; return p.f.bp;
  }
}

// The snapshot in one launch: the first `nc` blocks copy halo columns (those
// of one boundary over kSnapRows rows each), the next `nw` blocks copy warm-up
// / trailing rows (kSnapThreads columns of one row of one boundary each), and
// the rest collect the push's current.  A thread copies its element of all six
// arrays, loads first: bound by latency, 8.9 us at 2048^2 without a collection
// (18.4 with an array per thread).
constexpr int kSnapThreads = kCollectThreads;
constexpr int kSnapRows = kSnapThreads / (2 * kFuseHalo);
template <typename R>
__global__ void __launch_bounds__(kSnapThreads) k_fuse_prepare(const __grid_constant__ Params<R> p, R *snap_c,
                                                               R *snap_r, int seg_rows, int own_cols, int nc, int nw) {
  int blk = blockIdx.x;
  int ld, rows, cols;
  if (blk < nc) {
    const int per = (p.nr + kSnapRows) / kSnapRows, ba = blk / per;
    const int rr = threadIdx.x / (2 * kFuseHalo), cc = threadIdx.x - rr * (2 * kFuseHalo);
    const int row = (blk - ba * per) * kSnapRows + rr;
    if (row > p.nr || rr >= kSnapRows) return;
    const int col = (ba + 1) * own_cols - kFuseHalo + cc;
    R v[kFuseArrays];
#pragma unroll
    for (int a = 0; a < kFuseArrays; ++a) {
      const R *src = fuse_array(p, a, ld, rows, cols);
      v[a] = (row < rows && col >= 0 && col < cols) ? src[(int64_t)row * ld + col] : R(0);
    }
#pragma unroll
    for (int a = 0; a < kFuseArrays; ++a)
      snap_c[((int64_t)(ba * kFuseArrays + a) * (p.nr + 1) + row) * (2 * kFuseHalo) + cc] = v[a];
    return;
  }
  blk -= nc;
  if (blk < nw) {
    const int per = p.nt / kSnapThreads + 1, w = blk / per;
    const int col = (blk - w * per) * kSnapThreads + threadIdx.x;
    if (col > p.nt) return;
    const int rr = w % (kFuseWarm + kFuseTrail), ba = w / (kFuseWarm + kFuseTrail);
    const int row = (ba + 1) * seg_rows - kFuseWarm + rr;
    R v[kFuseArrays];
#pragma unroll
    for (int a = 0; a < kFuseArrays; ++a) {
      const R *src = fuse_array(p, a, ld, rows, cols);
      v[a] = (row >= 0 && row < rows && col < cols) ? src[(int64_t)row * ld + col] : R(0);
    }
#pragma unroll
    for (int a = 0; a < kFuseArrays; ++a)
      snap_r[((int64_t)(ba * kFuseArrays + a) * (kFuseWarm + kFuseTrail) + rr) * (p.nt + 1) + col] = v[a];
    return;
  }
  blk -= nw;
  const int cx = collect_blocks_x(p);
  collect_block(p, blk % cx, blk / cx);
}

// a value of the column to the right / left
template <typename T> __device__ __forceinline__ T right(T v) { return __shfl_down_sync(0xffffffffu, v, 1); }
template <typename T> __device__ __forceinline__ T left(T v) { return __shfl_up_sync(0xffffffffu, v, 1); }
__device__ __forceinline__ float2 right(float2 v) { return make_float2(right(v.x), right(v.y)); }

// What a row step reads, staged in shared memory by its own lane: E^n, dB^n,
// B_0 of the row (half rows: the half row above the node row), J_PIC and
// curl B_0 at the E locations of the row below, Psi of the row.
enum FuseInput { IN_ER, IN_ET, IN_EP, IN_BR, IN_BT, IN_BP, IN_B0R, IN_B0T, IN_B0P, IN_JR, IN_SR, IN_JT, IN_ST, IN_JP,
               IN_SP, IN_COUNT };
constexpr int kFuseStages = 4;        // rows staged: the two in use and two in flight
template <typename R> __host__ __device__ constexpr size_t fuse_stage_bytes() {
  return 32 * (IN_COUNT * sizeof(R) + 8);
}

// whether a step's rows (a warp's columns) are known to be interior
template <bool ROWS, bool COLS>
struct FuseTag {
  static constexpr bool rows = ROWS, cols = COLS;
};

template <typename R, bool FILT>
__global__ void __launch_bounds__(32 * fuse_warps(sizeof(R)), sizeof(R) == 4 ? 2 : 1)
    k_field_fused(const __grid_constant__ Params<R> p, R hdt, FuseGeom fg, const R *snap_c, const R *snap_r) {
  using P = typename PsiOf<R>::T;
  constexpr int H = fuse_halo(FILT), OWN = 32 - 2 * H, COLS = fuse_warps(sizeof(R)) * OWN, W = kFuseWarm;
  extern __shared__ __align__(16) unsigned char fsmem[];
  R *tab = reinterpret_cast<R *>(fsmem);
  const int nr = p.nr, nt = p.nt, n1 = nt + 1, seg_rows = fg.seg_rows;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, sx = blockIdx.x, sy = blockIdx.y;
  const int j = sx * COLS + warp * OWN - H + lane;                     // global column of this lane
  const bool jn_ = j >= 0 && j <= nt, jh_ = j >= 0 && j < nt;         // node / half column exists
  const bool own = lane >= H && lane < 32 - H && jn_;                 // column written by this lane
  const unsigned ju = jn_ ? j : 0;
  const bool mine = j >= sx * COLS && j < (sx + 1) * COLS;            // column of this block
  const int j0 = j - lane;                                            // first column of this warp
  const bool cin = j0 >= 2 && j0 + 31 <= nt - 3;                      // all columns away from the axis
  const bool live = __all_sync(0xffffffffu, mine);                    // all columns of this block
  const int i_s = sy * seg_rows;                                      // first output row
  if (i_s > nr) return;
  const int i_e = min(i_s + seg_rows, nr + 1);                        // one past the last output node row
  const int k0 = max(0, i_s - W), kl = min(nr, i_e) + 3;              // row steps
  const Fields<R> &f = p.f;
  const Tables<R> &t = p.t;
  const int t0 = k0 - 4;                                              // first row of the staged table
  {
    const R *src[TB_COUNT] = {t.rn, t.inv_rn, t.c_e2, t.c_ep2, t.sig_n, t.rho_a, t.rho_b, t.rh, t.inv_rh, t.c_b2,
                              t.c_bp2, t.sig_h, t.rh2};
    for (int w = 0; w < TB_COUNT; ++w) {
      const int last = w < TB_RH ? nr : nr - 1;
      for (int r = threadIdx.x; r <= kl - t0; r += blockDim.x) {
        const int row = t0 + r;
        tab[r * kTabN + w] = (row >= 0 && row <= last) ? src[w][row] : R(0);
      }
    }
  }
  __syncthreads();
  auto T = [&](int row, int w) -> R { return tab[(row - t0) * kTabN + w]; };
  // E^n and dB^n of node row k and half row k: live inside this block's own
  // area, from the snapshot in its outer halo columns and its warm-up /
  // trailing rows; then B_0 and Psi.  Steps come in versions for rows (and
  // columns) known to be in the grid's interior, where every condition on the
  // row (column) holds and the compiler drops it.
  int64_t sc0 = 0;
  if (!mine) {   // unused where the column is outside the grid
    const int b = (j < sx * COLS) ? sx : sx + 1;
    sc0 = (int64_t)(b - 1) * kFuseArrays * (nr + 1) * (2 * kFuseHalo) + (j - (b * COLS - kFuseHalo));
  }
  auto fetch = [&](int k, unsigned char *st, auto tag) {
    constexpr bool IN = decltype(tag)::rows, CI = decltype(tag)::cols, ALL = IN && CI;
    const bool jn = CI || jn_, jh = CI || jh_;
    const bool node = IN || k <= nr, half = IN || k < nr;
    const int64_t kn = (int64_t)k * n1, kh = (int64_t)k * nt;
    R *d = reinterpret_cast<R *>(st) + lane;
    auto get = [&](int a, const R *src, bool ok) {
      if constexpr (ALL) copy_async<sizeof(R)>(d + a * 32, src);
      else copy_async<sizeof(R)>(d + a * 32, ok ? src : f.ep, ok);
    };
    const bool cer = half && jn, cet = node && jh, cep = node && jn, cbr = node && jh, cbt = half && jn,
               cbp = half && jh;
    if ((live || mine) && k >= i_s && k < i_e) {
      get(IN_ER, f.er + kn + ju, cer);
      get(IN_ET, f.et + kh + ju, cet);
      get(IN_EP, f.ep + kn + ju, cep);
      get(IN_BR, f.br + kh + ju, cbr);
      get(IN_BT, f.bt + kn + ju, cbt);
      get(IN_BP, f.bp + kh + ju, cbp);
    } else {
      // array a of the snapshot at s + a as (see k_fuse_prepare)
      const R *s;
      int64_t as;
      if (mine) {
        const int b = (k < i_s) ? sy : sy + 1;
        s = snap_r + ((int64_t)(b - 1) * kFuseArrays * (W + kFuseTrail) + (k - (b * seg_rows - W))) * n1 + ju;
        as = (int64_t)(W + kFuseTrail) * n1;
      } else {
        s = snap_c + sc0 + (int64_t)k * (2 * kFuseHalo);
        as = (int64_t)(nr + 1) * (2 * kFuseHalo);
      }
      get(IN_ER, s, cer);
      get(IN_ET, s + as, cet);
      get(IN_EP, s + 2 * as, cep);
      get(IN_BR, s + 3 * as, cbr);
      get(IN_BT, s + 4 * as, cbt);
      get(IN_BP, s + 5 * as, cbp);
    }
    get(IN_B0R, f.br0 + kh + ju, cbr);
    get(IN_B0T, f.bt0 + kn + ju, cbt);
    get(IN_B0P, f.bp0 + kh + ju, cbp);
    {
      const bool up = IN || k >= 1, node1 = up && (IN || k - 1 <= nr), half1 = up && (IN || k - 1 < nr);
      const int64_t ln = kn - n1, lh = kh - nt;
      get(IN_JR, f.jr + ln + ju, half1 && jn);
      get(IN_SR, f.sr + ln + ju, half1 && jn);
      get(IN_JT, f.jt + lh + ju, node1 && jh);
      get(IN_ST, f.st + lh + ju, node1 && jh);
      get(IN_JP, f.jp + ln + ju, node1 && jn);
      get(IN_SP, f.sp + ln + ju, node1 && jn);
    }
    unsigned char *ps = st + 32 * IN_COUNT * sizeof(R) + lane * sizeof(P);
    const P *psi = f.psi + kn + ju;
    if constexpr (ALL) copy_async<sizeof(P)>(ps, psi);
    else copy_async<sizeof(P)>(ps, cep ? psi : f.psi, cep);
  };
  auto commit = [] { asm volatile("cp.async.commit_group;" ::: "memory"); };
  // theta tables of this column
  const R sn0 = jn_ ? t.sn[j] : R(0), sn1 = jh_ ? t.sn[j + 1] : R(0), idcp = jh_ ? t.inv_dcp[j] : R(0);
  const R sh0 = jh_ ? t.sh[j] : R(0), shm = (j >= 1 && j <= nt) ? t.sh[j - 1] : R(0);
  const R idch = jn_ ? t.inv_dch[j] : R(0);
  const R dt = p.dt, fp4 = R(4.0 * kPi) * p.dt;
  const bool lit = p.ff_interp_e == 1;
  unsigned nclamp = 0;
  // The blend weights are uniform where every Psi of the warp's two rows lies
  // on one side of all breakpoints by more than the rounding of a mean: the
  // usual case, and a mean in pairs with its search costs 35 instructions a
  // weight.
  R psi_lo = R(0), psi_hi = R(0), f_lo = R(0), f_hi = R(0);
  if (p.n_breaks > 0) {   // else f = 0 everywhere
    const R eps = R(1e-6), tiny = R(1e-30);
    psi_lo = psi_lead(p.psi_bk[0]);
    psi_lo -= eps * fabs(psi_lo) + tiny;
    f_lo = p.f_break[0];
    psi_hi = psi_lo;
    for (int q = 0; q < p.n_breaks; ++q) {
      const R b = psi_lead(p.psi_bk[q]);
      psi_hi = max(psi_hi, b + (eps * fabs(b) + tiny));
    }
    f_hi = p.f_break[p.n_breaks - 1];
  }
  bool lo1 = false, hi1 = false;   // every Psi of row k-1 below / above the breakpoints
  // the pipeline: suffix = rows behind k at the beginning of a step (half
  // rows: the half row above that node row)
  R tbt1 = 0, tbp1 = 0;                                  // B^n: B_th; B_ph, sum of two columns
  R jr1 = 0, jt1 = 0, jp1 = 0;                           // J_perp of row k-1
  R br1 = 0, br2 = 0, br3 = 0, ht2 = 0, ht3 = 0, ht4 = 0, hp2 = 0, hp3 = 0, hp4 = 0;   // dB^{n+1/2}
  R nb1 = 0, nb2 = 0, bb2 = 0, bb3 = 0, pp2 = 0, pp3 = 0;   // B^{n+1/2}: B_r at the node; B_th; B_ph, two columns
  R fr2 = 0, fr3 = 0, ft2 = 0, ft3 = 0, fn2 = 0, fn3 = 0;   // blend weights
  R ar2 = 0, ar3 = 0, ar4 = 0, ar5 = 0, at2 = 0, at3 = 0, ap2 = 0, ap3 = 0;   // E^{n+1} before the correction
  R dr3 = 0, mt3 = 0, dp3 = 0;                           // Delta E or E'': E_r, E_th (mean of two columns), E_ph
  R cd4 = 0, ct4 = 0, cp4 = 0;                           // corrected E: E_r (difference to the right), E_th, E_ph
  // step k: row k is staged at `at`, row k-1 at `below`, and `next` is free
  auto step = [&](int k, const unsigned char *at, const unsigned char *below, unsigned char *next, auto tag) {
    constexpr bool IN = decltype(tag)::rows, CI = decltype(tag)::cols;
    const bool jn = CI || jn_, jh = CI || jh_;
    const bool south = !CI && j == 0, north = !CI && j == nt, axis = south || north, inner = CI || (j > 0 && j < nt);
    if (k + kFuseStages - 2 <= kl) fetch(k + kFuseStages - 2, next, tag);
    commit();
    auto in = [&](int a) -> R { return reinterpret_cast<const R *>(at)[a * 32 + lane]; };
    auto in1 = [&](int a) -> R { return reinterpret_cast<const R *>(below)[a * 32 + lane]; };
    const R er = in(IN_ER), et = in(IN_ET), ep = in(IN_EP), dbr = in(IN_BR), dbt = in(IN_BT), dbp = in(IN_BP),
            b0r = in(IN_B0R), b0t = in(IN_B0T), b0p = in(IN_B0P);
    const P psi = reinterpret_cast<const P *>(at + 32 * IN_COUNT * sizeof(R))[lane];
    // row k-1
    const R er1 = in1(IN_ER), et1 = in1(IN_ET), ep1 = in1(IN_EP), bt1 = in1(IN_BT), bp1 = in1(IN_BP),
            b0r1 = in1(IN_B0R), b0t1 = in1(IN_B0T), b0p1 = in1(IN_B0P);
    const P psi1 = reinterpret_cast<const P *>(below + 32 * IN_COUNT * sizeof(R))[lane];
    // --------------------------------------------------------- F1, J_perp
    const R ep_r = right(ep);
    R bhr = dbr;   // B_r(k, j+1/2)
    if (jh) bhr -= hdt * (T(k, TB_INV_RN) * (sn1 * ep_r - sn0 * ep) * idcp);
    const R tbr = b0r + dbr, tbr_l = left(tbr), tbt = b0t + dbt, bpk = b0p + dbp, tbp = left(bpk) + bpk;
    const R et_l = left(et);
    R jx = 0, jy = 0, jz = 0;
    if ((IN || (k >= 1 && k < nr)) && jn) {
      const R e0 = R(0.5) * (er1 + er), e1 = axis ? R(0) : R(0.5) * (et_l + et), e2 = axis ? R(0) : ep;
      const R b0 = south ? tbr : north ? tbr_l : R(0.5) * (tbr_l + tbr);
      const R b1 = axis ? R(0) : R(0.5) * (tbt1 + tbt), b2 = axis ? R(0) : R(0.25) * (tbp1 + tbp);
      const R div = T(k, TB_RHO_A) * (T(k, TB_RH2) * er - T(k - 1, TB_RH2) * er1);
      R dth = 0;
      if (CI || j < nt) dth += sh0 * et;
      if (CI || j > 0) dth -= shm * et_l;
      const R rho = div + T(k, TB_RHO_B) * dth * idch;
      const R bsq = b0 * b0 + b1 * b1 + b2 * b2;
      if (bsq > b2min<R>()) {
        const R s = rho / bsq;
        jx = s * (e1 * b2 - e2 * b1);
        jy = s * (e2 * b0 - e0 * b2);
        jz = s * (e0 * b1 - e1 * b0);
      }
    }
    if (own && k >= i_s && k < i_e) {
      const int64_t kk = (int64_t)k * n1;
      (f.jpr + kk)[ju] = jx; (f.jpt + kk)[ju] = jy; (f.jpp + kk)[ju] = jz;
    }
    // half row k-1
    const int i1 = k - 1;
    R bht = R(0), bhp = R(0);
    const R er1_r = right(er1);
    if (IN || (k >= 1 && i1 < nr)) {
      const R cb2 = T(i1, TB_C_B2), rn0 = T(i1, TB_RN), rn1 = T(k, TB_RN);
      if (inner) bht = bt1 + hdt * cb2 * (rn1 * ep - rn0 * ep1);   // zero on the axis
      if (jh) {
        const R cu = cb2 * (rn1 * et - rn0 * et1) - T(i1, TB_C_BP2) * (er1_r - er1);
        bhp = bp1 - hdt * cu;
      }
    }
    // B^{n+1/2} for N: B_r at node row k, half row k-1
    const R hr = b0r + bhr, hr_l = left(hr);
    const R nb = south ? hr : north ? hr_l : R(0.5) * (hr_l + hr);
    const R bb1 = b0t1 + bht, hpk = b0p1 + bhp, pp1 = left(hpk) + hpk;
    // ------------------------------------------------------ A at row k-1
    const R bhp_l = left(bhp), br1_l = left(br1), jt1_r = right(jt1);
    const P psi1_r = right(psi1);
    R wr = f_lo, wt = f_lo, wn = f_lo;   // f at the E_r edge, the E_th edge and the node
    const bool lo0 = __all_sync(0xffffffffu, psi_lead(psi) < psi_lo);
    const bool hi0 = __all_sync(0xffffffffu, psi_lead(psi) > psi_hi);
    if (hi0 && hi1) {
      wr = wt = wn = f_hi;
    } else if (!(lo0 && lo1)) {
      wr = blend(p, psi_mean2(psi1, psi));
      wt = blend(p, psi_mean2(psi1, psi1_r));
      wn = blend(p, psi1);
    }
    lo1 = lo0;
    hi1 = hi0;
    R fr1 = 0, ft1 = 0, fn1 = 0, ar1 = 0, at1 = 0, ap1 = 0;
    if (IN || (k >= 1 && i1 <= nr)) {
      if ((IN || i1 < nr) && jn) {  // E_r(i+1/2, j)
        R cu = R(0);
        if (CI || j < nt) cu += sh0 * bhp;
        if (CI || j > 0) cu -= shm * bhp_l;
        cu *= T(i1, TB_INV_RH) * idch;
        fr1 = wr;
        const bool lo = IN || i1 >= 1, hi = IN || i1 + 1 <= nr - 1;
        R jm = R(0);
        if (lo) jm += jr1;
        if (hi) jm += jx;
        if (lo && hi) jm *= R(0.5);
        const R jt = (R(1) - fr1) * in(IN_JR) + fr1 * jm;
        ar1 = (er1 + dt * (cu + in(IN_SR)) - fp4 * jt) * (R(1) - T(i1, TB_SIG_H));
      }
      if (jh) {  // E_th(i, j+1/2)
        if (!IN && i1 == 0) {
          at1 = -p.omega * T(0, TB_RN) * sh0 * (b0r1 + br1);
        } else if (!IN && i1 == nr) {
          at1 = R(0);
        } else {
          const R cu = -T(i1, TB_C_E2) * (T(i1, TB_RH) * bhp - T(i1 - 1, TB_RH) * hp2);
          ft1 = wt;
          const R jt = (R(1) - ft1) * in(IN_JT) + ft1 * R(0.5) * (jt1 + jt1_r);
          at1 = (et1 + dt * (cu + in(IN_ST)) - fp4 * jt) * (R(1) - T(i1, TB_SIG_N));
        }
      }
      if ((IN || (i1 >= 1 && i1 < nr)) && inner) {  // E_ph(i, j)
        const R cu = T(i1, TB_C_E2) * (T(i1, TB_RH) * bht - T(i1 - 1, TB_RH) * ht2) - T(i1, TB_C_EP2) * (br1 - br1_l);
        fn1 = wn;
        const R jt = (R(1) - fn1) * in(IN_JP) + fn1 * jp1;
        ap1 = (ep1 + dt * (cu + in(IN_SP)) - fp4 * jt) * (R(1) - T(i1, TB_SIG_N));
      }
    }
    // ------------------------------------------------------ N at row k-2
    const int i2 = k - 2;
    const R at2_l = left(at2);
    R d0 = 0, d1 = 0, d2 = 0;
    if ((IN || (i2 >= 1 && i2 < nr)) && jn) {
      const R e0 = R(0.5) * (ar3 + ar2), e1 = axis ? R(0) : R(0.5) * (at2_l + at2), e2 = axis ? R(0) : ap2;
      const R b0 = nb2, b1 = axis ? R(0) : R(0.5) * (bb3 + bb2), b2 = axis ? R(0) : R(0.25) * (pp3 + pp2);
      const R bsq = b0 * b0 + b1 * b1 + b2 * b2;
      if (bsq > b2min<R>()) {
        const R sdot = (e0 * b0 + e1 * b1 + e2 * b2) / bsq;
        const R x = e0 - sdot * b0, y = e1 - sdot * b1, z = e2 - sdot * b2;
        const R esq = x * x + y * y + z * z;
        R sc = R(1);
        if (esq > bsq) {
          sc = sqrt(bsq / esq);
          if (own && i2 >= i_s && i2 < i_e) ++nclamp;
        }
        d0 = sc * x - e0;
        d1 = sc * y - e1;
        d2 = sc * z - e2;
      }
      if (lit) { d0 += e0; d1 += e1; d2 += e2; }
    }
    if (own && i2 >= i_s && i2 < i_e) {
      const int64_t kk = (int64_t)i2 * n1;
      (f.der + kk)[ju] = d0; (f.det + kk)[ju] = d1; (f.dep + kk)[ju] = d2;
    }
    const R mt2 = R(0.5) * (d1 + right(d1));
    // ------------------------------------------------------ C at row k-3
    const int i3 = k - 3;
    const bool out = own && i3 >= i_s && i3 < i_e;
    R f4 = R(0);
    if constexpr (FILT) {   // fourth difference of E_th along theta
      const R l1 = left(at3), l2 = __shfl_up_sync(0xffffffffu, at3, 2), r1 = right(at3),
              r2 = __shfl_down_sync(0xffffffffu, at3, 2);
      f4 = l2 - R(4) * l1 + R(6) * at3 - R(4) * r1 + r2;
    }
    R cr = ar3, ct = at3, cp = ap3;
    if (IN || (i3 >= 0 && i3 <= nr)) {
      if ((IN || i3 < nr) && jn) {  // E_r(i+1/2, j)
        if (fr3 != R(0)) {
          const bool lo = IN || i3 >= 1, hi = IN || i3 + 1 <= nr - 1;
          R m = R(0);
          if (lo) m += dr3;
          if (hi) m += d0;
          if (lo && hi) m *= R(0.5);
          if constexpr (FILT) {
            if (IN || (i3 >= 2 && i3 <= nr - 3))
              m -= p.ff_sigma16 * (ar5 - R(4) * ar4 + R(6) * ar3 - R(4) * ar2 + ar1);
          }
          cr += fr3 * (lit ? m - ar3 : m);
        }
        if (out) (f.er + (int64_t)i3 * n1)[ju] = cr;
      }
      if (jh) {  // E_th(i, j+1/2)
        if ((IN || (i3 >= 1 && i3 < nr)) && ft3 != R(0)) {
          R m = mt3;
          if (FILT && (CI || (j >= 2 && j <= nt - 3))) m -= p.ff_sigma16 * f4;
          ct += ft3 * (lit ? m - at3 : m);
        }
        if (out) (f.et + (int64_t)i3 * nt)[ju] = ct;
      }
      if (jn) {  // E_ph(i, j)
        if ((IN || (i3 >= 1 && i3 < nr)) && inner && fn3 != R(0)) cp += fn3 * (lit ? dp3 - ap3 : dp3);
        if (out) (f.ep + (int64_t)i3 * n1)[ju] = cp;
      }
    }
    // ----------------------------------- F2 at node row k-3, half row k-4
    const R cp_r = right(cp), cd = right(cr) - cr;
    if (out && jh) {
      const R cu = T(i3, TB_INV_RN) * (sn1 * cp_r - sn0 * cp) * idcp;
      R v = br3 - hdt * cu;
      const R sg = T(i3, TB_SIG_N);
      if (sg > R(0)) v -= sg * v;
      (f.br + (int64_t)i3 * nt)[ju] = v;
    }
    const int h = k - 4;
    if (own && h >= i_s && h < i_e && (IN || h < nr)) {
      const R sg = T(h, TB_SIG_H), cb2 = T(h, TB_C_B2), rn0 = T(h, TB_RN), rn1 = T(h + 1, TB_RN);
      R v = R(0);
      if (inner) {
        v = ht4 + hdt * cb2 * (rn1 * cp - rn0 * cp4);
        if (sg > R(0)) v -= sg * v;
      }
      (f.bt + (int64_t)h * n1)[ju] = v;
      if (jh) {
        const R cu = cb2 * (rn1 * ct - rn0 * ct4) - T(h, TB_C_BP2) * cd4;
        R w = hp4 - hdt * cu;
        if (sg > R(0)) w -= sg * w;
        (f.bp + (int64_t)h * nt)[ju] = w;
      }
    }
    // ------------------------------------------------------- one row on
    tbt1 = tbt; tbp1 = tbp; jr1 = jx; jt1 = jy; jp1 = jz;
    br3 = br2; br2 = br1; br1 = bhr; ht4 = ht3; ht3 = ht2; ht2 = bht; hp4 = hp3; hp3 = hp2; hp2 = bhp;
    nb2 = nb1; nb1 = nb; bb3 = bb2; bb2 = bb1; pp3 = pp2; pp2 = pp1;
    fr3 = fr2; fr2 = fr1; ft3 = ft2; ft2 = ft1; fn3 = fn2; fn2 = fn1;
    if constexpr (FILT) { ar5 = ar4; ar4 = ar3; }
    ar3 = ar2; ar2 = ar1; at3 = at2; at2 = at1; ap3 = ap2; ap2 = ap1;
    dr3 = d0; mt3 = mt2; dp3 = d2; cd4 = cd; ct4 = ct; cp4 = cp;
  };
  // interior steps: rows k-4 .. k+2 inside rows 2 .. nr-3
  const int kin0 = 6, kin1 = nr - 5;
  const bool some = j0 + H <= nt;   // this warp owns columns of the grid
  constexpr int kStage = (int)fuse_stage_bytes<R>();
  unsigned char *ring = fsmem + fuse_tab_rows(seg_rows) * kTabN * sizeof(R) + warp * (kFuseStages * kStage);
  static_assert((kFuseStages & (kFuseStages - 1)) == 0, "ring");
  auto slot = [&](int k) { return ring + (k & (kFuseStages - 1)) * kStage; };
  for (int w = lane; w < kStage / 4; w += 32) reinterpret_cast<int *>(slot(k0 - 1))[w] = 0;   // the row before the first
  __syncwarp();
  for (int k = k0; k < k0 + kFuseStages - 2; ++k) {
    if (some) fetch(k, slot(k), FuseTag<false, false>{});
    commit();
  }
  for (int k = k0; k <= kl; ++k) {
    asm volatile("cp.async.wait_group %0;" ::"n"(kFuseStages - 3) : "memory");
    if (((k - k0) & 3) == 3) __syncthreads();   // see above: neighbours' reads before this warp's writes
    if (!some) continue;
    const unsigned char *at = slot(k), *below = slot(k - 1);
    unsigned char *next = slot(k + kFuseStages - 2);
    if (k < kin0 || k > kin1) step(k, at, below, next, FuseTag<false, false>{});
    else if (cin) step(k, at, below, next, FuseTag<true, true>{});
    else step(k, at, below, next, FuseTag<true, false>{});
  }
  // running count of Eq. 26 activations (see k_node_b)
  unsigned tot = nclamp;
  for (int o = 16; o > 0; o >>= 1) tot += __shfl_down_sync(0xffffffffu, tot, o);
  if (lane == 0 && tot) atomicAdd(p.clamps, (unsigned long long)tot);
}

template <typename R> size_t field_fused_smem(int seg_rows) {
  return (size_t)fuse_tab_rows(seg_rows) * kTabN * sizeof(R) + fuse_warps(sizeof(R)) * kFuseStages * fuse_stage_bytes<R>();
}
template <typename R, bool F> const void *field_fused_fn() { return reinterpret_cast<const void *>(&k_field_fused<R, F>); }
template <typename R> cudaError_t set_field_fused_smem(size_t bytes) {
  const cudaError_t e = raise_smem_limit<field_fused_fn<R, false>>(bytes);
  return e != cudaSuccess ? e : raise_smem_limit<field_fused_fn<R, true>>(bytes);
}
// resident blocks per SM of the pass with segments of seg_rows rows; 0 on error
template <typename R> int field_fused_blocks_per_sm(int seg_rows, bool filt) {
  int n = 0;
  const void *f = filt ? field_fused_fn<R, true>() : field_fused_fn<R, false>();
  return cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, f, 32 * fuse_warps(sizeof(R)), field_fused_smem<R>(seg_rows)) == cudaSuccess ? n : 0;
}
// rows per segment: as many segments as fit the strips into wave_blocks
// resident blocks (one wave: every block walks its rows once, none waits
// for a second wave), at least 32 rows so that the warm-up stays a small
// share, and at most kFuseMaxRows (the staged radial tables)
int fuse_seg_rows(int nr, int nt, int wave_blocks, size_t real, bool filt) {
  const int cols = fuse_cols(real, filt), strips = (nt + 1 + cols - 1) / cols;
  const int segs = std::max(1, wave_blocks / strips);
  return std::min(kFuseMaxRows, std::max(32, (nr + 1 + segs - 1) / segs));
}
size_t fuse_snap_bytes(int nr, int nt, int seg_rows, size_t real, bool filt) {
  const FuseGeom fg = fuse_geom(nr, nt, seg_rows, fuse_cols(real, filt));
  return (size_t)(fuse_snap_cols(nr, fg.strips) + fuse_snap_rows(nt, fg.segs)) * real;
}
template <typename R> void launch_field_fused(const Params<R> &p, int seg_rows, void *snap, bool collect, cudaStream_t s) {
  const bool filt = p.ff_sigma16 != R(0);
  const int cols = fuse_cols(sizeof(R), filt);
  const FuseGeom fg = fuse_geom(p.nr, p.nt, seg_rows, cols);
  R *sc = reinterpret_cast<R *>(snap);
  R *sr = sc + fuse_snap_cols(p.nr, fg.strips);
  const int nc = (fg.strips - 1) * ((p.nr + kSnapRows) / kSnapRows);
  const int nw = (fg.segs - 1) * (kFuseWarm + kFuseTrail) * (p.nt / kSnapThreads + 1);
  const int nj = collect ? collect_blocks_x(p) * collect_blocks_y(p) : 0;
  if (nc + nw + nj > 0) k_fuse_prepare<R><<<nc + nw + nj, kSnapThreads, 0, s>>>(p, sc, sr, seg_rows, cols, nc, nw);
  const dim3 grid(fg.strips, fg.segs);
  const int threads = 32 * fuse_warps(sizeof(R));
  const size_t smem = field_fused_smem<R>(seg_rows);
  if (filt) k_field_fused<R, true><<<grid, threads, smem, s>>>(p, R(0.5) * p.dt, fg, sc, sr);
  else k_field_fused<R, false><<<grid, threads, smem, s>>>(p, R(0.5) * p.dt, fg, sc, sr);
}

// The per-cell pure force-free flag f(Psi_cell) >= 1 (used to remove
// particles, Eq. 29) on its own, for the fused field update, which computes
// J_perp itself: a thread walks kFfRows cells of one column, reading every
// node row of Psi once (the arithmetic of ff_cell).
constexpr int kFfRows = 16;
template <typename R>
__global__ void __launch_bounds__(kRowThreads) k_ffcell(Params<R> p) {
  using P = typename PsiOf<R>::T;
  const int nr = p.nr, nt = p.nt, n1 = nt + 1;
  const int j = blockIdx.x * blockDim.x + threadIdx.x, i0 = blockIdx.y * kFfRows;
  if (j >= nt || i0 >= nr) return;
  const int i1 = min(i0 + kFfRows, nr);
  const P *psi = p.f.psi + j;
  P a = psi[(int64_t)i0 * n1], b = psi[(int64_t)i0 * n1 + 1];
  for (int i = i0; i < i1; ++i) {
    const P c = psi[(int64_t)(i + 1) * n1], d = psi[(int64_t)(i + 1) * n1 + 1];
    p.f.ffcell[(int64_t)i * nt + j] = blend(p, psi_mean4(a, c, b, d)) >= R(1) ? 1 : 0;
    a = c;
    b = d;
  }
}

// The blend weights of the last flux prefix, on request (hff_fields): f at
// the E_r and E_th edges and at the nodes, and the force-free cell flags
// (outputs passed as null are skipped).
template <typename R>
__global__ void __launch_bounds__(kRowThreads) k_blend_out(Params<R> p, R *fr, R *ft, R *fn, uint8_t *cells) {
  const int i = blockIdx.y, j = blockIdx.x * blockDim.x + threadIdx.x;
  const int nr = p.nr, nt = p.nt, n1 = nt + 1;
  if (j > nt) return;
  if (fr && i < nr) fr[ix(i, j, n1)] = blend_redge(p, i, j);
  if (ft && j < nt) ft[ix(i, j, nt)] = blend_tedge(p, i, j);
  if (fn) fn[ix(i, j, n1)] = blend_node(p, i, j);
  if (cells && i < nr && j < nt) cells[ix(i, j, nt)] = ff_cell(p, i, j) ? 1 : 0;
}

static inline dim3 row_grid(int rows, int nt) { return dim3((nt + 1 + kRowThreads - 1) / kRowThreads, rows); }

template <typename R> size_t psi_smem(int nt) { return (size_t)(psi_pad(nt) + 2) * 8; }
template <typename R> void launch_psi(const Params<R> &p, cudaStream_t s) {
  const size_t smem = psi_smem<R>(p.nt);
  k_psi<R><<<p.nr + 1, kPsiThreads, smem, s>>>(p);
}
template <typename R> const void *psi_fn() { return reinterpret_cast<const void *>(&k_psi<R>); }
template <typename R> cudaError_t set_psi_smem(size_t bytes) { return raise_smem_limit<psi_fn<R>>(bytes); }
template <typename R> void launch_node_a(const Params<R> &p, cudaStream_t s) {
  k_node_a<R><<<row_grid(p.nr + 1, p.nt), kRowThreads, 0, s>>>(p);
}
template <typename R> void launch_ffcell(const Params<R> &p, cudaStream_t s) {
  k_ffcell<R><<<dim3((p.nt + kRowThreads - 1) / kRowThreads, (p.nr + kFfRows - 1) / kFfRows), kRowThreads, 0, s>>>(p);
}
template <typename R> bool faraday_carries_collect(const Params<R> &p) {
  return p.nr + 1 + collect_blocks_y(p) <= 65535;  // gridDim.y
}
template <typename R> void launch_faraday(const Params<R> &p, R half, bool absorb, bool collect, cudaStream_t s) {
  dim3 g = row_grid(p.nr + 1, p.nt);
  if (collect) {
    g.x = std::max<unsigned>(g.x, collect_blocks_x(p));
    g.y += collect_blocks_y(p);
  }
  k_faraday<R><<<g, kRowThreads, 0, s>>>(p, half * p.dt, absorb);
}
template <typename R> void launch_ampere(const Params<R> &p, cudaStream_t s) {
  k_ampere<R><<<row_grid(p.nr + 1, p.nt), kRowThreads, 0, s>>>(p);
}
template <typename R> void launch_correct(const Params<R> &p, cudaStream_t s) {
  k_node_b<R><<<row_grid(p.nr + 1, p.nt), kRowThreads, 0, s>>>(p);
  k_correct<R><<<row_grid(p.nr + 1, p.nt), kRowThreads, 0, s>>>(p);
}

template <typename R> void launch_blend_out(const Params<R> &p, R *fr, R *ft, R *fn, uint8_t *cells, cudaStream_t s) {
  k_blend_out<R><<<row_grid(p.nr + 1, p.nt), kRowThreads, 0, s>>>(p, fr, ft, fn, cells);
}

template <typename R>
__global__ void k_combine(R *dst, const R *a, const R *b, int64_t n, R sign) {
  for (int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; k < n; k += (int64_t)gridDim.x * blockDim.x)
    dst[k] = a[k] + sign * b[k];
}
template <typename R> void launch_combine(R *dst, const R *a, const R *b, int64_t n, int sign, cudaStream_t s) {
  if (n <= 0) return;
  const int64_t blocks = (n + 255) / 256;
  k_combine<R><<<(unsigned)(blocks < 65536 ? blocks : 65536), 256, 0, s>>>(dst, a, b, n, (R)sign);
}

#define HFF_INST(R)                                                            \
  template void launch_combine<R>(R *, const R *, const R *, int64_t, int, cudaStream_t); \
  template void launch_psi<R>(const Params<R> &, cudaStream_t);                \
  template cudaError_t set_psi_smem<R>(size_t);                                \
  template size_t psi_smem<R>(int);                                            \
  template void launch_node_a<R>(const Params<R> &, cudaStream_t);             \
  template void launch_ffcell<R>(const Params<R> &, cudaStream_t);             \
  template bool faraday_carries_collect<R>(const Params<R> &);                 \
  template void launch_faraday<R>(const Params<R> &, R, bool, bool, cudaStream_t); \
  template void launch_ampere<R>(const Params<R> &, cudaStream_t);             \
  template void launch_correct<R>(const Params<R> &, cudaStream_t);            \
  template void launch_blend_out<R>(const Params<R> &, R *, R *, R *, uint8_t *, cudaStream_t); \
  template void launch_field_fused<R>(const Params<R> &, int, void *, bool, cudaStream_t);      \
  template size_t field_fused_smem<R>(int);                                                         \
  template cudaError_t set_field_fused_smem<R>(size_t);                        \
  template int field_fused_blocks_per_sm<R>(int, bool);
HFF_INST(float)
HFF_INST(double)
#undef HFF_INST

}  // namespace hff
