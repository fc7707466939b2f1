// particles.cu -- particle side of the hybrid step: linear gather from the
// staggered mesh, modified Boris push with radiation reaction (Eqs. 15-17),
// removal of u_perp near the star (Sect. 5.1), straight-line move in the
// local Cartesian frame, charge-conserving (Esirkepov) deposit of J_PIC, and
// the surface pair injection (Sects. 4 and 5.1).
//
// Two drivers share one per-particle routine:
//  * k_push_tiled -- persistent blocks take (species, tile, chunk) work items
//    from a list built by the sort.  The block stages E, B and the force-free
//    flags of the tile plus a halo (the farthest a particle can drift between
//    sorts) into shared memory.  Particles of a tile are contiguous, so the
//    particle stream is read and written once, fully coalesced.
//    Particles appended since the last sort (injection, created pairs) follow
//    in the same launch, gathering through L1/L2.
//  * k_push_tail -- all particles of the no-sort configuration, the same way.
// Both deposit into the flux accumulators in global memory (see deposit);
// those become J_PIC at the end of the push stage (collect.cuh).
#include <type_traits>

#include "collect.cuh"
#include "fastmath.cuh"
#include "hff_common.cuh"

namespace hff {

// -------------------------------------------------------------- accessors
// Global-memory view of the mesh.
template <typename R>
struct GlobalMesh {
  const Params<R> &p;
  __device__ GlobalMesh(const Params<R> &pp) : p(pp) {}
  __device__ __forceinline__ R er(int i, int j) const { return p.f.er[ix(i, j, p.nt + 1)]; }
  __device__ __forceinline__ R et(int i, int j) const { return p.f.et[ix(i, j, p.nt)]; }
  __device__ __forceinline__ R ep(int i, int j) const { return p.f.ep[ix(i, j, p.nt + 1)]; }
  // B = B_0 + dB
  __device__ __forceinline__ R br(int i, int j) const { const int64_t k = ix(i, j, p.nt); return p.f.br0[k] + p.f.br[k]; }
  __device__ __forceinline__ R bt(int i, int j) const { const int64_t k = ix(i, j, p.nt + 1); return p.f.bt0[k] + p.f.bt[k]; }
  __device__ __forceinline__ R bp(int i, int j) const { const int64_t k = ix(i, j, p.nt); return p.f.bp0[k] + p.f.bp[k]; }
  __device__ __forceinline__ bool ff(int i, int j) const { return p.f.ffcell[ix(i, j, p.nt)] != 0; }
  __device__ __forceinline__ R rn(int i) const { return p.t.rn[i]; }
  __device__ __forceinline__ R sn(int j) const { return p.t.sn[j]; }
  __device__ __forceinline__ R cn(int j) const { return p.t.cn[j]; }
};

// Shared-memory view of a tile region [i0, i0 + LR) x [j0, j0 + LT) of every
// component (indices are global; the caller guarantees they fall inside).
// FP64: one array per component.
template <typename R>
struct SharedMesh {
  R *s_er, *s_et, *s_ep, *s_br, *s_bt, *s_bp;
  R *s_rn, *s_sn, *s_cn;   // row / column tables of the region
  uint8_t *s_ff;
  int i0, j0, lt;
  static size_t bytes_per_location() { return 6 * sizeof(R) + 1; }
  __device__ __forceinline__ unsigned char *carve(unsigned char *base, int area) {
    R *b = reinterpret_cast<R *>(base);
    s_er = b; s_et = b + area; s_ep = b + 2 * area; s_br = b + 3 * area; s_bt = b + 4 * area; s_bp = b + 5 * area;
    return reinterpret_cast<unsigned char *>(b + 6 * area);
  }
  __device__ __forceinline__ void put(int k, int, R er, R et, R ep, R br, R bt, R bp) const {
    s_er[k] = er; s_et[k] = et; s_ep[k] = ep; s_br[k] = br; s_bt[k] = bt; s_bp[k] = bp;
  }
  __device__ __forceinline__ int o(int i, int j) const { return (i - i0) * lt + (j - j0); }
  __device__ __forceinline__ bool ff(int i, int j) const { return s_ff[o(i, j)] != 0; }
  __device__ __forceinline__ R rn(int i) const { return s_rn[i - i0]; }
  __device__ __forceinline__ R sn(int j) const { return s_sn[j - j0]; }
  __device__ __forceinline__ R cn(int j) const { return s_cn[j - j0]; }
};
// FP32: the components that share their locations side by side, and E_ph and
// B_ph with their right-hand neighbours, so that the gather's corners are
// 8-byte loads: 12 a particle instead of 24.
template <>
struct SharedMesh<float> {
  float2 *s_a, *s_b;       // (E_r, B_th) and (E_th, B_r)
  float2 *s_p, *s_q;       // E_ph and B_ph at columns j, j + 1
  float *s_rn, *s_sn, *s_cn;
  uint8_t *s_ff;
  int i0, j0, lt;
  static size_t bytes_per_location() { return 4 * sizeof(float2) + 1; }
  __device__ __forceinline__ unsigned char *carve(unsigned char *base, int area) {
    s_a = reinterpret_cast<float2 *>(base); s_b = s_a + area;
    s_p = s_b + area; s_q = s_p + area;
    return reinterpret_cast<unsigned char *>(s_q + area);
  }
  // location k, column c of the region: its own slot and the left neighbour's
  // second half (the last column's second half is never read)
  __device__ __forceinline__ void put(int k, int c, float er, float et, float ep, float br, float bt, float bp) const {
    s_a[k] = make_float2(er, bt);
    s_b[k] = make_float2(et, br);
    s_p[k].x = ep;
    s_q[k].x = bp;
    if (c > 0) {
      s_p[k - 1].y = ep;
      s_q[k - 1].y = bp;
    }
  }
  __device__ __forceinline__ int o(int i, int j) const { return (i - i0) * lt + (j - j0); }
  __device__ __forceinline__ bool ff(int i, int j) const { return s_ff[o(i, j)] != 0; }
  __device__ __forceinline__ float rn(int i) const { return s_rn[i - i0]; }
  __device__ __forceinline__ float sn(int j) const { return s_sn[j - j0]; }
  __device__ __forceinline__ float cn(int j) const { return s_cn[j - j0]; }
};

// two FP32 values in the packed arithmetic (one issue slot for two additions,
// multiplications or multiply-adds), used where pairs fall together anyway
struct F2 {
  float2 v;
};
__device__ __forceinline__ F2 operator-(F2 a, F2 b) { return {__ffma2_rn(b.v, make_float2(-1.f, -1.f), a.v)}; }
// w a + b
__device__ __forceinline__ F2 vfma(float w, F2 a, F2 b) { return {__ffma2_rn(make_float2(w, w), a.v, b.v)}; }
__device__ __forceinline__ float vfma(float a, float b, float c) { return fmaf(a, b, c); }
__device__ __forceinline__ double vfma(double a, double b, double c) { return fma(a, b, c); }

// Comparisons of doubles on the integer pipe (a comparison costs the FP64
// pipe as much as an addition): x >= c for a positive constant c whose lower
// word is zero, the sign, finiteness, and |a| well below b.
__device__ __forceinline__ bool at_least(float x, float c) { return x >= c; }
__device__ __forceinline__ bool at_least(double x, double c) { return __double2hiint(x) >= __double2hiint(c); }
__device__ __forceinline__ bool below_zero(float x) { return x < 0.f; }
__device__ __forceinline__ bool below_zero(double x) { return __double2hiint(x) < 0 && ((__double2hiint(x) << 1) | __double2loint(x)) != 0; }
__device__ __forceinline__ bool finite(float x) { return fabsf(x) <= 3.402823466e38f; }
__device__ __forceinline__ bool finite(double x) { return exponent_field(x) != 2047u; }
// inside [0, 1) as an offset that needs no look at the cell: one comparison of
// the bits (-0 and values outside go the long way)
__device__ __forceinline__ bool stays(float x) { return (unsigned)__float_as_int(x) < 0x3f800000u; }
__device__ __forceinline__ bool stays(double x) { return (unsigned)__double2hiint(x) < 0x3ff00000u; }
__device__ __forceinline__ bool all_finite(float X, float Y, const float u[3]) {
  return finite((X + Y) + ((u[0] + u[1]) + u[2]));   // a sum is finite unless a term is not (none is near the range's end)
}
__device__ __forceinline__ bool all_finite(double X, double Y, const double u[3]) {
  return finite(X) && finite(Y) && finite(u[0]) && finite(u[1]) && finite(u[2]);
}
// |a| < 0.03 b (implies b > 0).  FP64: the high words, read as integers, are
// piecewise linear in the logarithm (within 0.0861 octaves), so a difference
// of 5.2 octaves means a ratio below 2^-5.11 = 0.029; ratios between 0.025 and
// 0.03 may be refused, which only sends the move to its general form.
constexpr double kSmall = 0.03;
__device__ __forceinline__ bool well_below(float a, float b) { return fabsf(a) < float(kSmall) * b; }
__device__ __forceinline__ bool well_below(double a, double b) {
  const int hb = __double2hiint(b);   // negative for b < 0
  return hb >= 0 && hb < 0x7ff00000 && hb - (__double2hiint(a) & 0x7fffffff) >= 0x00533333;
}

// Small-argument Taylor expansions about 0, for the per-step increments that
// the Courant condition keeps small; callers switch to the library functions
// outside |x| < kSmall (log1p outside 0.03125), where every truncation error is
// below 2e-13 of the value (for cosm, of the cosine) in FP64 (log1p's, x^8 / 9;
// the others below 1e-15) and 5e-10 in FP32 (the binomial ones, (35/64) q^3; a
// hundredth of its rounding).
// c[0] + c[1] x + .. by Horner's rule
template <typename R, int N>
__device__ __forceinline__ R poly(R x, const double (&c)[N]) {
  R t = R(c[N - 1]);
#pragma unroll
  for (int k = N - 2; k >= 0; --k) t = vfma(t, x, R(c[k]));
  return t;
}
// sin x / x, (cos x - 1) / x^2 and atan t / t as series in the square,
// log1p(x) / x and (exp x - 1) / x in x, and for q = tan^2 of an angle
// (1 - cos) / q = (1 - (1 + q)^(-1/2)) / q and ((1 + q)^(1/2) - 1) / q
// (binomial series)
template <typename R> struct Series {
  static __device__ __forceinline__ R sinc(R x2) { const double c[] = {1.0, -1.0 / 6, 1.0 / 120, -1.0 / 5040}; return poly(x2, c); }
  static __device__ __forceinline__ R cosm(R x2) { const double c[] = {-0.5, 1.0 / 24, -1.0 / 720}; return poly(x2, c); }
  static __device__ __forceinline__ R atanc(R t2) { const double c[] = {1.0, -1.0 / 3, 0.2, -1.0 / 7, 1.0 / 9}; return poly(t2, c); }
  static __device__ __forceinline__ R log1pc(R x) {
    const double c[] = {1.0, -0.5, 1.0 / 3, -0.25, 0.2, -1.0 / 6, 1.0 / 7, -0.125};
    return poly(x, c);
  }
  static __device__ __forceinline__ R expm1c(R x) {
    const double c[] = {1.0, 0.5, 1.0 / 6, 1.0 / 24, 1.0 / 120, 1.0 / 720, 1.0 / 5040};
    return poly(x, c);
  }
  static __device__ __forceinline__ R omc(R q) { const double c[] = {0.5, -3.0 / 8, 5.0 / 16, -35.0 / 128, 63.0 / 256}; return poly(q, c); }
  static __device__ __forceinline__ R sqm(R q) { const double c[] = {0.5, -1.0 / 8, 1.0 / 16, -5.0 / 128, 7.0 / 256}; return poly(q, c); }
};
template <> struct Series<float> {
  using R = float;
  static __device__ __forceinline__ R sinc(R x2) { const double c[] = {1.0, -1.0 / 6, 1.0 / 120}; return poly(x2, c); }
  static __device__ __forceinline__ R cosm(R x2) { const double c[] = {-0.5, 1.0 / 24}; return poly(x2, c); }
  static __device__ __forceinline__ R atanc(R t2) { const double c[] = {1.0, -1.0 / 3, 0.2}; return poly(t2, c); }
  static __device__ __forceinline__ R log1pc(R x) { const double c[] = {1.0, -0.5, 1.0 / 3, -0.25, 0.2, -1.0 / 6}; return poly(x, c); }
  static __device__ __forceinline__ R expm1c(R x) { const double c[] = {1.0, 0.5, 1.0 / 6, 1.0 / 24, 1.0 / 120}; return poly(x, c); }
  static __device__ __forceinline__ R omc(R q) { const double c[] = {0.5, -3.0 / 8, 5.0 / 16}; return poly(q, c); }
  static __device__ __forceinline__ R sqm(R q) { const double c[] = {0.5, -1.0 / 8, 1.0 / 16}; return poly(q, c); }
};

// ------------------------------------------------------------------ gather
// 1D linear weights for a component at positions k + a (a = 0 or 1/2),
// k = 0 .. n-1, constant beyond the ends.
template <typename R>
__device__ __forceinline__ void stag(int c, R o, bool half, int n, int &k0, R &w) {
  if (!half) { k0 = c; w = o; }
  else if (o >= R(0.5)) { k0 = c; w = o - R(0.5); }
  else { k0 = c - 1; w = o + R(0.5); }
  if (k0 < 0) { k0 = 0; w = R(0); }
  if (k0 > n - 2) { k0 = n - 2; w = R(1); }
}

template <typename R, typename M, typename Get>
__device__ __forceinline__ R interp(const M &m, Get g, int i, R wi, int j, R wj) {
  const R a0 = g(m, i, j), a1 = g(m, i, j + 1), b0 = g(m, i + 1, j), b1 = g(m, i + 1, j + 1);
  const R lo = a0 + wj * (a1 - a0), hi = b0 + wj * (b1 - b0);
  return lo + wi * (hi - lo);
}

template <typename R>
__device__ __forceinline__ void gather(const GlobalMesh<R> &m, int i, int j, R xo, R yo, R e[3], R b[3]) {
  using M = GlobalMesh<R>;
  const int nr = m.p.nr, nt = m.p.nt;
  // the four (node | half) x (node | half) weight sets, each shared by the
  // components that live there
  int kin, kih, kjn, kjh;
  R win, wih, wjn, wjh;
  stag(i, xo, false, nr + 1, kin, win);
  stag(i, xo, true, nr, kih, wih);
  stag(j, yo, false, nt + 1, kjn, wjn);
  stag(j, yo, true, nt, kjh, wjh);
  e[0] = interp(m, [](const M &q, int a, int c) { return q.er(a, c); }, kih, wih, kjn, wjn);
  b[1] = interp(m, [](const M &q, int a, int c) { return q.bt(a, c); }, kih, wih, kjn, wjn);
  e[1] = interp(m, [](const M &q, int a, int c) { return q.et(a, c); }, kin, win, kjh, wjh);
  b[0] = interp(m, [](const M &q, int a, int c) { return q.br(a, c); }, kin, win, kjh, wjh);
  e[2] = interp(m, [](const M &q, int a, int c) { return q.ep(a, c); }, kin, win, kjn, wjn);
  b[2] = interp(m, [](const M &q, int a, int c) { return q.bp(a, c); }, kih, wih, kjh, wjh);
}

// Shared-memory versions of the gather: every access is a constant offset
// from one base offset per weight set, and the staged region replicates the
// edge values of each array, which reproduces the constant extrapolation of
// stag() without clamping.
template <typename R>
__device__ __forceinline__ R lerp4(const R *a, int o, int lt, R wi, R wj) {
  const R a0 = a[o], a1 = a[o + 1], b0 = a[o + lt], b1 = a[o + lt + 1];
  const R lo = a0 + wj * (a1 - a0), hi = b0 + wj * (b1 - b0);
  return lo + wi * (hi - lo);
}
__device__ __forceinline__ void gather(const SharedMesh<double> &m, int i, int j, double xo, double yo, double e[3],
                                       double b[3]) {
  const bool hx = at_least(xo, 0.5), hy = at_least(yo, 0.5);
  const int oc = m.o(i, j), lt = m.lt;
  const int onn = oc, onh = oc - (hy ? 0 : 1), ohn = oc - (hx ? 0 : lt), ohh = ohn - (hy ? 0 : 1);
  const double win = xo, wjn = yo, wih = xo + (hx ? -0.5 : 0.5), wjh = yo + (hy ? -0.5 : 0.5);
  e[0] = lerp4(m.s_er, ohn, lt, wih, wjn);
  b[1] = lerp4(m.s_bt, ohn, lt, wih, wjn);
  e[1] = lerp4(m.s_et, onh, lt, win, wjh);
  b[0] = lerp4(m.s_br, onh, lt, win, wjh);
  e[2] = lerp4(m.s_ep, onn, lt, win, wjn);
  b[2] = lerp4(m.s_bp, ohh, lt, wih, wjh);
}
// (u, v) pairs of two components at the four corners: packed over components
__device__ __forceinline__ F2 lerp_pair(const float2 *a, int o, int lt, float wi, float wj) {
  const F2 a0{a[o]}, a1{a[o + 1]}, b0{a[o + lt]}, b1{a[o + lt + 1]};
  const F2 lo = vfma(wj, a1 - a0, a0), hi = vfma(wj, b1 - b0, b0);
  return vfma(wi, hi - lo, lo);
}
// one component: packed over the columns first
__device__ __forceinline__ float lerp_one(const float2 *a, int o, int lt, float wi, float wj) {
  const F2 r0{a[o]}, r1{a[o + lt]}, t = vfma(wi, r1 - r0, r0);
  return fmaf(wj, t.v.y - t.v.x, t.v.x);
}
__device__ __forceinline__ void gather(const SharedMesh<float> &m, int i, int j, float x, float y, float e[3],
                                       float b[3]) {
  const bool hx = x >= 0.5f, hy = y >= 0.5f;
  const int oc = m.o(i, j), lt = m.lt;
  const int onh = oc - (hy ? 0 : 1), ohn = oc - (hx ? 0 : lt), ohh = ohn - (hy ? 0 : 1);
  const float wih = x + (hx ? -0.5f : 0.5f), wjh = y + (hy ? -0.5f : 0.5f);
  const F2 a = lerp_pair(m.s_a, ohn, lt, wih, y), c = lerp_pair(m.s_b, onh, lt, x, wjh);
  e[0] = a.v.x; b[1] = a.v.y;
  e[1] = c.v.x; b[0] = c.v.y;
  e[2] = lerp_one(m.s_p, oc, lt, x, y);
  b[2] = lerp_one(m.s_q, ohh, lt, wih, wjh);
}

// ------------------------------------------------------------------- push
template <typename R> __device__ __forceinline__ R dot3(const R a[3], const R b[3], R c) {
  return vfma(a[2], b[2], vfma(a[1], b[1], vfma(a[0], b[0], c)));
}
template <typename R> __device__ __forceinline__ R dot3(const R a[3], const R b[3]) {
  return vfma(a[2], b[2], vfma(a[1], b[1], a[0] * b[0]));
}
// component k of a x b, plus c
template <int k, typename R> __device__ __forceinline__ R cross(const R a[3], const R b[3], R c) {
  constexpr int i = (k + 1) % 3, j = (k + 2) % 3;
  return vfma(a[i], b[j], vfma(-a[j], b[i], c));
}

// Modified Boris step (Eqs. 15-17, c = 1): Lorentz Boris gives u_L, the
// radiation-reaction kick K F_RR is evaluated at the time-centred momentum
// (u + u_L)/2 and limited to half of |u_L| per step.  Bperp^2 of Eq. 17 is
// evaluated as |F x beta|^2 + |F|^2 / gamma^2 with F = E + beta x B, which
// equals |F|^2 - (beta.F)^2 = |F|^2 - (beta.E)^2 without cancellation.
// Returns 1/gamma of the new momentum; dgam is the energy radiated.
template <typename R>
__device__ __forceinline__ R boris_rr(R qm, R krr, R dt, const R u[3], const R e[3], const R b[3], R out[3], R &dgam) {
  const R one = R(1), a = R(0.5) * qm * dt;
  R um[3], t[3], v[3], w[3], ul[3];
#pragma unroll
  for (int k = 0; k < 3; ++k) um[k] = vfma(a, e[k], u[k]);
  const R at = a * rsq(dot3(um, um, one));
#pragma unroll
  for (int k = 0; k < 3; ++k) t[k] = at * b[k];
  const R sc = R(2) * rcp(dot3(t, t, one));
  // u+ = u- + sc (u- + u- x t) x t
  v[0] = cross<0>(um, t, um[0]); v[1] = cross<1>(um, t, um[1]); v[2] = cross<2>(um, t, um[2]);
  w[0] = cross<0>(v, t, R(0)); w[1] = cross<1>(v, t, R(0)); w[2] = cross<2>(v, t, R(0));
#pragma unroll
  for (int k = 0; k < 3; ++k) ul[k] = vfma(sc, w[k], vfma(a, e[k], um[k]));
  if (krr == R(0)) {
#pragma unroll
    for (int k = 0; k < 3; ++k) out[k] = ul[k];
    dgam = R(0);
    return rsq(dot3(ul, ul, one));
  }
  R us[3], be[3], f[3], c[3], du[3];
#pragma unroll
  for (int k = 0; k < 3; ++k) us[k] = u[k] + ul[k];   // twice the centred momentum
  const R g2 = vfma(R(0.25), dot3(us, us), one), ig = rsq(g2), hb = R(0.5) * ig;
#pragma unroll
  for (int k = 0; k < 3; ++k) be[k] = hb * us[k];
  f[0] = cross<0>(be, b, e[0]); f[1] = cross<1>(be, b, e[1]); f[2] = cross<2>(be, b, e[2]);
  c[0] = cross<0>(f, be, R(0)); c[1] = cross<1>(f, be, R(0)); c[2] = cross<2>(f, be, R(0));
  const R bp2 = dot3(c, c, dot3(f, f) * (ig * ig));
  const R bdot = dot3(be, e), k = dt * krr, gb = -(g2 * bp2);
  du[0] = k * cross<0>(f, b, vfma(bdot, e[0], gb * be[0]));
  du[1] = k * cross<1>(f, b, vfma(bdot, e[1], gb * be[1]));
  du[2] = k * cross<2>(f, b, vfma(bdot, e[2], gb * be[2]));
  const R dn2 = dot3(du, du), ul2 = dot3(ul, ul);
  R lim = one;
  if (dn2 > R(0.25) * ul2) lim = R(0.5) * rsq(dn2 * rcp(ul2));
#pragma unroll
  for (int q = 0; q < 3; ++q) out[q] = vfma(lim, du[q], ul[q]);
  const R gl = one + ul2, go = dot3(out, out, one), rgo = rsq(go);
  dgam = vfma(gl, rsq(gl), -(go * rgo));
  return rgo;
}

// Straight-line move x' = x + (u/gamma) c dt in the local Cartesian frame at
// azimuth 0; the azimuthal displacement is rotated away (axisymmetry) and u
// re-expressed in the basis of the new point.  Increments only, no
// subtraction of absolute radii.  General form (any displacement).
template <typename R>
__device__ __forceinline__ void move_general(R r, R sn, R cs, R dt, const R u[3], R &dr, R &dth, R uo[3]) {
  const R ig = dt / sqrt(R(1) + u[0] * u[0] + u[1] * u[1] + u[2] * u[2]);
  const R d0 = u[0] * ig, d1 = u[1] * ig, d2 = u[2] * ig;
  const R x = (r + d0) * sn + d1 * cs;
  const R rc = sqrt(x * x + d2 * d2);
  const R dR = (x > R(0)) ? d2 * d2 / (rc + x) : rc - x;
  const R pa = d0 + dR * sn;
  const R a = r + pa, bb = d1 + dR * cs;
  const R rnew = sqrt(a * a + bb * bb);
  dr = (pa * (R(2) * r + pa) + bb * bb) / (rnew + r);
  const R al = atan2(bb, a);
  const R ph = atan2(d2, x);
  dth = al;
  const R uR = u[0] * sn + u[1] * cs;
  R sp, cp, sa, ca;
  sincos(ph, &sp, &cp);
  sincos(al, &sa, &ca);
  const R s1 = sn * ca + cs * sa, c1 = cs * ca - sn * sa;  // angle of the new point
  const R h = sin(R(0.5) * ph);
  const R duR = uR * (R(-2) * h * h) + u[2] * sp;
  uo[0] = u[0] * ca + u[1] * sa + duR * s1;
  uo[1] = -u[0] * sa + u[1] * ca + duR * c1;
  uo[2] = -uR * sp + u[2] * cp;
}

// The same move for the usual case of a displacement much smaller than the
// distance to the axis (|d_phi| < 0.03 X and |b| < 0.03 a), where both
// rotation angles are small: with t = tan(angle) and q = t^2, 1 - cos and
// sqrt(1 + q) - 1 are short series in q and sin = t cos.  xr = dr / r.
// A displacement that is not small takes the general form; `small` says that
// no particle of the tile can have one (see TileFacts).
template <typename R>
__device__ __forceinline__ void move(bool small, R r, R sn, R cs, R ginv, R dt, const R u[3], R &xr, R &dth, R uo[3]) {
  using P = Series<R>;
  const R one = R(1), ig = dt * ginv;
  const R d0 = u[0] * ig, d1 = u[1] * ig, d2 = u[2] * ig;
  const R x = vfma(r + d0, sn, d1 * cs);
  const R tp = d2 * rcp(x), qp = tp * tp;
  const R omc = qp * P::omc(qp), cp = one - omc, sp = tp * cp;   // 1 - cos, cos and sin of phi
  const R dR = x * (qp * P::sqm(qp));                             // sqrt(x^2 + d2^2) - x
  const R pa = vfma(dR, sn, d0), bb = vfma(dR, cs, d1), a = r + pa;
  const R ta = bb * rcp(a), qa = ta * ta;
  const R ca = vfma(-qa, P::omc(qa), one), sa = ta * ca;
  // dr = (pa (2 r + pa) + b^2) / (r' + r) with r' = a sqrt(1 + q)
  const R ar = a + r, den = r * vfma(a, qa * P::sqm(qa), ar);
  xr = vfma(pa, ar, bb * bb) * rcp(den);
  dth = ta * P::atanc(qa);
  const R uR = vfma(u[0], sn, u[1] * cs);
  const R s1 = vfma(sn, ca, cs * sa), c1 = vfma(cs, ca, -(sn * sa));
  const R duR = vfma(u[2], sp, -(uR * omc));
  uo[0] = vfma(duR, s1, vfma(u[0], ca, u[1] * sa));
  uo[1] = vfma(duR, c1, vfma(-u[0], sa, u[1] * ca));
  uo[2] = vfma(u[2], cp, -(uR * sp));
  if (small || (well_below(d2, x) && well_below(bb, a))) return;
  R dr;
  move_general<R>(r, sn, cs, dt, u, dr, dth, uo);
  xr = dr / r;
}

// ----------------------------------------------------------------- deposit
// Charge-conserving deposit for linear shapes (Esirkepov decomposition) in
// the logical (xi, eta) plane.  (x0, y0) in [0,1) is the start offset in cell
// (i0, j0) and (X1, Y1) the end point relative to node (i0, j0), in (-1, 2).
// With S0, S1 the start and end weights on the nodes and dS = S1 - S0, the
// charge through the radial dual face between nodes a and a+1 in row b is
// -q (dS_x[0] + .. + dS_x[a]) (S0_y[b] + S1_y[b]) / 2, and likewise in theta;
// J_ph uses the mid-point weights.  For linear weights and a move of less
// than a cell this has a closed form.  With Xc = X1 clamped to [0, 1], the
// flux is x0 - Xc through the face of the start cell and Xc - X1 through the
// face of the cell entered (if any); the mean weights are 1 - m - max(h, 0) and
// m + min(h, 0) on the start cell's nodes, with m = (x0 + Xc) / 2 and
// h = (Xc - X1) / 2, and |h| on the far node of the cell entered.
// The accumulators hold raw charge fluxes (charge x velocity for J_ph); the
// collection (collect.cuh) applies the face areas, node volumes and dt.
//
// FP32: one 32-byte record per cell,
//   [J_r(i+1/2; j, j+1) | J_th(j+1/2; i, i+1) | J_ph(i,j; i,j+1; i+1,j; i+1,j+1)],
// so that a particle that stays in its cell (most do: a step moves it by at
// most half of the innermost cell) deposits with two 16-byte vector
// reductions performed by the L2, and a crossing adds one more per cell
// entered.  Nothing waits for them.  FP32 adds in shared memory are compiled
// to retry loops (load, add, compare-and-swap, test) and cost a third of the
// push's issue slots.  Measured alone, in ns per 1000 particles: two vector
// reductions 10.7 (random cells of a tile) to 11.9 (consecutive particles in
// one cell), eight shared adds 11.8 and 140; eight scalar reductions 51.
__device__ __forceinline__ void red_add4(float *p, float a, float b, float c, float d) {
  asm volatile("red.relaxed.gpu.global.add.v4.f32 [%0], {%1, %2, %3, %4};" ::"l"(p), "f"(a), "f"(b), "f"(c), "f"(d)
               : "memory");
}
// FP64: three arrays of (nr+2) x (nt+2) values (the window of a particle next
// to the outer walls reaches one past the mesh), one scalar reduction each;
// the L2 adds, not the SM, whose FP64 pipe bounds the FP64 push.
__device__ __forceinline__ int64_t acc_index(const Params<float> &p, int i, int j) { return 8 * ix(i, j, p.nt + 1); }
__device__ __forceinline__ int64_t acc_index(const Params<double> &p, int i, int j) { return ix(i, j, p.nt + 2); }
// Where a particle deposits: the mesh's accumulators (FP32 and FP64), or, in
// crowded work items (FP32, see push_item), the block's own records of the
// tile's region, and then summed by cell within the warp first where `share`.
template <typename R>
struct MeshAcc {
  static constexpr bool kShare = false;
  const Params<R> &p;
  __device__ __forceinline__ R *at(int i, int j) const { return p.jacc + acc_index(p, i, j); }
};
struct TileAcc {
  static constexpr bool kShare = true;
  float *base;
  int i0, j0, ld;
  bool share;
  __device__ __forceinline__ float *at(int i, int j) const { return base + 8 * ix(i - i0, j - j0, ld); }
};
// fluxes of one cell: J_r through its radial face at its two nodes, J_th
// through its polar face at its two nodes
template <typename A>
__device__ __forceinline__ void add_faces(const Params<float> &, const A &acc, int i, int j, float r0, float r1,
                                          float t0, float t1) {
  red_add4(acc.at(i, j), r0, r1, t0, t1);
}
template <typename A>
__device__ __forceinline__ void add_faces(const Params<double> &p, const A &acc, int i, int j, double r0, double r1,
                                          double t0, double t1) {
  const int ld = p.nt + 2;
  double *q = acc.at(i, j), *t = q + (int64_t)(p.nr + 2) * ld;
  atomicAdd(q, r0); atomicAdd(q + 1, r1);
  atomicAdd(t, t0); atomicAdd(t + ld, t1);
}
template <typename A>
__device__ __forceinline__ void add_corners(const Params<float> &, const A &acc, int i, int j, float a, float b,
                                            float c, float d) {
  red_add4(acc.at(i, j) + 4, a, b, c, d);
}
template <typename A>
__device__ __forceinline__ void add_corners(const Params<double> &p, const A &acc, int i, int j, double a, double b,
                                            double c, double d) {
  const int ld = p.nt + 2;
  double *q = acc.at(i, j) + 2 * (int64_t)(p.nr + 2) * ld;
  atomicAdd(q, a); atomicAdd(q + 1, b); atomicAdd(q + ld, c); atomicAdd(q + ld + 1, d);
}

// Items whose particles fill few cells: lanes of a warp that deposit into the
// same cell are summed first, wherever they sit in the warp, and one of them
// issues the reduction.  The record of a full cell then sees a tenth of the
// additions: fewer in the L2's queue, and a shorter chain of FP32 roundings
// (3,300 equal contributions added one by one lose 3e-5 of their sum, in the
// L2 as in any FP32 accumulator).  The sums are the tree reduction by key of
// E. Westphal ("Voting and Shuffling to Optimize Atomic Operations", NVIDIA
// developer blog, 2015).  Decided once per work item, from sampled pairs of
// particles kShareDist apart: equal cells there mean more particles in a cell
// than an accumulator should take singly; elsewhere the reductions are cheaper
// alone (2e7 particles in cell order, ten to a cell, on 2048^2: push 0.53 ms
// alone, 0.60 summed), and left out where fewer than kShareMin lanes of the
// warp share.
constexpr int kShareMin = 4;
constexpr int kShareDist = 64;
constexpr int kShareItemMin = 16;  // equal cells among 256 sampled pairs of a work item
// returns whether this lane issues the (summed) values
template <int N>
__device__ __forceinline__ bool sum_by_cell(int key, float (&v)[N]) {
  const unsigned act = __activemask(), peers = __match_any_sync(act, key);
  const unsigned sharing = __ballot_sync(act, (peers & (peers - 1)) != 0);
  if (__popc(sharing) < kShareMin) return true;  // the same decision in every lane of act
  const int lane = threadIdx.x & 31;
  const unsigned below = (1u << lane) - 1u;
  unsigned rest = peers & ~below & ~(1u << lane);   // members after this lane still holding a partial sum
  int rank = __popc(peers & below);
  const bool first = rank == 0;
  while (__any_sync(act, rest != 0)) {
    const int next = __ffs(rest);
#pragma unroll
    for (int k = 0; k < N; ++k) {
      const float y = __shfl_sync(act, v[k], next ? next - 1 : lane);
      if (next) v[k] += y;
    }
    // members of odd rank have been taken; the others meet the next of theirs
    rest &= __ballot_sync(act, (rank & 1) == 0);
    rank >>= 1;
  }
  return first;
}
__device__ __forceinline__ void add_faces_shared(const Params<float> &p, const TileAcc &acc, int i, int j, float r0,
                                                 float r1, float t0, float t1) {
  float v[4] = {r0, r1, t0, t1};
  if (!acc.share || sum_by_cell((int)ix(i, j, p.nt + 1), v)) add_faces(p, acc, i, j, v[0], v[1], v[2], v[3]);
}

// sx, sy: the cell entered in either direction (-1, 0, 1)
template <typename R, typename A>
__device__ __forceinline__ void deposit(const Params<R> &p, const A &acc, R qw, int i, int j, int sx, int sy, R x0, R y0,
                                        R X1, R Y1, R vphi) {
  const R nq = -qw;
  R gx = nq * (x0 - X1), gy = nq * (y0 - Y1);
  R mx1 = R(0.5) * (x0 + X1), my1 = R(0.5) * (y0 + Y1), mx0 = R(1) - mx1, my0 = R(1) - my1;
  R wx = mx1, wy = my1;          // J_ph: mid-point weights in the cell (ic, jc)
  int ic = i, jc = j;
  if ((sx | sy) != 0) {
    const R Xc = sx == 0 ? X1 : (sx < 0 ? R(0) : R(1)), Yc = sy == 0 ? Y1 : (sy < 0 ? R(0) : R(1));
    const R hx = R(0.5) * (Xc - X1), hy = R(0.5) * (Yc - Y1);
    const R ax0 = sx < 0 ? hx : R(0), ax1 = sx > 0 ? -hx : R(0);   // far-node weights of the cell entered
    const R ay0 = sy < 0 ? hy : R(0), ay1 = sy > 0 ? -hy : R(0);
    const R gxo = nq * (Xc - X1), gyo = nq * (Yc - Y1);
    const R mxc = R(0.5) * (x0 + Xc), myc = R(0.5) * (y0 + Yc);
    gx = nq * (x0 - Xc); gy = nq * (y0 - Yc);
    mx0 = R(1) - mxc - ax0; mx1 = mxc - ax1; my0 = R(1) - myc - ay0; my1 = myc - ay1;
    if constexpr (A::kShare) {
      if (sx) add_faces_shared(p, acc, i + sx, j, gxo * my0, gxo * my1, gy * ax0, gy * ax1);
      if (sy) add_faces_shared(p, acc, i, j + sy, gx * ay0, gx * ay1, gyo * mx0, gyo * mx1);
      if (sx && sy) add_faces_shared(p, acc, i + sx, j + sy, gxo * ay0, gxo * ay1, gyo * ax0, gyo * ax1);
    } else {
      if (sx) add_faces(p, acc, i + sx, j, gxo * my0, gxo * my1, gy * ax0, gy * ax1);
      if (sy) add_faces(p, acc, i, j + sy, gx * ay0, gx * ay1, gyo * mx0, gyo * mx1);
      if (sx && sy) add_faces(p, acc, i + sx, j + sy, gxo * ay0, gxo * ay1, gyo * ax0, gyo * ax1);
    }
    if (sx && (below_zero(wx) || at_least(wx, R(1)))) { ic += sx; wx -= R(sx); }
    if (sy && (below_zero(wy) || at_least(wy, R(1)))) { jc += sy; wy -= R(sy); }
  }
  const R qv = qw * vphi, a1 = qv * wx, a0 = qv - a1, a01 = a0 * wy, a11 = a1 * wy;
  if constexpr (A::kShare) {
    if (acc.share) {
      float v[8] = {gx * my0, gx * my1, gy * mx0, gy * mx1, a0 - a01, a01, a1 - a11, a11};
      if (ic != i || jc != j) {   // mid-point in the cell entered: on its own
        add_corners(p, acc, ic, jc, v[4], v[5], v[6], v[7]);
        v[4] = v[5] = v[6] = v[7] = 0.f;
      }
      if (sum_by_cell(i * p.nt + j, v)) {
        add_faces(p, acc, i, j, v[0], v[1], v[2], v[3]);
        add_corners(p, acc, i, j, v[4], v[5], v[6], v[7]);
      }
      return;
    }
  }
  add_faces(p, acc, i, j, gx * my0, gx * my1, gy * mx0, gy * mx1);
  add_corners(p, acc, ic, jc, a0 - a01, a01, a1 - a11, a11);
}

template <typename R> __device__ __forceinline__ R one_minus_ulp();
template <> __device__ __forceinline__ float one_minus_ulp<float>() { return 0.99999994f; }
template <> __device__ __forceinline__ double one_minus_ulp<double>() { return 0.99999999999999989; }

// per-thread counters in the working precision (FP64 only in the warp and
// global sums)
template <typename R>
struct Tally {
  R killed, radiated;
  unsigned nonfinite;
  unsigned pushed;
  __device__ __forceinline__ void add(const Tally &t) {
    killed += t.killed; radiated += t.radiated;
    nonfinite += t.nonfinite; pushed += t.pushed;
  }
};

// per-species constants of a push, loaded once per work item.  The arrays
// read (in) and written (out) are the same, except in the first push after a
// sort, which reads the unsorted parity through the sorted order sidx.  xo,
// yo, ur, ut, up, w of a species lie p.pstride elements apart, so that one
// address serves all six.
template <typename R>
struct SpeciesConst {
  const int32_t *cell_in;
  int32_t *cell_out;
  const R *x_in;
  R *x_out;
  int64_t stride;
  const uint32_t *sidx;
  R qm, krr, q, m;
  uint32_t key_hi;   // species in the top bit of a pair-creation event key
  bool creates;      // a lepton of a run with pair creation
  __device__ __forceinline__ SpeciesConst(const Params<R> &p, int s, bool gather = false)
      : cell_in(gather ? p.src[s].cell : p.sp[s].cell), cell_out(p.sp[s].cell), x_in(gather ? p.src[s].xo : p.sp[s].xo),
        x_out(p.sp[s].xo), stride(p.pstride), sidx(p.sidx[s]), qm(p.qm[s]), krr(p.krr[s] * (R)(*p.rr_scale)), q(p.q[s]),
        m(p.m[s]), key_hi((uint32_t)s << 31), creates(p.pairs != 0 && s < 2) {}
  __device__ __forceinline__ R in(int k, int q) const { return x_in[q + k * stride]; }
  __device__ __forceinline__ R &out(int k, int q) const { return x_out[q + k * stride]; }
};

// Sect. 5.1: a lepton above the threshold Lorentz factor creates a pair at
// its new position, along its direction of motion, with gamma_s.  Recorded
// as an event here (slot order of the atomic is arbitrary; the key restores
// the parent order when the pairs are appended).
template <typename R>
__device__ __forceinline__ void record_pair(const Params<R> &p, const SpeciesConst<R> &K, int q, int cell, R xn,
                                            R yn, const R uo[3], R w) {
  const R u2 = uo[0] * uo[0] + uo[1] * uo[1] + uo[2] * uo[2];
  if (!(R(1) + u2 > p.gamma_th2)) return;
  const unsigned e = atomicAdd(p.pe_count, 1u);
  if ((int64_t)e >= p.pe_cap) { atomicOr(p.status, kStCapacity); return; }
  const R a = p.u_s * rsq(u2);
  p.ev_key[e] = K.key_hi | (uint32_t)q;
  p.ev_cell[e] = cell;
  p.ev_xo[e] = xn; p.ev_yo[e] = yn;
  p.ev_ur[e] = a * uo[0]; p.ev_ut[e] = a * uo[1]; p.ev_up[e] = a * uo[2];
  p.ev_w[e] = w;
}

// What holds for every particle of a work item (or, outside the tiles, what
// cannot be assumed), so that most particles skip the tests:
//   small  a step's displacement is small against the distance to the axis:
//          |d_phi|, |b| <= dt < 0.028 (r sin(theta) - 2 dt) over the region;
//   shell  some may lie inside shell_r;
//   edge   some may reach a wall, the axis or the absorber.
struct TileFacts {
  bool small, shell, edge;
};

// One particle in cell (i, j): gather, push, move, kill rules, deposit, and
// its new state in slot q (the slot it came from, unless the push also
// performs a sort's payload gather, kGather, which writes w too).
template <typename R, bool kGather, typename M, typename A>
__device__ __forceinline__ void push_one(const M &m, const A &acc, const TileFacts &F, const Params<R> &p, const SpeciesConst<R> &K,
                                         int q, int i, int j, R xo, R yo, R w, const R u[3], Tally<R> &tl) {
  using P = Series<R>;
  const int nt = p.nt;
  R e[3], b[3], un[3], uo[3], dg;
  gather(m, i, j, xo, yo, e, b);
  R ginv = boris_rr<R>(K.qm, K.krr, p.dt, u, e, b, un, dg);
  tl.pushed += 1;
  if (K.krr != R(0)) tl.radiated += w * K.m * dg;
  // position of the particle: r = r_i exp(xo D), theta = theta_j + yo dtheta
  const R xl = xo * p.dlog, ya = yo * p.dth;
  R ex, sa0, ca0;
  if (p.small_grid) {
    const R y2 = ya * ya;
    sa0 = ya * P::sinc(y2);
    ca0 = vfma(y2, P::cosm(y2), R(1));
    ex = vfma(xl, P::expm1c(xl), R(1));
  } else {
    sincos(ya, &sa0, &ca0);
    ex = exp(xl);
  }
  const R r = m.rn(i) * ex, snj = m.sn(j), cnj = m.cn(j);
  const R sn = vfma(snj, ca0, cnj * sa0), cs = vfma(cnj, ca0, -(snj * sa0));
  if (F.shell && r * r < p.shell_r2) {  // Sect. 5.1: no momentum across B near the star
    const R b2 = dot3(b, b);
    if (b2 > R(1e-30)) {
      const R ub = dot3(un, b) * rcp(b2);
#pragma unroll
      for (int k = 0; k < 3; ++k) un[k] = ub * b[k];
      ginv = rsq(dot3(un, un, R(1)));
    }
  }
  R xr, dth;
  move<R>(F.small, r, sn, cs, ginv, p.dt, un, xr, dth, uo);
  const R lg = (F.small || !at_least(fabs(xr), R(0.03125))) ? xr * P::log1pc(xr) : R(log1p(xr));
  R X1 = vfma(lg, p.inv_dlog, xo), Y1 = vfma(dth, p.inv_dth, yo);
  if (!all_finite(X1, Y1, uo)) {
    K.cell_out[q] = -1;
    tl.nonfinite += 1;
    return;
  }
  bool dead = F.edge && i >= p.i_abs && R(i) + X1 > p.xi_abs;
  int sx = 0, sy = 0, i1 = i, j1 = j;
  R xn = X1, yn = Y1;
  // A step moves a particle by less than a cell in either direction (Courant
  // number <= 0.9 at the innermost cells, the smallest; at most 0.965 cells
  // over all grids with nt >= 8), so the entered cell is a neighbour.
  if (!(stays(X1) && stays(Y1))) {
    bool lo = below_zero(X1), yl = below_zero(Y1), yh = at_least(Y1, R(1));
    const bool hi = at_least(X1, R(1));
    if (F.edge) {
      if (j == 0 && yl) { Y1 = -Y1; yl = false; }
      if (j == nt - 1 && yh && Y1 > R(1)) { Y1 = R(2) - Y1; yh = false; }
      if (i == 0 && lo) { X1 = R(0); lo = false; dead = true; }
    }
    sx = lo ? -1 : (hi ? 1 : 0);
    sy = yl ? -1 : (yh ? 1 : 0);
    xn = X1 - R(sx);
    yn = Y1 - R(sy);
    // a tiny step below the node, rounded back to it, stays in the cell
    if (lo && at_least(xn, R(1))) { xn = R(0); sx = 0; }
    if (yl && at_least(yn, R(1))) { yn = R(0); sy = 0; }
    i1 += sx;
    j1 += sy;
    if (j1 >= nt) { j1 = nt - 1; yn = one_minus_ulp<R>(); sy = 0; }
    // the deposit ends where the particle is stored (its offset was rounded
    // on the way down; these sums are exact), or Gauss's law would drift
    X1 = xn + R(sx);
    Y1 = yn + R(sy);
  }
  // off the mesh (no absorber), or force-free
  if (!dead) dead = (F.edge && i1 >= p.nr) || m.ff(i1, j1);
  deposit<R>(p, acc, K.q * w, i, j, sx, sy, xo, yo, X1, Y1, un[2] * ginv);
  if (dead) {
    K.cell_out[q] = -1;
    tl.killed += w;
    return;
  }
  K.cell_out[q] = i1 * nt + j1;
  K.out(0, q) = xn; K.out(1, q) = yn;
  K.out(2, q) = uo[0]; K.out(3, q) = uo[1]; K.out(4, q) = uo[2];
  if constexpr (kGather) K.out(5, q) = w;
  if (F.edge && i1 == 0 && p.inject) atomicAdd(&p.surf[j1], 1);
  if (K.creates) record_pair(p, K, q, i1 * nt + j1, xn, yn, uo, w);
}

// one particle outside the tiles (appended since the sort, drifted out of the
// staged region, or the no-sort configuration).  It returns its counts by
// value and takes the species index rather than the species constants:
// arguments passed by reference to an out-of-line call would have to live
// in local memory for the whole work item.
template <typename R, bool kGather>
__device__ __noinline__ Tally<R> push_one_global(const Params<R> &p, int s, int slot, int from, int cell) {
  const SpeciesConst<R> K(p, s, kGather);
  GlobalMesh<R> g(p);
  Tally<R> tl{R(0), R(0), 0u, 0u};
  int i, j;
  decode_cell(p, cell, i, j);
  const R u[3] = {K.in(2, from), K.in(3, from), K.in(4, from)};
  push_one<R, kGather>(g, MeshAcc<R>{p}, TileFacts{false, true, true}, p, K, slot, i, j, K.in(0, from), K.in(1, from), K.in(5, from), u, tl);
  return tl;
}

template <typename R>
__device__ __forceinline__ void flush_tally(const Tally<R> &tl, const Tally<R> &tail, double *acc, unsigned *status,
                                            unsigned long long *pushed) {
  // FP64 only for the warp and global sums
  double k = (double)tl.killed + (double)tail.killed, r = (double)tl.radiated + (double)tail.radiated;
  unsigned nf = tl.nonfinite + tail.nonfinite, np = tl.pushed, nt = tail.pushed;
  for (int o = 16; o > 0; o >>= 1) {
    k += __shfl_down_sync(0xffffffffu, k, o);
    r += __shfl_down_sync(0xffffffffu, r, o);
    nf += __shfl_down_sync(0xffffffffu, nf, o);
    np += __shfl_down_sync(0xffffffffu, np, o);
    nt += __shfl_down_sync(0xffffffffu, nt, o);
  }
  if ((threadIdx.x & 31) == 0) {
    if (k != 0.0) atomicAdd(&acc[1], k);
    if (r != 0.0) atomicAdd(&acc[2], r);
    if (nf) { atomicAdd(&acc[3], (double)nf); atomicOr(status, kStNonfinite); }
    if (np) atomicAdd(&pushed[0], (unsigned long long)np);
    if (nt) atomicAdd(&pushed[1], (unsigned long long)nt);
  }
}

// ----------------------------------------------------------- tail kernel
// slots count_sorted .. count of every species, one list over the species, a
// warp at a time over the grid from its last block (which the tiled kernel
// gives a work item last): they wait on their own loads, so they are spread
// over the SMs.  With blocks of 256 of one species after the other, and every
// block taking its first work item from the queue, a step on 96 x 80 with
// 1.2e4 particles took 42.4 us, now 35.0; 500 x 380 with three species 143,
// now 138; 256 x 128 in FP64 187, now 182; 1024^2 with 5e7 1132, now 1124.
template <typename R>
__device__ __forceinline__ Tally<R> push_tail(const Params<R> &p) {
  Tally<R> tl{R(0), R(0), 0u, 0u};
  const int warps = blockDim.x >> 5, warp = threadIdx.x >> 5;
  for (int64_t g = ((int64_t)warp * gridDim.x + (gridDim.x - 1 - blockIdx.x)) * 32 + (threadIdx.x & 31);;
       g += (int64_t)gridDim.x * warps * 32) {
    int64_t q = g;
    int s = 0;
    for (; s < p.n_species; ++s) {
      const int64_t n0 = p.count_sorted[s], n = p.count[s] - n0;
      if (q < n) { q += n0; break; }
      q -= n > 0 ? n : 0;
    }
    if (s == p.n_species) break;
    const int c = p.sp[s].cell[q];
    if (c >= 0) tl.add(push_one_global<R, false>(p, s, (int)q, (int)q, c));
  }
  return tl;
}
template <typename R>
__global__ void __launch_bounds__(256) k_push_tail(const __grid_constant__ Params<R> p) {
  flush_tally(Tally<R>{R(0), R(0), 0u, 0u}, push_tail(p), p.acc, p.status, p.pushed);
}

// ---------------------------------------------------------- tiled kernel
static_assert(kPushThreads * 32 >= kMaxItem, "one bit per round of a work item");
// The next round's particles are copied to shared memory while this round's
// are pushed (one slot per thread and array, read back by the thread that
// copied it): the loads' latency, lengthened by the reductions in the L2's
// queues, was the largest stall, and registers have no room for them.
template <typename R>
struct Prefetch {
  R *slot;   // 7 arrays of kPushThreads slots (the first holds the cells)
  __device__ __forceinline__ void start(const SpeciesConst<R> &K, int q, bool any) const {
    if (any) {
      R *d = slot + threadIdx.x;
      copy_async<4>(d, K.cell_in + q);
      const R *a = K.x_in + q;
#pragma unroll
      for (int k = 1; k < 7; ++k, a += K.stride) copy_async<sizeof(R)>(d + k * kPushThreads, a);
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
  }
  __device__ __forceinline__ void wait() const { asm volatile("cp.async.wait_group 0;" ::: "memory"); }
  __device__ __forceinline__ int cell() const { return *reinterpret_cast<const int *>(slot + threadIdx.x); }
  __device__ __forceinline__ R get(int k) const { return slot[(k + 1) * kPushThreads + threadIdx.x]; }
};

// particles of slots q0 .. q1 of a work item, one per thread and round
template <typename R, bool kGather, typename A>
__device__ __forceinline__ void push_item(const SharedMesh<R> &m, const A &acc, const TileFacts &F, const Params<R> &p,
                                          const SpeciesConst<R> &K, const Prefetch<R> &pre, int s, int q0, int q1, int lr,
                                          Tally<R> &tl) {
  // rounds whose particle was left for the global path: an item has at most
  // kMaxItem particles, 32 rounds
  unsigned left = 0, bit = 1;
  for (int slot = q0 + (int)threadIdx.x; slot < q1; slot += kPushThreads, bit <<= 1) {
    int c;
    R x, y, w, u[3];
    if constexpr (kGather) {
      const int from = (int)K.sidx[slot];
      c = K.cell_in[from];
      if (c < 0) K.cell_out[slot] = -1;
      x = K.in(0, from); y = K.in(1, from); w = K.in(5, from);
      u[0] = K.in(2, from); u[1] = K.in(3, from); u[2] = K.in(4, from);
    } else {
      pre.wait();
      c = pre.cell();
      x = pre.get(0); y = pre.get(1); u[0] = pre.get(2); u[1] = pre.get(3); u[2] = pre.get(4); w = pre.get(5);
      pre.start(K, slot + kPushThreads, slot + kPushThreads < q1);
    }
    if (c < 0) continue;
    int i, j;
    decode_cell(p, c, i, j);
    // a particle is handled in shared memory when its gather stencil and the
    // cells it can reach (start cell -1 .. +1) lie inside the region
    if ((unsigned)(i - m.i0 - 1) < (unsigned)(lr - 2) && (unsigned)(j - m.j0 - 1) < (unsigned)(m.lt - 2))
      push_one<R, kGather>(m, acc, F, p, K, slot, i, j, x, y, w, u, tl);
    else
      left |= bit;
  }
  for (; left; left &= left - 1) {
    const int slot = q0 + (int)threadIdx.x + kPushThreads * (__ffs(left) - 1);
    const int from = kGather ? (int)K.sidx[slot] : slot;
    tl.add(push_one_global<R, kGather>(p, s, slot, from, K.cell_in[from]));
  }
}

// Crowded items (FP32).  An FP32 accumulator that takes the particles of a tile
// one by one, over all its work items, loses more of their sum than one that
// takes the sums of its items.  Relative error of J_r, against FP64, one by one
// and by items: momenta at random 4.8e-7 and 4.6e-7 at 24 particles per cell and
// species, 4.8 and 4.6 at 48, 5.3 and 4.8 at 100, 7.0 and 4.6 at 500, 14.4 and
// 4.8 at 3000; equal momenta 1.2e-7 and 1.1e-7, 1.3 and 0.9, 1.6 and 0.8, 3.6 and
// 0.8, 7.6 and 1.2.  So where an accumulator expects more than kCrowdMin
// additions, the item deposits into the block's own records of its region (in
// the sort's scratch: 20 to 30 KB, in the L2), which it adds to the mesh's at
// its end.  What an accumulator expects is the tile's particles (all species; kept
// in the list by the sort) times the chance that two particles of the item share
// a cell, taken from how many sampled ones meet their like within their warp.
// The push of 5e7 particles on 1024^2, 177 to a cell, takes 1.08 ms so and 1.02
// one by one; 3e8 on 4096^2, where the current sheet (a fifth) is crowded and
// the rest has 68 to a cell, 6.39 and 6.22 ms, and 6.75 with a limit of 64 (the
// reductions at the end of an item are as many as those of 500 particles).
constexpr float kCrowdMin = 96.f;
constexpr float kCrowdItem = 4.f;
// place of thread t's sample among the 256: a fixed permutation without pattern
__device__ __forceinline__ int sample_place(int t) {
  t = (t * 167 + 13) & 255;
  t ^= t >> 4;
  t = (t * 89 + 71) & 255;
  return t ^ (t >> 3);
}
// met: sampled particles that share their cell with another one of their warp's,
// in two samples of up to 256 (fewer in an item of w < 320 particles); n:
// particles of the tile.  An item that itself brings an accumulator fewer than
// kCrowdItem particles does without: its sums would be hardly fewer additions
// than its particles, and cost as much.
__device__ __forceinline__ bool crowded(int met, int w, int n) {
  const int lanes = min(kPushThreads, w - kShareDist) / 8;   // sampled per warp
  if (lanes < 2) return false;
  const float got = (float)met / (float)(16 * lanes);        // chance to meet one's like among lanes - 1
  auto chance = [&](float c) { return c < 1.f ? 1.f - exp2f((float)(lanes - 1) * log2f(1.f - c)) : 2.f; };
  return got > chance(max(kCrowdMin / (float)max(n, 1), kCrowdItem / (float)w));
}
// A block's first crowded item: one of the sets of records (n floats each),
// cleared (they lie in the sort's scratch).  A small instance may have fewer
// sets than blocks; a block that finds none left deposits into the mesh's.
__device__ __noinline__ void claim_records(float *records, int sets, int *claimed, int n, int *which) {
  __syncthreads();   // *which has been read by all
  if (threadIdx.x == 0) {
    const int k = atomicAdd(claimed, 1);
    *which = k < sets ? k : -2;
  }
  __syncthreads();
  if (*which < 0) return;
  float4 *rec = reinterpret_cast<float4 *>(records + (int64_t)*which * n);
  for (int k = threadIdx.x; k < n / 4; k += kPushThreads) __stcg(rec + k, make_float4(0.f, 0.f, 0.f, 0.f));
  __syncthreads();   // before any thread's reductions
}
// the block's records of the region added to the mesh's, and cleared
__device__ __forceinline__ void flush_records(const Params<float> &p, const TileAcc &t, int lr) {
  const float4 z = make_float4(0.f, 0.f, 0.f, 0.f);
  __syncthreads();   // every thread's reductions are visible to the block
  for (int k = threadIdx.x; k < lr * t.ld; k += kPushThreads) {
    float4 *rec = reinterpret_cast<float4 *>(t.base + 8 * k);
    const float4 a = __ldcg(rec), c = __ldcg(rec + 1);
    const int r = k / t.ld, i = t.i0 + r, j = t.j0 + k - r * t.ld;
    if (i < 0 || j < 0 || i > p.nr || j > p.nt) continue;   // never deposited into
    float *q = p.jacc + acc_index(p, i, j);
    if (a.x != 0.f || a.y != 0.f || a.z != 0.f || a.w != 0.f) { __stcg(rec, z); red_add4(q, a.x, a.y, a.z, a.w); }
    if (c.x != 0.f || c.y != 0.f || c.z != 0.f || c.w != 0.f) { __stcg(rec + 1, z); red_add4(q + 4, c.x, c.y, c.z, c.w); }
  }
}

// Order of the work items: the list is by species and tile, so a tile with
// many particles (the current sheet: 36 items on the 1024^2 workload) would
// be pushed by many blocks at once, whose reductions then queue at the few
// records of its cells.  Within windows of kOrderWindow items an odd stride
// (a permutation of the window) spreads them; the window keeps the tiles at
// work, and their fields in the L2, close together.  Push of 5e7 particles on
// 1024^2: 1.07 ms in list order, 1.03 with 2048 or 4096, 1.05 unlimited.
constexpr int kOrderWindow = 2048, kOrderStride = 1013;
__device__ __forceinline__ int item_order(int it, int n) {
  const int w = it & ~(kOrderWindow - 1);
  return w + kOrderWindow <= n ? w + ((it * kOrderStride) & (kOrderWindow - 1)) : it;
}

// Region of a tile: cells [ti*TR - H, ti*TR + TR + H) (and likewise in theta)
// widened by the gather's stencil: one node on either side.
// Blocks of 256 per SM, measured on 2e7 FP32 particles (2048^2) and 4.6e6
// FP64 ones (512^2): FP32 with 3, 4, 5 blocks (80, 64, 48 registers) 0.486,
// 0.478, 0.53 ms; FP64 with 2, 3 (128, 80 registers) 2.93, 2.98 ms.
template <typename R> constexpr int push_tiled_min_blocks() { return sizeof(R) == 4 ? 4 : 2; }
template <typename R, bool kGather>
__global__ void __launch_bounds__(kPushThreads, push_tiled_min_blocks<R>())
    k_push_tiled(const __grid_constant__ Params<R> p, WorkList wl, int halo) {
  extern __shared__ __align__(16) unsigned char smem[];
  const int lrm = p.tile_r + 2 * halo + 2, ltm = p.tile_t + 2 * halo + 2;   // the largest region
  SharedMesh<R> m;
  Prefetch<R> pre;
  pre.slot = reinterpret_cast<R *>(smem);
  m.s_rn = reinterpret_cast<R *>(m.carve(smem + 7 * kPushThreads * sizeof(R), lrm * ltm));
  m.s_sn = m.s_rn + lrm; m.s_cn = m.s_sn + ltm;
  m.s_ff = reinterpret_cast<uint8_t *>(m.s_cn + ltm);
  __shared__ int s_item, s_records;   // which records are the block's (-1: none yet, -2: none left)
  if (threadIdx.x == 0) s_records = -1;   // read behind the first staging's barrier
  const int nr = p.nr, nt = p.nt, n1 = nt + 1;
  Tally<R> tl{R(0), R(0), 0u, 0u};
  const int ni = *wl.n_items;
  for (int it = blockIdx.x; it < ni;) {   // the first item by block, later ones from the queue
    const int4 item = wl.items[item_order(it, ni)];
    const int s = item.x & 3, tile = item.y;
    const int ti = tile / p.ntt, tj = tile - ti * p.ntt;
    // a step's drift in cells falls like 1 / r (or faster), and so does the halo
    // (particles beyond it would take the global path)
    const int hl = min(halo, (int)ceil((R)halo * p.r_min / p.t.rn[max(ti * p.tile_r - halo, 0)]));
    const int lr = p.tile_r + 2 * hl + 2, lt = p.tile_t + 2 * hl + 2, area = lr * lt;
    m.i0 = ti * p.tile_r - hl - 1;
    m.j0 = tj * p.tile_t - hl - 1;
    m.lt = lt;
    const SpeciesConst<R> K(p, s, kGather);
    int ca = -1, cb = -2;   // cells of a sampled pair of particles (read here, behind the staging too)
    if constexpr (sizeof(R) == 4) {
      const int qa = item.z + kShareDist + sample_place(threadIdx.x) * max(1, (item.w - kShareDist) / kPushThreads);
      if (qa < item.z + item.w) {
        ca = K.cell_in[kGather ? (int)K.sidx[qa] : qa];
        cb = K.cell_in[kGather ? (int)K.sidx[qa - kShareDist] : qa - kShareDist];
      }
    }
    if constexpr (!kGather)   // the first round's particles, behind the staging
      pre.start(K, item.z + (int)threadIdx.x, (int)threadIdx.x < item.w);
    // stage E, B, flags (edge values replicated outside each array)
    for (int k = threadIdx.x; k < area; k += blockDim.x) {
      const int a = k / lt, c = k - a * lt;
      const int gi = m.i0 + a, gj = m.j0 + c;
      const int in = min(max(gi, 0), nr), ih = min(max(gi, 0), nr - 1);   // node / half rows
      const int jn = min(max(gj, 0), nt), jh = min(max(gj, 0), nt - 1);   // node / half columns
      const int64_t kb = ix(in, jh, nt), kt = ix(ih, jn, n1), kp = ix(ih, jh, nt), kn = ix(in, jn, n1);
      m.put(k, c, p.f.er[kt], p.f.et[kb], p.f.ep[kn], p.f.br0[kb] + p.f.br[kb],   // B = B_0 + dB
            p.f.bt0[kt] + p.f.bt[kt], p.f.bp0[kp] + p.f.bp[kp]);
      m.s_ff[k] = (gi >= 0 && gj >= 0 && gi < nr && gj < nt) ? p.f.ffcell[ix(gi, gj, nt)] : 1;
    }
    for (int k = threadIdx.x; k < lr; k += blockDim.x) {
      const int gi = m.i0 + k;
      m.s_rn[k] = (gi >= 0 && gi <= nr) ? p.t.rn[gi] : R(1);
    }
    for (int k = threadIdx.x; k < lt; k += blockDim.x) {
      const int gj = m.j0 + k;
      m.s_sn[k] = (gj >= 0 && gj <= nt) ? p.t.sn[gj] : R(0);
      m.s_cn[k] = (gj >= 0 && gj <= nt) ? p.t.cn[gj] : R(1);
    }
    TileFacts F;
    // many particles in few cells?  (the barrier also completes the staged region)
    const bool share = __syncthreads_count(ca == cb && ca >= 0) >= kShareItemMin;
    {
      // over the region's nodes inside the mesh
      const int ra = max(m.i0, 0), rb = min(m.i0 + lr, nr), ca = max(m.j0, 0), cb = min(m.j0 + lt - 1, nt);
      const R r0 = p.t.rn[ra], sm = min(p.t.sn[ca], p.t.sn[cb]);
      F.small = p.dt < R(0.028) * (r0 * sm - R(2) * p.dt);
      F.shell = r0 * r0 < p.shell_r2 * R(1.001);
      F.edge = ra == 0 || rb == nr || ca == 0 || cb == nt || rb >= p.i_abs;
    }
    bool plain = true;
    if constexpr (sizeof(R) == 4) {
      bool own = item.x & kItemOwn;
      if (!(item.x & (kItemDirect | kItemOwn))) {   // the list's first push decides for the later ones
        const unsigned pa = __match_any_sync(0xffffffffu, ca >= 0 ? ca : -1 - (int)threadIdx.x);
        const unsigned pb = __match_any_sync(0xffffffffu, cb >= 0 ? cb : -1 - (int)threadIdx.x);
        const int met = __syncthreads_count((pa & (pa - 1)) != 0) + __syncthreads_count((pb & (pb - 1)) != 0);
        own = crowded(met, item.w, item.x / kItemTotal);
        if (threadIdx.x == 0) wl.items[item_order(it, ni)].x = item.x | (own ? kItemOwn : kItemDirect);
      }
      if (own && s_records == -1) claim_records(wl.records, wl.record_sets, wl.claimed, 8 * lrm * ltm, &s_records);
      own = own && s_records >= 0;
      plain = !own && !share;
      if (!plain) {
        const TileAcc t = own ? TileAcc{wl.records + (int64_t)s_records * (8 * lrm * ltm), m.i0, m.j0, lt, share}
                              : TileAcc{p.jacc, 0, 0, n1, share};
        push_item<R, kGather>(m, t, F, p, K, pre, s, item.z, item.z + item.w, lr, tl);
        if (own) flush_records(p, t, lr);
      }
    }
    if (plain) push_item<R, kGather>(m, MeshAcc<R>{p}, F, p, K, pre, s, item.z, item.z + item.w, lr, tl);
    if (threadIdx.x == 0) s_item = (int)gridDim.x + atomicAdd(wl.next, 1);
    __syncthreads();
    it = s_item;   // next written after the barrier behind the next staging
  }
  flush_tally(tl, push_tail(p), p.acc, p.status, p.pushed);
  // the last block to finish rewinds the work queue for the next push
  __syncthreads();
  if (threadIdx.x == 0 && atomicAdd(wl.done, 1) == (int)gridDim.x - 1) {
    *wl.next = 0;
    *wl.done = 0;
    if constexpr (sizeof(R) == 4) *wl.claimed = 0;
  }
}

template <typename R> size_t push_tiled_smem(int tile_r, int tile_t, int halo) {
  const size_t lr = tile_r + 2 * halo + 2, lt = tile_t + 2 * halo + 2, area = lr * lt;
  return 7 * kPushThreads * sizeof(R) + area * SharedMesh<R>::bytes_per_location() +
         (lr + 2 * lt) * sizeof(R);
}
template <typename R> size_t push_tiled_smem(const Params<R> &p, int halo) {
  return push_tiled_smem<R>(p.tile_r, p.tile_t, halo);
}

// what the records of a block's largest region take
size_t push_record_bytes(int tile_r, int tile_t, int halo) {
  return (size_t)(tile_r + 2 * halo + 2) * (tile_t + 2 * halo + 2) * 32;
}

// The tiles and cadences that hff_init accepts: those whose region, two
// cells wider than the gather needs and with nine values and a flag per
// location, fits 200 KB.  The kernel's own need is always below that.
template <typename R> bool push_tile_fits(const Params<R> &p, int halo) {
  const size_t lr = p.tile_r + 2 * halo + 4, lt = p.tile_t + 2 * halo + 4;
  return lr * lt * (9 * sizeof(R) + 1) + (lr + 2 * lt) * sizeof(R) <= 200 * 1024;
}

template <typename R>
__global__ void __launch_bounds__(kCollectThreads) k_collect(const __grid_constant__ Params<R> p) {
  collect_block(p, blockIdx.x, blockIdx.y);
}
template <typename R> void launch_collect(const Params<R> &p, cudaStream_t s) {
  k_collect<R><<<dim3(collect_blocks_x(p), collect_blocks_y(p)), kCollectThreads, 0, s>>>(p);
}
size_t push_acc_bytes(int nr, int nt, size_t real) {
  return real == 4 ? (size_t)(nr + 1) * (nt + 1) * 32 : (size_t)3 * (nr + 2) * (nt + 2) * 8;
}

template <typename R> void launch_push_tail(const Params<R> &p, cudaStream_t s, int grid) {
  k_push_tail<R><<<grid, 256, 0, s>>>(p);
}
template <typename R> void launch_push_tiled(const Params<R> &p, const WorkList &wl, int halo,
                                             cudaStream_t s, int grid, bool gather) {
  if (gather) k_push_tiled<R, true><<<grid, kPushThreads, push_tiled_smem(p, halo), s>>>(p, wl, halo);
  else k_push_tiled<R, false><<<grid, kPushThreads, push_tiled_smem(p, halo), s>>>(p, wl, halo);
}

// ------------------------------------------------------------- injection
// Top-up of each eligible surface cell to its target (fixed at init from
// kappa n_GJ V / w, Sects. 4 and 5.1): n_new(j) = max(0, target_j - surf_j/2)
// co-located pairs, offsets from Philox4x32-10 keyed (seed; step, j, k),
// corotating momentum, appended in (j, k) order.
__device__ __forceinline__ void philox4x32_10(uint32_t c[4], uint32_t k0, uint32_t k1) {
#pragma unroll
  for (int r = 0; r < 10; ++r) {
    const uint32_t lo0 = 0xD2511F53u * c[0], hi0 = __umulhi(0xD2511F53u, c[0]);
    const uint32_t lo1 = 0xCD9E8D57u * c[2], hi1 = __umulhi(0xCD9E8D57u, c[2]);
    const uint32_t n0 = hi1 ^ c[1] ^ k0, n2 = hi0 ^ c[3] ^ k1;
    c[0] = n0; c[1] = lo1; c[2] = n2; c[3] = lo0;
    k0 += 0x9E3779B9u;
    k1 += 0xBB67AE85u;
  }
}

// one block: exclusive scan of the per-cell counts, reserve slots
template <typename R>
__global__ void __launch_bounds__(1024) k_inject_scan(Params<R> p) {
  __shared__ int s_w[32];
  __shared__ int s_carry;
  const int nt = p.nt;
  if (threadIdx.x == 0) s_carry = 0;
  __syncthreads();
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  for (int seg = 0; seg < nt; seg += blockDim.x) {
    const int j = seg + threadIdx.x;
    int v = 0;
    if (j < nt) {
      const int need = p.target[j] - p.surf[j] / 2;
      v = need > 0 ? need : 0;
      p.surf[j] = 0;  // consumed: cleared for the next step
    }
    int x = v;
    for (int o = 1; o < 32; o <<= 1) {
      const int y = __shfl_up_sync(0xffffffffu, x, o);
      if (lane >= o) x += y;
    }
    if (lane == 31) s_w[wid] = x;
    __syncthreads();
    int off = s_carry;
    for (int w = 0; w < wid; ++w) off += s_w[w];
    if (j < nt) p.inj_prefix[j] = off + x - v;
    __syncthreads();
    if (threadIdx.x == blockDim.x - 1) s_carry = off + x;
    __syncthreads();
  }
  if (threadIdx.x == 0) {
    const int total = s_carry;
    p.inj_prefix[nt] = total;
    for (int k = 0; k < p.n_inj; ++k) {
      const int s = p.inj_sp[k];
      const long long base = p.count[s];
      p.inj_base[s] = base;
      long long end = base + total;
      if (end > p.cap) { end = p.cap; atomicOr(p.status, kStCapacity); }
      p.count[s] = end;
    }
    atomicAdd(&p.acc[0], (double)total * (double)p.w_inj * p.n_inj);
    *p.step += 1;  // the step is counted here (k_step_done does without injection)
  }
}

template <typename R>
__global__ void __launch_bounds__(128) k_inject_write(Params<R> p) {
  const int j = blockIdx.x * blockDim.x + threadIdx.x;
  const int nt = p.nt;
  if (j < nt) {
    const int k0 = p.inj_prefix[j], n = p.inj_prefix[j + 1] - k0;
    const long long step = *p.step - 1;  // the scan has counted this step
    for (int k = 0; k < n; ++k) {
      uint32_t c[4] = {(uint32_t)step, (uint32_t)((unsigned long long)step >> 32), (uint32_t)j, (uint32_t)k};
      philox4x32_10(c, p.seed_lo, p.seed_hi);
      const R ox = (R)(c[0] >> 8) * R(1.0 / 16777216.0);
      const R oy = (R)(c[1] >> 8) * R(1.0 / 16777216.0);
      const R r = p.t.rn[0] * exp(ox * p.dlog);
      const R v = p.omega * r * sin((R(j) + oy) * p.dth);
      const R uphi = v / sqrt(R(1) - v * v);
      for (int k2 = 0; k2 < p.n_inj; ++k2) {
        const int s = p.inj_sp[k2];
        const long long q = p.inj_base[s] + k0 + k;
        if (q >= p.count[s]) continue;  // capacity reached (flagged by the scan)
        Species<R> S = p.sp[s];
        S.cell[q] = j;
        S.xo[q] = ox; S.yo[q] = oy;
        S.ur[q] = R(0); S.ut[q] = R(0); S.up[q] = uphi;
        S.w[q] = p.w_inj;
      }
    }
  }
}

// The pairs of this step's events, appended to species 0 and 1 after the
// injected particles, in parent order (species 0 by slot, then species 1):
// each event is ranked by counting the smaller keys, for up to kRankMax
// events (a larger number, far beyond the parity cases, keeps the arbitrary
// event order).  One block.
constexpr int kRankMax = 4096;
template <typename R>
__global__ void __launch_bounds__(1024) k_pairs_append(Params<R> p) {
  __shared__ uint32_t skey[kRankMax];
  __shared__ long long base[2];
  __shared__ double wsum[32];
  const unsigned n_raw = *p.pe_count;
  const int64_t n = (int64_t)n_raw < p.pe_cap ? (int64_t)n_raw : p.pe_cap;
  const bool ranked = n <= kRankMax;
  if (threadIdx.x < 2) base[threadIdx.x] = p.count[threadIdx.x];
  if (ranked)
    for (int64_t e = threadIdx.x; e < n; e += blockDim.x) skey[e] = p.ev_key[e];
  __syncthreads();
  double ws = 0.0;
  for (int64_t e = threadIdx.x; e < n; e += blockDim.x) {
    int64_t rank = e;
    if (ranked) {
      const uint32_t k = skey[e];
      rank = 0;
      for (int64_t f = 0; f < n; ++f) rank += skey[f] < k;
    }
    ws += (double)p.ev_w[e];
    for (int s = 0; s < 2; ++s) {
      const int64_t q = base[s] + rank;
      if (q >= p.cap) continue;
      Species<R> S = p.sp[s];
      S.cell[q] = p.ev_cell[e];
      S.xo[q] = p.ev_xo[e]; S.yo[q] = p.ev_yo[e];
      S.ur[q] = p.ev_ur[e]; S.ut[q] = p.ev_ut[e]; S.up[q] = p.ev_up[e];
      S.w[q] = p.ev_w[e];
    }
  }
  for (int o = 16; o > 0; o >>= 1) ws += __shfl_down_sync(0xffffffffu, ws, o);
  if ((threadIdx.x & 31) == 0) wsum[threadIdx.x >> 5] = ws;
  __syncthreads();
  if (threadIdx.x == 0) {
    double t = 0.0;
    for (int k = 0; k < (int)(blockDim.x >> 5); ++k) t += wsum[k];
    for (int s = 0; s < 2; ++s) {
      long long end = base[s] + n;
      if (end > p.cap) { end = p.cap; atomicOr(p.status, kStCapacity); }
      p.count[s] = end;
    }
    p.acc[4] += 2.0 * t;
    *p.pe_count = 0u;
  }
}

template <typename R>
__global__ void k_step_done(Params<R> p) {
  if (threadIdx.x == 0 && blockIdx.x == 0) *p.step += 1;
}

template <typename R> void launch_inject(const Params<R> &p, cudaStream_t s) {
  if (p.inject) {
    k_inject_scan<R><<<1, 1024, 0, s>>>(p);
    k_inject_write<R><<<(p.nt + 127) / 128, 128, 0, s>>>(p);
  }
  if (p.pairs) k_pairs_append<R><<<1, 1024, 0, s>>>(p);
  if (!p.inject) k_step_done<R><<<1, 32, 0, s>>>(p);
}
template <typename R> void launch_step_done(const Params<R> &p, cudaStream_t s) {
  k_step_done<R><<<1, 32, 0, s>>>(p);
}
template <typename R, bool G> const void *push_tiled_fn() { return reinterpret_cast<const void *>(&k_push_tiled<R, G>); }
template <typename R> cudaError_t set_push_smem(size_t bytes) {
  const cudaError_t e = raise_smem_limit<push_tiled_fn<R, false>>(bytes);
  return e != cudaSuccess ? e : raise_smem_limit<push_tiled_fn<R, true>>(bytes);
}
// resident blocks of the tiled push per SM with `bytes` of shared memory
// (registers and shared memory both counted); 0 on error
template <typename R> int push_tiled_blocks_per_sm(size_t bytes) {
  int a = 0, b = 0;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&a, k_push_tiled<R, false>, kPushThreads, bytes) != cudaSuccess ||
      cudaOccupancyMaxActiveBlocksPerMultiprocessor(&b, k_push_tiled<R, true>, kPushThreads, bytes) != cudaSuccess)
    return 0;
  return a < b ? a : b;
}

#define HFF_INST(R)                                                                         \
  template size_t push_tiled_smem<R>(const Params<R> &, int);                               \
  template bool push_tile_fits<R>(const Params<R> &, int);                                  \
  template void launch_collect<R>(const Params<R> &, cudaStream_t);                         \
  template void launch_push_tail<R>(const Params<R> &, cudaStream_t, int);                  \
  template void launch_push_tiled<R>(const Params<R> &, const WorkList &, int, cudaStream_t, int, bool); \
  template void launch_inject<R>(const Params<R> &, cudaStream_t);                          \
  template void launch_step_done<R>(const Params<R> &, cudaStream_t);                       \
  template cudaError_t set_push_smem<R>(size_t);                                            \
  template int push_tiled_blocks_per_sm<R>(size_t);
HFF_INST(float)
HFF_INST(double)
#undef HFF_INST

}  // namespace hff
