// diag.cu -- FP64 diagnostics of Sect. 4, on request only (not in the step):
// Psi in FP64 (Eq. 27), spin-down power L(r) through each half-node sphere
// (Eq. 35), Gauss's-law residual div E / 4 pi - rho on interior nodes, field
// energies, kinetic energy and live counts per species.
// All of it is bound by the FP64 pipe (two operations per clock and SM), not
// by memory, so what can be is kept off it: conversions and tests are integer
// work, roots and divisions are the short forms of fastmath.cuh, factors of a
// row are multiplied in once per row, and the spectrum takes its bins in FP32
// wherever that cannot change them.  On 1.25e7 FP32 particles of each of two
// species, 1024^2, before and after: node charges and kinetic energies 1.58 and
// 1.17 ms, maps 0.73 and 0.50 per species, spectrum 1.40 and 0.12 per species,
// row sums 0.30 and 0.15.
#include "diag.cuh"
#include "fastmath.cuh"

namespace hff {

// Psi in FP64 at every node (one block per row)
template <typename R>
__global__ void __launch_bounds__(256) k_psi64(Params<R> p, double *out) {
  const int i = blockIdx.x, nt = p.nt;
  const R *br = p.f.br + (int64_t)i * nt, *br0 = p.f.br0 + (int64_t)i * nt;
  double *psi = out + (int64_t)i * (nt + 1);
  const double r2 = p.t.r2n[i];
  __shared__ double warp_tot[8];
  __shared__ double carry;
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  if (threadIdx.x == 0) { carry = 0.0; psi[0] = 0.0; }
  __syncthreads();
  for (int seg = 0; seg < nt; seg += 256) {
    const int j = seg + threadIdx.x;
    double v = (j < nt) ? ((double)br0[j] + (double)br[j]) * p.t.dcp[j] : 0.0;
    for (int o = 1; o < 32; o <<= 1) {
      const double y = __shfl_up_sync(0xffffffffu, v, o);
      if (lane >= o) v += y;
    }
    if (lane == 31) warp_tot[wid] = v;
    __syncthreads();
    double off = carry;
    for (int w = 0; w < wid; ++w) off += warp_tot[w];
    if (j < nt) psi[j + 1] = r2 * (off + v);
    __syncthreads();
    if (threadIdx.x == 255) carry = off + v;
    __syncthreads();
  }
}

// CIC node charges of the live particles (FP64 accumulation)
template <typename R>
__global__ void __launch_bounds__(256) k_node_charge(Params<R> p, double *q, double *kin, double *cnt) {
  const int nt = p.nt, n1 = nt + 1;
  for (int s = 0; s < p.n_species; ++s) {
    double ke = 0.0;
    unsigned c = 0;
    const int64_t n = p.count[s];
    const double qs = p.q[s], ms = p.m[s];
    for (int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; k < n; k += (int64_t)gridDim.x * blockDim.x) {
      const int cell = p.sp[s].cell[k];
      if (cell < 0) continue;
      int i, j;
      decode_cell(p, cell, i, j);
      const double x = to_double(p.sp[s].xo[k]), y = to_double(p.sp[s].yo[k]), w = to_double(p.sp[s].w[k]);
      const double qw = qs * w, q1 = qw * x, q0 = qw - q1, q01 = q0 * y, q11 = q1 * y;
      double *a = q + ix(i, j, n1);
      atomicAdd(a, q0 - q01);
      atomicAdd(a + n1, q1 - q11);
      atomicAdd(a + 1, q01);
      atomicAdd(a + n1 + 1, q11);
      const double u0 = to_double(p.sp[s].ur[k]), u1 = to_double(p.sp[s].ut[k]), u2 = to_double(p.sp[s].up[k]);
      const double g2 = fma(u2, u2, fma(u1, u1, fma(u0, u0, 1.0)));
      // gamma - 1; an infinite g2 keeps an infinite root (infinity times rsq would not)
      ke = fma(w * ms, mid_range(g2) ? fma(g2, rsq(g2), -1.0) : sqrt(g2) - 1.0, ke);
      c += 1;
    }
    for (int o = 16; o > 0; o >>= 1) {
      ke += __shfl_down_sync(0xffffffffu, ke, o);
      c += __shfl_down_sync(0xffffffffu, c, o);
    }
    if ((threadIdx.x & 31) == 0) { atomicAdd(&kin[s], ke); atomicAdd(&cnt[s], (double)c); }
  }
}

__device__ __forceinline__ double block_sum(double v, double *sh) {
  for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
  if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = v;
  __syncthreads();
  double t = 0.0;
  if (threadIdx.x == 0) for (int w = 0; w < (int)(blockDim.x >> 5); ++w) t += sh[w];
  __syncthreads();
  return t;
}
__device__ __forceinline__ double block_max(double v, double *sh) {
  for (int o = 16; o > 0; o >>= 1) v = fmax(v, __shfl_down_sync(0xffffffffu, v, o));
  if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = v;
  __syncthreads();
  double t = 0.0;
  if (threadIdx.x == 0) for (int w = 0; w < (int)(blockDim.x >> 5); ++w) t = fmax(t, sh[w]);
  __syncthreads();
  return t;
}

// per row i (0..nr): [L(r_{i+1/2}), U_E part, U_B part, gauss max, gauss sum2,
// gauss count, rho max, unused], all FP64.  Geometry in FP64 from the row and
// column tables of the working precision, which were themselves rounded from
// FP64 (the relative error is that of R).
template <typename R>
__global__ void __launch_bounds__(256) k_diag_rows(Params<R> p, DiagGeom g, const double *q, double *rows) {
  __shared__ double sh[8];
  const int i = blockIdx.x, nr = p.nr, nt = p.nt, n1 = nt + 1;
  const Fields<R> &f = p.f;
  // B = B_0 + dB, summed in FP64
  auto Bt = [&](int64_t k) { return to_double(f.bt0[k]) + to_double(f.bt[k]); };
  auto Bp = [&](int64_t k) { return to_double(f.bp0[k]) + to_double(f.bp[k]); };
  auto Br = [&](int64_t k) { return to_double(f.br0[k]) + to_double(f.br[k]); };
  auto odd = [](R x) { return !isfinite(x) ? 1u : 0u; };
  // sums over the row without the row's own factors: L, the energies of the
  // six components, and the Gauss residual times the row's volume factor
  double l0 = 0, l1 = 0, er2 = 0, et2 = 0, ep2 = 0, br2 = 0, bt2 = 0, bp2 = 0, gmax = 0, g2 = 0, rmax = 0;
  unsigned bad = 0, gcnt = 0;
  const double rlo = g.rlo[i], rhi = g.rhi[i], rni = g.rn[i];
  const bool gauss = i >= 2 && i <= g.imax;
  const double c1 = gauss ? 2 * kPi * g.rh[i] * g.rh[i] : 0.0, c0 = gauss ? 2 * kPi * g.rh[i - 1] * g.rh[i - 1] : 0.0;
  const double ct = kPi * (rhi * rhi - rlo * rlo), fourpi = 4 * kPi;
  const double vrow = 2.0 * kPi / 3.0 * (rhi * rhi * rhi - rlo * rlo * rlo);
  for (int j = threadIdx.x; j <= nt; j += blockDim.x) {
    const R ep_ = f.ep[ix(i, j, n1)];
    const double ep = to_double(ep_), dch = g.dch[j], snw = g.sn[j] * (g.thi[j] - g.tlo[j]);
    bad += odd(ep_);   // non-finite field values owned by (i, j) (failure detection)
    ep2 = fma(ep * ep, snw, ep2);
    R et_ = R(0);
    double et = 0, er = 0;
    if (j < nt) {
      et_ = f.et[ix(i, j, nt)];
      et = to_double(et_);
      bad += odd(et_) + odd(f.br[ix(i, j, nt)]);
      const double br = Br(ix(i, j, nt));
      et2 = fma(et * et, g.sh[j], et2);
      br2 = fma(br * br, g.dcp[j], br2);
    }
    if (i < nr) {
      const R er_ = f.er[ix(i, j, n1)];
      er = to_double(er_);
      bad += odd(er_) + odd(f.bt[ix(i, j, n1)]);
      const double bt = Bt(ix(i, j, n1));
      er2 = fma(er * er, dch, er2);
      bt2 = fma(bt * bt, snw, bt2);
      l1 = fma((ep + to_double(f.ep[ix(i + 1, j, n1)])) * bt, dch, l1);
      if (j < nt) {
        bad += odd(f.bp[ix(i, j, nt)]);
        const double bp = Bp(ix(i, j, nt));
        bp2 = fma(bp * bp, g.sh[j], bp2);
        l0 = fma((et + to_double(f.et[ix(i + 1, j, nt)])) * bp, g.dcp[j], l0);
      }
    }
    if (gauss) {
      double flux = dch * fma(c1, er, -(c0 * to_double(f.er[ix(i - 1, j, n1)])));
      double th = j < nt ? g.sh[j] * et : 0.0;
      if (j > 0) th = fma(-g.sh[j - 1], to_double(f.et[ix(i, j - 1, nt)]), th);
      flux = fma(ct, th, flux);
      const double qq = q[ix(i, j, n1)], iv = rcp(vrow * dch);
      const double res = fma(flux, 1.0 / fourpi, -qq) * iv;
      gmax = fmax(gmax, fabs(res));
      rmax = fmax(rmax, fabs(qq * iv));
      g2 = fma(res, res, g2);
      gcnt += 1;
    }
  }
  double L = 0, ue = 0, ub = 0;
  if (i < nr) {
    const double r = g.rh[i], dr = g.rn[i + 1] - rni, dr2 = g.rn[i + 1] * g.rn[i + 1] - rni * rni;
    L = (l0 - l1) * kPi * r * r;
    ue = er2 * 2 * kPi * r * r * dr;
    ub = bt2 * kPi * dr2 * r + bp2 * 0.5 * dr2 * g.dth * 2 * kPi * r;
  }
  ue += et2 * ct * rni * g.dth + ep2 * ct * rni;
  ub += br2 * 2 * kPi * rni * rni * (rhi - rlo);
  L = block_sum(L, sh);
  ue = block_sum(ue, sh);
  ub = block_sum(ub, sh);
  g2 = block_sum(g2, sh);
  const double ngauss = block_sum((double)gcnt, sh);
  gmax = block_max(gmax, sh);
  rmax = block_max(rmax, sh);
  const double nbad = block_sum((double)bad, sh);
  if (threadIdx.x == 0) {
    double *o = rows + (int64_t)i * 8;
    o[0] = L / (4 * kPi); o[1] = ue; o[2] = ub; o[3] = gmax; o[4] = g2; o[5] = ngauss; o[6] = rmax; o[7] = nbad;
  }
}

// Sect. 5.2 maps: sums of w and w m (gamma - 1) per cell, then divided by
// the exact cell volume (2 pi / 3)(r_{i+1}^3 - r_i^3)(cos th_j - cos th_{j+1})
template <typename R>
__global__ void __launch_bounds__(256) k_species_sums(Params<R> p, int s, double m, double *dens, double *ener) {
  const int64_t n = p.count[s];
  for (int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; k < n; k += (int64_t)gridDim.x * blockDim.x) {
    const int c = p.sp[s].cell[k];
    if (c < 0) continue;
    const double w = to_double(p.sp[s].w[k]), u0 = to_double(p.sp[s].ur[k]), u1 = to_double(p.sp[s].ut[k]),
                 u2 = to_double(p.sp[s].up[k]);
    const double uu = fma(u2, u2, fma(u1, u1, u0 * u0)), g2 = 1.0 + uu;
    atomicAdd(&dens[c], w);
    atomicAdd(&ener[c], (w * m) * (uu * rcp(fma(g2, rsq(g2), 1.0))));  // gamma - 1 = u^2 / (gamma + 1), without cancellation
  }
}
template <typename R>
__global__ void __launch_bounds__(256) k_per_volume(Params<R> p, DiagGeom g, double *dens, double *ener) {
  for (int i = blockIdx.x; i < p.nr; i += gridDim.x) {
    const double a = g.rn[i], b = g.rn[i + 1], vrow = 2.0 * kPi / 3.0 * (b * b * b - a * a * a);
    for (int j = threadIdx.x; j < p.nt; j += blockDim.x) {
      const double iv = rcp(vrow * g.dcp[j]);
      const int64_t c = ix(i, j, p.nt);
      dens[c] *= iv;
      ener[c] *= iv;
    }
  }
}
// The bin of a particle is floor((log10 gamma - lg0) inv) in FP64.  An FP32
// evaluation is within `off` bins of that (its rounding: u^2 and the logarithm
// to a few ulp, 2e-6 of 1 + |log10 gamma|, and 1e-6 of the bin number), so it
// decides wherever it is further than that from the next bin; the others, and
// momenta whose square leaves the FP32 range, are evaluated in FP64.  The
// block's histogram has 2^shift copies, one per lane modulo that, so that the
// lanes of a warp seldom meet (FP64 adds in shared memory retry).
template <typename R>
__global__ void __launch_bounds__(256) k_spectrum(Params<R> p, int s, int nbins, double lg0, double inv, int shift,
                                                  double *out) {
  extern __shared__ double hist[];
  const int copies = 1 << shift;
  for (int b = threadIdx.x; b < nbins << shift; b += blockDim.x) hist[b] = 0.0;
  __syncthreads();
  const int64_t n = p.count[s];
  const float lg0f = (float)lg0, invf = (float)inv;
  double *mine = hist + (threadIdx.x & (copies - 1));
  for (int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; k < n; k += (int64_t)gridDim.x * blockDim.x) {
    if (p.sp[s].cell[k] < 0) continue;
    const R v0 = p.sp[s].ur[k], v1 = p.sp[s].ut[k], v2 = p.sp[s].up[k];
    const float a0 = (float)v0, a1 = (float)v1, a2 = (float)v2;
    const float g2 = fmaf(a2, a2, fmaf(a1, a1, fmaf(a0, a0, 1.f)));
    const float lgf = 0.5f * log10f(g2), xf = (lgf - lg0f) * invf;
    const float off = fmaf(2e-6f * (1.f + fabsf(lgf) + fabsf(lg0f)), invf, 1e-6f * (1.f + fabsf(xf)));
    const float fl = floorf(xf), fr = xf - fl;
    int bin;
    if (g2 < 1e37f && fr > off && fr < 1.f - off && fabsf(xf) < 1e6f) {
      bin = (int)fl;
      bin = bin < 0 ? 0 : (bin > nbins - 1 ? nbins - 1 : bin);
    } else {
      const double u0 = v0, u1 = v1, u2 = v2;
      const double lg = log10(sqrt(1.0 + u0 * u0 + u1 * u1 + u2 * u2));
      double x = floor((lg - lg0) * inv);
      x = x < 0.0 ? 0.0 : (x > nbins - 1 ? (double)(nbins - 1) : x);
      bin = (int)x;
    }
    atomicAdd(&mine[bin << shift], to_double(p.sp[s].w[k]));
  }
  __syncthreads();
  for (int b = threadIdx.x; b < nbins; b += blockDim.x) {
    double t = 0.0;
    for (int c = 0; c < copies; ++c) t += hist[(b << shift) + c];
    if (t != 0.0) atomicAdd(&out[b], t);
  }
}

template <typename R> void launch_maps(const Params<R> &p, const DiagGeom &g, int species, double mass,
                                       double *dens, double *ener, cudaStream_t s) {
  const size_t n = (size_t)p.nr * p.nt;
  cudaMemsetAsync(dens, 0, n * sizeof(double), s);
  cudaMemsetAsync(ener, 0, n * sizeof(double), s);
  k_species_sums<R><<<1216, 256, 0, s>>>(p, species, mass, dens, ener);
  k_per_volume<R><<<(unsigned)(p.nr < 4864 ? p.nr : 4864), 256, 0, s>>>(p, g, dens, ener);
}
template <typename R> void launch_spectrum(const Params<R> &p, int species, int nbins, double lg_min,
                                           double lg_max, double *out, cudaStream_t s) {
  cudaMemsetAsync(out, 0, (size_t)nbins * sizeof(double), s);
  int shift = 0;   // copies of the histogram in 32 KB, at most one per lane
  while (shift < 5 && ((size_t)nbins << (shift + 1)) * sizeof(double) <= 32 * 1024) ++shift;
  k_spectrum<R><<<912, 256, ((size_t)nbins << shift) * sizeof(double), s>>>(p, species, nbins, lg_min,
                                                                             nbins / (lg_max - lg_min), shift, out);
}

template <typename R> void launch_psi64(const Params<R> &p, double *out, cudaStream_t s) {
  k_psi64<R><<<p.nr + 1, 256, 0, s>>>(p, out);
}
template <typename R> void launch_diag(const Params<R> &p, const DiagGeom &g, double *q, double *kin,
                                       double *cnt, double *rows, cudaStream_t s) {
  cudaMemsetAsync(q, 0, sizeof(double) * (size_t)(p.nr + 1) * (p.nt + 1), s);
  cudaMemsetAsync(kin, 0, sizeof(double) * 2 * kMaxSpecies, s);
  k_node_charge<R><<<1216, 256, 0, s>>>(p, q, kin, cnt);
  k_diag_rows<R><<<p.nr + 1, 256, 0, s>>>(p, g, q, rows);
}

template void launch_maps<float>(const Params<float> &, const DiagGeom &, int, double, double *, double *,
                                 cudaStream_t);
template void launch_maps<double>(const Params<double> &, const DiagGeom &, int, double, double *, double *,
                                  cudaStream_t);
template void launch_spectrum<float>(const Params<float> &, int, int, double, double, double *, cudaStream_t);
template void launch_spectrum<double>(const Params<double> &, int, int, double, double, double *, cudaStream_t);
template void launch_psi64<float>(const Params<float> &, double *, cudaStream_t);
template void launch_psi64<double>(const Params<double> &, double *, cudaStream_t);
template void launch_diag<float>(const Params<float> &, const DiagGeom &, double *, double *, double *,
                                 double *, cudaStream_t);
template void launch_diag<double>(const Params<double> &, const DiagGeom &, double *, double *, double *,
                                  double *, cudaStream_t);

}  // namespace hff
