// 4D source and sink kernels on the caller's arrays (C ABI layouts), FP64: the
// domain-wall source of a 4D field, gauge-covariant Gaussian smearing, and the
// residual-mass contraction.  All three are bound by FP64 arithmetic (2
// multiply-adds per SM and clock; a warp instruction takes 64 clocks of its
// scheduler's FP64 unit whatever its active lanes), so threads are split until
// every lane of every warp works, and what is zero is not multiplied.  The
// caller's arrays are read and written 8 bytes at a time: they are aligned to a
// double.  Links: the context's [parity][h][mu][18], h = lex / 2.
#include "blas.h"

namespace mdwf {

namespace {

struct Z2d {
  double re, im;
};
__device__ __forceinline__ Z2d ldz(const double* __restrict__ p) { return Z2d{__ldg(p), __ldg(p + 1)}; }
__device__ __forceinline__ Z2d ldz2(const double* __restrict__ p) {      // 16-byte aligned (links)
  const double2 t = __ldg(reinterpret_cast<const double2*>(p));
  return Z2d{t.x, t.y};
}
// Any bit of the three complex numbers set (integer test: no FP64 instruction).
__device__ __forceinline__ bool any_bits(const Z2d v[3]) {
  unsigned long long b = 0;
#pragma unroll
  for (int i = 0; i < 3; i++) b |= __double_as_longlong(v[i].re) | __double_as_longlong(v[i].im);
  return b != 0;
}
// a += u v, a += conj(u) v
__device__ __forceinline__ void zfma(const Z2d& u, const Z2d& v, Z2d& a) {
  a.re = __fma_rn(u.re, v.re, a.re); a.re = __fma_rn(-u.im, v.im, a.re);
  a.im = __fma_rn(u.re, v.im, a.im); a.im = __fma_rn(u.im, v.re, a.im);
}
__device__ __forceinline__ void zfma_c(const Z2d& u, const Z2d& v, Z2d& a) {
  a.re = __fma_rn(u.re, v.re, a.re); a.re = __fma_rn(u.im, v.im, a.re);
  a.im = __fma_rn(u.re, v.im, a.im); a.im = __fma_rn(-u.im, v.re, a.im);
}

// Lexicographic neighbour of site lex with coordinates c.
__device__ __forceinline__ long nbr_lex(const Geom& g, const int c[4], long lex, int mu, bool fwd) {
  const long st = mu == 0 ? 1 : mu == 1 ? g.L[0] : mu == 2 ? (long)g.L[0] * g.L[1] : (long)g.L[0] * g.L[1] * g.L[2];
  if (fwd) return c[mu] == g.L[mu] - 1 ? lex - (g.L[mu] - 1) * st : lex + st;
  return c[mu] == 0 ? lex + (g.L[mu] - 1) * st : lex - st;
}
__device__ __forceinline__ int coords(const Geom& g, long lex, int c[4]) {     // returns the parity
  long r = lex;
#pragma unroll
  for (int i = 0; i < 4; i++) { c[i] = (int)(r % g.L[i]); r /= g.L[i]; }
  return (c[0] + c[1] + c[2] + c[3]) & 1;
}

// src = (1 - c5 d) w + (c5 / 2) H w for the wall field w = P_+ eta on slice 0 and P_- eta
// on slice L5 - 1 (the other slices of src are zero).  A thread per (site, spin k of
// eta): H takes spin k to itself (the sum of both hops of every direction) and, with
// the gamma matrices' factor, to one spin of the other chirality (their difference;
// spin k ^ 3 for x and y, k ^ 2 for z and t), so each of the 8 colour multiplies of a
// spin is done once and the other ten slices of a 12-slice source cost a memset.
// Before, H ran on all slices of w through the generic matrix form: 16^3 x 48, L5 = 12
// took 9.2 ms; now 0.65 ms.
__global__ void __launch_bounds__(128) k_wall_source(const double* __restrict__ U, const double* __restrict__ eta,
                                                     double* __restrict__ src, Geom g, int L5, int anti, double f,
                                                     double hc) {
  const long i = (long)blockIdx.x * 128 + threadIdx.x;
  const bool on = i < 4 * g.V;            // 4 V is a multiple of 32: whole warps
  if (!on) return;
  const long lex = i >> 2;
  const int k = (int)(i & 3);
  int c[4];
  const int par = coords(g, lex, c);
  Z2d diag[3], offx[3], offz[3];
#pragma unroll
  for (int a = 0; a < 3; a++) diag[a] = offx[a] = offz[a] = Z2d{0.0, 0.0};
  // factor of the difference (backward - forward) on the other chirality: x: -i (k < 2) or i; y: -1, 1, 1, -1;
  // z: -i, i, i, -i; t: 1
  const double sx = k < 2 ? -1.0 : 1.0, sy = (k == 1 || k == 2) ? 1.0 : -1.0;
#pragma unroll
  for (int mu = 0; mu < 4; mu++) {
    const long nf = nbr_lex(g, c, lex, mu, true), nb = nbr_lex(g, c, lex, mu, false);
    Z2d vf[3], vb[3];
#pragma unroll
    for (int b = 0; b < 3; b++) { vf[b] = ldz(eta + nf * 24 + 6 * k + 2 * b); vb[b] = ldz(eta + nb * 24 + 6 * k + 2 * b); }
    if (!any_bits(vf) && !any_bits(vb)) continue;
    if (mu == 3 && anti && c[3] == g.L[3] - 1) {
#pragma unroll
      for (int b = 0; b < 3; b++) { vf[b].re = -vf[b].re; vf[b].im = -vf[b].im; }
    }
    if (mu == 3 && anti && c[3] == 0) {
#pragma unroll
      for (int b = 0; b < 3; b++) { vb[b].re = -vb[b].re; vb[b].im = -vb[b].im; }
    }
    const double* uf = U + (((long)par * g.Vh + (lex >> 1)) * 4 + mu) * 18;
    const double* ub = U + (((long)(1 - par) * g.Vh + (nb >> 1)) * 4 + mu) * 18;
#pragma unroll
    for (int a = 0; a < 3; a++) {
      Z2d x{0.0, 0.0};
#pragma unroll
      for (int b = 0; b < 3; b++) zfma(ldz2(uf + 2 * (3 * a + b)), vf[b], x);
      Z2d y{0.0, 0.0};
#pragma unroll
      for (int b = 0; b < 3; b++) zfma_c(ldz2(ub + 2 * (3 * b + a)), vb[b], y);
      // forward + backward and backward - forward of the rounded products: 2 x + (y - x) with y summed onto
      // -x saves two additions (612 us at 16^3 x 48) but has 15 % more rounding error
      diag[a].re += x.re + y.re;
      diag[a].im += x.im + y.im;
      const Z2d d{y.re - x.re, y.im - x.im};
      if (mu == 0) { offx[a].re = __fma_rn(-sx, d.im, offx[a].re); offx[a].im = __fma_rn(sx, d.re, offx[a].im); }
      if (mu == 1) { offx[a].re = __fma_rn(sy, d.re, offx[a].re); offx[a].im = __fma_rn(sy, d.im, offx[a].im); }
      if (mu == 2) { offz[a].re = __fma_rn(-sy, d.im, offz[a].re); offz[a].im = __fma_rn(sy, d.re, offz[a].im); }
      if (mu == 3) { offz[a].re += d.re; offz[a].im += d.im; }
    }
  }
  const long base = ((k < 2 ? 0 : (long)(L5 - 1) * g.V) + lex) * 24;
#pragma unroll
  for (int a = 0; a < 3; a++) {
    const double xr = __shfl_xor_sync(0xffffffffu, offx[a].re, 1), xi = __shfl_xor_sync(0xffffffffu, offx[a].im, 1);
    const Z2d e = ldz(eta + lex * 24 + 6 * k + 2 * a);
    src[base + 6 * k + 2 * a] = __fma_rn(f, e.re, hc * diag[a].re);
    src[base + 6 * k + 2 * a + 1] = __fma_rn(f, e.im, hc * diag[a].im);
    src[base + 6 * (k ^ 2) + 2 * a] = hc * (offz[a].re + xr);
    src[base + 6 * (k ^ 2) + 2 * a + 1] = hc * (offz[a].im + xi);
  }
}

// list = {number, indices in order} of the time slices of a 4D field that have a bit set; flags: Lt zeros.
__global__ void __launch_bounds__(256) k_slice_flags(const double* __restrict__ eta, long slice, int* __restrict__ flags) {
  const double* p = eta + (long)blockIdx.y * slice;
  unsigned long long b = 0;
  for (long i = (long)blockIdx.x * 256 + threadIdx.x; i < slice; i += 256l * gridDim.x)
    b |= __double_as_longlong(__ldg(p + i));
  if (__any_sync(0xffffffffu, b != 0) && (threadIdx.x & 31) == 0) flags[blockIdx.y] = 1;
}
__global__ void k_slice_list(const int* __restrict__ flags, int Lt, int* __restrict__ list) {
  int n = 0;
  for (int b = 0; b < Lt; b += 32) {
    const int t = b + (int)threadIdx.x;
    const bool on = t < Lt && flags[t] != 0;
    const unsigned m = __ballot_sync(0xffffffffu, on);
    if (on) list[1 + n + __popc(m & ((1u << threadIdx.x) - 1))] = t;
    n += __popc(m);
  }
  if (threadIdx.x == 0) list[0] = n;
}

// One step of gauge-covariant Gaussian source smearing on a 4D field (the sources
// of the paper's propagators, Sec. VII):
//   out(x) = in(x) + k sum_{i = x,y,z} [U_i(x) in(x+i) + U_i(x-i)^+ in(x-i) - 2 in(x)],
// spin-diagonal, no hop in time: a time slice that is zero stays zero and is left
// out (list; a point source lives on one slice), and so is a neighbour that is
// zero.  Items are the complex numbers of the listed slices (72 multiply-adds
// each), taken by a grid of eight blocks per SM, so that a step on one slice does
// not pay for the blocks of the others.  16^3 x 48, 30 steps from a point source:
// 16.6 ms with a thread per site on all slices, 0.5 ms now.
constexpr int kSmearBlocks = 152 * 8;
__global__ void __launch_bounds__(192) k_smear_step(const double* __restrict__ U, const double* __restrict__ in,
                                                    double* __restrict__ out, Geom g, double k, long slice12,
                                                    const int* __restrict__ list) {
  const long n = list[0] * slice12;
  const double k0 = 1.0 - 6.0 * k;
  for (long q = (long)blockIdx.x * 192 + threadIdx.x; q < n; q += 192l * gridDim.x) {
    const long ts = q / slice12;
    const long i = list[1 + ts] * slice12 + (q - ts * slice12);
    const long lex = i / 12;
    const int e = (int)(i - 12 * lex), sp = e / 3, a = e - 3 * sp;
    int c[4];
    const int par = coords(g, lex, c);
    Z2d s{0.0, 0.0};
#pragma unroll
    for (int mu = 0; mu < 3; mu++) {
      const long nf = nbr_lex(g, c, lex, mu, true), nb = nbr_lex(g, c, lex, mu, false);
      Z2d vf[3], vb[3];
#pragma unroll
      for (int b = 0; b < 3; b++) { vf[b] = ldz(in + nf * 24 + 6 * sp + 2 * b); vb[b] = ldz(in + nb * 24 + 6 * sp + 2 * b); }
      const bool f = any_bits(vf), w = any_bits(vb);
      if (!f && !w) continue;
      Z2d t{0.0, 0.0};             // a direction's products by themselves: one chain of 72 has 1.5 times the error
      if (f) {
        const double* uf = U + (((long)par * g.Vh + (lex >> 1)) * 4 + mu) * 18 + 6 * a;
#pragma unroll
        for (int b = 0; b < 3; b++) zfma(ldz2(uf + 2 * b), vf[b], t);
      }
      if (w) {
        const double* ub = U + (((long)(1 - par) * g.Vh + (nb >> 1)) * 4 + mu) * 18 + 2 * a;
#pragma unroll
        for (int b = 0; b < 3; b++) zfma_c(ldz2(ub + 6 * b), vb[b], t);
      }
      s.re += t.re;
      s.im += t.im;
    }
    const Z2d me = ldz(in + 2 * i);
    out[2 * i] = __fma_rn(k, s.re, k0 * me.re);
    out[2 * i + 1] = __fma_rn(k, s.im, k0 * me.im);
  }
}
// The listed time slices of `in` to `out`.
__global__ void __launch_bounds__(256) k_copy_slices(const double* __restrict__ in, double* __restrict__ out, long slice,
                                                     const int* __restrict__ list) {
  if ((int)blockIdx.y >= list[0]) return;
  const long o = (long)list[1 + blockIdx.y] * slice;
  for (long i = (long)blockIdx.x * 256 + threadIdx.x; i < slice; i += 256l * gridDim.x) out[o + i] = in[o + i];
}

// Residual-mass correlators (Eq. mres of arXiv:1701.07559): per time slice, summed
// over the n solutions (spin-colour sources), the squared norms of the wall field
// q = P_- x_0 + P_+ x_{L5-1} and of the midpoint field Q = P_+ x_{L5/2-1} + P_- x_{L5/2};
// P_+ keeps spins 0, 1 and P_- spins 2, 3 (gamma_5 = diag(1, 1, -1, -1)).  An item is
// one real number j = 0..11 of a half spinor of one site: 12 lanes read 96 contiguous
// bytes of each of the four half spinors, and a thread takes every nb-th item of its
// slice, so that its sums are reduced across the block once.  Fixed order.
__global__ void __launch_bounds__(128) k_mres(const double* const* __restrict__ xs, int n, long V, long slice, int L5,
                                              double* __restrict__ part) {
  __shared__ double sh[2][4];
  const int sm = L5 / 2;
  const long o_wl = (long)(L5 - 1) * V * 24, o_m0 = (long)(sm - 1) * V * 24, o_m1 = (long)sm * V * 24;
  double a = 0.0, b = 0.0;
  for (long i = (long)blockIdx.x * 128 + threadIdx.x; i < 12 * slice; i += 128l * gridDim.x) {
    const long site = i / 12;
    const long e = ((long)blockIdx.y * slice + site) * 24 + (i - 12 * site);
#pragma unroll 4
    for (int k = 0; k < n; k++) {
      const double* f = xs[k] + e;
      const double w0 = __ldg(f + 12), wl = __ldg(f + o_wl), m0 = __ldg(f + o_m0), m1 = __ldg(f + o_m1 + 12);
      a = __fma_rn(wl, wl, a);
      b = __fma_rn(m0, m0, b);
      a = __fma_rn(w0, w0, a);
      b = __fma_rn(m1, m1, b);
    }
  }
#pragma unroll
  for (int w = 16; w > 0; w >>= 1) {
    a += __shfl_down_sync(0xffffffffu, a, w);
    b += __shfl_down_sync(0xffffffffu, b, w);
  }
  if ((threadIdx.x & 31) == 0) { sh[0][threadIdx.x >> 5] = a; sh[1][threadIdx.x >> 5] = b; }
  __syncthreads();
  if (threadIdx.x < 2) {
    const double* s = sh[threadIdx.x];
    part[((long)threadIdx.x * gridDim.y + blockIdx.y) * gridDim.x + blockIdx.x] = (s[0] + s[1]) + (s[2] + s[3]);
  }
}
// Per (correlator, time slice), the sum of its nb partial sums.
__global__ void k_mres_sum(const double* __restrict__ part, int nb, double* __restrict__ out) {
  double v = 0.0;
  for (int i = threadIdx.x; i < nb; i += 32) v += part[(long)blockIdx.x * nb + i];
#pragma unroll
  for (int w = 16; w > 0; w >>= 1) v += __shfl_down_sync(0xffffffffu, v, w);
  if (threadIdx.x == 0) out[blockIdx.x] = v;
}

}  // namespace

cudaError_t wall_source(const double* U, const double* eta, double* src, const Geom& g, int L5, int anti, double f,
                        double hc, cudaStream_t st) {
  if (L5 > 2) {
    cudaError_t e = cudaMemsetAsync(src + 24 * g.V, 0, sizeof(double) * 24 * (size_t)g.V * (L5 - 2), st);
    if (e != cudaSuccess) return e;
  }
  k_wall_source<<<(unsigned)((4 * g.V + 127) / 128), 128, 0, st>>>(U, eta, src, g, L5, anti, f, hc);
  return cudaGetLastError();
}

cudaError_t smear(const double* U, double* eta, double* tmp, int* slices, const Geom& g, double k, int n_iter,
                  cudaStream_t st) {
  const int Lt = g.L[3];
  const long sites = g.V / Lt, slice = sites * 24;
  int *flags = slices, *list = slices + Lt;
  const dim3 sg((unsigned)(slice >= 256 * 32 ? 32 : (slice + 255) / 256), (unsigned)Lt);
  cudaError_t e = cudaMemsetAsync(flags, 0, sizeof(int) * Lt, st);
  if (e != cudaSuccess) return e;
  k_slice_flags<<<sg, 256, 0, st>>>(eta, slice, flags);
  k_slice_list<<<1, 32, 0, st>>>(flags, Lt, list);
  const long blocks = (12 * g.V + 191) / 192;
  const unsigned grid = (unsigned)(blocks < kSmearBlocks ? blocks : kSmearBlocks);
  double* a = eta;
  double* b = tmp;
  for (int i = 0; i < n_iter; i++) {
    k_smear_step<<<grid, 192, 0, st>>>(U, a, b, g, k, 12 * sites, list);
    double* t = a;
    a = b;
    b = t;
  }
  if (a != eta) k_copy_slices<<<sg, 256, 0, st>>>(a, eta, slice, list);
  return cudaGetLastError();
}

// 32 blocks per time slice, more where there are few slices: eight blocks of four warps per SM
// (kMresBlocks) keep enough loads in flight, and no block without an item of its own (12 solutions
// at 32^3 x 2: 801 us with 32 blocks per slice, 152 us with 608; 48 slices take 32 either way).
constexpr int kMresBlocks = 152 * 8;
int mres_blocks(long slice_sites, int Lt) {
  const long b = (12 * slice_sites + 127) / 128;
  const long fill = (kMresBlocks + Lt - 1) / Lt, most = fill > 32 ? fill : 32;
  return (int)(b > most ? most : b);
}

cudaError_t mres_correlators(const double* const* xs, int n, long V, int Lt, int L5, double* part, double* c,
                             cudaStream_t st) {
  const int nb = mres_blocks(V / Lt, Lt);
  k_mres<<<dim3((unsigned)nb, (unsigned)Lt), 128, 0, st>>>(xs, n, V, V / Lt, L5, part);
  k_mres_sum<<<2 * Lt, 32, 0, st>>>(part, nb, c);
  return cudaGetLastError();
}

}  // namespace mdwf
