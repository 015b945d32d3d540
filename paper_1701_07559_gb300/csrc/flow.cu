// Wilson (gradient) flow of a gauge field on the device, FP64.
//
// The paper smooths its ensembles' links by the gradient flow to t_gf = 1
// (Sec. III, citing Luscher, JHEP 08 (2010) 071) before the domain-wall
// solves.  Here: dV/dt = Z(V) V with Z = -P_TA(Omega), Omega_mu(x) the sum of
// the six plaquettes that start with V_mu(x) (Wilson plaquette action) and
// P_TA(M) = (M - M^+)/2 - tr(M - M^+)/6, integrated by Luscher's three-stage
// Runge-Kutta scheme:
//   W1 = exp(Z0 / 4) W0,  W2 = exp(8/9 Z1 - 17/36 Z0) W1,
//   W3 = exp(3/4 Z2 - 8/9 Z1 + 17/36 Z0) W2,   Z_i = eps Z(W_i).
//
// Both kernels are bound by FP64 arithmetic (2 multiply-adds per SM and clock on
// this part), so they are written for few of them and for full warps:
// * Z: the six staples of a link are summed first and multiplied by the link
//   once (13 matrix products instead of 18), by three threads per link, one per
//   matrix row (a staple's rows are independent; only the last product needs the
//   other rows, through shared memory): a third of the registers of a thread per
//   link and three times the warps.
// * exp(X) of an anti-Hermitian traceless X: X^3 = (tr X^2 / 2) X + det X
//   (Cayley-Hamilton), so the Taylor polynomial is summed as f0 + f1 X + f2 X^2 by
//   Horner's rule on three complex numbers, four multiply-adds per term, instead
//   of matrix products.  |X|_F is first scaled to at most 1/2 by 2^-k (k squarings
//   of the result; none for the usual steps); 17 terms leave a remainder below
//   (1/2)^18 / 18! < 1e-21.
// * U <- exp(X) U as U + (exp(X) - 1) U: for the usual steps the second term is small, and a stage rounds U once at its
//   own size.  Error of 10 steps of 0.01 against extended precision: 1.96e-16 of the links, where the chain of
//   multiply-adds of exp(X) U left 5.35e-16 and the matrix products before it 4.65e-16; it costs 1 % of a step.
// Z keeps the nine independent reals of an anti-Hermitian matrix, one plane each.
// Ten steps at 16^3 x 48: 297 ms with a thread per link and the matrix Taylor series
// (which spilled), 72 ms so (2.4 ms per stage; its 1800 FP64 instructions per link take 2.25 ms
// at 6.3e11 per second, two lanes per SM and clock at 2070 MHz).
//
// Layout of U: the C ABI's gauge layout U[t][z][y][x][mu][a][b], complex (re, im).
// Input preparation: the solver reads links only through mdwf_load_gauge.
#include "mdwf_internal.h"

namespace mdwf {

namespace {

struct C2 {
  double re, im;
};
struct M3 {
  C2 m[9];
};

__device__ __forceinline__ void cfma(const C2& x, const C2& y, C2& a) {         // a += x y
  a.re = __fma_rn(x.re, y.re, a.re); a.re = __fma_rn(-x.im, y.im, a.re);
  a.im = __fma_rn(x.re, y.im, a.im); a.im = __fma_rn(x.im, y.re, a.im);
}
__device__ __forceinline__ void cfma_c(const C2& x, const C2& y, C2& a) {       // a += x conj(y)
  a.re = __fma_rn(x.re, y.re, a.re); a.re = __fma_rn(x.im, y.im, a.re);
  a.im = __fma_rn(x.im, y.re, a.im); a.im = __fma_rn(-x.re, y.im, a.im);
}
// 8-byte accesses: U is the caller's array, aligned to a double (the kernels are bound by FP64, not by loads).
__device__ __forceinline__ C2 ldc(const double* __restrict__ p) { return C2{p[0], p[1]}; }
// c = a b
__device__ __forceinline__ void mmul(const M3& a, const M3& b, M3& c) {
  M3 t;
#pragma unroll
  for (int i = 0; i < 3; i++)
#pragma unroll
    for (int j = 0; j < 3; j++) {
      C2 s{0.0, 0.0};
#pragma unroll
      for (int k = 0; k < 3; k++) cfma(a.m[3 * i + k], b.m[3 * k + j], s);
      t.m[3 * i + j] = s;
    }
  c = t;
}

// Row vector times a stored matrix: o = v M (DAG: v M^+), added to o when ADD.
template <bool DAG, bool ADD>
__device__ __forceinline__ void vmul(const C2 v[3], const double* __restrict__ p, C2 o[3]) {
  if (!ADD) {
#pragma unroll
    for (int j = 0; j < 3; j++) o[j] = C2{0.0, 0.0};
  }
#pragma unroll
  for (int i = 0; i < 3; i++)
#pragma unroll
    for (int j = 0; j < 3; j++) {
      const C2 y = ldc(p + 2 * (3 * i + j));            // M_ij
      if (DAG) cfma_c(v[j], y, o[i]);                   // (M^+)_ji = conj(M_ij)
      else cfma(v[i], y, o[j]);
    }
}

struct Lat {
  int L[4];
  long V;
};

__device__ __forceinline__ long lat_nbr(const Lat& g, const int c[4], int mu, int dir) {
  int d[4] = {c[0], c[1], c[2], c[3]};
#pragma unroll
  for (int i = 0; i < 4; i++)
    if (i == mu) {
      d[i] += dir;
      if (d[i] < 0) d[i] += g.L[i];
      if (d[i] >= g.L[i]) d[i] -= g.L[i];
    }
  return d[0] + (long)g.L[0] * (d[1] + (long)g.L[1] * (d[2] + (long)g.L[2] * d[3]));
}

__device__ __forceinline__ const double* lnk(const double* U, long s, int mu) { return U + 18 * (4 * s + mu); }

constexpr int kZLinks = 32;             // links per block of k_flow_Z (three threads each: three full warps)

// Z = eps * (-P_TA(Omega_mu(x))) for every link, as nine planes of nlink reals: the
// imaginary diagonal (0..2) and re, im of the elements (0,1), (0,2), (1,2) (3..8).
__global__ void __launch_bounds__(3 * kZLinks) k_flow_Z(const double* __restrict__ U, double* __restrict__ Z, Lat g,
                                                       double eps) {
  __shared__ double2 st[3 * kZLinks][3];
  const long nlink = 4 * g.V;
  const int kl = threadIdx.x / 3, row = threadIdx.x - 3 * kl;
  const long k = (long)blockIdx.x * kZLinks + kl;
  const bool on = k < nlink;
  const long s = on ? k >> 2 : 0;
  const int mu = on ? (int)(k & 3) : 0;
  C2 acc[3] = {{0.0, 0.0}, {0.0, 0.0}, {0.0, 0.0}};      // row of the sum of the staples
  if (on) {
    int c[4];
    long r = s;
    for (int i = 0; i < 4; i++) { c[i] = (int)(r % g.L[i]); r /= g.L[i]; }
    const long xp = lat_nbr(g, c, mu, +1);
    int cp[4];
#pragma unroll
    for (int i = 0; i < 4; i++) cp[i] = i == mu ? (c[i] + 1 == g.L[i] ? 0 : c[i] + 1) : c[i];
    for (int p = 1; p < 4; p++) {
      const int nu = (mu + p) & 3;
      const long xn = lat_nbr(g, c, nu, +1), xm = lat_nbr(g, c, nu, -1), xpm = lat_nbr(g, cp, nu, -1);
      C2 v[3], w[3];
      // U_nu(x+mu) U_mu(x+nu)^+ U_nu(x)^+
      const double* a = lnk(U, xp, nu) + 6 * row;
#pragma unroll
      for (int j = 0; j < 3; j++) v[j] = ldc(a + 2 * j);
      vmul<true, false>(v, lnk(U, xn, mu), w);
      vmul<true, true>(w, lnk(U, s, nu), acc);
      // U_nu(x+mu-nu)^+ U_mu(x-nu)^+ U_nu(x-nu)
      const double* b = lnk(U, xpm, nu) + 2 * row;
#pragma unroll
      for (int j = 0; j < 3; j++) { v[j] = ldc(b + 6 * j); v[j].im = -v[j].im; }
      vmul<true, false>(v, lnk(U, xm, mu), w);
      vmul<false, true>(w, lnk(U, xm, nu), acc);
    }
  }
#pragma unroll
  for (int j = 0; j < 3; j++) st[threadIdx.x][j] = make_double2(acc[j].re, acc[j].im);
  __syncthreads();
  // row of Omega = U_mu(x) (sum of staples)
  C2 om[3] = {{0.0, 0.0}, {0.0, 0.0}, {0.0, 0.0}};
  if (on) {
    const double* u = lnk(U, s, mu) + 6 * row;
#pragma unroll
    for (int i = 0; i < 3; i++) {
      const C2 ui = ldc(u + 2 * i);
#pragma unroll
      for (int j = 0; j < 3; j++) {
        const double2 q = st[3 * kl + i][j];
        cfma(ui, C2{q.x, q.y}, om[j]);
      }
    }
  }
  __syncthreads();
#pragma unroll
  for (int j = 0; j < 3; j++) st[threadIdx.x][j] = make_double2(om[j].re, om[j].im);
  __syncthreads();
  if (!on) return;
  // -eps P_TA: thread `row` writes its diagonal and one off-diagonal element
  const double2 d0 = st[3 * kl][0], d1 = st[3 * kl + 1][1], d2 = st[3 * kl + 2][2];
  const double tr = (d0.y + d1.y + d2.y) / 3.0;
  const double dg = row == 0 ? d0.y : row == 1 ? d1.y : d2.y;
  const int i = row == 2 ? 1 : 0, j = row == 0 ? 1 : 2;   // (0,1), (0,2), (1,2)
  const double2 x = st[3 * kl + i][j], y = st[3 * kl + j][i];
  Z[(long)row * nlink + k] = -eps * (dg - tr);
  Z[(long)(3 + 2 * row) * nlink + k] = -eps * (0.5 * (x.x - y.x));
  Z[(long)(4 + 2 * row) * nlink + k] = -eps * (0.5 * (x.y + y.y));
}

// F = exp(X) - 1 of the anti-Hermitian traceless X with diagonal i d[0..2] and elements (0,1), (0,2), (1,2) = o[0..2].
// Without the unit matrix its small elements keep their digits.
__device__ __forceinline__ void mexpm1(const double d_in[3], const C2 o_in[3], M3& F) {
  double n2 = 0.0;
#pragma unroll
  for (int i = 0; i < 3; i++)
    n2 += d_in[i] * d_in[i] + 2.0 * (o_in[i].re * o_in[i].re + o_in[i].im * o_in[i].im);
  int sq = 0;
  while (n2 > 0.25 && sq < 64) { n2 *= 0.25; sq++; }
  const double sc = ldexp(1.0, -sq);
  double d[3];
  C2 o[3];
#pragma unroll
  for (int i = 0; i < 3; i++) { d[i] = d_in[i] * sc; o[i] = C2{o_in[i].re * sc, o_in[i].im * sc}; }
  // X^2 (Hermitian): diagonal -q[i], elements (0,1), (0,2), (1,2) = y[i]
  const double a01 = o[0].re * o[0].re + o[0].im * o[0].im;
  const double a02 = o[1].re * o[1].re + o[1].im * o[1].im;
  const double a12 = o[2].re * o[2].re + o[2].im * o[2].im;
  const double q[3] = {d[0] * d[0] + a01 + a02, d[1] * d[1] + a01 + a12, d[2] * d[2] + a02 + a12};
  C2 y[3];
  // (0,1): i (d0 + d1) o01 - o02 conj(o12);  (0,2): i (d0 + d2) o02 + o01 o12;  (1,2): i (d1 + d2) o12 - conj(o01) o02
  const double s01 = d[0] + d[1], s02 = d[0] + d[2], s12 = d[1] + d[2];
  y[0].re = -s01 * o[0].im - (o[1].re * o[2].re + o[1].im * o[2].im);
  y[0].im = s01 * o[0].re - (o[1].im * o[2].re - o[1].re * o[2].im);
  y[1].re = -s02 * o[1].im + (o[0].re * o[2].re - o[0].im * o[2].im);
  y[1].im = s02 * o[1].re + (o[0].re * o[2].im + o[0].im * o[2].re);
  y[2].re = -s12 * o[2].im - (o[0].re * o[1].re + o[0].im * o[1].im);
  y[2].im = s12 * o[2].re - (o[0].re * o[1].im - o[0].im * o[1].re);
  // X^3 = c1 X + i dt:  c1 = tr X^2 / 2,  det X = i dt,
  // dt = -d0 d1 d2 + d0 a12 + d1 a02 + d2 a01 - 2 Im(o01 o12 conj(o02))
  const double c1 = -0.5 * (q[0] + q[1] + q[2]);
  const C2 t{o[0].re * o[2].re - o[0].im * o[2].im, o[0].re * o[2].im + o[0].im * o[2].re};
  const double dt = -d[0] * d[1] * d[2] + d[0] * a12 + d[1] * a02 + d[2] * a01 -
                    2.0 * (t.im * o[1].re - t.re * o[1].im);
  // Horner on p0 + p1 X + p2 X^2:  p <- p X + 1/k!, the last step (k = 0) without its 1
  constexpr int kTerms = 17;
  const double invf[kTerms + 1] = {1.0, 1.0, 1.0 / 2, 1.0 / 6, 1.0 / 24, 1.0 / 120, 1.0 / 720, 1.0 / 5040, 1.0 / 40320,
                                   1.0 / 362880, 1.0 / 3628800, 1.0 / 39916800, 1.0 / 479001600, 1.0 / 6227020800.0,
                                   1.0 / 87178291200.0, 1.0 / 1307674368000.0, 1.0 / 20922789888000.0,
                                   1.0 / 355687428096000.0};
  C2 p0{invf[kTerms], 0.0}, p1{0.0, 0.0}, p2{0.0, 0.0};
#pragma unroll
  for (int k = kTerms - 1; k >= 0; k--) {
    const C2 n0{k > 0 ? __fma_rn(-dt, p2.im, invf[k]) : -dt * p2.im, dt * p2.re};
    const C2 n1{__fma_rn(c1, p2.re, p0.re), __fma_rn(c1, p2.im, p0.im)};
    p2 = p1;
    p1 = n1;
    p0 = n0;
  }
  // F = p0 + p1 X + p2 X^2
#pragma unroll
  for (int i = 0; i < 3; i++) {
    C2 e = p0;
    e.re = __fma_rn(-p1.im, d[i], e.re); e.im = __fma_rn(p1.re, d[i], e.im);
    e.re = __fma_rn(-p2.re, q[i], e.re); e.im = __fma_rn(-p2.im, q[i], e.im);
    F.m[4 * i] = e;
  }
#pragma unroll
  for (int i = 0; i < 3; i++) {
    const int a = i == 2 ? 1 : 0, b = i == 0 ? 1 : 2;
    C2 u{0.0, 0.0}, l{0.0, 0.0};
    cfma(p1, o[i], u);
    cfma(p2, y[i], u);
    cfma(p1, C2{-o[i].re, o[i].im}, l);                  // X_ba = -conj(X_ab)
    cfma(p2, C2{y[i].re, -y[i].im}, l);                  // (X^2)_ba = conj((X^2)_ab)
    F.m[3 * a + b] = u;
    F.m[3 * b + a] = l;
  }
  for (int k = 0; k < sq; k++) {                         // (1 + F)^2 - 1 = F^2 + 2 F
    M3 t;
    mmul(F, F, t);
#pragma unroll
    for (int i = 0; i < 9; i++) F.m[i] = C2{__fma_rn(2.0, F.m[i].re, t.m[i].re), __fma_rn(2.0, F.m[i].im, t.m[i].im)};
  }
}

// U <- exp(c0 Z0 + c1 Z1 + c2 Z2) U for every link, as U + F U.
template <int NZ>
__global__ void __launch_bounds__(128) k_flow_update(double* __restrict__ U, const double* __restrict__ Z, long nlink,
                                                    double c0, double c1, double c2) {
  const long k = (long)blockIdx.x * blockDim.x + threadIdx.x;
  if (k >= nlink) return;
  double x[9];
#pragma unroll
  for (int i = 0; i < 9; i++) {
    double v = c0 * Z[(long)i * nlink + k];
    if (NZ > 1) v += c1 * Z[(long)(9 + i) * nlink + k];
    if (NZ > 2) v += c2 * Z[(long)(18 + i) * nlink + k];
    x[i] = v;
  }
  const double d[3] = {x[0], x[1], x[2]};
  const C2 o[3] = {{x[3], x[4]}, {x[5], x[6]}, {x[7], x[8]}};
  M3 F;
  mexpm1(d, o, F);
  // column by column of U (three complex numbers live at a time)
  double* u = U + 18 * k;
#pragma unroll
  for (int j = 0; j < 3; j++) {
    const C2 v[3] = {ldc(u + 2 * j), ldc(u + 6 + 2 * j), ldc(u + 12 + 2 * j)};
#pragma unroll
    for (int i = 0; i < 3; i++) {
      C2 s{0.0, 0.0};
#pragma unroll
      for (int m = 0; m < 3; m++) cfma(F.m[3 * i + m], v[m], s);
      u[6 * i + 2 * j] = v[i].re + s.re;
      u[6 * i + 2 * j + 1] = v[i].im + s.im;
    }
  }
}

// Re tr of a plaquette is Re tr(A B^+) with A = U_mu(x) U_nu(x+mu), B = U_nu(x) U_mu(x+nu):
// two matrix products and a contraction.  A thread per (site, plane); a block writes the
// sum of its threads in a fixed order.
__global__ void __launch_bounds__(192) k_plaq(const double* __restrict__ U, double* __restrict__ part, Lat g) {
  __shared__ double sh[192];
  const long i = (long)blockIdx.x * 192 + threadIdx.x;
  double tot = 0.0;
  if (i < 6 * g.V) {
    const long s = i / 6;
    const int pl = (int)(i - 6 * s);
    const int mu = pl < 3 ? 0 : pl < 5 ? 1 : 2;
    const int nu = pl < 3 ? pl + 1 : pl < 5 ? pl - 1 : 3;
    int c[4];
    long r = s;
    for (int k = 0; k < 4; k++) { c[k] = (int)(r % g.L[k]); r /= g.L[k]; }
    const double* um = lnk(U, s, mu);
    const double* un = lnk(U, s, nu);
    const double* unp = lnk(U, lat_nbr(g, c, mu, +1), nu);
    const double* ump = lnk(U, lat_nbr(g, c, nu, +1), mu);
#pragma unroll
    for (int row = 0; row < 3; row++) {
      C2 v[3], a[3], b[3];
#pragma unroll
      for (int j = 0; j < 3; j++) v[j] = ldc(um + 6 * row + 2 * j);
      vmul<false, false>(v, unp, a);
#pragma unroll
      for (int j = 0; j < 3; j++) v[j] = ldc(un + 6 * row + 2 * j);
      vmul<false, false>(v, ump, b);
#pragma unroll
      for (int j = 0; j < 3; j++) tot = __fma_rn(a[j].re, b[j].re, __fma_rn(a[j].im, b[j].im, tot));
    }
  }
  sh[threadIdx.x] = tot;
  __syncthreads();
  for (int w = 96; w >= 3; w >>= 1) {
    if ((int)threadIdx.x < w) sh[threadIdx.x] += sh[threadIdx.x + w];
    __syncthreads();
  }
  if (threadIdx.x == 0) part[blockIdx.x] = sh[0] + sh[1] + sh[2];
}

// Fixed-order sum of n doubles by one block.
__global__ void __launch_bounds__(1024) k_sum(const double* __restrict__ v, long n, double* out) {
  __shared__ double sh[1024];
  double s = 0.0;
  for (long i = threadIdx.x; i < n; i += 1024) s += v[i];
  sh[threadIdx.x] = s;
  __syncthreads();
  for (int w = 512; w > 0; w >>= 1) {
    if ((int)threadIdx.x < w) sh[threadIdx.x] += sh[threadIdx.x + w];
    __syncthreads();
  }
  if (threadIdx.x == 0) *out = sh[0];
}

}  // namespace

cudaError_t wilson_flow(double* U, const int L[4], double eps, int nsteps, double* Z, cudaStream_t st) {
  Lat g;
  for (int i = 0; i < 4; i++) g.L[i] = L[i];
  g.V = (long)L[0] * L[1] * L[2] * L[3];
  const long nlink = 4 * g.V;
  const unsigned gz = (unsigned)((nlink + kZLinks - 1) / kZLinks), gu = (unsigned)((nlink + 127) / 128);
  for (int n = 0; n < nsteps; n++) {
    k_flow_Z<<<gz, 3 * kZLinks, 0, st>>>(U, Z, g, eps);
    k_flow_update<1><<<gu, 128, 0, st>>>(U, Z, nlink, 0.25, 0.0, 0.0);
    k_flow_Z<<<gz, 3 * kZLinks, 0, st>>>(U, Z + 9 * nlink, g, eps);
    k_flow_update<2><<<gu, 128, 0, st>>>(U, Z, nlink, -17.0 / 36.0, 8.0 / 9.0, 0.0);
    k_flow_Z<<<gz, 3 * kZLinks, 0, st>>>(U, Z + 18 * nlink, g, eps);
    k_flow_update<3><<<gu, 128, 0, st>>>(U, Z, nlink, 17.0 / 36.0, -8.0 / 9.0, 0.75);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

cudaError_t plaquette(const double* U, const int L[4], double* part, double* out, cudaStream_t st) {
  Lat g;
  for (int i = 0; i < 4; i++) g.L[i] = L[i];
  g.V = (long)L[0] * L[1] * L[2] * L[3];
  const long nb = (6 * g.V + 191) / 192;
  k_plaq<<<(unsigned)nb, 192, 0, st>>>(U, part, g);
  k_sum<<<1, 1024, 0, st>>>(part, nb, out);
  return cudaGetLastError();
}

}  // namespace mdwf
