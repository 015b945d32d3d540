// FP64 Wilson hop on all L5 slices x RHS slots with the fifth-dimension epilogues
// (the forms E_RAW ... E_AINVD_SAME, see hop_fast.cu), on the solver's parity
// fields or directly on the caller's arrays (C ABI layout).
//
// What bounds it: an FP64 instruction of a warp occupies its scheduler's FP64
// unit for 64 clocks however many of its lanes are active (two lanes per SM and clock: 6.3e11
// instructions per second on 152 SMs at 2070 MHz), 40 times the cost of anything else the kernel does.  So
// the kernel is built for full warps and few FP64 instructions, and spends loads,
// shuffles and integer work freely:
// * eight lanes per unit (site, s, r): lane (mu, j) does both hops of direction mu
//   for the projected spin j.  A warp holds four units whatever L5, N and the
//   lattice are (a thread per unit left half of the lanes idle at N = 1, L5 = 8, and
//   a 4^3 x 8 lattice on a few schedulers); on small lattices the work spreads eight
//   times wider.
// * x_b = U^+ h_b and x_f = U h_f, each rounded by itself, then S = x_b + x_f and D = x_b - x_f: the
//   upper spins sum S over the directions, the lower ones D with the gamma matrices' factors: 105
//   instructions per lane, 840 per unit (896 by ncu, with the signs of the projections), where the
//   accumulation of every product into all four spins took 864.  Chaining U h_f onto x_b and taking D = 2 x_b - S saves 6 of the 105, but rounds at the size of
//   the sum: 1.05 times the error of that accumulation in H (1.57e-16 against 1.49e-16, rms of the result,
//   extended precision as the reference), this order 0.93 times (1.38e-16).
// * the sums over the directions are a reduce-scatter by shuffles; factors 1, -1, i, -i
//   are exchanges and sign bits.
// * slots whose mask is off are left out of the enumeration, so a re-reference of a
//   few systems costs what they need.
// * the epilogues run over (unit, component) or (column, component) items of a
//   shared-memory tile, with the coefficients folded (3 to 4 instructions per
//   component).
// * three blocks of eight warps per SM (80 registers, with up to 20 bytes of spills per thread, 60 to 68 in three
//   of the column epilogues): 24 warps hide the loads and shuffles better than the 16 of an unbounded kernel (104
//   registers; D below, measured with the chained products: 4.50 ms with 24 warps, 4.68 with 16); 32 (64
//   registers) measured the same as 24.
// D of one field at 16^3 x 48, L5 = 12: 6.61 ms with a thread per unit and packing to parity fields, 4.73 so,
// of which 3.9 ms are FP64 (962 instructions per unit here, 72 in B in); H^+ at 6 x 4 x 2 x 10, L5 = 5:
// 138 -> 26 us; an FP64 solve at 4^3 x 8, L5 = 4: 28.2 -> 8.7 ms.
// A unit's result depends on nothing but its inputs: every block shape, slot count
// and mask, the decomposed lattice (halo terms) and both layouts give the same bits.
#include "mdwf_internal.h"
#include "hop_common.cuh"

namespace mdwf {

namespace {

// Element index of component cp of slice s, slot r at a site.
template <bool API>
struct Map;
template <>
struct Map<false> {      // parity field: planes of 16-byte words, unit (h L5 + s) N + r
  static __device__ __forceinline__ long at(const FastArgs<double, double>& a, long lex, int s, int r, int cp) {
    return 2 * ((cp >> 1) * plane_of(a) + ((lex >> 1) * a.L5 + s) * a.N + r) + (cp & 1);
  }
  // the six reals of a spin
  static __device__ __forceinline__ void load6(const FastArgs<double, double>& a, const double* __restrict__ f, long lex,
                                               int s, int r, int spin, double* v) {
    const long pl = plane_of(a);
    const double2* p = reinterpret_cast<const double2*>(f) + 3 * spin * pl + ((lex >> 1) * a.L5 + s) * a.N + r;
#pragma unroll
    for (int i = 0; i < 3; i++) {
      const double2 t = __ldg(p + i * pl);
      v[2 * i] = t.x;
      v[2 * i + 1] = t.y;
    }
  }
};
template <>
struct Map<true> {       // the caller's layout [s][lex][24], one slot; aligned to a double
  static __device__ __forceinline__ long at(const FastArgs<double, double>& a, long lex, int s, int, int cp) {
    return ((long)s * a.g.V + lex) * 24 + cp;
  }
  static __device__ __forceinline__ void load6(const FastArgs<double, double>& a, const double* __restrict__ f, long lex,
                                               int s, int r, int spin, double* v) {
    const double* p = f + at(a, lex, s, r, 6 * spin);
#pragma unroll
    for (int i = 0; i < 6; i++) v[i] = __ldg(p + i);
  }
};

struct Shape64 {
  int nsb;               // sites per block
  int rt;                // slots per block
};

__device__ __forceinline__ double flip(double v, unsigned bit31) {      // v or -v
  return __hiloint2double(__double2hiint(v) ^ (int)bit31, __double2loint(v));
}
__device__ __forceinline__ double sx(double v, int m) { return __shfl_xor_sync(0xffffffffu, v, m); }

// o = M v with M_ab = l[a][b] (DAG: conj(l[b][a])), the operations of a colour multiply in their
// usual order: one multiply and five multiply-adds per real output.
template <bool DAG>
__device__ __forceinline__ void colour_mul(const double* __restrict__ l, const double* v, double* o) {
#pragma unroll
  for (int a = 0; a < 3; a++) {
    double re, im;
#pragma unroll
    for (int b = 0; b < 3; b++) {
      const double2 u = __ldg(reinterpret_cast<const double2*>(l) + (DAG ? 3 * b + a : 3 * a + b));
      const double ui = DAG ? -u.y : u.y;
      if (b == 0) { re = u.x * v[0]; im = u.x * v[1]; }
      else { re = __fma_rn(u.x, v[2 * b], re); im = __fma_rn(u.x, v[2 * b + 1], im); }
      re = __fma_rn(-ui, v[2 * b + 1], re);
      im = __fma_rn(ui, v[2 * b], im);
    }
    o[2 * a] = re;
    o[2 * a + 1] = im;
  }
}

// B y_k = b5 x_k + c5 x_{k-1} and A^-1 along a column of the tile (k along the recursion direction,
// stride st doubles; see hop_fast.cu).
__device__ __forceinline__ void col_ainv64(double* c, long st, int L, const Fifth<double>& f, double m) {
  double z = 0.0;
  for (int k = 0; k < L; k++) { z = __fma_rn(-f.kap, z, c[k * st] * f.inv_alpha); c[k * st] = z; }
  const double yl = z / __fma_rn(m, f.powL, 1.0);
  c[(L - 1) * st] = yl;
  double w = m * yl * -f.kap;
  for (int k = 0; k < L - 1; k++) { c[k * st] -= w; w *= -f.kap; }
}
__device__ __forceinline__ void col_bop64(double* c, long st, int L, const Fifth<double>& f, double m) {
  double prev = -m * c[(L - 1) * st];
  for (int k = 0; k < L; k++) { const double x = c[k * st]; c[k * st] = __fma_rn(f.c5, prev, f.b5 * x); prev = x; }
}
// The same with the column in registers (compile-time length).
template <int EPI, int L>
__device__ __forceinline__ void col_regs64(double* c, long st, const Fifth<double>& f, double m) {
  double v[L];
#pragma unroll
  for (int k = 0; k < L; k++) v[k] = c[k * st];
  auto bop = [&]() {
    double prev = -m * v[L - 1];
#pragma unroll
    for (int k = 0; k < L; k++) { const double x = v[k]; v[k] = __fma_rn(f.c5, prev, f.b5 * x); prev = x; }
  };
  auto ainv = [&]() {
    double z = 0.0;
#pragma unroll
    for (int k = 0; k < L; k++) { z = __fma_rn(-f.kap, z, v[k] * f.inv_alpha); v[k] = z; }
    v[L - 1] = z / __fma_rn(m, f.powL, 1.0);
    double w = m * v[L - 1] * -f.kap;
#pragma unroll
    for (int k = 0; k < L - 1; k++) { v[k] -= w; w *= -f.kap; }
  };
  if (EPI == E_BAINV) { ainv(); bop(); }
  else if (EPI == E_AINVD_BD) { bop(); ainv(); }
  else ainv();
#pragma unroll
  for (int k = 0; k < L; k++) c[k * st] = v[k];
}
// FP64 Schur operator of four fields at 8^3 x 16, register columns against the tile: 467.7 against 470.1 us at L5 = 6,
// 591 against 593 at 8, 730 against 734 at 10, 840 against 853 at 12, 1092 against 1099 at 16.
template <int EPI>
__device__ __forceinline__ void column64(double* c, long st, int L, const Fifth<double>& f, double m) {
  switch (L) {
#define MDWF_CASE(L) case L: col_regs64<EPI, L>(c, st, f, m); break;
    MDWF_COLUMN_LENGTHS(MDWF_CASE)
#undef MDWF_CASE
    default:
      if (EPI == E_BAINV) { col_ainv64(c, st, L, f, m); col_bop64(c, st, L, f, m); }
      else if (EPI == E_AINVD_BD) { col_bop64(c, st, L, f, m); col_ainv64(c, st, L, f, m); }
      else col_ainv64(c, st, L, f, m);
  }
}

constexpr int kRow64 = 25;       // doubles between the rows of the tile (odd: lanes of one component hit all banks)

template <int EPI, bool API>
__global__ void __launch_bounds__(256, 3) hop64_kernel(FastArgs<double, double> a, Shape64 p) {
  extern __shared__ __align__(16) double tile[];            // [nsb L5 rt][kRow64], then the slot list
  constexpr bool kCols = (EPI == E_BAINV || EPI == E_AINVD_BD || EPI == E_AINV_SAME || EPI == E_SAME_AINV ||
                          EPI == E_AINVD_SAME);
  constexpr bool kSameFirst = (EPI == E_AINV_SAME || EPI == E_AINVD_SAME);
  constexpr bool kBdag = (EPI == E_AD_SAME_BD || EPI == E_SAME_BD);
  const int L5 = a.L5;
  int* slots = reinterpret_cast<int*>(tile + (size_t)p.nsb * L5 * p.rt * kRow64);
  const int nthr = blockDim.x, tid = threadIdx.x, lane = tid & 31;
  const int par = API && a.out_par < 0 ? (int)blockIdx.z : a.out_par;
  // the group's active slots, in order
  if (tid < 32) {
    int n = 0;
    for (int b = 0; b < p.rt; b += 32) {
      const int r = blockIdx.y * p.rt + b + lane;
      const bool on = b + lane < p.rt && r < a.N && (a.active == nullptr || a.active[r] != 0);
      const unsigned m = __ballot_sync(0xffffffffu, on);
      if (on) slots[1 + n + __popc(m & ((1u << lane) - 1))] = r;
      n += __popc(m);
    }
    if (lane == 0) slots[0] = n;
  }
  __syncthreads();
  const int na = slots[0];
  if (na == 0) return;
  const long h0 = (long)blockIdx.x * p.nsb;
  const int ns = (int)(a.g.Vh - h0 < p.nsb ? a.g.Vh - h0 : p.nsb);
  const int nu = ns * L5 * na;                              // units of the block: (site, s, active slot)

  if (a.in != nullptr) {
    const int mu = (lane >> 1) & 3, j = lane & 1;
    const bool xy = mu < 2, sw = (mu & 1) == 0;             // x, y exchange spins; x, z carry an i
    // h = p_j + sg sigma (i) p_partner, sigma = -1 for (y, 0) and (z, 1), else 1
    const double sgf = a.dagger ? 1.0 : -1.0;
    const double sig = (mu == 1 && j == 0) || (mu == 2 && j == 1) ? -1.0 : 1.0;
    const int spin_p = xy ? 3 - j : 2 + j;
    // factor of sg_b D on the lower spin (3 - j for x, y; 2 + j for z, t): x: -i; y: 1 (j = 1), -1 (j = 0);
    // z: -i (j = 0), i (j = 1); t: 1.  With re and im exchanged for -i and i.
    const bool neg = (mu == 1 && j == 0) != (a.dagger != 0);             // the sign of sg_b = -sgf folded in
    const bool pos_i = mu == 2 && j == 1;                                // +i, else -i (x, z)
    const unsigned fr = sw ? ((pos_i != (a.dagger != 0)) ? 0x80000000u : 0u) : (neg ? 0x80000000u : 0u);
    const unsigned fi = sw ? ((pos_i != (a.dagger != 0)) ? 0u : 0x80000000u) : (neg ? 0x80000000u : 0u);
    const int st = mu == 0 ? 1 : mu == 1 ? a.g.L[0] : mu == 2 ? a.g.L[0] * a.g.L[1] : a.g.L[0] * a.g.L[1] * a.g.L[2];
    const int Lm = mu == 0 ? a.g.L[0] : mu == 1 ? a.g.L[1] : mu == 2 ? a.g.L[2] : a.g.L[3];
    for (int q = tid >> 5; q * 4 < nu; q += nthr >> 5) {
      const int i = q * 4 + (lane >> 3);
      const int ul = i < nu ? i : nu - 1;
      const int k = ul / na, r = slots[1 + ul - k * na];
      const int site_l = k / L5, s = k - site_l * L5;
      const long h = h0 + site_l;
      int c[4];
      site_coords(a.g, par, h, c);
      const long lex = lex_index(a.g, c);
      const int cm = mu == 0 ? c[0] : mu == 1 ? c[1] : mu == 2 ? c[2] : c[3];
      const bool ef = cm == Lm - 1, eb = cm == 0;
      const long nf = ef ? lex - (long)(Lm - 1) * st : lex + st;
      const long nb = eb ? lex + (long)(Lm - 1) * st : lex - st;
      const bool halo = API && mu == 3 && a.halo_fwd != nullptr, hf = halo && ef, hb = halo && eb;
      const bool flf = mu == 3 && ef && a.antiperiodic, flb = mu == 3 && eb && a.antiperiodic;
      // projected neighbours
      auto project = [&](long n, double sg, double* v) {
        double e[6];
        Map<API>::load6(a, a.in, n, s, r, j, v);
        Map<API>::load6(a, a.in, n, s, r, spin_p, e);
        const double f = sg * sig, f0 = sw ? -f : f;
#pragma unroll
        for (int b = 0; b < 3; b++) {
          v[2 * b] = __fma_rn(f0, sw ? e[2 * b + 1] : e[2 * b], v[2 * b]);
          v[2 * b + 1] = __fma_rn(f, sw ? e[2 * b] : e[2 * b + 1], v[2 * b + 1]);
        }
      };
      const long lex3 = lex - (long)c[3] * a.g.L[0] * a.g.L[1] * a.g.L[2];
      double v[6], xb[6], xf[6], S[6], D[6];
      if (hb) {
        const double* hp = a.halo_bwd + ((lex3 * L5 + s) * a.N + r) * 12 + 6 * j;
#pragma unroll
        for (int b = 0; b < 6; b++) xb[b] = hp[b] * a.halo_sgn_bwd;
      } else {
        project(nb, -sgf, v);
        if (flb) {
#pragma unroll
          for (int b = 0; b < 6; b++) v[b] = flip(v[b], 0x80000000u);
        }
        colour_mul<true>(a.U + (((long)(1 - par) * a.g.Vh + (nb >> 1)) * 4 + mu) * 18, v, xb);
      }
      if (hf) {
        const double* hp = a.halo_fwd + ((lex3 * L5 + s) * a.N + r) * 12 + 6 * j;
#pragma unroll
        for (int b = 0; b < 6; b++) v[b] = hp[b] * a.halo_sgn_fwd;
      } else {
        project(nf, sgf, v);
        if (flf) {
#pragma unroll
          for (int b = 0; b < 6; b++) v[b] = flip(v[b], 0x80000000u);
        }
      }
      colour_mul<false>(a.U + (((long)par * a.g.Vh + h) * 4 + mu) * 18, v, xf);
#pragma unroll
      for (int b = 0; b < 6; b++) { S[b] = xb[b] + xf[b]; D[b] = xb[b] - xf[b]; }
      // factor on the lower spin, then x, y lanes hand theirs to the lane of its spin
      double E[6];
#pragma unroll
      for (int b = 0; b < 3; b++) {
        E[2 * b] = flip(sw ? D[2 * b + 1] : D[2 * b], fr);
        E[2 * b + 1] = flip(sw ? D[2 * b] : D[2 * b + 1], fi);
      }
#pragma unroll
      for (int b = 0; b < 6; b++) { const double o = sx(E[b], 1); E[b] = xy ? o : E[b]; }
      // sum over the four directions: mu < 2 keep S (upper spin j), mu >= 2 keep E (lower spin 2 + j),
      // then even mu the first three reals, odd mu the last three
      double w[6], z[3];
#pragma unroll
      for (int b = 0; b < 6; b++) { const double o = sx(xy ? E[b] : S[b], 4); w[b] = (xy ? S[b] : E[b]) + o; }
#pragma unroll
      for (int b = 0; b < 3; b++) { const double o = sx((mu & 1) ? w[b] : w[3 + b], 2); z[b] = ((mu & 1) ? w[3 + b] : w[b]) + o; }
      if (i < nu) {
        double* t = tile + (size_t)ul * kRow64 + 6 * (xy ? j : 2 + j) + 3 * (mu & 1);
#pragma unroll
        for (int b = 0; b < 3; b++) t[b] = z[b];
      }
    }
    __syncthreads();
  }

  // (unit ul, component): ul = (site_l L5 + s) na + slot
  auto site_of = [&](int k, long* lex) {
    int c[4];
    const long h = h0 + k;
    site_coords(a.g, par, h, c);
    *lex = lex_index(a.g, c);
  };
  if (kCols) {
    // v = kappa H (+ same), then the recursion along s
    const long st = (long)na * kRow64;
    for (int it = tid; it < ns * na * 24; it += nthr) {
      const int cp = it % 24, k = it / 24, site_l = k / na, rl = k - site_l * na, r = slots[1 + rl];
      double* col = tile + ((size_t)site_l * L5 * na + rl) * kRow64 + cp;
      long lex = 0;
      if (kSameFirst) site_of(site_l, &lex);
      if (kSameFirst || a.kappa != 1.0)
        for (int s = 0; s < L5; s++) {
          const double hv = a.in != nullptr ? col[s * st] : 0.0;
          col[s * st] = kSameFirst ? __fma_rn(a.kappa, hv, a.same[Map<API>::at(a, lex, s, r, cp)]) : a.kappa * hv;
        }
      const bool upper = cp < 12, down = (EPI == E_AINVD_BD || EPI == E_AINVD_SAME) ? !upper : upper;
      column64<EPI>(down ? col : col + (L5 - 1) * st, down ? st : -st, L5, a.f, a.f.mass[r]);
    }
    __syncthreads();
  }
  constexpr bool kAdd = EPI == E_RAW || EPI == E_A_SAME || EPI == E_AD_SAME_BD || EPI == E_SAME_AINV || EPI == E_SAME_BD;
  const bool norm = a.partials != nullptr;
  const double ga = a.g_same * a.f.alpha, gb = a.g_same * a.f.beta, kc = a.kappa * a.f.c5, kb = a.kappa * a.f.b5;
  for (int it = tid; it < nu * 24; it += nthr) {
    const int ul = it / 24, cp = it - 24 * ul;
    const int k = ul / na, r = slots[1 + ul - k * na], site_l = k / L5, s = k - site_l * L5;
    long lex;
    site_of(site_l, &lex);
    const bool upper = cp < 12;
    double* t = tile + (size_t)ul * kRow64 + cp;
    double o = a.in != nullptr || kSameFirst ? *t : 0.0;
    // neighbour slices with the wall factor -m
    const int sd = s == 0 ? L5 - 1 : s - 1, sp = s == L5 - 1 ? 0 : s + 1;
    if (kBdag) {
      // B^+ (kappa H): P_+ half from slice s + 1, P_- half from slice s - 1
      const int sn = upper ? sp : sd;
      double cw = kc;
      if (upper ? s == L5 - 1 : s == 0) cw = kc * -a.f.mass[r];
      const double hn = a.in != nullptr ? t[(sn - s) * (long)na * kRow64] : 0.0;
      o = __fma_rn(cw, hn, kb * o);
    } else if ((EPI == E_RAW || EPI == E_A_SAME) && a.kappa != 1.0) {
      o = a.kappa * o;
    }
    if ((EPI == E_A_SAME || EPI == E_AD_SAME_BD) && a.g_same != 0.0) {
      // g A y: P_+ half alpha y_s + beta y_{s-1} (A) or y_{s+1} (A^+), P_- half the other neighbour
      const bool from_up = upper == (EPI == E_AD_SAME_BD);
      const int sn = from_up ? sp : sd;
      double gw = gb;
      if (from_up ? s == L5 - 1 : s == 0) gw = gb * -a.f.mass[r];
      const double y = a.same[Map<API>::at(a, lex, s, r, cp)];
      const double yn = a.same[Map<API>::at(a, lex, sn, r, cp)];
      o = __fma_rn(ga, y, __fma_rn(gw, yn, o));
    }
    if ((EPI == E_SAME_AINV || EPI == E_SAME_BD) && a.g_same != 0.0)
      o = __fma_rn(a.g_same, a.same[Map<API>::at(a, lex, s, r, cp)], o);
    if (kAdd && a.add != nullptr) o += a.add[Map<API>::at(a, lex, s, r, cp)];
    a.out[Map<API>::at(a, lex, s, r, cp)] = o;
    // the B^+ forms still read the tile of other units: their norms are formed from the stored output
    if (norm && !kBdag) *t = o;
  }
  if (norm) {
    // per-site, per-slot sums over the L5 slices (fixed order), stored as partials[r][h]: eight lanes per
    // unit, three components each, then the slices in order
    __syncthreads();
    for (int q = tid >> 5; q * 4 < nu; q += nthr >> 5) {
      const int i = q * 4 + (lane >> 3), ul = i < nu ? i : nu - 1;
      double* t = tile + (size_t)ul * kRow64 + 3 * (lane & 7);
      double n2 = 0.0;
      if (kBdag) {
        const int k = ul / na, r = slots[1 + ul - k * na], site_l = k / L5, s = k - site_l * L5;
        long lex;
        site_of(site_l, &lex);
#pragma unroll
        for (int b = 0; b < 3; b++) {
          const double o = a.out[Map<API>::at(a, lex, s, r, 3 * (lane & 7) + b)];
          n2 = __fma_rn(o, o, n2);
        }
      } else {
#pragma unroll
        for (int b = 0; b < 3; b++) n2 = __fma_rn(t[b], t[b], n2);
      }
      n2 += sx(n2, 1);
      n2 += sx(n2, 2);
      n2 += sx(n2, 4);
      if (i < nu && (lane & 7) == 0) tile[(size_t)ul * kRow64 + 24] = n2;       // the row's padding
    }
    __syncthreads();
    for (int it = tid; it < ns * na; it += nthr) {
      const int site_l = it / na, rl = it - site_l * na;
      double sum = 0.0;
      for (int s = 0; s < L5; s++) sum += tile[((size_t)(site_l * L5 + s) * na + rl) * kRow64 + 24];
      a.partials[(long)slots[1 + rl] * a.g.Vh + h0 + site_l] = sum;
    }
  }
}

template <int EPI, bool API>
cudaError_t launch64_one(const FastArgs<double, double>& a, const Tiling& t, cudaStream_t st) {
  const int warps = (t.threads + 3) / 4;                   // four units per warp
  // at least three warps: the epilogue's items (24 per unit) fill them where the units don't
  // (4^3 x 8, L5 = 4: 9.1 ms per FP64 solve with one warp per block, 8.7 with three)
  const int threads = 32 * (warps > 8 ? 8 : warps < 3 ? 3 : warps);
  const size_t smem = (size_t)t.threads * kRow64 * sizeof(double) + sizeof(int) * (t.rt + 1);
  auto* kern = hop64_kernel<EPI, API>;
  if (smem > 48 * 1024) {
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
  }
  const dim3 grid((unsigned)t.ntiles, (unsigned)t.ngroups, API && a.out_par < 0 ? 2u : 1u);
  kern<<<grid, threads, smem, st>>>(a, Shape64{t.nsb, t.rt});
  return cudaGetLastError();
}

// (b5 + c5 P) x of one component on the caller's layout: the elements of P_+ from slice s - 1, of P_- from s + 1.
__global__ void __launch_bounds__(256) k_bop_api(const double* __restrict__ x, double* __restrict__ u, long n, int L5,
                                                 double b5, double c5, double m) {
  const long i = (long)blockIdx.x * 256 + threadIdx.x;      // element of one slice
  if (i >= n) return;
  const bool upper = i % 24 < 12;
  const int s = blockIdx.y;
  const int sn = upper ? (s == 0 ? L5 - 1 : s - 1) : (s == L5 - 1 ? 0 : s + 1);
  const bool wall = upper ? s == 0 : s == L5 - 1;
  double cw = c5;
  if (wall) cw = c5 * -m;
  u[(long)s * n + i] = bop_term(b5, x[(long)s * n + i], cw, x[(long)sn * n + i]);
}

// A column (one component of one site, all slices) per thread, read once into shared memory.
constexpr int kLocal5 = 128;
__global__ void __launch_bounds__(kLocal5) k_local5_api(const double* __restrict__ in, double* __restrict__ out,
                                                        const double* __restrict__ G, long n, int L5) {
  extern __shared__ double col[];      // [slice][thread]
  const long i = (long)blockIdx.x * kLocal5 + threadIdx.x;
  if (i >= n) return;
  for (int s = 0; s < L5; s++) col[s * kLocal5 + threadIdx.x] = in[(long)s * n + i];
  const double* M = G + (i % 24 < 12 ? 0 : L5 * L5);
  for (int s = 0; s < L5; s++) {
    double o = 0.0;
    for (int k = 0; k < L5; k++) o = __fma_rn(__ldg(M + s * L5 + k), col[k * kLocal5 + threadIdx.x], o);
    out[(long)s * n + i] = o;
  }
}

}  // namespace

// Sites and slots per block: about 32 units (one pass of eight warps, a tile of 6.4 KB), whole sites; large sites
// are split into slot groups so that the tile stays within 100 KB, two blocks per SM.  nsb: that many sites
// instead, as far as such a tile holds them; 0: the choice made here.
Tiling hop64_tiling(long Vh, int L5, int N, int nsb) {
  const size_t unit = kRow64 * sizeof(double), most = 100 * 1024;
  Tiling t;
  t.ngroups = 1;
  while (t.ngroups < N && (size_t)((N + t.ngroups - 1) / t.ngroups) * L5 * unit > most) t.ngroups++;
  t.rt = (N + t.ngroups - 1) / t.ngroups;
  t.ngroups = (N + t.rt - 1) / t.rt;
  t.nsb = nsb > 0 ? (nsb < 64 ? nsb : 64) : 32 / (L5 * t.rt);
  if (nsb > 0) {
    while (t.nsb > 1 && (size_t)t.nsb * L5 * t.rt * unit > most) t.nsb--;
  } else {
    // small lattices: fewer sites per block while that leaves schedulers idle (152 SMs x 4)
    while (t.nsb > 1 && (Vh / t.nsb) * ((t.nsb * L5 * t.rt + 3) / 4) * t.ngroups < 608) t.nsb--;
  }
  if (t.nsb < 1) t.nsb = 1;
  t.ntiles = (Vh + t.nsb - 1) / t.nsb;
  t.threads = t.nsb * L5 * t.rt;                           // units of a block
  return t;
}

cudaError_t launch_hop64(const FastArgs<double, double>& a, const Tiling& t, int epi, cudaStream_t st) {
  if (a.N < 1 || a.L5 < 1 || a.g.Vh < 1) return cudaErrorInvalidValue;
  switch (epi) {
    case E_RAW: return launch64_one<E_RAW, false>(a, t, st);
    case E_BAINV: return launch64_one<E_BAINV, false>(a, t, st);
    case E_AINVD_BD: return launch64_one<E_AINVD_BD, false>(a, t, st);
    case E_A_SAME: return launch64_one<E_A_SAME, false>(a, t, st);
    case E_AD_SAME_BD: return launch64_one<E_AD_SAME_BD, false>(a, t, st);
    case E_AINV_SAME: return launch64_one<E_AINV_SAME, false>(a, t, st);
    case E_SAME_AINV: return launch64_one<E_SAME_AINV, false>(a, t, st);
    case E_SAME_BD: return launch64_one<E_SAME_BD, false>(a, t, st);
    case E_AINVD_SAME: return launch64_one<E_AINVD_SAME, false>(a, t, st);
    default: return cudaErrorInvalidValue;
  }
}

cudaError_t launch_hop64_api(const FastArgs<double, double>& a, int epi, cudaStream_t st) {
  if (a.N != 1 || a.L5 < 1 || a.g.Vh < 1) return cudaErrorInvalidValue;
  const Tiling t = hop64_tiling(a.g.Vh, a.L5, 1, 0);
  switch (epi) {
    case E_RAW: return launch64_one<E_RAW, true>(a, t, st);
    case E_A_SAME: return launch64_one<E_A_SAME, true>(a, t, st);
    case E_AD_SAME_BD: return launch64_one<E_AD_SAME_BD, true>(a, t, st);
    default: return cudaErrorInvalidValue;
  }
}

cudaError_t bop_api(const double* x, double* u, long V, int L5, double b5, double c5, double m, cudaStream_t st) {
  const long n = 24 * V;
  k_bop_api<<<dim3((unsigned)((n + 255) / 256), (unsigned)L5), 256, 0, st>>>(x, u, n, L5, b5, c5, m);
  return cudaGetLastError();
}

cudaError_t local5_api(const double* in, double* out, const double* G, long V, int L5, cudaStream_t st) {
  const long n = 24 * V;
  const size_t smem = sizeof(double) * kLocal5 * L5;
  k_local5_api<<<(unsigned)((n + kLocal5 - 1) / kLocal5), kLocal5, smem, st>>>(in, out, G, n, L5);
  return cudaGetLastError();
}

}  // namespace mdwf
