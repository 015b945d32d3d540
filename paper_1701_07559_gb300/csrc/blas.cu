// Vector kernels of the solver: layout conversion, precision conversion,
// the CG updates with their fused norms, and the fixed-order reductions.
//
// All unit-wise kernels use the tile mapping of the hop kernel (tile of nsb
// sites x L5 slices x rt slots per block), so per-slot partial sums are formed
// per tile in a fixed order and the final sum over tiles is also fixed: a
// slot's result does not depend on how many other slots share the launch.
#include <cooperative_groups.h>

#include "blas.h"

namespace mdwf {

struct Unit {
  long h;
  int s, r, site_l, r_l;
  bool valid;
  long u;
};

__device__ __forceinline__ Unit unit_of(const Tiling& tl, long Vh, int L5, int N) {
  Unit x;
  const int tid = threadIdx.x;
  x.r_l = tid % tl.rt;
  x.s = (tid / tl.rt) % L5;
  x.site_l = tid / (tl.rt * L5);
  x.h = (long)blockIdx.x * tl.nsb + x.site_l;
  x.r = blockIdx.y * tl.rt + x.r_l;
  x.valid = (x.h < Vh) && (x.r < N);
  x.u = (x.h * L5 + x.s) * N + x.r;
  return x;
}

// Per-site, per-slot sum of `v` over the L5 slices (fixed order), written to
// partials[r][h]; the final sum over sites is then independent of the tiling.
__device__ __forceinline__ void block_partial(double v, const Unit& x, const Tiling& tl, int L5, long Vh,
                                              double* __restrict__ partials) {
  __shared__ double sred[1024];
  sred[threadIdx.x] = v;
  __syncthreads();
  if (x.s == 0 && x.valid) {
    double sum = 0.0;
    for (int k = 0; k < L5; k++) sum += sred[(x.site_l * L5 + k) * tl.rt + x.r_l];
    partials[(long)x.r * Vh + x.h] = sum;
  }
}

// The caller's fields (C ABI layout, aligned to a double) of the slots r0 .. r0 + nr - 1 <-> one parity of a field.
// kPackUnits units per block, slots fastest (the words of consecutive slots are contiguous in the planes), through
// a shared-memory tile: the caller's side moves the 24 doubles of a unit as one 192-byte run, the field's side
// consecutive units of a plane.  Four FP64 fields of 8^3 x 16, L5 = 8: 8 us to unpack a parity, 32 us with a thread per
// unit that moves its 24 doubles by itself (192 bytes between the lanes of a warp).
constexpr int kPtrs = 64;
template <typename P>
struct Ptrs {
  P p[kPtrs];
};
constexpr int kPackUnits = 64;
constexpr int kPackRow = 25;

// Offset of a unit in its field, and the field, for the units of the block.
struct PackMap {
  long off[kPackUnits];
  long u[kPackUnits];
  int k[kPackUnits];
};
__device__ __forceinline__ int pack_map(PackMap& m, const Geom& g, int L5, int N, int par, int r0, int nr) {
  const long base = (long)blockIdx.x * kPackUnits, total = g.Vh * L5 * nr;
  const int n = total - base < kPackUnits ? (int)(total - base) : kPackUnits;
  if (threadIdx.x < n) {
    const long idx = base + threadIdx.x, hs = idx / nr, h = hs / L5;
    const int k = (int)(idx - hs * nr), s = (int)(hs - h * L5);
    int c[4];
    site_coords(g, par, h, c);
    m.off[threadIdx.x] = ((long)s * g.V + lex_index(g, c)) * 24;
    m.u[threadIdx.x] = hs * N + r0 + k;
    m.k[threadIdx.x] = k;
  }
  __syncthreads();
  return n;
}

template <typename S>
__global__ void __launch_bounds__(256) k_pack(Ptrs<const double*> api, S* __restrict__ out, float* __restrict__ out_nrm,
                                              Geom g, int L5, int N, int par, int r0, int nr) {
  using T = typename StoreTraits<S>::T;
  __shared__ PackMap m;
  __shared__ double tile[kPackUnits * kPackRow];
  const int n = pack_map(m, g, L5, N, par, r0, nr);
  for (int i = threadIdx.x; i < n * 24; i += 256) {
    const int u = i / 24, c = i - 24 * u;
    tile[u * kPackRow + c] = __ldg(api.p[m.k[u]] + m.off[u] + c);
  }
  __syncthreads();
  const long pl = g.Vh * L5 * N;
  if constexpr (std::is_same<S, double>::value) {
    for (int i = threadIdx.x; i < kPackUnits * 12; i += 256) {
      const int u = i % kPackUnits, w = i / kPackUnits;
      if (u < n)
        reinterpret_cast<double2*>(out)[w * pl + m.u[u]] =
            make_double2(tile[u * kPackRow + 2 * w], tile[u * kPackRow + 2 * w + 1]);
    }
  } else if (threadIdx.x < n) {
    T a[24];
#pragma unroll
    for (int i = 0; i < 24; i++) a[i] = (T)tile[threadIdx.x * kPackRow + i];
    store24<S, T>(out, out_nrm, pl, m.u[threadIdx.x], a);
  }
}

// in == null: zeros.
template <typename S>
__global__ void __launch_bounds__(256) k_unpack(const S* __restrict__ in, const float* __restrict__ in_nrm,
                                                Ptrs<double*> api, Geom g, int L5, int N, int par, int r0, int nr) {
  using T = typename StoreTraits<S>::T;
  __shared__ PackMap m;
  __shared__ double tile[kPackUnits * kPackRow];
  const int n = pack_map(m, g, L5, N, par, r0, nr);
  const long pl = g.Vh * L5 * N;
  if (in != nullptr) {
    if constexpr (std::is_same<S, double>::value) {
      for (int i = threadIdx.x; i < kPackUnits * 12; i += 256) {
        const int u = i % kPackUnits, w = i / kPackUnits;
        if (u < n) {
          const double2 v = __ldg(reinterpret_cast<const double2*>(in) + w * pl + m.u[u]);
          tile[u * kPackRow + 2 * w] = v.x;
          tile[u * kPackRow + 2 * w + 1] = v.y;
        }
      }
    } else if (threadIdx.x < n) {
      T a[24];
      load24<S, T>(in, in_nrm, pl, m.u[threadIdx.x], a);
#pragma unroll
      for (int i = 0; i < 24; i++) tile[threadIdx.x * kPackRow + i] = (double)a[i];
    }
    __syncthreads();
  }
  for (int i = threadIdx.x; i < n * 24; i += 256) {
    const int u = i / 24, c = i - 24 * u;
    api.p[m.k[u]][m.off[u] + c] = in != nullptr ? tile[u * kPackRow + c] : 0.0;
  }
}

template <typename Si, typename So>
__global__ void k_convert(const Si* __restrict__ in, const float* __restrict__ in_nrm, So* __restrict__ out,
                          float* __restrict__ out_nrm, Tiling tl, long Vh, int L5, int N, const int* __restrict__ mask) {
  const Unit x = unit_of(tl, Vh, L5, N);
  const long pl = Vh * L5 * N;
  if (!x.valid || (mask && !mask[x.r])) return;
  using Ti = typename StoreTraits<Si>::T;
  using To = typename StoreTraits<So>::T;
  Ti a[24];
  load24<Si, Ti>(in, in_nrm, pl, x.u, a);
  To b[24];
#pragma unroll
  for (int i = 0; i < 24; i++) b[i] = (To)a[i];
  store24<So, To>(out, out_nrm, pl, x.u, b);
}

__device__ __forceinline__ float axpy_fma(float a, float b, float c) { return __fmaf_rn(a, b, c); }
__device__ __forceinline__ double axpy_fma(double a, double b, double c) { return __fma_rn(a, b, c); }

// x += alpha_r p ; rho -= alpha_r q ; |rho|^2 of one unit, explicit roundings.
template <typename TX, typename T>
__device__ __forceinline__ T axpy_unit(T a, const T* pv, const T* qv, T* rv, TX* xv) {
  T n2t = 0;
#pragma unroll
  for (int i = 0; i < 24; i++) {
    xv[i] = axpy_fma((TX)a, (TX)pv[i], xv[i]);
    rv[i] = axpy_fma(-a, qv[i], rv[i]);
    n2t = axpy_fma(rv[i], rv[i], n2t);
  }
  return n2t;
}

template <typename SX, typename S>
__global__ void k_axpy_x_rho(SX* __restrict__ xv, const S* __restrict__ p, const float* __restrict__ p_nrm,
                             S* __restrict__ rho, float* __restrict__ rho_nrm, const S* __restrict__ q,
                             const float* __restrict__ q_nrm, const double* __restrict__ alpha, Tiling tl, long Vh,
                             int L5, int N, const int* __restrict__ active, double* __restrict__ partials) {
  using T = typename StoreTraits<S>::T;
  using TX = typename StoreTraits<SX>::T;
  const Unit x = unit_of(tl, Vh, L5, N);
  const long pl = Vh * L5 * N;
  double n2 = 0.0;
  if (x.valid && active[x.r]) {
    const T a = (T)alpha[x.r];
    T pv[24], qv[24], rv[24];
    TX xv_[24];
    load24<S, T>(p, p_nrm, pl, x.u, pv);
    load24<S, T>(q, q_nrm, pl, x.u, qv);
    load24<S, T>(rho, rho_nrm, pl, x.u, rv);
    load24<SX, SX>(xv, nullptr, pl, x.u, xv_);
    n2 = (double)axpy_unit<TX, T>(a, pv, qv, rv, xv_);
    store24<SX, SX>(xv, nullptr, pl, x.u, xv_);
    store24<S, T>(rho, rho_nrm, pl, x.u, rv);
  }
  block_partial(n2, x, tl, L5, Vh, partials);
}

// rho -= alpha_r q, |rho|^2, with the roundings of axpy_unit.
template <typename S>
__global__ void k_axpy_rho(S* __restrict__ rho, float* __restrict__ rho_nrm, const S* __restrict__ q,
                           const float* __restrict__ q_nrm, const double* __restrict__ alpha, Tiling tl, long Vh,
                           int L5, int N, const int* __restrict__ active, double* __restrict__ partials) {
  using T = typename StoreTraits<S>::T;
  const Unit x = unit_of(tl, Vh, L5, N);
  const long pl = Vh * L5 * N;
  double n2 = 0.0;
  if (x.valid && active[x.r]) {
    const T a = (T)alpha[x.r];
    T qv[24], rv[24];
    load24<S, T>(q, q_nrm, pl, x.u, qv);
    load24<S, T>(rho, rho_nrm, pl, x.u, rv);
    T n2t = 0;
#pragma unroll
    for (int i = 0; i < 24; i++) {
      rv[i] = axpy_fma(-a, qv[i], rv[i]);
      n2t = axpy_fma(rv[i], rv[i], n2t);
    }
    n2 = (double)n2t;
    store24<S, T>(rho, rho_nrm, pl, x.u, rv);
  }
  block_partial(n2, x, tl, L5, Vh, partials);
}

// x += alpha_r[i] p_i for the iterations i < taken[r] of a group, in their order (the
// same roundings as an update per iteration).  Bound by memory: x is read and written
// once per group of kGroup iterations instead of in each, and the search directions of a
// group, which lie in fields that the iterations don't use, are read once: 465 B per unit
// and iteration of fp16 vectors for all vector updates together instead of 609.  63 us per
// group at 995,000 units, 6.3 TB/s; a propagator at 16^3 x 32, L5 = 12, 12 systems:
// 1258 ms per solve with x updated in every iteration, 1222 in groups of two, 1206 of four.
template <typename SX, typename S>
__global__ void __launch_bounds__(sizeof(S) == 8 ? 512 : 1024) k_axpy_group(SX* __restrict__ xv, PGroup<S> p, int m,
                                                     const double* __restrict__ alpha, const int* __restrict__ taken,
                                                     Tiling tl, long Vh, int L5, int N) {
  using T = typename StoreTraits<S>::T;
  using TX = typename StoreTraits<SX>::T;
  const Unit x = unit_of(tl, Vh, L5, N);
  const long pl = Vh * L5 * N;
  if (!x.valid) return;
  const int k = taken[x.r] < m ? taken[x.r] : m;
  if (k == 0) return;
  TX xs[24];
  load24<SX, SX>(xv, nullptr, pl, x.u, xs);
#pragma unroll
  for (int j = 0; j < kGroup; j++) {
    if (j >= k) break;
    T pv[24];
    load24<S, T>(p.v[j], p.n[j], pl, x.u, pv);
    const T a = (T)alpha[(long)j * N + x.r];
#pragma unroll
    for (int i = 0; i < 24; i++) xs[i] = axpy_fma((TX)a, (TX)pv[i], xs[i]);
  }
  store24<SX, SX>(xv, nullptr, pl, x.u, xs);
}

// xhi += xlo ; xlo = 0
template <typename SX>
__global__ void k_accum_xhi(double* __restrict__ xhi, SX* __restrict__ xlo, Tiling tl, long Vh, int L5, int N,
                            const int* __restrict__ mask) {
  using TX = typename StoreTraits<SX>::T;
  const Unit x = unit_of(tl, Vh, L5, N);
  const long pl = Vh * L5 * N;
  if (!x.valid || (mask && !mask[x.r])) return;
  double h[24];
  TX l[24];
  load24<double, double>(xhi, nullptr, pl, x.u, h);
  load24<SX, SX>(xlo, nullptr, pl, x.u, l);
#pragma unroll
  for (int i = 0; i < 24; i++) { h[i] += (double)l[i]; l[i] = 0; }
  store24<double, double>(xhi, nullptr, pl, x.u, h);
  store24<SX, SX>(xlo, nullptr, pl, x.u, l);
}

template <typename S>
__global__ void k_norm2(const S* __restrict__ v, const float* __restrict__ v_nrm, Tiling tl, long Vh, int L5, int N,
                        const int* __restrict__ mask, double* __restrict__ partials) {
  using T = typename StoreTraits<S>::T;
  const Unit x = unit_of(tl, Vh, L5, N);
  const long pl = Vh * L5 * N;
  double n2 = 0.0;
  if (x.valid && (!mask || mask[x.r])) {
    T a[24];
    load24<S, T>(v, v_nrm, pl, x.u, a);
    T n2t = 0;
#pragma unroll
    for (int i = 0; i < 24; i++) n2t += a[i] * a[i];
    n2 = (double)n2t;
  }
  block_partial(n2, x, tl, L5, Vh, partials);
}

// The scalar steps of a CG iteration.
//
// |rho|^2: the low-precision residual recursion can stagnate for a system whose
// residual is already tiny: it neither reaches the stopping norm nor drops by
// delta, so no update would ever come.  After stag_max iterations without an
// update one is forced; it is followed by an FP64 re-reference and a restart of
// the search direction (beta = 0).
// The slot's scalars are loaded while the partial sums are.
struct Slot {
  int active, flags, since;
  double gamma, rho2_max, stop2, bhat2;
};
template <int OP>
__device__ __forceinline__ Slot load_slot(const Scal& c, int r) {
  Slot s{};
  if (OP != FIN_STORE) {
    s.active = c.active[r];
    s.gamma = c.gamma[r];
  }
  if (OP == FIN_RHO_BETA) {
    s.flags = c.flags[r];
    s.since = c.since[r];
    s.rho2_max = c.rho2_max[r];
    s.stop2 = c.stop2[r];
    s.bhat2 = c.bhat2[r];
  }
  return s;
}
// |rho|^2 = v: true while the slot goes on.
__device__ __forceinline__ bool rho_step(const Scal& c, const Slot& s, int r, double v) {
  c.tmp[r] = v;
  if (!s.active) return false;
  c.rho2[r] = v;
  double top = s.rho2_max;
  if (v > top) c.rho2_max[r] = top = v;
  if (v <= s.stop2) {
    c.active[r] = 0;
    c.flags[r] = s.flags | FLAG_INNER_DONE;
    return false;
  }
  if (v < c.delta2 * top || v <= c.tau2 * s.bhat2) c.flags[r] = s.flags | FLAG_UPDATE;
  else if (s.since >= c.stag_max) c.flags[r] = s.flags | FLAG_UPDATE | FLAG_STAG;
  return true;
}
// The scalar step of a CG iteration that needs slot r's sums v (and w).
template <int OP>
__device__ __forceinline__ void cg_step(const Scal& c, const Slot& s, int r, double v, double w, double* out) {
  if (OP == FIN_STORE) out[r] = v;
  if (OP == FIN_ALPHA) {
    if (s.active) c.alpha[r] = v > 0.0 ? s.gamma / v : 0.0;
    if (s.active) c.taken[r] = c.pos + 1;
    else if (c.pos == 0) c.taken[r] = 0;
  }
  if (OP == FIN_RHO_BETA) {
    // a slot that stopped on |rho|^2 keeps its search direction
    const bool go = rho_step(c, s, r, v);
    c.rr[r] = w;
    if (go) {
      c.beta[r] = s.gamma > 0.0 ? w / s.gamma : 0.0;
      c.gamma_prev[r] = s.gamma;
      c.gamma[r] = w;
      c.iters[r] += 1;
      c.since[r] = s.since + 1;
    }
  }
}

// Sums of one or two arrays (OP) over their sites, in an order that depends on their number only.
// Thread t adds the sites t, t + 256, ... of [beg, end): eight loads at a time, then their additions.
template <bool TWO>
__device__ __forceinline__ void site_sums(const double* __restrict__ p, const double* __restrict__ p2, long beg, long end,
                                          double* s) {
  constexpr int B = 8;
  for (long k = beg + threadIdx.x; k < end; k += B * 256) {
    double v[B], w[B];
#pragma unroll
    for (int j = 0; j < B; j++) {
      const bool in = k + j * 256 < end;
      v[j] = in ? p[k + j * 256] : 0.0;
      if (TWO) w[j] = in ? p2[k + j * 256] : 0.0;
    }
#pragma unroll
    for (int j = 0; j < B; j++) {
      if (k + j * 256 >= end) break;
      s[0] += v[j];
      if (TWO) s[1] += w[j];
    }
  }
}
// Tree over W lanes for each of two values: the lower and the upper W / 2 lanes take one each after the
// first step; an FP64 instruction costs a warp 64 clocks whatever its active lanes.
template <bool TWO, int W>
__device__ __forceinline__ double lane_sum(double v, double w) {
  if (TWO) {
    const bool up = (threadIdx.x & (W / 2)) != 0;
    const double give = up ? v : w;
    v = (up ? w : v) + __shfl_xor_sync(0xffffffffu, give, W / 2);
  } else {
    v += __shfl_down_sync(0xffffffffu, v, W / 2);
  }
#pragma unroll
  for (int k = W / 4; k > 0; k >>= 1) v += __shfl_down_sync(0xffffffffu, v, k);
  return v;
}
// Sums of a block's 256 values by its first warp, after one exchange: of the first value in lane 0, of the
// second in lane 8.
template <bool TWO>
__device__ __forceinline__ double block_sum256(const double* s, double* sh) {
  const double t = lane_sum<TWO, 32>(s[0], TWO ? s[1] : 0.0);
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  if (lane == 0) sh[warp] = t;
  if (TWO && lane == 16) sh[8 + warp] = t;
  __syncthreads();
  double u = 0.0;
  if (threadIdx.x < 32) {
    u = lane < (TWO ? 16 : 8) ? sh[lane] : 0.0;
#pragma unroll
    for (int k = 4; k > 0; k >>= 1) u += __shfl_down_sync(0xffffffffu, u, k);
  }
  return u;
}

// The sums of slot r over its sites, then the scalar step.  A cluster of kFinCluster
// blocks per slot: block c sums the c-th contiguous chunk, and block 0 adds the blocks'
// sums, which they put into its shared memory behind one barrier.  What bounds it is
// latency: the barrier that shows that block 0 has started is taken while the partial
// sums load, and the slot's scalars load with them (a session on 8^3 x 24: 54.2 ms with a
// barrier on both sides of block 0's reads and the scalars loaded after it, 53.5 ms; 51.0 ms
// with |rho|^2 and |r|^2 added up in one launch).  Spreading a slot over several SMs matters on a part with few FP64 adders per SM; up to kFinSmall sites a single block is
// faster than the cluster's barriers (5.6 us for the cluster and 3 us for a scalar kernel
// after it at 2048 sites; 4096 sites are 16 additions per thread).
constexpr int kFinCluster = 8;
constexpr long kFinSmall = 4096;
template <int OP>
__global__ void __cluster_dims__(kFinCluster, 1, 1) __launch_bounds__(256)
    k_finalize(const double* __restrict__ partials, const double* __restrict__ partials2, long nsites, Scal sc,
               double* __restrict__ out) {
  namespace cg = cooperative_groups;
  constexpr bool TWO = OP == FIN_RHO_BETA;
  __shared__ double sh[16];
  __shared__ double total[2 * kFinCluster];
  cg::cluster_group cluster = cg::this_cluster();
  const int r = blockIdx.y;
  const int c = (int)cluster.block_rank();
  asm volatile("barrier.cluster.arrive.relaxed.aligned;" ::: "memory");
  const Slot slot = load_slot<OP>(sc, r);
  const long len = (nsites + kFinCluster - 1) / kFinCluster;
  const long beg = (long)c * len;
  const long end = beg + len < nsites ? beg + len : nsites;
  double s[2] = {0.0, 0.0};
  site_sums<TWO>(partials + (long)r * nsites, partials2 + (long)r * nsites, beg, end, s);
  const double t = block_sum256<TWO>(s, sh);
  asm volatile("barrier.cluster.wait.aligned;" ::: "memory");
  if (threadIdx.x == 0) *cluster.map_shared_rank(&total[c], 0) = t;
  if (TWO && threadIdx.x == 8) *cluster.map_shared_rank(&total[kFinCluster + c], 0) = t;
  cluster.sync();
  if (c == 0 && threadIdx.x < 32) {
    double tot = threadIdx.x < (TWO ? 2 : 1) * kFinCluster ? total[threadIdx.x] : 0.0;
#pragma unroll
    for (int w = kFinCluster / 2; w > 0; w >>= 1) tot += __shfl_down_sync(0xffffffffu, tot, w);
    const double second = __shfl_sync(0xffffffffu, tot, kFinCluster);
    if (threadIdx.x == 0) cg_step<OP>(sc, slot, r, tot, second, out);
  }
}
template <int OP>
__global__ void __launch_bounds__(256) k_finalize_small(const double* __restrict__ partials,
                                                        const double* __restrict__ partials2, int nsites, Scal sc,
                                                        double* __restrict__ out) {
  constexpr bool TWO = OP == FIN_RHO_BETA;
  __shared__ double sh[16];
  const int r = blockIdx.x;
  const Slot slot = load_slot<OP>(sc, r);
  double s[2] = {0.0, 0.0};
  site_sums<TWO>(partials + (long)r * nsites, partials2 + (long)r * nsites, 0, nsites, s);
  const double t = block_sum256<TWO>(s, sh);
  if (threadIdx.x < 32) {
    const double second = __shfl_sync(0xffffffffu, t, 8);
    if (threadIdx.x == 0) cg_step<OP>(sc, slot, r, t, second, out);
  }
}

// u = B x on one parity: P_+ half b5 x_s + c5 x_{s-1}, P_- half b5 x_s + c5 x_{s+1},
// with x_{-1} = -m x_{L5-1} and x_{L5} = -m x_0.
template <typename S>
__global__ void k_bop(const S* __restrict__ xv, const float* __restrict__ x_nrm, S* __restrict__ uv,
                      float* __restrict__ u_nrm, Fifth<typename StoreTraits<S>::T> f, Tiling tl, long Vh, int L5, int N,
                      const int* __restrict__ mask) {
  using T = typename StoreTraits<S>::T;
  const Unit x = unit_of(tl, Vh, L5, N);
  const long pl = Vh * L5 * N;
  if (!x.valid || (mask && !mask[x.r])) return;
  const T m = f.mass[x.r];
  const int s_dn = x.s == 0 ? L5 - 1 : x.s - 1, s_up = x.s == L5 - 1 ? 0 : x.s + 1;
  const T w_dn = x.s == 0 ? -m : T(1), w_up = x.s == L5 - 1 ? -m : T(1);
  T y[24], up[12], lo[12];
  load24<S, T>(xv, x_nrm, pl, x.u, y);
  load_part<S, T>(xv, x_nrm, pl, (x.h * L5 + s_dn) * N + x.r, 0, up);
  load_part<S, T>(xv, x_nrm, pl, (x.h * L5 + s_up) * N + x.r, 1, lo);
#pragma unroll
  for (int i = 0; i < 12; i++) y[i] = bop_term(f.b5, y[i], f.c5 * w_dn, up[i]);
#pragma unroll
  for (int i = 0; i < 12; i++) y[12 + i] = bop_term(f.b5, y[12 + i], f.c5 * w_up, lo[i]);
  store24<S, T>(uv, u_nrm, pl, x.u, y);
}

// p = r + beta_r p0, then u = B p (the new p of the neighbouring slices comes from
// shared memory: a block holds every slice of its sites).  p may be p0.  taken: the
// iterations a slot has done in its group; a slot that stopped in it hands p0 on.
template <typename S>
__global__ void k_xpay_b(const S* __restrict__ r, const float* __restrict__ r_nrm, const S* p0, const float* p0_nrm, S* p,
                         float* p_nrm, S* __restrict__ uv, float* __restrict__ u_nrm,
                         const double* __restrict__ beta, Fifth<typename StoreTraits<S>::T> f, Tiling tl, long Vh,
                         int L5, int N, const int* __restrict__ active, const int* __restrict__ taken) {
  using T = typename StoreTraits<S>::T;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  T* sP = reinterpret_cast<T*>(smem_raw);
  const Unit x = unit_of(tl, Vh, L5, N);
  const long pl = Vh * L5 * N;
  const bool act = x.valid && active[x.r];
  T pv[24];
#pragma unroll
  for (int i = 0; i < 24; i++) pv[i] = 0;
  if (act) {
    const T b = (T)beta[x.r];
    T rv[24];
    load24<S, T>(r, r_nrm, pl, x.u, rv);
    load24<S, T>(p0, p0_nrm, pl, x.u, pv);
#pragma unroll
    for (int i = 0; i < 24; i++) pv[i] = rv[i] + b * pv[i];
    store24<S, T>(p, p_nrm, pl, x.u, pv);
  } else if (x.valid && taken != nullptr && taken[x.r] > 0) {
    load24<S, T>(p0, p0_nrm, pl, x.u, pv);
    store24<S, T>(p, p_nrm, pl, x.u, pv);
  }
#pragma unroll
  for (int i = 0; i < 24; i++) sP[threadIdx.x * 25 + i] = pv[i];
  __syncthreads();
  if (!act) return;
  const T m = f.mass[x.r];
  const int s_dn = x.s == 0 ? L5 - 1 : x.s - 1, s_up = x.s == L5 - 1 ? 0 : x.s + 1;
  const T w_dn = x.s == 0 ? -m : T(1), w_up = x.s == L5 - 1 ? -m : T(1);
  const T* nd = sP + (size_t)((x.site_l * L5 + s_dn) * tl.rt + x.r_l) * 25;
  const T* nu = sP + (size_t)((x.site_l * L5 + s_up) * tl.rt + x.r_l) * 25;
  T y[24];
#pragma unroll
  for (int i = 0; i < 12; i++) y[i] = f.b5 * pv[i] + f.c5 * w_dn * nd[i];
#pragma unroll
  for (int i = 12; i < 24; i++) y[i] = f.b5 * pv[i] + f.c5 * w_up * nu[i];
  store24<S, T>(uv, u_nrm, pl, x.u, y);
}

// FP64 forms of the two updates.  A warp's FP64 instruction takes 64 clocks, so a thread that walks
// through the 24 components of its unit spends 3 us on them alone, with most schedulers idle on a small
// lattice.  Four lanes per unit with three of its 12 words each; a quarter warp reads eight consecutive units of
// one plane.  The sum of a unit (two steps of shuffles) and of a site do not depend on the other slots.
// 4^3 x 8, L5 = 4, one system:
// 8.45 ms per solve with a thread per unit, 7.84 with these; 8^3 x 16, L5 = 8, one to four systems: the same.
struct Item64 {
  Unit x;
  int ul;        // unit of the tile
  bool in;       // of the tile and of the lattice
};
__device__ __forceinline__ Item64 item64(const Tiling& tl, int ul, long Vh, int L5, int N) {
  Item64 i;
  i.ul = ul;
  Unit& x = i.x;
  x.r_l = ul % tl.rt;
  x.s = (ul / tl.rt) % L5;
  x.site_l = ul / (tl.rt * L5);
  x.h = (long)blockIdx.x * tl.nsb + x.site_l;
  x.r = blockIdx.y * tl.rt + x.r_l;
  i.in = ul < tl.threads && x.h < Vh && x.r < N;
  x.u = (x.h * L5 + x.s) * N + x.r;
  return i;
}
constexpr int kMax64 = 512;      // threads; larger tiles take several passes

// rho -= alpha_r q, |rho|^2; X: x += alpha_r p too.
template <bool X>
__global__ void __launch_bounds__(kMax64)
    k_axpy64(double2* __restrict__ xv, const double2* __restrict__ p, double2* __restrict__ rho,
             const double2* __restrict__ q, const double* __restrict__ alpha, Tiling tl, long Vh, int L5, int N,
             const int* __restrict__ active, double* __restrict__ partials) {
  extern __shared__ double sunit[];
  const long pl = Vh * L5 * N;
  const int lane = threadIdx.x & 31, w0 = lane >> 3;
  for (int base = (threadIdx.x >> 5) * 8; base < tl.threads; base += blockDim.x / 4) {
    const Item64 it = item64(tl, base + (lane & 7), Vh, L5, N);
    double n2 = 0.0;
    if (it.in && active[it.x.r]) {
      const double a = alpha[it.x.r];
      double2 qv[3], rv[3], pv[3], xs[3];
#pragma unroll
      for (int j = 0; j < 3; j++) {
        const long o = (w0 + 4 * j) * pl + it.x.u;
        qv[j] = __ldg(q + o);
        rv[j] = rho[o];
        if (X) {
          pv[j] = __ldg(p + o);
          xs[j] = xv[o];
        }
      }
#pragma unroll
      for (int j = 0; j < 3; j++) {
        const long o = (w0 + 4 * j) * pl + it.x.u;
        rv[j].x = __fma_rn(-a, qv[j].x, rv[j].x);
        rv[j].y = __fma_rn(-a, qv[j].y, rv[j].y);
        n2 = __fma_rn(rv[j].x, rv[j].x, n2);
        n2 = __fma_rn(rv[j].y, rv[j].y, n2);
        rho[o] = rv[j];
        if (X) {
          xs[j].x = __fma_rn(a, pv[j].x, xs[j].x);
          xs[j].y = __fma_rn(a, pv[j].y, xs[j].y);
          xv[o] = xs[j];
        }
      }
    }
    n2 += __shfl_xor_sync(0xffffffffu, n2, 8);
    n2 += __shfl_xor_sync(0xffffffffu, n2, 16);
    if (w0 == 0 && it.ul < tl.threads) sunit[it.ul] = n2;
  }
  __syncthreads();
  for (int k = threadIdx.x; k < tl.nsb * tl.rt; k += blockDim.x) {
    const int site_l = k / tl.rt, r_l = k - site_l * tl.rt;
    const long h = (long)blockIdx.x * tl.nsb + site_l;
    const int r = blockIdx.y * tl.rt + r_l;
    if (h >= Vh || r >= N) continue;
    double sum = 0.0;
    for (int s = 0; s < L5; s++) sum += sunit[(site_l * L5 + s) * tl.rt + r_l];
    partials[(long)r * Vh + h] = sum;
  }
}

// k_xpay_b in FP64.
__global__ void __launch_bounds__(kMax64)
    k_xpay64(const double2* __restrict__ r, const double2* p0, double2* p, double2* __restrict__ uv,
             const double* __restrict__ beta, Fifth<double> f, Tiling tl, long Vh, int L5, int N,
             const int* __restrict__ active, const int* __restrict__ taken) {
  extern __shared__ __align__(16) double2 sP2[];      // [word][unit of the tile]
  const long pl = Vh * L5 * N;
  const int lane = threadIdx.x & 31, w0 = lane >> 3, nu = tl.threads;
  for (int base = (threadIdx.x >> 5) * 8; base < nu; base += blockDim.x / 4) {
    const Item64 it = item64(tl, base + (lane & 7), Vh, L5, N);
    if (!it.in) continue;
    const bool act = active[it.x.r];
    if (!act && !(taken != nullptr && taken[it.x.r] > 0)) continue;
    const double b = beta[it.x.r];
    double2 pv[3], rv[3];
#pragma unroll
    for (int j = 0; j < 3; j++) {
      const long o = (w0 + 4 * j) * pl + it.x.u;
      pv[j] = p0[o];
      if (act) rv[j] = __ldg(r + o);
    }
#pragma unroll
    for (int j = 0; j < 3; j++) {
      if (act) {
        pv[j].x = __fma_rn(b, pv[j].x, rv[j].x);
        pv[j].y = __fma_rn(b, pv[j].y, rv[j].y);
      }
      p[(w0 + 4 * j) * pl + it.x.u] = pv[j];
      sP2[(w0 + 4 * j) * nu + it.ul] = pv[j];
    }
  }
  __syncthreads();
  for (int base = (threadIdx.x >> 5) * 8; base < nu; base += blockDim.x / 4) {
    const Item64 it = item64(tl, base + (lane & 7), Vh, L5, N);
    if (!it.in || !active[it.x.r]) continue;
    const int s = it.x.s;
    const double m = f.mass[it.x.r];
    const int dn = it.ul + ((s == 0 ? L5 : 0) - 1) * tl.rt, up = it.ul + (1 - (s == L5 - 1 ? L5 : 0)) * tl.rt;
    const double c_dn = f.c5 * (s == 0 ? -m : 1.0), c_up = f.c5 * (s == L5 - 1 ? -m : 1.0);
#pragma unroll
    for (int j = 0; j < 3; j++) {
      const int w = w0 + 4 * j;
      const double c = w < 6 ? c_dn : c_up;
      const double2 a = sP2[w * nu + it.ul], b = sP2[w * nu + (w < 6 ? dn : up)];
      uv[w * pl + it.x.u] = make_double2(__fma_rn(f.b5, a.x, c * b.x), __fma_rn(f.b5, a.y, c * b.y));
    }
  }
}

// Zero the units of the slots in mask.
template <typename S>
__global__ void k_zero_masked(S* __restrict__ v, float* __restrict__ nrm, Tiling tl, long Vh, int L5, int N,
                              const int* __restrict__ mask) {
  using T = typename StoreTraits<S>::T;
  const Unit x = unit_of(tl, Vh, L5, N);
  const long pl = Vh * L5 * N;
  if (!x.valid || !mask[x.r]) return;
  T z[24];
#pragma unroll
  for (int i = 0; i < 24; i++) z[i] = 0;
  store24<S, T>(v, nrm, pl, x.u, z);
}

// Z2 noise source: complex element k of a 4D field ([t][z][y][x][spin][colour],
// k = 0 .. 12V-1) is (+1, 0) or (-1, 0) by the top bit of the k-th output of
// SplitMix64 from state `seed` (Steele, Lea and Flood, OOPSLA 2014): the state
// advances by the 64-bit golden-ratio increment and each output is the state
// passed through the 64-bit mixing finaliser of that generator.
__global__ void k_z2(unsigned long long seed, double* __restrict__ eta, long n) {
  long k = (long)blockIdx.x * blockDim.x + threadIdx.x;
  if (k >= n) return;
  unsigned long long z = seed + (unsigned long long)(k + 1) * 0x9E3779B97F4A7C15ull;
  z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
  z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
  z = z ^ (z >> 31);
  eta[2 * k] = (z >> 63) ? -1.0 : 1.0;
  eta[2 * k + 1] = 0.0;
}

// rho = S(bhat - q) with bhat in FP64 and q in FP32 (the residual of a reliable
// update computed with FP32 arithmetic); partial |bhat - q|^2 in FP64.
template <typename S>
__global__ void k_resid_update(const double* __restrict__ bhat, const float* __restrict__ q, S* __restrict__ rho,
                               float* __restrict__ rho_nrm, Tiling tl, long Vh, int L5, int N,
                               const int* __restrict__ mask, double* __restrict__ partials) {
  using T = typename StoreTraits<S>::T;
  const Unit x = unit_of(tl, Vh, L5, N);
  const long pl = Vh * L5 * N;
  double n2 = 0.0;
  if (x.valid && (!mask || mask[x.r])) {
    double b[24];
    float qv[24];
    load24<double, double>(bhat, nullptr, pl, x.u, b);
    load24<float, float>(q, nullptr, pl, x.u, qv);
    T o[24];
#pragma unroll
    for (int i = 0; i < 24; i++) {
      double v = b[i] - (double)qv[i];
      n2 += v * v;
      o[i] = (T)v;
    }
    store24<S, T>(rho, rho_nrm, pl, x.u, o);
  }
  block_partial(n2, x, tl, L5, Vh, partials);
}

// ---------------------------------------------------------------------------
// launchers
// ---------------------------------------------------------------------------
static inline dim3 tile_grid(const Tiling& t) { return dim3((unsigned)t.ntiles, (unsigned)t.ngroups); }

int pack_launches(int nr) { return (nr + kPtrs - 1) / kPtrs; }

template <typename S>
cudaError_t pack_rhs(const double* const* api, S* out, float* out_nrm, const Geom& g, int L5, int N, int par, int r0,
                     int nr, cudaStream_t st) {
  for (int b = 0; b < nr; b += kPtrs) {
    const int m = nr - b < kPtrs ? nr - b : kPtrs;
    Ptrs<const double*> p;
    for (int k = 0; k < kPtrs; k++) p.p[k] = k < m ? api[b + k] : nullptr;
    k_pack<S><<<(unsigned)((g.Vh * L5 * m + kPackUnits - 1) / kPackUnits), 256, 0, st>>>(p, out, out_nrm, g, L5, N, par, r0 + b, m);
  }
  return cudaGetLastError();
}

template <typename S>
cudaError_t unpack_rhs(const S* in, const float* in_nrm, double* const* api, const Geom& g, int L5, int N, int par,
                       int r0, int nr, cudaStream_t st) {
  for (int b = 0; b < nr; b += kPtrs) {
    const int m = nr - b < kPtrs ? nr - b : kPtrs;
    Ptrs<double*> p;
    for (int k = 0; k < kPtrs; k++) p.p[k] = k < m ? api[b + k] : nullptr;
    k_unpack<S><<<(unsigned)((g.Vh * L5 * m + kPackUnits - 1) / kPackUnits), 256, 0, st>>>(in, in_nrm, p, g, L5, N, par, r0 + b, m);
  }
  return cudaGetLastError();
}

// A launch takes the slots that follow while their arrays share nothing: its threads write in no order.
template <typename S>
cudaError_t unpack_all(const S* even, const float* even_nrm, const S* odd, const float* odd_nrm, double* const* api,
                       const Geom& g, int L5, int N, long long* launches, cudaStream_t st) {
  const uintptr_t bytes = sizeof(double) * 24 * (uintptr_t)g.V * L5;
  for (int b = 0, m; b < N; b += m) {
    for (m = 1; m < kPtrs && b + m < N; m++) {
      const uintptr_t x = (uintptr_t)api[b + m];
      bool shares = false;
      for (int k = b; k < b + m; k++) {
        const uintptr_t y = (uintptr_t)api[k];
        shares = shares || (x < y + bytes && y < x + bytes);
      }
      if (shares) break;
    }
    cudaError_t e = unpack_rhs<S>(even, even_nrm, api + b, g, L5, N, 0, b, m, st);
    if (e == cudaSuccess) e = unpack_rhs<S>(odd, odd_nrm, api + b, g, L5, N, 1, b, m, st);
    if (e != cudaSuccess) return e;
    if (launches) *launches += 2;
  }
  return cudaSuccess;
}

template <typename Si, typename So>
cudaError_t convert(const Si* in, const float* in_nrm, So* out, float* out_nrm, const Tiling& t, long Vh, int L5,
                    int N, const int* mask, cudaStream_t st) {
  k_convert<Si, So><<<tile_grid(t), t.threads, 0, st>>>(in, in_nrm, out, out_nrm, t, Vh, L5, N, mask);
  return cudaGetLastError();
}

// Tile and block of the FP64 forms.
static Tiling tiling64(long Vh, int L5, int N, int* threads) {
  const Tiling t = blas_tiling(Vh, L5, N, kMax64, 4);
  const int n = (t.threads + 7) / 8 * 32;
  *threads = n < kMax64 ? n : kMax64;
  return t;
}
static cudaError_t room64(const void* kern, size_t smem) {
  return smem <= 48 * 1024 ? cudaSuccess
                           : cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
}
template <bool X>
static cudaError_t axpy64(double* x, const double* p, double* rho, const double* q, const double* alpha, long Vh, int L5,
                          int N, const int* active, double* partials, cudaStream_t st) {
  int threads;
  const Tiling t = tiling64(Vh, L5, N, &threads);
  k_axpy64<X><<<tile_grid(t), threads, sizeof(double) * t.threads, st>>>(
      reinterpret_cast<double2*>(x), reinterpret_cast<const double2*>(p), reinterpret_cast<double2*>(rho),
      reinterpret_cast<const double2*>(q), alpha, t, Vh, L5, N, active, partials);
  return cudaGetLastError();
}

template <typename SX, typename S>
cudaError_t axpy_x_rho(SX* x, const S* p, const float* p_nrm, S* rho, float* rho_nrm, const S* q, const float* q_nrm,
                       const double* alpha, const Tiling& t, long Vh, int L5, int N, const int* active,
                       double* partials, cudaStream_t st) {
  if constexpr (std::is_same<S, double>::value) {
    return axpy64<true>(x, p, rho, q, alpha, Vh, L5, N, active, partials, st);
  } else {
    k_axpy_x_rho<SX, S><<<tile_grid(t), t.threads, 0, st>>>(x, p, p_nrm, rho, rho_nrm, q, q_nrm, alpha, t, Vh, L5, N,
                                                             active, partials);
    return cudaGetLastError();
  }
}

template <typename S>
cudaError_t axpy_rho(S* rho, float* rho_nrm, const S* q, const float* q_nrm, const double* alpha, const Tiling& t,
                     long Vh, int L5, int N, const int* active, double* partials, cudaStream_t st) {
  if constexpr (std::is_same<S, double>::value) {
    return axpy64<false>(nullptr, nullptr, rho, q, alpha, Vh, L5, N, active, partials, st);
  } else {
    k_axpy_rho<S><<<tile_grid(t), t.threads, 0, st>>>(rho, rho_nrm, q, q_nrm, alpha, t, Vh, L5, N, active, partials);
    return cudaGetLastError();
  }
}

template <typename SX, typename S>
cudaError_t axpy_group(SX* x, const PGroup<S>& p, int m, const double* alpha, const int* taken, const Tiling& t, long Vh,
                       int L5, int N, cudaStream_t st) {
  k_axpy_group<SX, S><<<tile_grid(t), t.threads, 0, st>>>(x, p, m, alpha, taken, t, Vh, L5, N);
  return cudaGetLastError();
}

template <typename SX>
cudaError_t accum_xhi(double* xhi, SX* xlo, const Tiling& t, long Vh, int L5, int N, const int* mask,
                      cudaStream_t st) {
  k_accum_xhi<SX><<<tile_grid(t), t.threads, 0, st>>>(xhi, xlo, t, Vh, L5, N, mask);
  return cudaGetLastError();
}

template <typename S>
cudaError_t norm2_partials(const S* v, const float* v_nrm, const Tiling& t, long Vh, int L5, int N, const int* mask,
                           double* partials, cudaStream_t st) {
  k_norm2<S><<<tile_grid(t), t.threads, 0, st>>>(v, v_nrm, t, Vh, L5, N, mask, partials);
  return cudaGetLastError();
}

template <typename S>
cudaError_t bop(const S* x, const float* x_nrm, S* u, float* u_nrm, const Fifth<typename StoreTraits<S>::T>& f,
                const Tiling& t, long Vh, int L5, int N, const int* mask, cudaStream_t st) {
  k_bop<S><<<tile_grid(t), t.threads, 0, st>>>(x, x_nrm, u, u_nrm, f, t, Vh, L5, N, mask);
  return cudaGetLastError();
}

template <typename S>
cudaError_t xpay_b(const S* r, const float* r_nrm, const S* p0, const float* p0_nrm, S* p, float* p_nrm, S* u,
                   float* u_nrm, const double* beta, const Fifth<typename StoreTraits<S>::T>& f, const Tiling& t,
                   long Vh, int L5, int N, const int* active, const int* taken, cudaStream_t st) {
  if constexpr (std::is_same<S, double>::value) {
    int threads;
    const Tiling t4 = tiling64(Vh, L5, N, &threads);
    const size_t smem = sizeof(double2) * 12 * (size_t)t4.threads;
    cudaError_t e = room64((const void*)k_xpay64, smem);
    if (e != cudaSuccess) return e;
    k_xpay64<<<tile_grid(t4), threads, smem, st>>>(
        reinterpret_cast<const double2*>(r), reinterpret_cast<const double2*>(p0), reinterpret_cast<double2*>(p),
        reinterpret_cast<double2*>(u), beta, f, t4, Vh, L5, N, active, taken);
    return cudaGetLastError();
  } else {
    using T = typename StoreTraits<S>::T;
    size_t smem = (size_t)t.threads * 25 * sizeof(T);
    if (smem > 48 * 1024) {
      cudaError_t e = cudaFuncSetAttribute(k_xpay_b<S>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
      if (e != cudaSuccess) return e;
    }
    k_xpay_b<S><<<tile_grid(t), t.threads, smem, st>>>(r, r_nrm, p0, p0_nrm, p, p_nrm, u, u_nrm, beta, f, t, Vh, L5, N, active,
                                                      taken);
    return cudaGetLastError();
  }
}

template <typename S>
cudaError_t resid_update(const double* bhat, const float* q, S* rho, float* rho_nrm, const Tiling& t, long Vh, int L5,
                         int N, const int* mask, double* partials, cudaStream_t st) {
  k_resid_update<S><<<tile_grid(t), t.threads, 0, st>>>(bhat, q, rho, rho_nrm, t, Vh, L5, N, mask, partials);
  return cudaGetLastError();
}

template <typename S>
cudaError_t zero_masked(S* v, float* nrm, const Tiling& t, long Vh, int L5, int N, const int* mask, cudaStream_t st) {
  k_zero_masked<S><<<tile_grid(t), t.threads, 0, st>>>(v, nrm, t, Vh, L5, N, mask);
  return cudaGetLastError();
}

cudaError_t z2_source(unsigned long long seed, double* eta, long V, cudaStream_t st) {
  const long n = V * 12;
  k_z2<<<(unsigned)((n + 255) / 256), 256, 0, st>>>(seed, eta, n);
  return cudaGetLastError();
}

template <int OP>
static cudaError_t finalize_one(const double* partials, const double* partials2, long nsites, int N, const Scal& c,
                                double* out, cudaStream_t st) {
  if (nsites <= kFinSmall) k_finalize_small<OP><<<N, 256, 0, st>>>(partials, partials2, (int)nsites, c, out);
  else k_finalize<OP><<<dim3(kFinCluster, (unsigned)N), 256, 0, st>>>(partials, partials2, nsites, c, out);
  return cudaGetLastError();
}
cudaError_t finalize(const double* partials, long ntiles, int N, double* out, cudaStream_t st) {
  return finalize_one<FIN_STORE>(partials, partials, ntiles, N, Scal(), out, st);
}
cudaError_t finalize_alpha(const double* qq, long nsites, int N, const Scal& c, cudaStream_t st) {
  return finalize_one<FIN_ALPHA>(qq, qq, nsites, N, c, nullptr, st);
}
cudaError_t finalize_rho_beta(const double* rho2, const double* rr, long nsites, int N, const Scal& c,
                              cudaStream_t st) {
  return finalize_one<FIN_RHO_BETA>(rho2, rr, nsites, N, c, nullptr, st);
}

Tiling blas_tiling(long Vh, int L5, int N, int max_units, int lanes) {
  // the threads wanted: 256, fewer on lattices that would leave SMs without a block
  const long units = Vh * L5 * N;
  const long hi = 256 / lanes, lo = 32 / lanes;
  long want = units / 152;
  want = want > hi ? hi : want < lo ? lo : want;
  // the number of sites per block with the best-filled warps among those near that size
  int best = 1;
  double score = -1.0;
  for (int nsb = 1; nsb <= 64 && nsb * L5 <= max_units; nsb++) {
    const Tiling t = make_tiling(Vh, L5, N, nsb, max_units);
    if (nsb > 1 && (t.ngroups > 1 || t.threads > 1.5 * want)) break;
    const int n = t.threads * lanes;
    const double fill = (double)n / ((n + 31) / 32 * 32);
    const double size = t.threads < want ? (double)t.threads / want : 1.0;
    if (fill * size > score + 1e-9) { score = fill * size; best = nsb; }
  }
  return make_tiling(Vh, L5, N, best, max_units);
}

#define MDWF_INST_S(S)                                                                                          \
  template cudaError_t pack_rhs<S>(const double* const*, S*, float*, const Geom&, int, int, int, int, int,      \
                                   cudaStream_t);                                                               \
  template cudaError_t unpack_rhs<S>(const S*, const float*, double* const*, const Geom&, int, int, int, int,   \
                                     int, cudaStream_t);                                                        \
  template cudaError_t unpack_all<S>(const S*, const float*, const S*, const float*, double* const*, const Geom&, \
                                     int, int, long long*, cudaStream_t);                                       \
  template cudaError_t norm2_partials<S>(const S*, const float*, const Tiling&, long, int, int, const int*,      \
                                         double*, cudaStream_t);

#define MDWF_INST_B(S)                                                                                           \
  template cudaError_t bop<S>(const S*, const float*, S*, float*, const Fifth<StoreTraits<S>::T>&, const Tiling&,  \
                              long, int, int, const int*, cudaStream_t);                                          \
  template cudaError_t xpay_b<S>(const S*, const float*, const S*, const float*, S*, float*, S*, float*,          \
                                 const double*, const Fifth<StoreTraits<S>::T>&, const Tiling&, long, int, int,   \
                                 const int*, const int*, cudaStream_t);                                           \
  template cudaError_t axpy_rho<S>(S*, float*, const S*, const float*, const double*, const Tiling&, long, int, int, \
                                   const int*, double*, cudaStream_t);                                            \
  template cudaError_t resid_update<S>(const double*, const float*, S*, float*, const Tiling&, long, int, int,      \
                                       const int*, double*, cudaStream_t);
template cudaError_t zero_masked<double>(double*, float*, const Tiling&, long, int, int, const int*, cudaStream_t);
template cudaError_t zero_masked<float>(float*, float*, const Tiling&, long, int, int, const int*, cudaStream_t);
template cudaError_t zero_masked<__half>(__half*, float*, const Tiling&, long, int, int, const int*, cudaStream_t);
template cudaError_t zero_masked<__nv_bfloat16>(__nv_bfloat16*, float*, const Tiling&, long, int, int, const int*,
                                                cudaStream_t);

MDWF_INST_B(double)
MDWF_INST_B(float)
MDWF_INST_B(__half)
MDWF_INST_B(__nv_bfloat16)

MDWF_INST_S(double)
MDWF_INST_S(float)
MDWF_INST_S(__half)
MDWF_INST_S(__nv_bfloat16)

#define MDWF_INST_CONV(A, B)                                                                                  \
  template cudaError_t convert<A, B>(const A*, const float*, B*, float*, const Tiling&, long, int, int,       \
                                     const int*, cudaStream_t);
MDWF_INST_CONV(double, float)
MDWF_INST_CONV(double, __half)
MDWF_INST_CONV(double, __nv_bfloat16)
MDWF_INST_CONV(double, double)

#define MDWF_INST_AXPY(SX, S)                                                                                    \
  template cudaError_t axpy_x_rho<SX, S>(SX*, const S*, const float*, S*, float*, const S*, const float*,        \
                                         const double*, const Tiling&, long, int, int, const int*, double*,      \
                                         cudaStream_t);                                                          \
  template cudaError_t axpy_group<SX, S>(SX*, const PGroup<S>&, int, const double*, const int*, const Tiling&,   \
                                         long, int, int, cudaStream_t);
MDWF_INST_AXPY(double, double)
MDWF_INST_AXPY(float, float)
MDWF_INST_AXPY(float, __half)
MDWF_INST_AXPY(float, __nv_bfloat16)

template cudaError_t accum_xhi<double>(double*, double*, const Tiling&, long, int, int, const int*, cudaStream_t);
template cudaError_t accum_xhi<float>(double*, float*, const Tiling&, long, int, int, const int*, cudaStream_t);

}  // namespace mdwf
