// Declarations of the vector kernels in blas.cu.
#pragma once
#include "mdwf_internal.h"

namespace mdwf {

// Tiling of the unit-wise kernels: whole sites per block, 32 to 256 threads in full warps where the
// sizes allow it.
// lanes: threads per unit.
Tiling blas_tiling(long Vh, int L5, int N, int max_units, int lanes = 1);

constexpr int kGroup = 4;
// The search directions of a group.
template <typename S>
struct PGroup {
  const S* v[kGroup];
  const float* n[kGroup];
};

// Per-slot scalars of the batched CG.
struct Scal {
  double *gamma, *gamma_prev, *alpha, *beta, *rho2, *rho2_max, *stop2, *rr, *tmp, *bhat2, *upd2;
  int *active, *flags, *iters;
  int* since;     // CG iterations since the last reliable update of the slot
  int stag_max;   // that many without one: the inner recursion stagnates
  double delta2;  // periodic reliable update when |rho|^2 < delta2 * max |rho|^2 since the last one
  // The iterations of a chunk run in groups of up to kGroup.  The i-th of a group (pos = i) keeps its search
  // direction and, in alpha (the i-th row of kGroup), its step; x takes them together at the group's end.
  int* taken;     // iterations that the slot has done in the group
  int pos;
  double tau2;    // FP64 re-reference when |rho|^2 <= tau2 * |bhat|^2 (bhat = current reference residual)
};
enum { FLAG_INNER_DONE = 1, FLAG_UPDATE = 2, FLAG_DONE = 4, FLAG_REREF = 8, FLAG_STAG = 16 };
// The reductions of a CG iteration with the scalar steps that they feed: |q|^2 and alpha; |rho|^2 with the
// stopping and update decisions, and |r|^2 with beta, in one launch.
enum FinOp { FIN_STORE = 0, FIN_ALPHA = 1, FIN_RHO_BETA = 2 };
cudaError_t finalize_alpha(const double* qq, long nsites, int N, const Scal& c, cudaStream_t st);
cudaError_t finalize_rho_beta(const double* rho2, const double* rr, long nsites, int N, const Scal& c,
                              cudaStream_t st);

// API layout (one field per RHS, [s][t][z][y][x][spin][colour][re,im], FP64, device) <-> slots r0 .. r0 + nr - 1
// of a parity field; api: nr device pointers (host array).  unpack_rhs with in == null writes zeros.
template <typename S>
cudaError_t pack_rhs(const double* const* api, S* out, float* out_nrm, const Geom& g, int L5, int N, int par, int r0,
                     int nr, cudaStream_t st);
template <typename S>
cudaError_t unpack_rhs(const S* in, const float* in_nrm, double* const* api, const Geom& g, int L5, int N, int par,
                       int r0, int nr, cudaStream_t st);

// Kernels that pack_rhs launches for nr fields.
int pack_launches(int nr);
// Both parities of slots 0 .. N - 1 into the caller's arrays (odd == null: zeros on the odd sites).  Arrays that
// coincide or overlap are written one after the other, as if slot by slot: what they share holds the last
// slot's values.  Adds the kernels launched to *launches, if given.
template <typename S>
cudaError_t unpack_all(const S* even, const float* even_nrm, const S* odd, const float* odd_nrm, double* const* api,
                       const Geom& g, int L5, int N, long long* launches, cudaStream_t st);

template <typename Si, typename So>
cudaError_t convert(const Si* in, const float* in_nrm, So* out, float* out_nrm, const Tiling& t, long Vh, int L5,
                    int N, const int* mask, cudaStream_t st);

template <typename SX, typename S>
cudaError_t axpy_x_rho(SX* x, const S* p, const float* p_nrm, S* rho, float* rho_nrm, const S* q, const float* q_nrm,
                       const double* alpha, const Tiling& t, long Vh, int L5, int N, const int* active,
                       double* partials, cudaStream_t st);
template <typename S>
cudaError_t axpy_rho(S* rho, float* rho_nrm, const S* q, const float* q_nrm, const double* alpha, const Tiling& t,
                     long Vh, int L5, int N, const int* active, double* partials, cudaStream_t st);
template <typename SX, typename S>
cudaError_t axpy_group(SX* x, const PGroup<S>& p, int m, const double* alpha, const int* taken, const Tiling& t, long Vh,
                       int L5, int N, cudaStream_t st);

template <typename SX>
cudaError_t accum_xhi(double* xhi, SX* xlo, const Tiling& t, long Vh, int L5, int N, const int* mask,
                      cudaStream_t st);
template <typename S>
cudaError_t norm2_partials(const S* v, const float* v_nrm, const Tiling& t, long Vh, int L5, int N, const int* mask,
                           double* partials, cudaStream_t st);

template <typename S>
cudaError_t bop(const S* x, const float* x_nrm, S* u, float* u_nrm, const Fifth<typename StoreTraits<S>::T>& f,
                const Tiling& t, long Vh, int L5, int N, const int* mask, cudaStream_t st);

template <typename S>
cudaError_t xpay_b(const S* r, const float* r_nrm, const S* p0, const float* p0_nrm, S* p, float* p_nrm, S* u,
                   float* u_nrm, const double* beta, const Fifth<typename StoreTraits<S>::T>& f, const Tiling& t,
                   long Vh, int L5, int N, const int* active, const int* taken, cudaStream_t st);

template <typename S>
cudaError_t resid_update(const double* bhat, const float* q, S* rho, float* rho_nrm, const Tiling& t, long Vh, int L5,
                         int N, const int* mask, double* partials, cudaStream_t st);

template <typename S>
cudaError_t zero_masked(S* v, float* nrm, const Tiling& t, long Vh, int L5, int N, const int* mask, cudaStream_t st);

cudaError_t z2_source(unsigned long long seed, double* eta, long V, cudaStream_t st);

// 4D sources and sinks (sources.cu).
// src = f w + hc H w, w = P_+ eta on slice 0 and P_- eta on slice L5 - 1.
cudaError_t wall_source(const double* U, const double* eta, double* src, const Geom& g, int L5, int anti, double f,
                        double hc, cudaStream_t st);
// n_iter smearing steps of eta in place; tmp: V * 24 doubles, slices: 2 Lt + 1 ints.
cudaError_t smear(const double* U, double* eta, double* tmp, int* slices, const Geom& g, double k, int n_iter,
                  cudaStream_t st);
// c[2][Lt]: the two residual-mass correlators; part: 2 Lt mres_blocks(V / Lt, Lt) doubles.
int mres_blocks(long slice_sites, int Lt);
cudaError_t mres_correlators(const double* const* xs, int n, long V, int Lt, int L5, double* part, double* c,
                             cudaStream_t st);

cudaError_t finalize(const double* partials, long ntiles, int N, double* out, cudaStream_t st);

}  // namespace mdwf
