// GenEO coarse space, coarse operators and PCG vector kernels (Section 2.3).
#pragma once

#include "factor.h"

namespace gl {

// Element -> local-index maps of every subdomain (for local products with the
// element matrices): n_pairs entries of (element id, subdomain, 81 local
// indices or -1).
struct LocalElems {
    int64_t n_pairs = 0;
    DBuf<int> elem, sub;
    DBuf<int> loc;   // 81 per pair
};

// y_s += S (K_s) S x_s for every subdomain s: S = diag(xi) if xi != NULL,
// K_s = sum of the subdomain's element matrices (applied matrix-free from C_e
// and the Gauss-point geometry); x, y multi-vectors of nv columns in the
// per-subdomain layout of FactorPlan (x[vec_off*nv + v*n + i]).
void local_K_apply(const FactorPlan &P, const LocalElems &E, const double *C, const double *geo, const double *xi,
                   const double *x, double *y, int nv, cudaStream_t s);

// Block Krylov eigensolver of the pencils B p = mu M p (problem.cu), its basis
// V (with M V and B V) with KRY_MAX columns at most, grown by blocks of KRY_B
// (the sweeps' widest multi-vector, and more than the six rigid modes; where an
// eigenvalue has more copies, random columns take the place of those that the
// basis already holds).  V: FactorPlan layout with ldv columns; blocks W: KRY_B
// columns.
constexpr int KRY_B = 8, KRY_MAX = 96;
// Up to three bases and the blocks that go with them.
struct KryBlocks {
    int count = 0;
    double *V[3] = {}, *W[3] = {};
};
// G_s[a ldg + j] += A_s[:, a]^T B_s[:, j] for a < ma, j < KRY_B (subdomain stride gs)
void kry_gram(const FactorPlan &P, const double *A, int lda, int ma, const double *B, double *G, int64_t gs, int ldg,
              cudaStream_t s);
// W -= V H for every pair (H_s row-major m x KRY_B, leading dimension ldh)
void kry_project(const FactorPlan &P, const KryBlocks &K, int ldv, int m, const double *H, int64_t hs, int ldh,
                 cudaStream_t s);
// R_s orthonormalising a block with Gram matrix G_s; H, m: what its projection took away
void kry_orth(int n_sub, bool first, const double *G, const double *H, int64_t hs, int ldh, int m, double drop,
              double *R, int *d_err, cudaStream_t s);
// W <- W R for every pair; also stored at column col of V unless col < 0.  refill != 0: the columns that
// R leaves zero are random ones instead (refill: their seed)
void kry_scale(const FactorPlan &P, const KryBlocks &K, const double *R, int ldv, int col, cudaStream_t s,
               uint64_t refill = 0);
// Ritz pairs of T_s (leading dimension ldt, m rows), largest first; *worst = the largest relative residual
// of the first nev (bits of a non-negative double).  Y: KRY_MAX x ldy per subdomain, mu: ldy per subdomain.
void kry_ritz(const FactorPlan &P, const double *T, int ldt, int m, const double *G, int nev, int keep, double *Y,
              int ldy, double *mu, unsigned long long *worst, cudaStream_t s);
void kry_diag(int n_sub, double *T, int ldt, const double *mu, int ldm, int k, cudaStream_t s);
// out_s[:, 0..k) = V_s[:, 0..m) Y_s
void kry_combine(const FactorPlan &P, const double *V, int ldv, int m, const double *Y, int64_t ys, int ldy, int k,
                 double *out, int ldo, cudaStream_t s);

// Deterministic pseudo-random fill of a multi-vector (splitmix64 hash of the index).
void fill_random(double *x, int64_t n, uint64_t seed, cudaStream_t s);

// Coarse operators: Z stored per subdomain as n_s x m column-major (FactorPlan
// layout with nv = m).  c[s*m + a] = sum_i Z_s[i, a] r[gdof_s[i]];
// z[gdof_s[i]] += sum_a Z_s[i, a] y[s*m + a].
void coarse_restrict(const FactorPlan &P, const double *Z, int m, const double *r, double *c, cudaStream_t s);
void coarse_prolong(const FactorPlan &P, const double *Z, int m, const double *y, double *z, cudaStream_t s);

// Scales a multi-vector by xi row-wise: X[:, a] *= xi.
void scale_rows(const FactorPlan &P, double *X, const double *xi, int k, cudaStream_t s);

// ---------------------------------------------------------------- many laminates at once
struct PartDesc {
    int64_t elem_off, dof_off, n_dof;
    int nx, ny, NX, NY;
};
void launch_ku_batch(const PartDesc *d_parts, int n_parts, int64_t n_elem, int64_t n_dof, const double *C,
                     const double *geo, const double *x, double *y, cudaStream_t s);

// Per-part PCG state (structure of arrays, n parts each).
struct SegScalars {
    double *rho, *rho_new, *pq, *rr, *ff, *rz_old;
    int *active, *iters;
};
constexpr int SEG_BLOCKS = 64;
// out[i] = sum over part i's range of a*b   (partials: n * SEG_BLOCKS)
void seg_dot(const double *a, const double *b, const PartDesc *parts, int n, double *partials, double *out,
             cudaStream_t s);
// x += alpha_i p, r -= alpha_i q (alpha_i = rho_i/pq_i for active parts, else 0); rr_i = r.r
void seg_update_xr(double *x, double *r, const double *p, const double *q, const PartDesc *parts, int n,
                   SegScalars S, double *partials, cudaStream_t s);
// p = z + beta_i p, beta_i = (rho_new_i - rz_old_i) / rho_i; then rho_i = rho_new_i
void seg_update_p(double *p, const double *z, const PartDesc *parts, int n, SegScalars S, cudaStream_t s);
// for active parts: iters_i += 1, deactivate when rr_i <= tol^2 ff_i or iters_i >= max_iter; *n_active = count
void seg_check(SegScalars S, int n, double tol, int max_iter, int *n_active, cudaStream_t s);
// with rr_i the FP64 true residual of every part: reactivate the inactive parts that stopped below
// max_iter on a recurrence residual whose true residual misses tol (rr_i > tol^2 ff_i, finite);
// *n_active = how many were reactivated
void seg_confirm(SegScalars S, int n, double tol, int max_iter, int *n_active, cudaStream_t s);

// ---------------------------------------------------------------- PCG vector kernels
struct CGScalars {
    double rho, rho_new, pq, rr, rz_old, alpha, beta, ff;
};
// Partial sums of a reduction, one per block, and the count of blocks done
// (zero between launches: the last block of each resets it).
constexpr int RED_BLOCKS = 1024, RED_SCRATCH = RED_BLOCKS + 1;

// out = sum a_i b_i written to *out (device); the order of the sum depends on n only.
// partials: RED_SCRATCH entries, the last one zero.
void dot(const double *a, const double *b, int64_t n, double *partials, double *out, cudaStream_t s);
// x += alpha p; r -= alpha q (0 where mask), alpha = S->rho / S->pq; r.r -> S->rr; z = 0 unless z is NULL
void cg_update_xr(double *x, double *r, const double *p, const double *q, const uint8_t *mask, double *z, int64_t n,
                  CGScalars *S, double *partials, cudaStream_t s);
// beta = rho_new / rho (or flexible), p = z + beta p, q = 0, rho = rho_new
void cg_update_p(double *p, const double *z, double *q, int64_t n, CGScalars *S, double *partials, cudaStream_t s);
// y[dof[i]] = val (val = 0 or from array)
void set_entries(double *y, const int64_t *dof, int64_t n, const double *vals, cudaStream_t s);
// y = a - b
void sub(double *y, const double *a, const double *b, int64_t n, cudaStream_t s);
void axpy(double *y, double a, const double *x, int64_t n, cudaStream_t s);
// *out = the largest v where mask (NULL: everywhere); partials: 1024 entries
void max_where(const double *v, const uint8_t *mask, int64_t n, double *partials, double *out, cudaStream_t s);

}  // namespace gl
