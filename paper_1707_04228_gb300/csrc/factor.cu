// Batched multifrontal supernodal Cholesky and triangular solves.
//
// Section 2.3 solves each overlapping subdomain problem (zero displacement on
// the artificial boundary) with a sparse direct method.  Here every subdomain
// is ordered by geometric nested dissection (symbolic.cpp); the numeric phase
// walks the dissection trees of all subdomains together, one depth level at a
// time from the leaves up, so each launch covers every front of that depth in
// every subdomain:
//   1. zero the level's dense fronts (f x f, column-major, lower triangle);
//   2. add the element-matrix entries of the front's pivot columns;
//   3. extend-add the children's update matrices (child slot 0, then slot 1);
//   4. blocked right-looking partial Cholesky of the p pivot columns:
//      diagonal block (POTRF), panel below (TRSM), trailing lower triangle
//      (SYRK/GEMM) -- the trailing update also forms the update matrix;
//   5. write the front's panel to the factor array in inverse form:
//      L11^{-1} over W = L21 L11^{-1} (k_diag_inverse; FP32: k_tri_inverse,
//      k_wpanel; FP64: k_trinv_tc, k_wpanel_tc in gemm64_tc.cu).
// The solves walk the same levels, forward (leaves to root) and backward.  With
// the pivot block's inverse stored, a front's step is one product with its
// panel and no row of it waits for another.
#include <algorithm>
#include <cstdio>
#include <mutex>
#include <type_traits>

#include "factor.h"
#include "q2.cuh"
#include "slaves.h"
#include "warp.cuh"

namespace gl {

constexpr int NB = 32;        // pivot block
constexpr int TILE = 64;      // trailing-update tile

// ----------------------------------------------------------------- plan

void build_plan(const std::vector<SubSymbolic> &subs, FactorPlan &P, cudaStream_t s) {
    P.n_sub = (int)subs.size();
    P.vec_off.clear();
    P.vec_len.clear();
    P.fr.clear();
    P.levels.clear();
    P.h_gdof.clear();
    std::vector<int> rows, rel, pair_elem;
    std::vector<int16_t> pair_pos;
    int64_t voff = 0, loff = 0;
    int max_depth = 0;
    for (auto &S : subs) max_depth = std::max(max_depth, S.max_depth);
    P.levels.resize(max_depth + 1);
    for (int j = 0; j < P.n_sub; ++j) {
        const SubSymbolic &S = subs[j];
        P.vec_off.push_back(voff);
        P.vec_len.push_back(S.n);
        P.h_gdof.insert(P.h_gdof.end(), S.gdof.begin(), S.gdof.end());
        int base = (int)P.fr.size();
        int64_t row_base = (int64_t)rows.size(), rel_base = (int64_t)rel.size(),
                pair_base = (int64_t)pair_elem.size();
        for (size_t i = 0; i < S.sn.size(); ++i) {
            const Supernode &sn = S.sn[i];
            FrontDesc d{};
            d.l_off = loff + sn.l_off;
            d.row_off = row_base + sn.row_off;
            d.vec_off = voff;
            d.rel_off = rel_base + sn.rel_off;
            d.pair_off = pair_base + sn.emap_off;
            d.p = sn.p;
            d.q = sn.q;
            d.n_pairs = sn.n_elem_pairs;
            d.parent = sn.parent >= 0 ? base + sn.parent : -1;
            d.sub = j;
            d.slot = 0;
            if (sn.parent >= 0) d.slot = (S.sn[sn.parent].child[1] == (int)i) ? 1 : 0;
            d.first = sn.first;
            d.vlen = S.n;
            P.fr.push_back(d);
            Level &L = P.levels[sn.depth];
            L.fronts.push_back(base + (int)i);
            if (sn.parent >= 0) L.child_slot[d.slot].push_back(base + (int)i);
        }
        rows.insert(rows.end(), S.rows.begin(), S.rows.end());
        rel.insert(rel.end(), S.rel.begin(), S.rel.end());
        pair_elem.insert(pair_elem.end(), S.pair_elem.begin(), S.pair_elem.end());
        pair_pos.insert(pair_pos.end(), S.pair_pos.begin(), S.pair_pos.end());
        voff += S.n;
        loff += S.l_size;
    }
    P.n_local = voff;
    P.l_size = loff;
    P.nnz = 0;
    for (const FrontDesc &d : P.fr) P.nnz += (int64_t)d.p * (d.p + 1) / 2 + (int64_t)d.p * d.q;
    P.ws_max = 0;
    P.max_f = 0;
    for (auto &L : P.levels) {
        int64_t off = 0;
        for (int g : L.fronts) {
            FrontDesc &d = P.fr[g];
            int f = d.p + d.q;
            d.front_off = off;
            off += (int64_t)f * f;
            L.max_p = std::max(L.max_p, d.p);
            L.max_f = std::max(L.max_f, f);
        }
        L.ws = off;
        P.ws_max = std::max(P.ws_max, off);
        P.max_f = std::max(P.max_f, L.max_f);
        std::vector<int> v(L.fronts);
        L.d_fronts.upload(v, s);
        L.d_child[0].upload(L.child_slot[0], s);
        L.d_child[1].upload(L.child_slot[1], s);
    }
    // the first half of the subdomains: fronts are listed per level in subdomain order
    P.half_fronts.assign(P.levels.size(), 0);
    for (size_t d = 0; d < P.levels.size(); ++d)
        for (int g : P.levels[d].fronts)
            if (P.fr[g].sub < P.n_sub / 2) ++P.half_fronts[d];
    P.d_fr.upload(P.fr, s);
    P.d_rows.upload(rows, s);
    P.d_rel.upload(rel, s);
    P.d_pair_elem.upload(pair_elem, s);
    P.d_pair_pos.upload(pair_pos, s);
    P.d_gdof.upload(P.h_gdof, s);
    P.d_vec_off.upload(P.vec_off, s);
    P.d_vec_len.upload(P.vec_len, s);
    GL_CUDA(cudaStreamSynchronize(s));
}

// ----------------------------------------------------------------- numeric kernels

// One block per (front, element): the entries of K_e = sum_q w_q |J_q| B_q^T C_e B_q
// (FP64) in the front's pivot columns, added into the front.  With sigma != 0
// the entry (i, j) is scaled by 1 + sigma xi_i xi_j (the matrix A^N + sigma Xi
// A^N Xi of the GenEO pencil).  Every DOF is a pivot of one front, so over all
// fronts only half of the element's 81 x 81 entries are formed: the element's
// DOFs are sorted by their position in the front (pivots first), a warp takes
// a pivot column at a time -- its weighted stresses at the 27 Gauss points into
// shared memory, lane = point -- and its lanes the rows from the diagonal on,
// 81 FMAs an entry.  Bound by the FP64 pipe.  Forming all 6,561 entries of
// every pair took 3.5 ms a launch on the 63k-DOF corner.
constexpr int ASM_THREADS = 256;
constexpr size_t ASM_SMEM = sizeof(double) * (27 * 27 * 3 + (ASM_THREADS / 32) * 27 * 6);

template <class T>
__global__ void __launch_bounds__(ASM_THREADS) k_assemble(const int *__restrict__ fronts,
                                                          const FrontDesc *__restrict__ D,
                                                          const int *__restrict__ pair_elem,
                                                          const int16_t *__restrict__ pair_pos,
                                                          const int *__restrict__ rows, const double *__restrict__ C,
                                                          const double *__restrict__ geo,
                                                          const double *__restrict__ xi, double sigma, int s20,
                                                          T *__restrict__ ws) {
    const FrontDesc &d = D[fronts[blockIdx.x]];
    const int pr_i = blockIdx.y;
    if (pr_i >= d.n_pairs) return;
    extern __shared__ double sm[];
    double (*sG)[27][3] = reinterpret_cast<double (*)[27][3]>(sm);      // [q][node][axis]
    __shared__ int16_t spos[81], sdof[81];   // positions in the front, ascending; the element DOFs they belong to
    __shared__ double sx[81], sC[36], sw[27];
    __shared__ int16_t raw[81];
    __shared__ int cnt[2];                   // DOFs in the front, pivot columns among them
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int p = d.p, f = d.p + d.q;
    const int64_t e = pair_elem[d.pair_off + pr_i];
    if (tid < 2) cnt[tid] = 0;
    if (tid < 81) raw[tid] = pair_pos[(d.pair_off + pr_i) * 81 + tid];
    if (tid >= 96 && tid < 132) sC[tid - 96] = C[36 * e + tid - 96];
    if (tid >= 160 && tid < 187) sw[tid - 160] = geo[10 * (e * 27 + tid - 160) + 9];
    __syncthreads();
    if (tid < 81 && raw[tid] >= 0) {
        const int v = raw[tid];
        int r = 0;
        for (int i = 0; i < 81; ++i) r += raw[i] >= 0 && raw[i] < v;
        spos[r] = (int16_t)v;
        sdof[r] = (int16_t)tid;
        sx[r] = xi ? xi[d.vec_off + rows[d.row_off + v]] : 0.0;
        atomicAdd(&cnt[0], 1);
        if (v < p) atomicAdd(&cnt[1], 1);
    }
    // physical gradients of the 27 shape functions at the 27 Gauss points
    Q2Tables Tb;
    Tb.init();
    for (int idx = tid; idx < 27 * 27; idx += ASM_THREADS) {
        const int q = idx / 27, a = idx % 27;
        const int qx = q % 3, qy = (q / 3) % 3, qz = q / 9, i = a % 3, j = (a / 3) % 3, k = a / 9;
        const double *g = geo + 10 * (e * 27 + q);
        const double r0 = Tb.D[qx][i] * Tb.N[qy][j] * Tb.N[qz][k];
        const double r1 = Tb.N[qx][i] * Tb.D[qy][j] * Tb.N[qz][k];
        const double r2 = Tb.N[qx][i] * Tb.N[qy][j] * Tb.D[qz][k];
#pragma unroll
        for (int dd = 0; dd < 3; ++dd) sG[q][a][dd] = r0 * g[0 + dd] + r1 * g[3 + dd] + r2 * g[6 + dd];
    }
    __syncthreads();
    if (s20) {
        // serendipity element: the face and body centres follow the 20 nodes, whose shape functions
        // take their share of the centres' (the centres' DOFs are in no front)
        for (int idx = tid; idx < 27 * 27; idx += ASM_THREADS) {
            const int q = idx / 27, a = idx % 27;
            if (s20_is_slave(a)) continue;
            double v0 = sG[q][a][0], v1 = sG[q][a][1], v2 = sG[q][a][2];
            for (int b = 0; b < 27; ++b)
                if (s20_is_slave(b)) {
                    const double w = s20_weight(b, a);
                    v0 += w * sG[q][b][0];
                    v1 += w * sG[q][b][1];
                    v2 += w * sG[q][b][2];
                }
            sG[q][a][0] = v0;
            sG[q][a][1] = v1;
            sG[q][a][2] = v2;
        }
        __syncthreads();
    }
    const int n = cnt[0], nc = cnt[1];
    double (*sS)[6] = reinterpret_cast<double (*)[6]>(sm + 27 * 27 * 3 + warp * 27 * 6);
    T *F = ws + d.front_off;
    for (int j = warp; j < nc; j += ASM_THREADS / 32) {
        const int dof = sdof[j], node = dof / 3, c = dof % 3;
        __syncwarp();
        if (lane < 27) {
            // w C B_j at Gauss point `lane`: strain of the unit displacement c of the node
            const double gx = sG[lane][node][0], gy = sG[lane][node][1], gz = sG[lane][node][2], w = sw[lane];
            const int i0 = c, i1 = c == 0 ? 5 : (c == 1 ? 3 : 4), i2 = c == 0 ? 4 : (c == 1 ? 5 : 3);
            const double e0 = w * (c == 0 ? gx : (c == 1 ? gy : gz));          // normal strain
            const double e1 = w * (c == 0 ? gy : (c == 1 ? gz : gx));          // 12, 23, 13
            const double e2 = w * (c == 0 ? gz : (c == 1 ? gx : gy));          // 13, 12, 23
#pragma unroll
            for (int I = 0; I < 6; ++I) sS[lane][I] = sC[6 * I + i0] * e0 + sC[6 * I + i1] * e1 + sC[6 * I + i2] * e2;
        }
        __syncwarp();
        for (int i = j + lane; i < n; i += 32) {
            const int rd = sdof[i], a = rd / 3, rc = rd % 3;
            // row rc of the stress: components (rc, x), (rc, y), (rc, z)
            const int k0 = rc == 0 ? 0 : (rc == 1 ? 5 : 4), k1 = rc == 0 ? 5 : (rc == 1 ? 1 : 3),
                      k2 = rc == 0 ? 4 : (rc == 1 ? 3 : 2);
            double v0 = 0.0, v1 = 0.0, v2 = 0.0;
#pragma unroll 9
            for (int q = 0; q < 27; ++q) {
                v0 += sG[q][a][0] * sS[q][k0];
                v1 += sG[q][a][1] * sS[q][k1];
                v2 += sG[q][a][2] * sS[q][k2];
            }
            double v = v0 + v1 + v2;
            if (sigma != 0.0) v *= 1.0 + sigma * sx[i] * sx[j];
            atomicAdd(F + spos[i] + (int64_t)spos[j] * f, (T)v);
        }
    }
}

template <class T>
__global__ void k_extend_add(const int *__restrict__ children, const FrontDesc *__restrict__ D,
                             const int *__restrict__ rel, const T *__restrict__ ws_child, T *__restrict__ ws_par) {
    const FrontDesc c = D[children[blockIdx.x]];
    const int qc = c.q;
    if (qc == 0) return;
    const FrontDesc par = D[c.parent];
    const int fc = c.p + c.q, fp = par.p + par.q;
    const int *rm = rel + c.rel_off;
    const T *U = ws_child + c.front_off;
    T *F = ws_par + par.front_off;
    for (int j = blockIdx.y; j < qc; j += gridDim.y) {
        const int pj = rm[j];
        const T *Uc = U + (int64_t)(c.p + j) * fc + c.p;
        T *Fc = F + (int64_t)pj * fp;
        for (int i = j + threadIdx.x; i < qc; i += blockDim.x) Fc[rm[i]] += Uc[i];
    }
}

// Diagonal block Cholesky (kb <= 32) of each front at pivot offset k0.  A chain
// of 32 dependent steps whose FP64 instructions each hold an SM quarter's pipe
// for 64 clocks, so every step is cut to one reciprocal square root, one
// product and a quarter of the column updates per warp (the warps compute the
// column alike, lane = row, and share the updates), and one barrier.  With a
// square root and divisions in turn it took 53 us a launch, this form 32.
template <class T>
__global__ void __launch_bounds__(128) k_potrf(const int *__restrict__ fronts, const FrontDesc *__restrict__ D,
                                               T *__restrict__ ws, int k0, int *__restrict__ err, T drop,
                                               int *__restrict__ drops) {
    const FrontDesc &d = D[fronts[blockIdx.x]];
    if (k0 >= d.p) return;
    const int kb = min(NB, d.p - k0), f = d.p + d.q;
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    T *A = ws + d.front_off + k0 + (int64_t)k0 * f;
    __shared__ T a[NB][NB + 1];   // column-major: a[j][i]
    for (int j = w; j < NB; j += 4) a[j][lane] = j < kb && lane < kb && lane >= j ? A[lane + (int64_t)j * f] : T(0);
    __syncthreads();
    for (int j = 0; j < kb; ++j) {
        T v = a[j][j], l;
        if (drop > T(0) && fabs(v) <= drop) {
            // dependent column (drop mode): zero pivot, the column leaves the factor
            if (threadIdx.x == 0) atomicAdd(drops, 1);
            l = T(0);
        } else {
            if (!(v > T(0))) {
                if (threadIdx.x == 0) atomicExch(err, 1);
                v = T(1);
            }
            if (sizeof(T) == 8) {
                const T r = (T)rsqrt((double)v);
                l = lane == j ? v * r : a[j][lane] * r;
            } else {
                const T r = (T)sqrtf((float)v);
                l = lane == j ? r : a[j][lane] / r;
            }
        }
        if (lane < j) l = T(0);
        for (int k = j + 1 + w; k < kb; k += 4) {
            const T lk = __shfl_sync(0xffffffffu, l, k);
            if (lane >= k) a[k][lane] -= l * lk;
        }
        __syncthreads();          // every warp has read column j; its updates are in place
        if (w == 0) a[j][lane] = l;
    }
    __syncthreads();
    for (int j = w; j < kb; j += 4)
        if (lane < kb && lane >= j) A[lane + (int64_t)j * f] = a[j][lane];
}

// Panel below the diagonal block: rows r in [k0+kb, f) <- row * L_kk^{-T}, one
// row per thread.  The pivots' reciprocals are formed once per CTA (FP64): a
// division per entry, 32 of them against 500 FMAs, took most of the time (69
// us a launch on the 63k-DOF corner, now 48).
template <class T>
__global__ void __launch_bounds__(128) k_trsm(const int *__restrict__ fronts, const FrontDesc *__restrict__ D,
                                              T *__restrict__ ws, int k0) {
    const FrontDesc &d = D[fronts[blockIdx.x]];
    if (k0 >= d.p) return;
    const int kb = min(NB, d.p - k0), f = d.p + d.q;
    if (k0 + kb + (int)(blockIdx.y * blockDim.x) >= f) return;
    const int r = k0 + kb + blockIdx.y * blockDim.x + threadIdx.x;
    __shared__ T l[NB][NB + 1];   // l[j][i] = L[j, i], i < j; the diagonal holds the reciprocal (FP64) or the pivot
    T *F = ws + d.front_off;
    for (int idx = threadIdx.x; idx < NB * NB; idx += blockDim.x) {
        const int j = idx % NB, i = idx / NB;
        T v = j < kb && i <= j ? F[(k0 + j) + (int64_t)(k0 + i) * f] : T(0);
        if (sizeof(T) == 8 && i == j) v = v != T(0) ? T(1) / v : T(0);
        l[j][i] = v;
    }
    __syncthreads();
    if (r >= f) return;
    T x[NB];
#pragma unroll
    for (int j = 0; j < NB; ++j)
        if (j < kb) x[j] = F[r + (int64_t)(k0 + j) * f];
#pragma unroll
    for (int j = 0; j < NB; ++j) {
        if (j < kb) {
            T v = x[j], v1 = T(0);   // two chains
#pragma unroll
            for (int i = 0; i < NB; ++i)
                if (i < j) {
                    if (i & 1) v1 -= x[i] * l[j][i];
                    else v -= x[i] * l[j][i];
                }
            v += v1;
            if (sizeof(T) == 8) x[j] = v * l[j][j];                        // zero pivot: a dropped column
            else x[j] = l[j][j] != T(0) ? v / l[j][j] : T(0);
        }
    }
#pragma unroll
    for (int j = 0; j < NB; ++j)
        if (j < kb) F[r + (int64_t)(k0 + j) * f] = x[j];
}

// Trailing update of the lower triangle: F[r, c] -= sum_j P[r, j] P[c, j] for
// r >= c >= k0+kb, P the panel columns k0..k0+kb.  64x64 tiles, 256 threads.
// With cend > 0 only the columns c < min(cend, p) are updated (the rest of an
// outer panel whose trailing matrix is updated separately): the tiles are
// then those of the first column tiles of the trailing lower triangle.
template <class T>
__global__ void __launch_bounds__(256) k_syrk(const int *__restrict__ fronts, const FrontDesc *__restrict__ D,
                                              T *__restrict__ ws, int k0, int cend) {
    const FrontDesc d = D[fronts[blockIdx.x]];
    if (k0 >= d.p) return;
    const int kb = min(NB, d.p - k0), f = d.p + d.q;
    const int base = k0 + kb, m = f - base;
    if (m <= 0) return;
    const int nt = (m + TILE - 1) / TILE;
    int t = blockIdx.y, ti, tj;
    if (cend > 0) {
        const int cw = min(cend, d.p) - base;       // columns to update
        if (cw <= 0) return;
        const int ncw = (cw + TILE - 1) / TILE;
        // t -> (ti, tj), column-major over the tiles of the first ncw tile columns
        tj = 0;
        while (tj < ncw && t >= nt - tj) t -= nt - tj++;
        if (tj >= ncw) return;
        ti = tj + t;
    } else {
        if (t >= nt * (nt + 1) / 2) return;
        // t -> (ti, tj), ti >= tj, row-major over the lower triangle of tiles
        ti = (int)((sqrt(8.0 * t + 1.0) - 1.0) * 0.5);
        while ((ti + 1) * (ti + 2) / 2 <= t) ++ti;
        while (ti * (ti + 1) / 2 > t) --ti;
        tj = t - ti * (ti + 1) / 2;
    }
    const int cmax = cend > 0 ? min(cend, d.p) : f;   // columns c < cmax are updated
    const int r0 = base + ti * TILE, c0 = base + tj * TILE;
    T *F = ws + d.front_off;
    __shared__ T sa[NB][TILE + 1], sb[NB][TILE + 1];
    for (int idx = threadIdx.x; idx < NB * TILE; idx += blockDim.x) {
        int i = idx % TILE, j = idx / TILE;
        int r = r0 + i, c = c0 + i;
        sa[j][i] = (j < kb && r < f) ? F[r + (int64_t)(k0 + j) * f] : T(0);
        sb[j][i] = (j < kb && c < f) ? F[c + (int64_t)(k0 + j) * f] : T(0);
    }
    __syncthreads();
    const int tx = threadIdx.x % 16, ty = threadIdx.x / 16;
    T acc[4][4];
#pragma unroll
    for (int a = 0; a < 4; ++a)
#pragma unroll
        for (int b = 0; b < 4; ++b) acc[a][b] = T(0);
#pragma unroll 8
    for (int j = 0; j < NB; ++j) {
        T av[4], bv[4];
#pragma unroll
        for (int a = 0; a < 4; ++a) av[a] = sa[j][tx + 16 * a];
#pragma unroll
        for (int b = 0; b < 4; ++b) bv[b] = sb[j][ty + 16 * b];
#pragma unroll
        for (int a = 0; a < 4; ++a)
#pragma unroll
            for (int b = 0; b < 4; ++b) acc[a][b] += av[a] * bv[b];
    }
#pragma unroll
    for (int a = 0; a < 4; ++a)
#pragma unroll
        for (int b = 0; b < 4; ++b) {
            int r = r0 + tx + 16 * a, c = c0 + ty + 16 * b;
            if (r < f && c < cmax && r >= c) F[r + (int64_t)c * f] -= acc[a][b];
        }
}

// Blocked right-looking partial Cholesky of the p pivot columns of every front
// of a level, in blocks of NB = 32 pivots.  Without tc each block is followed
// by the rank-32 update of the whole trailing lower triangle.  With tc the
// blocks' updates stay inside an outer panel, and one update of the trailing
// matrix per panel runs on the tensor cores: FP32 with panels of 128 columns
// (syrk_tc.cu), FP64 with panels of 64 (gemm64_tc.cu; wider ones leave more to
// the FP64 pipe inside the panel than they save outside).
constexpr int PANEL64 = 64;

template <class T>
static void partial_cholesky_level(const int *d_fronts, int n_fronts, const FrontDesc *d_fr, int max_p, int max_f,
                                   T *ws, int *d_err, cudaStream_t s, T drop = T(0), int *d_drops = nullptr,
                                   bool tc = false) {
    const int PW = !tc ? NB : (sizeof(T) == 4 ? syrk_tc_panel() : PANEL64);
    for (int k0 = 0; k0 < max_p; k0 += PW) {
        const int kend = k0 + PW;
        for (int k1 = k0; k1 < std::min(kend, max_p); k1 += NB) {
            // upper bounds over the level's fronts (a front's last pivot block may be short)
            const int rows = std::max(1, max_f - k1);
            const int nt = (rows + TILE - 1) / TILE;
            k_potrf<T><<<n_fronts, 128, 0, s>>>(d_fronts, d_fr, ws, k1, d_err, drop, d_drops);
            k_trsm<T><<<dim3(n_fronts, (rows + 127) / 128), 128, 0, s>>>(d_fronts, d_fr, ws, k1);
            if (!tc) {
                k_syrk<T><<<dim3(n_fronts, nt * (nt + 1) / 2), 256, 0, s>>>(d_fronts, d_fr, ws, k1, 0);
            } else if (k1 + NB < kend) {
                const int ncw = std::min(nt, (kend - k1 - 1) / TILE + 1);    // column tiles inside the panel
                k_syrk<T><<<dim3(n_fronts, std::max(1, ncw * nt - ncw * (ncw - 1) / 2)), 256, 0, s>>>(d_fronts, d_fr, ws,
                                                                                                   k1, kend);
            }
            GL_CUDA(cudaGetLastError());
        }
        if (!tc) continue;
        if constexpr (sizeof(T) == 4) syrk_tc_level(d_fronts, n_fronts, d_fr, k0, max_f, ws, d_err, s);
        else syrk64_tc_level(d_fronts, n_fronts, d_fr, k0, PANEL64, max_f, ws, d_err, s);
    }
}

// ----------------------------------------------------------------- inverse form of the panels

// The sweeps read a front's panel as [L11^{-1}; W], W = L21 L11^{-1}, so that a
// forward step is y_1 = L11^{-1} x_1, x_2 -= W x_1 and a backward step
// x_1 = L11^{-T} y_1 - W^T x_2: products without a triangular solve, as many
// entries as the factor itself.  Both sweeps read the same numbers, so the
// preconditioner stays symmetric positive definite whatever their rounding.
// Computed in FP64 whatever the storage type.
constexpr int INV_THREADS = 256;

// Diagonal blocks: out[B, B] = L[B, B]^{-1}, the strict upper triangle zero.
// One warp per (front, 32-pivot block): lane j solves for column j.
template <class T>
__global__ void __launch_bounds__(32) k_diag_inverse(const int *__restrict__ fronts, const FrontDesc *__restrict__ D,
                                                     const T *__restrict__ ws, T *__restrict__ out) {
    const FrontDesc d = D[fronts[blockIdx.x]];
    const int jb = blockIdx.y * 32;
    if (jb >= d.p) return;
    const int kb = min(32, d.p - jb), f = d.p + d.q, j = threadIdx.x;
    const T *A = ws + d.front_off + jb + (int64_t)jb * f;
    __shared__ double Dk[32][33], Li[32][33];
    for (int c = 0; c < kb; ++c) Dk[j][c] = j < kb && j >= c ? (double)A[j + (int64_t)c * f] : 0.0;
    __syncwarp();
    const double rd = j < kb ? 1.0 / Dk[j][j] : 0.0;
    for (int i = 0; i < kb; ++i) {
        double a0 = i == j ? 1.0 : 0.0, a1 = 0.0;
        int k = 0;
        for (; k + 1 < i; k += 2) {
            a0 -= Dk[i][k] * Li[k][j];
            a1 -= Dk[i][k + 1] * Li[k + 1][j];
        }
        if (k < i) a0 -= Dk[i][k] * Li[k][j];
        Li[i][j] = (a0 + a1) * __shfl_sync(0xffffffffu, rd, i);   // zero above the diagonal: column j starts at e_j
    }
    __syncwarp();
    T *O = out + d.l_off + jb + (int64_t)jb * f;
    if (j < kb)
        for (int c = 0; c < kb; ++c) O[j + (int64_t)c * f] = j >= c ? (T)Li[j][c] : T(0);
}

// Column tile J of L11^{-1} below its diagonal block: block row k from the one
// above down, X_k = -L_kk^{-1} sum_{m=J}^{k-1} L_km X_m (the diagonal blocks'
// inverses are in place).  One CTA per (front, tile); the chain over k is the
// CTA's own, so tiles need no other synchronisation.  Rows above J are zeroed.
// (FP32 storage; FP64 on the tensor cores, k_trinv_tc.)
template <class T>
__global__ void __launch_bounds__(INV_THREADS) k_tri_inverse(const int *__restrict__ fronts,
                                                             const FrontDesc *__restrict__ D,
                                                             const T *__restrict__ ws, T *out) {
    const FrontDesc d = D[fronts[blockIdx.x]];
    const int p = d.p, f = d.p + d.q, j0 = blockIdx.y * 32;
    if (j0 >= p) return;
    const int jw = min(32, p - j0);
    const T *F = ws + d.front_off;
    T *O = out + d.l_off + (int64_t)j0 * f;
    __shared__ double A[32][33], B[32][33];
    const int c = threadIdx.x & 31, r4 = threadIdx.x >> 5;   // output column c, rows r4 + 8 t
    for (int idx = threadIdx.x; idx < j0 * jw; idx += INV_THREADS) O[idx % j0 + (int64_t)(idx / j0) * f] = T(0);
    for (int k0 = j0 + 32; k0 < p; k0 += 32) {
        const int kw = min(32, p - k0);
        double acc[4] = {0.0, 0.0, 0.0, 0.0};
        for (int m0 = j0; m0 < k0; m0 += 32) {
            // rows k0.. of L columns m0..  (A[row][col]) and X_m (B[row][col])
#pragma unroll
            for (int t = 0; t < 4; ++t) {
                const int col = r4 + 8 * t;
                A[c][col] = c < kw ? (double)F[k0 + c + (int64_t)(m0 + col) * f] : 0.0;
                B[c][col] = col < jw ? (double)O[m0 + c + (int64_t)col * f] : 0.0;
            }
            __syncthreads();
#pragma unroll 8
            for (int m = 0; m < 32; ++m) {
                const double b = B[m][c];
#pragma unroll
                for (int t = 0; t < 4; ++t) acc[t] += A[r4 + 8 * t][m] * b;
            }
            __syncthreads();
        }
        // X_k = -D_k acc
#pragma unroll
        for (int t = 0; t < 4; ++t) {
            B[r4 + 8 * t][c] = acc[t];
            const int col = r4 + 8 * t;
            A[c][col] = c < kw && col < kw ? (double)out[d.l_off + k0 + c + (int64_t)(k0 + col) * f] : 0.0;
        }
        __syncthreads();
        double x[4] = {0.0, 0.0, 0.0, 0.0};
#pragma unroll 8
        for (int m = 0; m < 32; ++m) {
            const double b = B[m][c];
#pragma unroll
            for (int t = 0; t < 4; ++t) x[t] += A[r4 + 8 * t][m] * b;
        }
        __syncthreads();
#pragma unroll
        for (int t = 0; t < 4; ++t) A[r4 + 8 * t][c] = -x[t];
        __syncthreads();
#pragma unroll
        for (int t = 0; t < 4; ++t) {
            const int col = r4 + 8 * t;
            if (c < kw && col < jw) O[k0 + c + (int64_t)col * f] = (T)A[c][col];
        }
        __syncthreads();   // block row k is read back by the next steps
    }
}

// W = L21 L11^{-1}: 64 x 64 tiles of the structure rows, 256 threads with 4 x 4
// outputs each; tile column c0 needs the pivots from c0 on.
template <class T>
__global__ void __launch_bounds__(256) k_wpanel(const int *__restrict__ fronts, const FrontDesc *__restrict__ D,
                                                const T *__restrict__ ws, T *out) {
    const FrontDesc d = D[fronts[blockIdx.x]];
    const int p = d.p, f = d.p + d.q;
    const int ntr = (d.q + TILE - 1) / TILE;
    if (ntr == 0) return;
    const int ti = blockIdx.y % ntr, tj = blockIdx.y / ntr;
    const int c0 = tj * TILE, r0 = p + ti * TILE;
    if (c0 >= p) return;
    const T *F = ws + d.front_off;
    T *O = out + d.l_off;
    __shared__ double sa[NB][TILE + 1], sb[NB][TILE + 1];
    const int tx = threadIdx.x % 16, ty = threadIdx.x / 16;
    double acc[4][4];
#pragma unroll
    for (int a = 0; a < 4; ++a)
#pragma unroll
        for (int b = 0; b < 4; ++b) acc[a][b] = 0.0;
    for (int m0 = c0; m0 < p; m0 += NB) {
        for (int idx = threadIdx.x; idx < NB * TILE; idx += 256) {
            const int i = idx % TILE, m = idx / TILE;
            sa[m][i] = m0 + m < p && r0 + i < f ? (double)F[r0 + i + (int64_t)(m0 + m) * f] : 0.0;
            const int mm = idx % NB, cc = idx / NB;
            sb[mm][cc] = m0 + mm < p && c0 + cc < p ? (double)O[m0 + mm + (int64_t)(c0 + cc) * f] : 0.0;
        }
        __syncthreads();
#pragma unroll 8
        for (int m = 0; m < NB; ++m) {
            double av[4], bv[4];
#pragma unroll
            for (int a = 0; a < 4; ++a) av[a] = sa[m][tx + 16 * a];
#pragma unroll
            for (int b = 0; b < 4; ++b) bv[b] = sb[m][ty + 16 * b];
#pragma unroll
            for (int a = 0; a < 4; ++a)
#pragma unroll
                for (int b = 0; b < 4; ++b) acc[a][b] += av[a] * bv[b];
        }
        __syncthreads();
    }
#pragma unroll
    for (int a = 0; a < 4; ++a)
#pragma unroll
        for (int b = 0; b < 4; ++b) {
            const int r = r0 + tx + 16 * a, c = c0 + ty + 16 * b;
            if (r < f && c < p) O[r + (int64_t)c * f] = (T)acc[a][b];
        }
}

template <class T>
static void inverse_form_level(const int *d_fronts, int nf, const FrontDesc *d_fr, int max_p, int max_f, T *ws,
                               T *L, int *d_err, cudaStream_t s) {
    const int nb = (max_p + 31) / 32;
    if (nb == 0) return;
    k_diag_inverse<T><<<dim3(nf, nb), 32, 0, s>>>(d_fronts, d_fr, ws, L);
    if constexpr (sizeof(T) == 8) {
        trinv_tc_level(d_fronts, nf, d_fr, max_p, ws, L, d_err, s);
        wpanel_tc_level(d_fronts, nf, d_fr, max_p, max_f, ws, L, d_err, s);
    } else {
        k_tri_inverse<T><<<dim3(nf, nb), INV_THREADS, 0, s>>>(d_fronts, d_fr, ws, L);
        // upper bound of row tiles x column tiles over the level's fronts (q <= max_f, p <= max_p)
        const int tiles = ((max_f + TILE - 1) / TILE) * ((max_p + TILE - 1) / TILE);
        k_wpanel<T><<<dim3(nf, tiles), 256, 0, s>>>(d_fronts, d_fr, ws, L);
    }
    GL_CUDA(cudaGetLastError());
}

// Subdomains are factorised in consecutive groups whose two live levels of
// dense fronts fit a workspace budget; inside a group every level is one set
// of batched launches.
template <class T>
void numeric_factor(FactorPlan &P, const double *C, const double *geo, const double *xi, double sigma, T *L,
                    int *d_err, cudaStream_t s) {
    const int nlev = (int)P.levels.size();
    const int64_t budget = (int64_t)(P.ws_budget_bytes / sizeof(T));   // entries per workspace buffer
    std::vector<int> depth_of(P.fr.size());
    for (int d = 0; d < nlev; ++d)
        for (int g : P.levels[d].fronts) depth_of[g] = d;
    std::vector<int64_t> sub_ws((size_t)P.n_sub * nlev, 0);
    for (size_t g = 0; g < P.fr.size(); ++g) {
        int64_t f = P.fr[g].p + P.fr[g].q;
        sub_ws[(size_t)P.fr[g].sub * nlev + depth_of[g]] += f * f;
    }
    std::vector<int> first_front(P.n_sub + 1, 0);
    for (size_t g = 0; g < P.fr.size(); ++g) first_front[P.fr[g].sub + 1] = (int)g + 1;
    for (int j = 1; j <= P.n_sub; ++j) first_front[j] = std::max(first_front[j], first_front[j - 1]);
    std::vector<FrontDesc> fr = P.fr;
    DBuf<FrontDesc> d_fr;
    DBuf<T> ws[2];
    int j0 = 0;
    P.last_groups = 0;
    while (j0 < P.n_sub) {
        ++P.last_groups;
        // grow the group while every level's total stays within the budget
        std::vector<int64_t> tot(nlev, 0);
        int j1 = j0;
        while (j1 < P.n_sub) {
            bool ok = true;
            for (int d = 0; d < nlev; ++d)
                if (tot[d] + sub_ws[(size_t)j1 * nlev + d] > budget) ok = false;
            if (!ok && j1 > j0) break;
            for (int d = 0; d < nlev; ++d) tot[d] += sub_ws[(size_t)j1 * nlev + d];
            ++j1;
        }
        // per-level lists of this group's fronts and their workspace offsets
        std::vector<std::vector<int>> lev(nlev), child[2];
        child[0].resize(nlev);
        child[1].resize(nlev);
        std::vector<int> max_p(nlev, 0), max_f(nlev, 0), max_pairs(nlev, 0);
        std::vector<int64_t> lev_ws(nlev, 0);
        for (int g = first_front[j0]; g < first_front[j1]; ++g) {
            int d = depth_of[g];
            int f = fr[g].p + fr[g].q;
            fr[g].front_off = lev_ws[d];
            lev_ws[d] += (int64_t)f * f;
            lev[d].push_back(g);
            if (fr[g].parent >= 0) child[fr[g].slot][d].push_back(g);
            max_p[d] = std::max(max_p[d], fr[g].p);
            max_f[d] = std::max(max_f[d], f);
            max_pairs[d] = std::max(max_pairs[d], fr[g].n_pairs);
        }
        int64_t need = 1;
        for (int d = 0; d < nlev; ++d) need = std::max(need, lev_ws[d]);
        if ((int64_t)ws[0].n < need) {
            ws[0].alloc(need);
            ws[1].alloc(need);
        }
        d_fr.upload(fr, s);
        std::vector<DBuf<int>> d_lev(nlev), d_ch0(nlev), d_ch1(nlev);
        for (int d = 0; d < nlev; ++d) {
            d_lev[d].upload(lev[d], s);
            d_ch0[d].upload(child[0][d], s);
            d_ch1[d].upload(child[1][d], s);
        }
        for (int dpt = nlev - 1; dpt >= 0; --dpt) {
            const int nf = (int)lev[dpt].size();
            if (nf == 0) continue;
            T *W = ws[dpt & 1].p;
            GL_CUDA(cudaMemsetAsync(W, 0, lev_ws[dpt] * sizeof(T), s));
            if (max_pairs[dpt] > 0) {
                k_assemble<T><<<dim3(nf, max_pairs[dpt]), ASM_THREADS, ASM_SMEM, s>>>(
                    d_lev[dpt].p, d_fr.p, P.d_pair_elem.p, P.d_pair_pos.p, P.d_rows.p, C, geo, xi, sigma, P.s20 ? 1 : 0,
                    W);
                GL_CUDA(cudaGetLastError());
            }
            if (dpt + 1 < nlev) {
                for (int slot = 0; slot < 2; ++slot) {
                    int nc = (int)child[slot][dpt + 1].size();
                    if (!nc) continue;
                    int ycols = std::min(std::max(1, max_f[dpt + 1] / 8), 1024);
                    k_extend_add<T><<<dim3(nc, ycols), 128, 0, s>>>(slot ? d_ch1[dpt + 1].p : d_ch0[dpt + 1].p,
                                                                  d_fr.p, P.d_rel.p, ws[(dpt + 1) & 1].p, W);
                    GL_CUDA(cudaGetLastError());
                }
            }
            partial_cholesky_level<T>(d_lev[dpt].p, nf, d_fr.p, max_p[dpt], max_f[dpt], W, d_err, s, T(0), nullptr,
                                      sizeof(T) == 8 || P.tc_update);
            inverse_form_level<T>(d_lev[dpt].p, nf, d_fr.p, max_p[dpt], max_f[dpt], W, L, d_err, s);
        }
        GL_CUDA(cudaStreamSynchronize(s));   // the group's lists are released at the end of this scope
        j0 = j1;
    }
}

template void numeric_factor<double>(FactorPlan &, const double *, const double *, const double *, double, double *,
                                     int *, cudaStream_t);
template void numeric_factor<float>(FactorPlan &, const double *, const double *, const double *, double, float *,
                                    int *, cudaStream_t);

// ----------------------------------------------------------------- solves

// Sweep kernels.  A level's work is cut into warp tasks over all its fronts
// (forward: 32 panel rows; backward: a tile of panel columns), which the
// inverse form makes independent of one another, so a level with a few large
// fronts fills the chip as well as one with thousands of small ones.  Where
// the level has fewer than SWEEP_WARPS tasks they are cut along the summed
// dimension too (to no less than 32 columns or 64 rows) and add their parts
// atomically: short tasks hide one another's loads and even out the SMs.  The
// solve of the 475k-DOF corner (FP32) took 66.9, 64.5, 61.6 and 57.5 ms with
// 12, 24, 48 and 96 tasks an SM, the 20k-DOF plate 11.3 to 10.4 ms.
constexpr int SWEEP_CTA = 128;            // four warp tasks
constexpr int SWEEP_WARPS = 152 * 96;

// Forward: panel rows [r0, r0 + 32 R), lane = row (R rows), the columns of blockIdx.z's
// chunk.  Pivot rows give y_1 = L11^{-1} b_1 (up to the diagonal block: zeros
// above it), structure rows subtract W b_1 from the ancestors' entries of b.
// FP64: one FMA per entry on a pipe of two per clock and SM binds it at every
// size that fills the chip; FP32 is bound by reading the panel once.  One CTA
// per front stepping through 32-pivot blocks took 74 us (FP64) and 62 us (FP32)
// a launch on the 308k- and 475k-DOF corners, this form 44 and 25 us.
// Rows per lane of a forward task: two in FP32, 256 contiguous bytes a column,
// which HBM likes better: 9.74 to 8.78 ms for all levels of the 12.2M-DOF corner
// (one level after another), 50.9 to 50.5 ms a solve on the 475k-DOF one.  Four
// rows gained 2% more on the former and cost 3% on the latter.
template <class T>
constexpr int FWD_ROWS = sizeof(T) == 4 ? 2 : 1;

template <class T>
__global__ void __launch_bounds__(SWEEP_CTA) k_fwd(const int *__restrict__ fronts, const FrontDesc *__restrict__ D,
                                                   const T *__restrict__ L, const int *__restrict__ rows, T *b,
                                                   T *y, int chunk) {
    __shared__ __align__(16) T sx[SWEEP_CTA / 32][32];
    const FrontDesc &d = D[fronts[blockIdx.x]];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int p = d.p, f = p + d.q;
    constexpr int R = FWD_ROWS<T>, RT = 32 * R;      // rows per lane, per warp task
    const int r0 = (blockIdx.y * (SWEEP_CTA / 32) + w) * RT;
    const int cb = blockIdx.z * chunk;
    // pivot rows need the columns up to their diagonal block, any structure row all of them
    const int cend = min(r0 + RT <= p ? r0 + RT : p, cb + chunk);
    if (r0 >= f || cb >= cend) {
        cudaGridDependencySynchronize();
        return;
    }
    const T *b1 = b + d.vec_off + d.first;
    const T *Lr[R];
#pragma unroll
    for (int q = 0; q < R; ++q) Lr[q] = L + d.l_off + min(r0 + lane + 32 * q, f - 1);
    constexpr int G = sizeof(T) == 4 ? 32 / R : 16;   // columns in flight per lane
    T l[R][G];
    // the panel does not depend on the launches before: its first columns are on their way during the wait
#pragma unroll
    for (int j = 0; j < G; ++j)
#pragma unroll
        for (int q = 0; q < R; ++q) l[q][j] = cb + j < cend ? Lr[q][(int64_t)(cb + j) * f] : T(0);
    cudaGridDependencySynchronize();
    T acc[R], acc2[R];
#pragma unroll
    for (int q = 0; q < R; ++q) acc[q] = acc2[q] = T(0);
    T *xs = sx[w];
    for (int c = cb; c < cend; c += 32) {
        const int kb = min(32, cend - c);
        __syncwarp();
        xs[lane] = lane < kb ? b1[c + lane] : T(0);
        __syncwarp();
        const int64_t cf = (int64_t)c * f;
#pragma unroll
        for (int g = 0; g < 32; g += G) {
            if (g >= kb) break;
            const bool have = g == 0 && c == cb;
            if (g + G <= kb) {
                if (!have) {
#pragma unroll
                    for (int j = 0; j < G; ++j)
#pragma unroll
                        for (int q = 0; q < R; ++q) l[q][j] = Lr[q][cf + (int64_t)(g + j) * f];
                }
#pragma unroll
                for (int j = 0; j < G; j += 2)
#pragma unroll
                    for (int q = 0; q < R; ++q) {
                        acc[q] += l[q][j] * xs[g + j];
                        acc2[q] += l[q][j + 1] * xs[g + j + 1];
                    }
            } else {
                // the last columns, in fours
                if (!have) {
#pragma unroll
                    for (int j = 0; j < G; ++j)
#pragma unroll
                        for (int q = 0; q < R; ++q) l[q][j] = g + j < kb ? Lr[q][cf + (int64_t)(g + j) * f] : T(0);
                }
#pragma unroll
                for (int h = 0; h < G; h += 4) {
                    if (g + h >= kb) break;
#pragma unroll
                    for (int j = h; j < h + 4; ++j)
#pragma unroll
                        for (int q = 0; q < R; ++q) acc[q] += l[q][j] * xs[g + j];
                }
            }
        }
    }
    cudaTriggerProgrammaticLaunchCompletion();
#pragma unroll
    for (int q = 0; q < R; ++q) {
        const int row = r0 + lane + 32 * q;
        if (row >= f) break;
        const T sum = acc[q] + acc2[q];
        if (row < p) {
            T *yo = y + d.vec_off + d.first + row;
            if (gridDim.z == 1) *yo = sum;
            else atomicAdd(yo, sum);
        } else {
            atomicAdd(b + d.vec_off + rows[d.row_off + row], -sum);
        }
    }
}

// Backward: x_1 = [L11^{-1}; -W]^T [y_1; x_2].  A warp task is a tile of 16
// panel columns over one chunk of the panel's rows, lane = row, one accumulator
// per column; the lanes are summed at the end (warp_sum_many).  With 32 columns
// the kernel took 226 registers and 74.6 us a launch against 54.5 on the
// 308k-DOF corner: too few warps on an SM to cover the loads.  One CTA per
// front took 85 us (FP64) and 68 us (FP32) a launch on the 308k- and 475k-DOF
// corners, this form 44 and 34 us.
constexpr int BWD_TILE = 16;

template <class T>
__global__ void __launch_bounds__(SWEEP_CTA) k_bwd(const int *__restrict__ fronts, const FrontDesc *__restrict__ D,
                                                   const T *__restrict__ L, const int *__restrict__ rows,
                                                   const T *__restrict__ y, T *x, int chunks) {
    constexpr int CT = BWD_TILE;
    const FrontDesc &d = D[fronts[blockIdx.x]];
    const int lane = threadIdx.x & 31;
    const int p = d.p, f = p + d.q;
    const int task = blockIdx.y * (SWEEP_CTA / 32) + (threadIdx.x >> 5);
    const int nct = (p + CT - 1) / CT;
    if (task >= nct * chunks) {
        cudaGridDependencySynchronize();
        return;
    }
    const int j0 = (task % nct) * CT, kb = min(CT, p - j0);
    // the tile's rows start at its diagonal block; chunks of whole 32-row steps
    const int steps = (f - j0 + 31) / 32, per = (steps + chunks - 1) / chunks;
    const int rb = j0 + 32 * per * (task / nct), re = min(f, rb + 32 * per);
    if (rb >= re) {
        cudaGridDependencySynchronize();
        return;
    }
    const T *y1 = y + d.vec_off + d.first, *xo = x + d.vec_off;
    const int *rw = rows + d.row_off;
    const T *Lt = L + d.l_off + (int64_t)j0 * f;
    T acc[CT];
#pragma unroll
    for (int i = 0; i < CT; ++i) acc[i] = T(0);
    // the rows' vector entries: where they are two steps ahead, their values one step ahead
    auto where = [&](int r) {
        const int i = min(r + lane, f - 1);
        return i < p ? y1 + i : xo + rw[i];
    };
    // y_1 or -x_2, zero past the chunk; by the bits, not by the FP64 pipe that binds the kernel
    auto fetch_v = [&](int r, const T *at) {
        const bool in = r + lane < re;
        const int flip = r + lane < p ? 0 : (int)0x80000000u;
        const T t = *at;
        if constexpr (sizeof(T) == 8)
            return in ? (T)__hiloint2double(__double2hiint(t) ^ flip, __double2loint(t)) : T(0);
        else
            return in ? (T)__int_as_float(__float_as_int(t) ^ flip) : T(0);
    };
    T v, vn, l[CT];
    auto fetch_l = [&](int r) {
        const T *Li = Lt + min(r + lane, f - 1);
#pragma unroll
        for (int j = 0; j < CT; ++j) l[j] = j < kb ? Li[(int64_t)j * f] : T(0);
    };
    // the panel does not depend on the launches before: its first rows are on their way during the wait
    fetch_l(rb);
    const T *at = where(rb);
    const T *at1 = where(rb + 32);
    cudaGridDependencySynchronize();
    v = fetch_v(rb, at);
    at = at1;
    for (int r = rb; r < re; r += 32) {
        auto step = [&](auto cols) {
            constexpr int G = decltype(cols)::value;
            if (r != rb) fetch_l(r);
            vn = fetch_v(r + 32, at);
            at = where(r + 64);
#pragma unroll
            for (int j = 0; j < G; ++j) acc[j] += l[j] * v;
        };
        if (kb <= CT / 2) step(std::integral_constant<int, CT / 2>());
        else step(std::integral_constant<int, CT>());
        v = vn;
    }
    cudaTriggerProgrammaticLaunchCompletion();
    warp_sum_many<T, CT>(acc, lane);
    const int j = lane >> 1;      // two lanes hold each sum
    if ((lane & 1) || j >= kb) return;
    T *out = x + d.vec_off + d.first + j0 + j;
    if (chunks == 1) *out = acc[0];
    else atomicAdd(out, acc[0]);
}

void level_clock_enable(FactorPlan &P, bool on) {
    LevelClock &K = P.clock;
    const size_t nlev = P.levels.size();
    if (on && K.ev.size() != 2 * nlev + 1) {
        for (cudaEvent_t e : K.ev)
            if (e) cudaEventDestroy(e);
        K.ev.assign(2 * nlev + 1, nullptr);
        for (cudaEvent_t &e : K.ev) GL_CUDA(cudaEventCreate(&e));
    }
    K.fwd_ms.assign(nlev, 0.0);
    K.bwd_ms.assign(nlev, 0.0);
    K.calls = 0;
    K.on = on;
}

// Events e[0..2 nlev]: e[nlev-1-d] before the forward launch of depth d,
// e[nlev+d] before its backward launch, e[2 nlev] after the last launch.
static void level_clock_fold(const FactorPlan &P) {
    LevelClock &K = P.clock;
    const int nlev = (int)P.levels.size();
    GL_CUDA(cudaEventSynchronize(K.ev[2 * nlev]));
    for (int d = 0; d < nlev; ++d) {
        float a = 0, b = 0;
        GL_CUDA(cudaEventElapsedTime(&a, K.ev[nlev - 1 - d], K.ev[nlev - d]));
        GL_CUDA(cudaEventElapsedTime(&b, K.ev[nlev + d], K.ev[nlev + d + 1]));
        K.fwd_ms[d] += a;
        K.bwd_ms[d] += b;
    }
    K.calls += 1;
}

// A level's launch may start while the one before it in the stream finishes
// (programmatic dependent launch): its CTAs read their descriptors and the
// first part of their panels, then wait for that launch's results.  A launch
// lets the next one start when its tasks reach their last additions (earlier,
// the waiting CTAs take the place of running ones: 12.2 instead of 9.0 ms on the
// 20k-DOF plate).  Every thread waits, also those without work, so that a launch
// never completes before the ones it follows.
template <class K, class... A>
static void launch_chained(K kernel, dim3 grid, cudaStream_t s, A... args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = dim3(SWEEP_CTA);
    cfg.stream = s;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    GL_CUDA(cudaLaunchKernelEx(&cfg, kernel, args...));
}

// One level's forward or backward sweep over the fronts fr[0..nf) of that level.
template <class T>
static void launch_fwd(const FactorPlan &P, const Level &Lv, const int *fr, unsigned nf, const T *L, T *b, T *y,
                       cudaStream_t s) {
    if (nf == 0 || Lv.max_p == 0) return;
    const int tiles = (Lv.max_f + 32 * FWD_ROWS<T> - 1) / (32 * FWD_ROWS<T>), blocks = (Lv.max_p + 31) / 32;
    // (the level's fronts, not nf: the arithmetic is the same however the level is split over streams)
    const int split = std::min<int64_t>(blocks, std::max<int64_t>(1, SWEEP_WARPS / ((int64_t)Lv.fronts.size() * tiles)));
    const int chunk = 32 * ((blocks + split - 1) / split);
    const dim3 g(nf, (tiles + SWEEP_CTA / 32 - 1) / (SWEEP_CTA / 32), (Lv.max_p + chunk - 1) / chunk);
    launch_chained(k_fwd<T>, g, s, fr, (const FrontDesc *)P.d_fr.p, L, (const int *)P.d_rows.p, b, y, chunk);
}

template <class T>
static void launch_bwd(const FactorPlan &P, const Level &Lv, const int *fr, unsigned nf, const T *L, const T *y, T *x,
                       cudaStream_t s) {
    if (nf == 0 || Lv.max_p == 0) return;
    const int tiles = (Lv.max_p + BWD_TILE - 1) / BWD_TILE;
    const int chunks = std::min<int64_t>((Lv.max_f + 63) / 64,
                                         std::max<int64_t>(1, SWEEP_WARPS / ((int64_t)Lv.fronts.size() * tiles)));
    const dim3 g(nf, (tiles * chunks + SWEEP_CTA / 32 - 1) / (SWEEP_CTA / 32));
    launch_chained(k_bwd<T>, g, s, fr, (const FrontDesc *)P.d_fr.p, L, (const int *)P.d_rows.p, y, x, chunks);
}

static HalfStreams &half_streams(const FactorPlan &P) {
    if (!P.hs) {
        auto h = std::make_unique<HalfStreams>();
        int lo = 0, hi = 0;
        GL_CUDA(cudaDeviceGetStreamPriorityRange(&lo, &hi));
        for (int k = 0; k < 2; ++k) {
            GL_CUDA(cudaStreamCreateWithPriority(&h->hi[k], cudaStreamNonBlocking, hi));
            GL_CUDA(cudaStreamCreateWithPriority(&h->lo[k], cudaStreamNonBlocking, lo));
        }
        GL_CUDA(cudaEventCreateWithFlags(&h->fork, cudaEventDisableTiming));
        for (cudaEvent_t &e : h->ev) GL_CUDA(cudaEventCreateWithFlags(&e, cudaEventDisableTiming));
        P.hs = std::move(h);
    }
    return *P.hs;
}

// Overlapped sweeps of the two halves of the subdomains (FactorPlan::overlap_top
// = k > 0).  Half h: deep forward levels (depth >= k) on lo[h], then its top
// levels (forward to the root and backward down to depth k - 1) on hi[h],
// then its deep backward levels on lo[h].  The second half's deep forward
// levels start when the first half enters its top levels.  The halves hold
// disjoint subdomains, so they share no data.
template <class T>
static void solve_levels_overlap(const FactorPlan &P, const T *L, T *b, T *y, T *x, cudaStream_t s) {
    HalfStreams &H = half_streams(P);
    const int nlev = (int)P.levels.size(), k = std::min(P.overlap_top, nlev);
    GL_CUDA(cudaEventRecord(H.fork, s));
    for (int h = 0; h < 2; ++h) {
        GL_CUDA(cudaStreamWaitEvent(H.lo[h], H.fork, 0));
        GL_CUDA(cudaStreamWaitEvent(H.hi[h], H.fork, 0));
    }
    auto part = [&](int h, int d, const int *&fr, unsigned &nf) {
        const Level &Lv = P.levels[d];
        const unsigned na = (unsigned)P.half_fronts[d];
        fr = Lv.d_fronts.p + (h == 0 ? 0 : na);
        nf = h == 0 ? na : (unsigned)Lv.fronts.size() - na;
    };
    // ev[3h]: half h reached its top levels; ev[3h+1]: its top levels are done; ev[3h+2]: all done
    for (int h = 0; h < 2; ++h) {
        if (h == 1) GL_CUDA(cudaStreamWaitEvent(H.lo[1], H.ev[0], 0));
        for (int d = nlev - 1; d >= k; --d) {
            const int *fr; unsigned nf;
            part(h, d, fr, nf);
            launch_fwd<T>(P, P.levels[d], fr, nf, L, b, y, H.lo[h]);
        }
        GL_CUDA(cudaEventRecord(H.ev[3 * h], H.lo[h]));
        GL_CUDA(cudaStreamWaitEvent(H.hi[h], H.ev[3 * h], 0));
        for (int d = k - 1; d >= 0; --d) {
            const int *fr; unsigned nf;
            part(h, d, fr, nf);
            launch_fwd<T>(P, P.levels[d], fr, nf, L, b, y, H.hi[h]);
        }
        for (int d = 0; d < k; ++d) {
            const int *fr; unsigned nf;
            part(h, d, fr, nf);
            launch_bwd<T>(P, P.levels[d], fr, nf, L, y, x, H.hi[h]);
        }
        GL_CUDA(cudaEventRecord(H.ev[3 * h + 1], H.hi[h]));
    }
    for (int h = 0; h < 2; ++h) {
        GL_CUDA(cudaStreamWaitEvent(H.lo[h], H.ev[3 * h + 1], 0));
        for (int d = k; d < nlev; ++d) {
            const int *fr; unsigned nf;
            part(h, d, fr, nf);
            launch_bwd<T>(P, P.levels[d], fr, nf, L, y, x, H.lo[h]);
        }
        GL_CUDA(cudaEventRecord(H.ev[3 * h + 2], H.lo[h]));
        GL_CUDA(cudaStreamWaitEvent(s, H.ev[3 * h + 2], 0));
    }
    GL_CUDA(cudaGetLastError());
}

template <class T>
void factor_solve(const FactorPlan &P, const T *L, T *b, T *y, T *x, cudaStream_t s) {
    const int nlev = (int)P.levels.size();
    const bool timed = P.clock.on && P.clock.ev.size() == 2 * (size_t)nlev + 1;
    if (P.overlap_top > 0 && !timed && P.n_sub >= 2) {
        solve_levels_overlap<T>(P, L, b, y, x, s);
        return;
    }
    auto mark = [&](int k) {
        if (timed) GL_CUDA(cudaEventRecord(P.clock.ev[k], s));
    };
    for (int dpt = nlev - 1; dpt >= 0; --dpt) {
        mark(nlev - 1 - dpt);
        const Level &Lv = P.levels[dpt];
        launch_fwd<T>(P, Lv, Lv.d_fronts.p, (unsigned)Lv.fronts.size(), L, b, y, s);
    }
    for (int dpt = 0; dpt < nlev; ++dpt) {
        mark(nlev + dpt);
        const Level &Lv = P.levels[dpt];
        launch_bwd<T>(P, Lv, Lv.d_fronts.p, (unsigned)Lv.fronts.size(), L, y, x, s);
    }
    GL_CUDA(cudaGetLastError());
    if (timed) {
        mark(2 * nlev);
        level_clock_fold(P);
    }
}

template void factor_solve<double>(const FactorPlan &, const double *, double *, double *, double *, cudaStream_t);
template void factor_solve<float>(const FactorPlan &, const float *, float *, float *, float *, cudaStream_t);

void factor_solve8(const FactorPlan &P, const double *L, double *b, double *y, double *x, int *d_err, cudaStream_t s) {
    const int nlev = (int)P.levels.size();
    for (int d = nlev - 1; d >= 0; --d) {
        const Level &Lv = P.levels[d];
        fwd_tc_level(Lv.d_fronts.p, (int)Lv.fronts.size(), P.d_fr.p, Lv.max_p, Lv.max_f, L, P.d_rows.p, b, y, d_err, s);
    }
    for (int d = 0; d < nlev; ++d) {
        const Level &Lv = P.levels[d];
        bwd_tc_level(Lv.d_fronts.p, (int)Lv.fronts.size(), P.d_fr.p, Lv.max_p, Lv.max_f, L, P.d_rows.p, y, x, d_err, s);
    }
}

// ----------------------------------------------------------------- local <-> global

// b = r at the local DOFs, y = x = 0 (the sweeps add into them)
template <class T>
__global__ void k_gather(int64_t n, const int64_t *__restrict__ gdof, const double *__restrict__ r, T *__restrict__ b,
                         T *__restrict__ y, T *__restrict__ x) {
    int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i >= n) return;
    b[i] = (T)r[gdof[i]];
    y[i] = x[i] = T(0);
}

template <class T>
__global__ void k_scatter_add(int64_t n, const int64_t *__restrict__ gdof, const T *__restrict__ xl, double *__restrict__ z) {
    int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i < n) atomicAdd(z + gdof[i], (double)xl[i]);
}

template <class T>
void gather_local(const FactorPlan &P, const double *r, T *b, T *y, T *x, cudaStream_t s) {
    if (!P.n_local) return;
    k_gather<T><<<(unsigned)((P.n_local + 255) / 256), 256, 0, s>>>(P.n_local, P.d_gdof.p, r, b, y, x);
    GL_CUDA(cudaGetLastError());
}
template <class T>
void scatter_add_local(const FactorPlan &P, const T *xl, double *z, cudaStream_t s) {
    if (!P.n_local) return;
    k_scatter_add<T><<<(unsigned)((P.n_local + 255) / 256), 256, 0, s>>>(P.n_local, P.d_gdof.p, xl, z);
    GL_CUDA(cudaGetLastError());
}
template void gather_local<double>(const FactorPlan &, const double *, double *, double *, double *, cudaStream_t);
template void gather_local<float>(const FactorPlan &, const double *, float *, float *, float *, cudaStream_t);
template void scatter_add_local<double>(const FactorPlan &, const double *, double *, cudaStream_t);
template void scatter_add_local<float>(const FactorPlan &, const float *, double *, cudaStream_t);

// ----------------------------------------------------------------- dense (coarse) inverse

// K^{-1} of a dense SPD matrix through the same partial Cholesky: factoring the
// p = n pivots of the 2n x 2n front [[A_s, I], [I, 0]] leaves the Schur
// complement 0 - I A_s^{-1} I = -A_s^{-1} in the trailing block, where
// A_s = D A D is A scaled to unit diagonal (D = diag(A)^{-1/2}); then
// A^{-1} = D A_s^{-1} D.  With drop > 0 a pivot of |v| <= drop (on the unit
// diagonal scale) marks its column as linearly dependent on the earlier ones:
// the column is left out of the factor, its row and column of the result are
// zero, and the result is the inverse of A on the kept columns -- a
// generalised inverse of A when the dropped columns lie in the span of the
// kept ones (a zero column of A has a zero scaled pivot and is dropped too).
__device__ __forceinline__ double unit_diag_scale(const double *A, int n, int64_t i) {
    const double d = A[i + i * (int64_t)n];
    return d > 0.0 ? 1.0 / sqrt(d) : 0.0;
}

__global__ void k_aug_init(const double *__restrict__ A, int n, double *__restrict__ F) {
    const int64_t m = 2 * (int64_t)n;
    for (int64_t idx = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; idx < m * m; idx += (int64_t)gridDim.x * blockDim.x) {
        int64_t i = idx % m, j = idx / m;
        double v = 0.0;
        if (i < n && j < n) {
            const double di = unit_diag_scale(A, n, i), dj = unit_diag_scale(A, n, j);
            v = (di == 0.0 || dj == 0.0) ? 0.0 : A[i + j * n] * di * dj;
        } else if (j < n && i - n == j) {
            v = 1.0;
        }
        F[idx] = v;
    }
}

__global__ void k_extract_inv(const double *__restrict__ A, const double *__restrict__ F, int n,
                              double *__restrict__ Ainv) {
    const int64_t m = 2 * (int64_t)n;
    for (int64_t idx = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; idx < (int64_t)n * n;
         idx += (int64_t)gridDim.x * blockDim.x) {
        int64_t i = idx % n, j = idx / n;
        int64_t a = i > j ? i : j, b = i > j ? j : i;   // lower triangle of the trailing block
        Ainv[idx] = -F[(n + a) + (n + b) * m] * unit_diag_scale(A, n, i) * unit_diag_scale(A, n, j);
    }
}

int dense_inverse(const double *A, int n, double *Ainv, int *d_err, cudaStream_t s, double drop) {
    DBuf<FrontDesc> d;
    DBuf<int> idx, drops;
    FrontDesc f{};
    f.p = n;
    f.q = n;
    f.vlen = 2 * n;
    f.parent = -1;
    d.upload(std::vector<FrontDesc>{f}, s);
    idx.upload(std::vector<int>{0}, s);
    drops.alloc(1);
    drops.zero(s);
    DBuf<double> F;
    F.alloc((size_t)4 * n * n);
    k_aug_init<<<1024, 256, 0, s>>>(A, n, F.p);
    GL_CUDA(cudaGetLastError());
    partial_cholesky_level<double>(idx.p, 1, d.p, n, 2 * n, F.p, d_err, s, drop, drops.p);
    k_extract_inv<<<1024, 256, 0, s>>>(A, F.p, n, Ainv);
    GL_CUDA(cudaGetLastError());
    int h = 0;
    GL_CUDA(cudaMemcpyAsync(&h, drops.p, sizeof(int), cudaMemcpyDeviceToHost, s));
    GL_CUDA(cudaStreamSynchronize(s));
    return h;
}

// Block-diagonal version: for each block b, y[o_b : o_b + n_b] = A_b x[o_b : o_b + n_b],
// A_b stored column-major at aoff[b]; one warp per output row.
__global__ void k_symv_blocks(const double *__restrict__ A, const int64_t *__restrict__ aoff,
                              const int *__restrict__ voff, const int *__restrict__ nb, int nblk,
                              const double *__restrict__ x, double *__restrict__ y, int total) {
    const int lane = threadIdx.x & 31;
    const int row = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
    if (row >= total) return;
    int lo = 0, hi = nblk - 1;   // block containing this row
    while (lo < hi) {
        int mid = (lo + hi + 1) >> 1;
        if (voff[mid] <= row) lo = mid;
        else hi = mid - 1;
    }
    const int b = lo, n = nb[b], i = row - voff[b];
    const double *col = A + aoff[b] + (int64_t)i * n;
    const double *xb = x + voff[b];
    double acc = 0.0;
    for (int j = lane; j < n; j += 32) acc += col[j] * xb[j];
    for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
    if (lane == 0) y[row] = acc;
}

void dense_symv_blocks(const double *A, const int64_t *aoff, const int *voff, const int *nb, int nblk, int total,
                       const double *x, double *y, cudaStream_t s) {
    if (total <= 0) return;
    k_symv_blocks<<<(total + 7) / 8, 256, 0, s>>>(A, aoff, voff, nb, nblk, x, y, total);
    GL_CUDA(cudaGetLastError());
}

}  // namespace gl
