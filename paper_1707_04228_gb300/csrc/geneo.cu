// GenEO coarse-space kernels, coarse restrict/prolong, PCG vector kernels.
//
// Section 2.3 (Fig. eig): on each subdomain a few of the lowest-energy modes
// of a local generalised eigenproblem are computed and glued with a
// partition of unity into the coarse space.  The eigenproblem solved here is
// A_j^N p = lambda B_j p with B_j = Xi_j A_j^N Xi_j, through the definite
// pencil B p = mu (A^N + sigma B) p (largest mu <-> smallest lambda), by a block
// Krylov (Lanczos) method; these are its batched pieces.
#include <algorithm>

#include "geneo.h"
#include "warp.cuh"

namespace gl {

constexpr int NV_MAX = 32;

// (local element products: local_K_apply in ku.cu, matrix-free)

// ---------------------------------------------------------------- block Krylov pieces

// G_s[a * ldg + j] += sum_i A_s[i, a] B_s[i, j], a < ma, j < KRY_B, over a chunk
// of GRAM_ROWS rows.  Warp w takes the columns a = w, w + 8, ... of A (each read
// once, coalesced), B's chunk sits in shared memory; bound by the FP64 pipe
// once there are rows enough.
constexpr int GRAM_ROWS = 512;

__global__ void __launch_bounds__(256) k_kry_gram(const int64_t *__restrict__ voff, const int64_t *__restrict__ vlen,
                                                  const double *__restrict__ A, int lda, int ma,
                                                  const double *__restrict__ B, double *__restrict__ G, int64_t gs,
                                                  int ldg) {
    const int s = blockIdx.x;
    const int64_t n = vlen[s];
    const int64_t r0 = (int64_t)blockIdx.y * GRAM_ROWS;
    if (r0 >= n) return;
    const int rows = (int)min((int64_t)GRAM_ROWS, n - r0);
    __shared__ double sb[KRY_B][GRAM_ROWS];
    const double *Bs = B + voff[s] * KRY_B + r0, *As = A + voff[s] * lda + r0;
    for (int idx = threadIdx.x; idx < KRY_B * GRAM_ROWS; idx += 256) {
        const int i = idx % GRAM_ROWS, j = idx / GRAM_ROWS;
        sb[j][i] = i < rows ? Bs[(int64_t)j * n + i] : 0.0;
    }
    __syncthreads();
    const int lane = threadIdx.x & 31;
    for (int a = threadIdx.x >> 5; a < ma; a += 8) {
        const double *Aa = As + (int64_t)a * n;
        double acc[KRY_B];
#pragma unroll
        for (int j = 0; j < KRY_B; ++j) acc[j] = 0.0;
#pragma unroll 4
        for (int i = lane; i < GRAM_ROWS; i += 32) {
            const double v = i < rows ? Aa[i] : 0.0;
#pragma unroll
            for (int j = 0; j < KRY_B; ++j) acc[j] += v * sb[j][i];
        }
        warp_sum_many<double, KRY_B>(acc, lane);
        if (lane % (32 / KRY_B) == 0) atomicAdd(G + s * gs + (int64_t)a * ldg + lane / (32 / KRY_B), acc[0]);
    }
}

static unsigned row_chunks(const FactorPlan &P, int rows) {
    int64_t maxn = 1;
    for (auto v : P.vec_len) maxn = std::max(maxn, v);
    return (unsigned)((maxn + rows - 1) / rows);
}

void kry_gram(const FactorPlan &P, const double *A, int lda, int ma, const double *B, double *G, int64_t gs, int ldg,
              cudaStream_t s) {
    if (ma <= 0) return;
    k_kry_gram<<<dim3(P.n_sub, row_chunks(P, GRAM_ROWS)), 256, 0, s>>>(P.d_vec_off.p, P.d_vec_len.p, A, lda, ma, B, G,
                                                                       gs, ldg);
    GL_CUDA(cudaGetLastError());
}

// W_z -= V_z H for the pairs z: one row per thread, H in shared memory.
__global__ void __launch_bounds__(256) k_kry_project(const int64_t *__restrict__ voff,
                                                     const int64_t *__restrict__ vlen, KryBlocks K, int ldv, int m,
                                                     const double *__restrict__ H, int64_t hs, int ldh) {
    const int s = blockIdx.x;
    const int64_t n = vlen[s], i = (int64_t)blockIdx.y * 256 + threadIdx.x;
    if ((int64_t)blockIdx.y * 256 >= n) return;
    __shared__ double sh[KRY_MAX * KRY_B];
    for (int idx = threadIdx.x; idx < m * KRY_B; idx += 256)
        sh[idx] = H[s * hs + (int64_t)(idx / KRY_B) * ldh + idx % KRY_B];
    __syncthreads();
    if (i >= n) return;
    double *out = K.W[blockIdx.z] + voff[s] * KRY_B + i;
    const double *Vi = K.V[blockIdx.z] + voff[s] * ldv + i;
    double w[KRY_B];
#pragma unroll
    for (int j = 0; j < KRY_B; ++j) w[j] = out[(int64_t)j * n];
#pragma unroll 4
    for (int c = 0; c < m; ++c) {
        const double v = Vi[(int64_t)c * n];
#pragma unroll
        for (int j = 0; j < KRY_B; ++j) w[j] -= v * sh[c * KRY_B + j];
    }
#pragma unroll
    for (int j = 0; j < KRY_B; ++j) out[(int64_t)j * n] = w[j];
}

void kry_project(const FactorPlan &P, const KryBlocks &K, int ldv, int m, const double *H, int64_t hs, int ldh,
                 cudaStream_t s) {
    if (m <= 0) return;
    k_kry_project<<<dim3(P.n_sub, row_chunks(P, 256), K.count), 256, 0, s>>>(P.d_vec_off.p, P.d_vec_len.p, K, ldv, m,
                                                                            H, hs, ldh);
    GL_CUDA(cudaGetLastError());
}

// Uniform in [-1, 1): splitmix64 of the seed and an index.
__device__ __forceinline__ double hash_uniform(uint64_t seed, int64_t i) {
    uint64_t z = seed + 0x9E3779B97F4A7C15ull * (uint64_t)(i + 1);
    z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
    z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
    z = z ^ (z >> 31);
    return (double)(z >> 11) * (2.0 / 9007199254740992.0) - 1.0;
}

// W_z <- W_z R in place; with col >= 0 the columns are also stored at column col
// of V_z.  With refill != 0 the columns that R drops become random ones: the
// block's image lies in the basis there, and without new directions an
// eigenvalue with more copies than the block has columns would come out with
// KRY_B of them only (Xi constant over the whole subdomain: every eigenvalue
// is the same one).
__global__ void __launch_bounds__(256) k_kry_scale(const int64_t *__restrict__ voff, const int64_t *__restrict__ vlen,
                                                   KryBlocks K, const double *__restrict__ R, int ldv, int col,
                                                   uint64_t refill) {
    const int s = blockIdx.x;
    const int64_t n = vlen[s], i = (int64_t)blockIdx.y * 256 + threadIdx.x;
    if ((int64_t)blockIdx.y * 256 >= n) return;
    __shared__ double sr[KRY_B * KRY_B];
    if (threadIdx.x < KRY_B * KRY_B) sr[threadIdx.x] = R[(int64_t)s * KRY_B * KRY_B + threadIdx.x];
    __syncthreads();
    if (i >= n) return;
    double *io = K.W[blockIdx.z] + voff[s] * KRY_B + i;
    double w[KRY_B], o[KRY_B];
#pragma unroll
    for (int j = 0; j < KRY_B; ++j) {
        w[j] = io[(int64_t)j * n];
        o[j] = 0.0;
    }
#pragma unroll
    for (int c = 0; c < KRY_B; ++c)
#pragma unroll
        for (int j = 0; j < KRY_B; ++j) o[j] += w[c] * sr[c * KRY_B + j];
    if (refill) {
#pragma unroll
        for (int j = 0; j < KRY_B; ++j) {
            bool dropped = true;
#pragma unroll
            for (int c = 0; c < KRY_B; ++c) dropped = dropped && sr[c * KRY_B + j] == 0.0;
            if (dropped) o[j] = hash_uniform(refill, (voff[s] + i) * KRY_B + j);
        }
    }
#pragma unroll
    for (int j = 0; j < KRY_B; ++j) io[(int64_t)j * n] = o[j];
    if (col >= 0) {
        double *dst = K.V[blockIdx.z] + voff[s] * ldv + (int64_t)col * n + i;
#pragma unroll
        for (int j = 0; j < KRY_B; ++j) dst[(int64_t)j * n] = o[j];
    }
}

void kry_scale(const FactorPlan &P, const KryBlocks &K, const double *R, int ldv, int col, cudaStream_t s,
               uint64_t refill) {
    k_kry_scale<<<dim3(P.n_sub, row_chunks(P, 256), K.count), 256, 0, s>>>(P.d_vec_off.p, P.d_vec_len.p, K, R, ldv,
                                                                          col, refill);
    GL_CUDA(cudaGetLastError());
}

// out[:, 0..k) = V[:, 0..m) Y (row-major m x k, leading dimension ldy), k <= KRY_MAX, eight columns at a time.
__global__ void __launch_bounds__(256) k_kry_combine(const int64_t *__restrict__ voff,
                                                     const int64_t *__restrict__ vlen, const double *__restrict__ V,
                                                     int ldv, int m, const double *__restrict__ Y, int64_t ys, int ldy,
                                                     int k, double *__restrict__ out, int ldo) {
    const int s = blockIdx.x, c0 = blockIdx.z * 8;
    const int64_t n = vlen[s], i = (int64_t)blockIdx.y * 256 + threadIdx.x;
    if ((int64_t)blockIdx.y * 256 >= n) return;
    __shared__ double sy[KRY_MAX * 8];
    for (int idx = threadIdx.x; idx < m * 8; idx += 256)
        sy[idx] = c0 + idx % 8 < k ? Y[s * ys + (int64_t)(idx / 8) * ldy + c0 + idx % 8] : 0.0;
    __syncthreads();
    if (i >= n) return;
    const double *Vi = V + voff[s] * ldv + i;
    double w[8];
#pragma unroll
    for (int j = 0; j < 8; ++j) w[j] = 0.0;
#pragma unroll 4
    for (int c = 0; c < m; ++c) {
        const double v = Vi[(int64_t)c * n];
#pragma unroll
        for (int j = 0; j < 8; ++j) w[j] += v * sy[c * 8 + j];
    }
    double *o = out + voff[s] * ldo + i;
#pragma unroll
    for (int j = 0; j < 8; ++j)
        if (c0 + j < k) o[(int64_t)(c0 + j) * n] = w[j];
}

void kry_combine(const FactorPlan &P, const double *V, int ldv, int m, const double *Y, int64_t ys, int ldy, int k,
                 double *out, int ldo, cudaStream_t s) {
    k_kry_combine<<<dim3(P.n_sub, row_chunks(P, 256), (k + 7) / 8), 256, 0, s>>>(P.d_vec_off.p, P.d_vec_len.p, V, ldv,
                                                                                m, Y, ys, ldy, k, out, ldo);
    GL_CUDA(cudaGetLastError());
}

// ---------------------------------------------------------------- small eigenproblems

// The projected problems are tiny (at most KRY_MAX rows), so their kernels are
// a chain of dependent steps: one CTA per subdomain with everything in shared
// memory, each Jacobi round applying half as many disjoint rotations as there
// are rows at once (round-robin pairs), every 2 x 2 block of C that a pair of
// rotations touches by one thread, two barriers per round.
constexpr int GENEIG_THREADS = 256;

// Pair i of round t in the round-robin tournament of m (even) players.
__device__ __forceinline__ void jacobi_pair(int m, int t, int i, int &p, int &q) {
    const int a = i == 0 ? m - 1 : (t + i) % (m - 1), b = (t + m - 1 - i) % (m - 1);
    p = min(a, b);
    q = max(a, b);
}

// Rotation (c, s) that annihilates apq between the diagonal entries app and
// aqq.  Only the angle may be rough (it leaves its error times apq, which the
// next sweep takes), so it is computed in FP32; c^2 + s^2 = 1 holds to T.
template <class T>
__device__ __forceinline__ void jacobi_rotation(T app, T aqq, T apq, T &c, T &s) {
    const float b = (float)apq;
    if (b == 0.0f) {
        c = T(1);
        s = T(0);
        return;
    }
    const float tau = (float)(aqq - app) / (2.0f * b);
    const T t = (T)(copysignf(1.0f, tau) / (fabsf(tau) + sqrtf(1.0f + tau * tau)));
    c = rsqrt(T(1) + t * t);
    s = t * c;
}

// Eigenvectors of the symmetric k x k matrix C by cyclic Jacobi, until the
// squares of the off-diagonal entries sum to at most tol of all: on return the
// diagonal of C holds the eigenvalues and Q the vectors as columns (times what
// it held, unless init).  All threads of the CTA take part; cs holds 2 numbers
// and pairs one per pair, red two per warp.
template <class T>
__device__ void cta_jacobi(T *C, T *Q, int ld, int k, T *cs, int *pairs, T *red, T tol, bool init) {
    const int m = k + (k & 1), np = m / 2, nt = blockDim.x, tid = threadIdx.x;
    if (init)
        for (int idx = tid; idx < k * k; idx += nt) Q[(idx / k) * ld + idx % k] = idx / k == idx % k ? T(1) : T(0);
    __syncthreads();
    for (int sweep = 0; sweep < 60; ++sweep) {
        T off = T(0), tot = T(0);
        for (int idx = tid; idx < k * k; idx += nt) {
            const T v = C[(idx / k) * ld + idx % k];
            tot += v * v;
            if (idx / k != idx % k) off += v * v;
        }
        for (int o = 16; o > 0; o >>= 1) {
            off += __shfl_xor_sync(0xffffffffu, off, o);
            tot += __shfl_xor_sync(0xffffffffu, tot, o);
        }
        if ((tid & 31) == 0) {
            red[2 * (tid >> 5)] = off;
            red[2 * (tid >> 5) + 1] = tot;
        }
        __syncthreads();
        off = tot = T(0);
        for (int w = 0; w < nt / 32; ++w) {
            off += red[2 * w];
            tot += red[2 * w + 1];
        }
        __syncthreads();
        if (!(off > tol * tot)) break;   // uniform: every thread adds the same numbers
        for (int t = 0; t < m - 1; ++t) {
            for (int i = tid; i < np; i += nt) {
                int p, q;
                jacobi_pair(m, t, i, p, q);
                T c = T(1), sn = T(0);
                if (q < k) jacobi_rotation(C[p * ld + p], C[q * ld + q], C[p * ld + q], c, sn);
                cs[2 * i] = c;
                cs[2 * i + 1] = sn;
                pairs[i] = p | (q << 16);
            }
            __syncthreads();
            // a warp per pair of rows (C) or row (Q), a lane per pair of columns
            for (int j = tid & 31; j < np; j += 32) {
                const int u = pairs[j] & 0xFFFF, v = pairs[j] >> 16;
                const T cj = cs[2 * j], sj = cs[2 * j + 1];
                for (int i = tid >> 5; i < np; i += nt >> 5) {
                    const int p = pairs[i] & 0xFFFF, q = pairs[i] >> 16;
                    const T ci = cs[2 * i], si = cs[2 * i + 1];
                    if (q < k && v < k) {
                        const T a = C[p * ld + u], b = C[p * ld + v], c = C[q * ld + u], d = C[q * ld + v];
                        const T a1 = cj * a - sj * b, b1 = sj * a + cj * b;
                        const T c1 = cj * c - sj * d, d1 = sj * c + cj * d;
                        C[p * ld + u] = ci * a1 - si * c1;
                        C[p * ld + v] = ci * b1 - si * d1;
                        C[q * ld + u] = si * a1 + ci * c1;
                        C[q * ld + v] = si * b1 + ci * d1;
                    } else if (q < k) {   // odd k: the player without a partner (u) is not rotated
                        const T a = C[p * ld + u], c = C[q * ld + u];
                        C[p * ld + u] = ci * a - si * c;
                        C[q * ld + u] = si * a + ci * c;
                    } else if (v < k) {
                        const T a = C[p * ld + u], b = C[p * ld + v];
                        C[p * ld + u] = cj * a - sj * b;
                        C[p * ld + v] = sj * a + cj * b;
                    }
                }
                if (v < k)
                    for (int r = tid >> 5; r < k; r += nt >> 5) {
                        const T a = Q[r * ld + u], b = Q[r * ld + v];
                        Q[r * ld + u] = cj * a - sj * b;
                        Q[r * ld + v] = sj * a + cj * b;
                    }
            }
            __syncthreads();
        }
    }
    __syncthreads();
}

// out = A^T B (at) or A B, m x m, leading dimension ld.
__device__ void cta_product(const double *A, const double *B, double *out, int ld, int m, bool at) {
    for (int idx = threadIdx.x; idx < m * m; idx += blockDim.x) {
        const int i = idx / m, j = idx % m;
        double v = 0.0;
        if (at)
            for (int k = 0; k < m; ++k) v += A[k * ld + i] * B[k * ld + j];
        else
            for (int k = 0; k < m; ++k) v += A[i * ld + k] * B[k * ld + j];
        out[i * ld + j] = v;
    }
    __syncthreads();
}

// Eigenpairs of the symmetric m x m matrix C in FP64: Jacobi in FP32 first,
// whose vectors, made orthonormal to FP64 rounding by two Newton-Schulz steps
// Q (3 - Q^T Q) / 2, leave C nearly diagonal, so that the FP64 sweeps (each
// some 6 m^3 FMAs at two per clock) are two or three instead of about nine.
// tmp: m x ld doubles.
__device__ void cta_eig(double *C, double *Q, double *tmp, int ld, int m, double *cs, int *pairs, double *red) {
    const int nt = blockDim.x, tid = threadIdx.x;
    float *Cf = reinterpret_cast<float *>(tmp), *Qf = Cf + m * ld;
    // C scaled by a power of two to FP32's range
    double big = 0.0;
    for (int idx = tid; idx < m * m; idx += nt) big = fmax(big, fabs(C[(idx / m) * ld + idx % m]));
    for (int o = 16; o > 0; o >>= 1) big = fmax(big, __shfl_xor_sync(0xffffffffu, big, o));
    if ((tid & 31) == 0) red[tid >> 5] = big;
    __syncthreads();
    big = 0.0;
    for (int w = 0; w < nt / 32; ++w) big = fmax(big, red[w]);
    __syncthreads();
    const int e = big > 0.0 && big < INFINITY ? -ilogb(big) : 0;
    for (int idx = tid; idx < m * m; idx += nt) {
        const int at = (idx / m) * ld + idx % m;
        C[at] = scalbn(C[at], e);
        Cf[at] = (float)C[at];
    }
    __syncthreads();
    cta_jacobi<float>(Cf, Qf, ld, m, reinterpret_cast<float *>(cs), pairs, reinterpret_cast<float *>(red), 1e-11f,
                      true);
    for (int idx = tid; idx < m * m; idx += nt) {
        const int at = (idx / m) * ld + idx % m;
        Q[at] = (double)Qf[at];
    }
    __syncthreads();
    for (int step = 0; step < 2; ++step) {
        cta_product(Q, Q, tmp, ld, m, true);
        // Q <- Q (3 I - tmp) / 2, nt / m rows at a time
        const int rows = max(1, nt / m);
        for (int r0 = 0; r0 < m; r0 += rows) {
            const int i = r0 + tid / m, j = tid % m;
            const bool on = tid < rows * m && i < m;
            double v = 0.0;
            if (on) {
                for (int k = 0; k < m; ++k) v -= Q[i * ld + k] * tmp[k * ld + j];
                v = 0.5 * (3.0 * Q[i * ld + j] + v);
            }
            __syncthreads();
            if (on) Q[i * ld + j] = v;
            __syncthreads();
        }
    }
    cta_product(C, Q, tmp, ld, m, false);
    cta_product(Q, tmp, C, ld, m, true);
    for (int idx = tid; idx < m * m; idx += nt) {
        const int i = idx / m, j = idx % m;
        if (i < j) C[i * ld + j] = C[j * ld + i] = 0.5 * (C[i * ld + j] + C[j * ld + i]);
    }
    __syncthreads();
    cta_jacobi<double>(C, Q, ld, m, cs, pairs, red, 1e-30, false);
    for (int i = tid; i < m; i += nt) C[i * ld + i] = scalbn(C[i * ld + i], -e);
    __syncthreads();
}

// R_s with W R_s orthonormal in the M inner product, from G_s = W^T M W: Q
// Lambda^{-1/2} of G's eigenpairs; directions at or below the noise become zero
// columns.  H holds the coefficients that W's projection took away.  FIRST:
// noise is drop times the block's squared norm before the projection.  Else (a
// block of near-unit columns and random ones of any length) every column is held
// to drop times its own, and those that stay are brought to a length near one
// by a power of two.
template <bool FIRST>
__global__ void __launch_bounds__(64) k_kry_orth(const double *__restrict__ G, const double *__restrict__ H, int64_t hs,
                                                 int ldh, int m, double drop, double *__restrict__ R,
                                                 int *__restrict__ err) {
    constexpr int ld = KRY_B + 1;
    __shared__ double C[KRY_B * ld], Q[KRY_B * ld], cs[KRY_B], red[4], lost[KRY_B], scale[KRY_B];
    __shared__ int pairs[KRY_B / 2];
    const int s = blockIdx.x, tid = threadIdx.x;
    if (tid < KRY_B) lost[tid] = 0.0;
    for (int idx = tid; idx < KRY_B * KRY_B; idx += 64) {
        const int i = idx / KRY_B, j = idx % KRY_B;
        const double *g = G + (int64_t)s * KRY_B * KRY_B;
        C[i * ld + j] = 0.5 * (g[idx] + g[j * KRY_B + i]);
    }
    __syncthreads();
    double h2 = 0.0;                                         // of column tid % KRY_B
    for (int idx = tid; idx < m * KRY_B; idx += 64) {
        const double h = H[s * hs + (int64_t)(idx / KRY_B) * ldh + idx % KRY_B];
        h2 += h * h;
    }
    if (tid < KRY_B) h2 += C[tid * ld + tid];
    atomicAdd(&lost[tid % KRY_B], h2);
    __syncthreads();
    if (tid < KRY_B) {
        const double g = C[tid * ld + tid];
        if (FIRST || !(fabs(g) < INFINITY)) scale[tid] = 1.0;
        else scale[tid] = g > drop * lost[tid] ? scalbn(1.0, -(ilogb(g) / 2)) : 0.0;
    }
    __syncthreads();
    const int ci = tid / KRY_B, cj = tid % KRY_B;            // 64 threads, 64 entries
    if (!FIRST) C[ci * ld + cj] *= scale[ci] * scale[cj];
    __syncthreads();
    double sum = 0.0, big = 0.0;
    for (int j = 0; j < KRY_B; ++j) sum += FIRST ? lost[j] : C[j * ld + j];
    const double floor_ = drop * sum;
    // scaled by a power of two to the range of the rotations' FP32 angles
    for (int idx = 0; idx < KRY_B * KRY_B; ++idx) big = fmax(big, fabs(C[(idx / KRY_B) * ld + idx % KRY_B]));
    const int e = big > 0.0 && big < INFINITY ? -ilogb(big) : 0;
    __syncthreads();
    C[ci * ld + cj] = scalbn(C[ci * ld + cj], e);
    __syncthreads();
    cta_jacobi<double>(C, Q, ld, KRY_B, cs, pairs, red, 1e-30, true);
    const double lam = scalbn(C[cj * ld + cj], -e);
    if (!(fabs(lam) < INFINITY)) atomicExch(err, 1);
    R[(int64_t)s * KRY_B * KRY_B + tid] = lam > floor_ && lam > 0.0 ? scale[ci] * Q[ci * ld + cj] / sqrt(lam) : 0.0;
}

void kry_orth(int n_sub, bool first, const double *G, const double *H, int64_t hs, int ldh, int m, double drop,
              double *R, int *d_err, cudaStream_t s) {
    if (first) k_kry_orth<true><<<n_sub, 64, 0, s>>>(G, H, hs, ldh, m, drop, R, d_err);
    else k_kry_orth<false><<<n_sub, 64, 0, s>>>(G, H, hs, ldh, m, drop, R, d_err);
    GL_CUDA(cudaGetLastError());
}

// Ritz pairs of the m x m projected matrix T_s (its upper triangle is read),
// largest first: keep values mu and vectors Y (row-major m x keep), and the
// largest relative residual of the first nev, sqrt(y^T G y) / mu with y the
// vector's part on the last block and G the squared norms of what that block's
// image has left outside the basis.  A value of exactly zero is that of a zero
// column: no pair yet, unless the basis holds the whole space of the subdomain.
__global__ void __launch_bounds__(GENEIG_THREADS) k_kry_ritz(const int64_t *__restrict__ vlen,
                                                             const double *__restrict__ T, int ldt, int m,
                                                             const double *__restrict__ G, int nev, int keep,
                                                             double *__restrict__ Y, int ldy, double *__restrict__ mu,
                                                             unsigned long long *__restrict__ worst) {
    extern __shared__ double sm[];
    const int ld = m + 1, s = blockIdx.x, tid = threadIdx.x, nt = blockDim.x;
    double *C = sm, *Q = C + m * ld, *tmp = Q + m * ld, *cs = tmp + m * ld, *red = cs + m + 2;
    __shared__ int rank[KRY_MAX];
    const double *Ts = T + (int64_t)s * ldt * ldt;
    for (int idx = tid; idx < m * m; idx += nt) {
        const int i = idx / m, j = idx % m;
        C[i * ld + j] = Ts[(int64_t)min(i, j) * ldt + max(i, j)];
    }
    __syncthreads();
    cta_eig(C, Q, tmp, ld, m, cs, rank, red);   // rank is free until the pairs are known
    for (int a = tid; a < m; a += nt) {
        const double me = C[a * ld + a];
        int r = 0;
        for (int i = 0; i < m; ++i) {
            const double v = C[i * ld + i];
            r += v > me || (v == me && i < a);
        }
        rank[a] = r;
    }
    __syncthreads();
    for (int a = tid; a < m; a += nt)
        if (rank[a] == 0) cs[m] = C[a * ld + a];
    __syncthreads();
    for (int idx = tid; idx < m * m; idx += nt) {
        const int r = rank[idx % m];
        if (r < keep) Y[((int64_t)s * KRY_MAX + idx / m) * ldy + r] = Q[(idx / m) * ld + idx % m];
    }
    for (int a = tid; a < m; a += nt) {
        const int r = rank[a];
        const double me = C[a * ld + a];
        if (r < keep) mu[(int64_t)s * ldy + r] = me;
        if (r >= nev) continue;
        const double *g = G + (int64_t)s * KRY_B * KRY_B;
        double res = 0.0;
        for (int i = 0; i < KRY_B; ++i)
            for (int j = 0; j < KRY_B; ++j) res += Q[(m - KRY_B + i) * ld + a] * g[i * KRY_B + j] * Q[(m - KRY_B + j) * ld + a];
        const double rel = me > 0.0 || m >= vlen[s] ? sqrt(fmax(res, 0.0)) / fmax(me, 1e-12 * cs[m]) : INFINITY;
        atomicMax(worst, (unsigned long long)__double_as_longlong(rel));   // rel >= 0: ordered like its bits
    }
}

static size_t ritz_smem(int m) { return sizeof(double) * ((size_t)3 * m * (m + 1) + m + 2 + 2 * (GENEIG_THREADS / 32)); }

void kry_ritz(const FactorPlan &P, const double *T, int ldt, int m, const double *G, int nev, int keep, double *Y,
              int ldy, double *mu, unsigned long long *worst, cudaStream_t s) {
    static SmemLimit limit;
    raise_smem_limit(limit, ritz_smem(KRY_MAX), [](size_t v) {
        GL_CUDA(cudaFuncSetAttribute(k_kry_ritz, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)v));
    });
    GL_CUDA(cudaMemsetAsync(worst, 0, sizeof(*worst), s));
    k_kry_ritz<<<P.n_sub, GENEIG_THREADS, ritz_smem(m), s>>>(P.d_vec_len.p, T, ldt, m, G, nev, keep, Y, ldy, mu, worst);
    GL_CUDA(cudaGetLastError());
}

// T_s = diag(mu_s) (k values), the rest of T_s zero.
__global__ void k_kry_diag(double *__restrict__ T, int ldt, const double *__restrict__ mu, int ldm, int k) {
    const int s = blockIdx.x;
    for (int idx = threadIdx.x; idx < ldt * ldt; idx += blockDim.x)
        T[(int64_t)s * ldt * ldt + idx] = idx / ldt == idx % ldt && idx / ldt < k ? mu[(int64_t)s * ldm + idx / ldt] : 0.0;
}

void kry_diag(int n_sub, double *T, int ldt, const double *mu, int ldm, int k, cudaStream_t s) {
    k_kry_diag<<<n_sub, 256, 0, s>>>(T, ldt, mu, ldm, k);
    GL_CUDA(cudaGetLastError());
}

// ---------------------------------------------------------------- scaling, random

__global__ void k_scale_rows(const int64_t *__restrict__ voff, const int64_t *__restrict__ vlen, double *__restrict__ X,
                             const double *__restrict__ xi, int k) {
    const int s = blockIdx.x;
    const int64_t n = vlen[s], base = voff[s] * k;
    for (int64_t i = (int64_t)blockIdx.y * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.y * blockDim.x) {
        double w = xi[voff[s] + i];
        for (int a = 0; a < k; ++a) X[base + a * n + i] *= w;
    }
}

void scale_rows(const FactorPlan &P, double *X, const double *xi, int k, cudaStream_t s) {
    k_scale_rows<<<dim3(P.n_sub, 64), 256, 0, s>>>(P.d_vec_off.p, P.d_vec_len.p, X, xi, k);
    GL_CUDA(cudaGetLastError());
}

__global__ void k_fill_random(double *x, int64_t n, uint64_t seed) {
    int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i < n) x[i] = hash_uniform(seed, i);
}

void fill_random(double *x, int64_t n, uint64_t seed, cudaStream_t s) {
    if (!n) return;
    k_fill_random<<<(unsigned)((n + 255) / 256), 256, 0, s>>>(x, n, seed);
    GL_CUDA(cudaGetLastError());
}

// ---------------------------------------------------------------- coarse restrict / prolong

// c = Z^T r: a CTA gathers its chunk of r once, its warps take the columns of Z
// in turn (contiguous reads, one FMA an entry).  Bound by reading Z; with the
// column sums of all m columns in one thread (local memory) it took 157 us a
// launch on the batch of five plates.
constexpr int RESTRICT_ROWS = 256;

__global__ void __launch_bounds__(256) k_coarse_restrict(const int64_t *__restrict__ voff, const int64_t *__restrict__ vlen,
                                                         const int64_t *__restrict__ gdof, const double *__restrict__ Z,
                                                         int m, const double *__restrict__ r, double *__restrict__ c) {
    const int s = blockIdx.x;
    const int64_t n = vlen[s], r0 = (int64_t)blockIdx.y * RESTRICT_ROWS;
    if (r0 >= n) return;
    const int rows = (int)min((int64_t)RESTRICT_ROWS, n - r0);
    __shared__ double sr[RESTRICT_ROWS];
    const int64_t *gd = gdof + voff[s] + r0;
    for (int i = threadIdx.x; i < RESTRICT_ROWS; i += 256) sr[i] = i < rows ? r[gd[i]] : 0.0;
    __syncthreads();
    const int lane = threadIdx.x & 31;
    for (int a = threadIdx.x >> 5; a < m; a += 8) {
        const double *Za = Z + voff[s] * m + (int64_t)a * n + r0;
        double v0 = 0.0, v1 = 0.0;
#pragma unroll 8
        for (int i = lane; i < RESTRICT_ROWS; i += 64) {
            v0 += (i < rows ? Za[i] : 0.0) * sr[i];
            v1 += (i + 32 < rows ? Za[i + 32] : 0.0) * sr[i + 32];
        }
        double v = v0 + v1;
        for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
        if (lane == 0) atomicAdd(c + (int64_t)s * m + a, v);
    }
}

void coarse_restrict(const FactorPlan &P, const double *Z, int m, const double *r, double *c, cudaStream_t s) {
    GL_CUDA(cudaMemsetAsync(c, 0, sizeof(double) * P.n_sub * m, s));
    k_coarse_restrict<<<dim3(P.n_sub, row_chunks(P, RESTRICT_ROWS)), 256, 0, s>>>(P.d_vec_off.p, P.d_vec_len.p,
                                                                                 P.d_gdof.p, Z, m, r, c);
    GL_CUDA(cudaGetLastError());
}

__global__ void k_coarse_prolong(const int64_t *__restrict__ voff, const int64_t *__restrict__ vlen,
                                 const int64_t *__restrict__ gdof, const double *__restrict__ Z, int m,
                                 const double *__restrict__ y, double *__restrict__ z) {
    const int s = blockIdx.x;
    const int64_t n = vlen[s], base = voff[s] * m;
    const int64_t *gd = gdof + voff[s];
    __shared__ double sy[NV_MAX];
    if (threadIdx.x < m) sy[threadIdx.x] = y[(int64_t)s * m + threadIdx.x];
    __syncthreads();
    for (int64_t i = (int64_t)blockIdx.y * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.y * blockDim.x) {
        double v = 0.0;
#pragma unroll 4
        for (int a = 0; a < m; ++a) v += Z[base + a * n + i] * sy[a];
        atomicAdd(z + gd[i], v);
    }
}

void coarse_prolong(const FactorPlan &P, const double *Z, int m, const double *y, double *z, cudaStream_t s) {
    k_coarse_prolong<<<dim3(P.n_sub, 32), 256, 0, s>>>(P.d_vec_off.p, P.d_vec_len.p, P.d_gdof.p, Z, m, y, z);
    GL_CUDA(cudaGetLastError());
}

// ---------------------------------------------------------------- PCG vector kernels

__device__ __forceinline__ double block_sum(double v) {
    __shared__ double red[32];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    __syncthreads();
    if (lane == 0) red[w] = v;
    __syncthreads();
    double t = 0.0;
    if (w == 0) {
        t = lane < (int)(blockDim.x >> 5) ? red[lane] : 0.0;
        for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
    }
    return t;
}

// Blocks of a reduction over n entries: four a thread at least.  (1,024 blocks
// whatever n took 8.7 us on 20k entries, most of it their 8,192 divisions.)
static int red_blocks(int64_t n) { return (int)std::min<int64_t>(RED_BLOCKS, std::max<int64_t>(1, (n + 1023) / 1024)); }

// Sum over the grid of the blocks' v: the block that finishes last adds the
// partial sums in block order and returns true with the total in its thread 0
// -- a second launch for it cost 3 us and a gap.
__device__ __forceinline__ bool grid_sum(double v, double *partials, double &total) {
    __shared__ bool last;
    unsigned int *done = reinterpret_cast<unsigned int *>(partials + RED_BLOCKS);
    v = block_sum(v);
    if (threadIdx.x == 0) {
        partials[blockIdx.x] = v;
        __threadfence();
        last = atomicAdd(done, 1u) == gridDim.x - 1;
    }
    __syncthreads();
    if (!last) return false;
    __threadfence();
    double t = 0.0;
    for (int i = threadIdx.x; i < gridDim.x; i += blockDim.x) t += __ldcg(partials + i);
    total = block_sum(t);
    if (threadIdx.x == 0) *done = 0u;
    return true;
}

__global__ void __launch_bounds__(256) k_dot(const double *__restrict__ a, const double *__restrict__ b, int64_t n,
                                             double *partials, double *__restrict__ out) {
    double v = 0.0, t;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
        v += a[i] * b[i];
    if (grid_sum(v, partials, t) && threadIdx.x == 0) *out = t;
}

void dot(const double *a, const double *b, int64_t n, double *partials, double *out, cudaStream_t s) {
    k_dot<<<red_blocks(n), 256, 0, s>>>(a, b, n, partials, out);
    GL_CUDA(cudaGetLastError());
}

__global__ void __launch_bounds__(256) k_update_xr(double *__restrict__ x, double *__restrict__ r,
                                                   const double *__restrict__ p, const double *__restrict__ q,
                                                   const uint8_t *__restrict__ mask, double *__restrict__ z, int64_t n,
                                                   CGScalars *__restrict__ S, double *partials) {
    __shared__ double sa;
    if (threadIdx.x == 0) sa = S->rho / S->pq;
    __syncthreads();
    const double alpha = sa;
    double v = 0.0, t;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        x[i] += alpha * p[i];
        const double ri = mask[i] ? 0.0 : r[i] - alpha * q[i];
        r[i] = ri;
        if (z) z[i] = 0.0;
        v += ri * ri;
    }
    if (grid_sum(v, partials, t) && threadIdx.x == 0) {
        S->rr = t;
        S->alpha = alpha;
    }
}

void cg_update_xr(double *x, double *r, const double *p, const double *q, const uint8_t *mask, double *z, int64_t n,
                  CGScalars *S, double *partials, cudaStream_t s) {
    k_update_xr<<<red_blocks(n), 256, 0, s>>>(x, r, p, q, mask, z, n, S, partials);
    GL_CUDA(cudaGetLastError());
}

// beta = (rho_new - rz_old) / rho  (rz_old = 0 gives the standard recurrence);
// the block that finishes last moves rho on
__global__ void __launch_bounds__(256) k_update_p(double *__restrict__ p, const double *__restrict__ z,
                                                  double *__restrict__ q, int64_t n, CGScalars *S, double *partials) {
    __shared__ double sb;
    __shared__ bool last;
    if (threadIdx.x == 0) sb = (S->rho_new - S->rz_old) / S->rho;
    __syncthreads();
    const double beta = sb;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        p[i] = z[i] + beta * p[i];
        q[i] = 0.0;
    }
    if (threadIdx.x == 0) {
        unsigned int *done = reinterpret_cast<unsigned int *>(partials + RED_BLOCKS);
        __threadfence();
        last = atomicAdd(done, 1u) == gridDim.x - 1;
        if (last) {
            S->beta = beta;
            S->rho = S->rho_new;
            *done = 0u;
        }
    }
}

void cg_update_p(double *p, const double *z, double *q, int64_t n, CGScalars *S, double *partials, cudaStream_t s) {
    k_update_p<<<red_blocks(n), 256, 0, s>>>(p, z, q, n, S, partials);
    GL_CUDA(cudaGetLastError());
}

// ---- per-part (segmented) versions for many laminates solved together

__global__ void __launch_bounds__(256) k_seg_dot(const double *__restrict__ a, const double *__restrict__ b,
                                                 const PartDesc *__restrict__ parts, double *__restrict__ partials) {
    const PartDesc pd = parts[blockIdx.x];
    double v = 0.0;
    for (int64_t i = (int64_t)blockIdx.y * blockDim.x + threadIdx.x; i < pd.n_dof; i += (int64_t)gridDim.y * blockDim.x)
        v += a[pd.dof_off + i] * b[pd.dof_off + i];
    v = block_sum(v);
    if (threadIdx.x == 0) partials[blockIdx.x * SEG_BLOCKS + blockIdx.y] = v;
}

__global__ void k_seg_final(const double *__restrict__ partials, double *__restrict__ out) {
    const int lane = threadIdx.x;   // 64 threads
    double v = partials[blockIdx.x * SEG_BLOCKS + lane];
    v += __shfl_xor_sync(0xffffffffu, v, 16);
    v += __shfl_xor_sync(0xffffffffu, v, 8);
    v += __shfl_xor_sync(0xffffffffu, v, 4);
    v += __shfl_xor_sync(0xffffffffu, v, 2);
    v += __shfl_xor_sync(0xffffffffu, v, 1);
    __shared__ double w[2];
    if ((lane & 31) == 0) w[lane >> 5] = v;
    __syncthreads();
    if (lane == 0) out[blockIdx.x] = w[0] + w[1];
}

void seg_dot(const double *a, const double *b, const PartDesc *parts, int n, double *partials, double *out,
             cudaStream_t s) {
    k_seg_dot<<<dim3(n, SEG_BLOCKS), 256, 0, s>>>(a, b, parts, partials);
    k_seg_final<<<n, SEG_BLOCKS, 0, s>>>(partials, out);
    GL_CUDA(cudaGetLastError());
}

__global__ void __launch_bounds__(256) k_seg_update_xr(double *__restrict__ x, double *__restrict__ r,
                                                       const double *__restrict__ p, const double *__restrict__ q,
                                                       const PartDesc *__restrict__ parts, SegScalars S,
                                                       double *__restrict__ partials) {
    const int ip = blockIdx.x;
    const PartDesc pd = parts[ip];
    const double alpha = S.active[ip] ? S.rho[ip] / S.pq[ip] : 0.0;
    double v = 0.0;
    for (int64_t i = (int64_t)blockIdx.y * blockDim.x + threadIdx.x; i < pd.n_dof; i += (int64_t)gridDim.y * blockDim.x) {
        const int64_t g = pd.dof_off + i;
        x[g] += alpha * p[g];
        const double ri = r[g] - alpha * q[g];
        r[g] = ri;
        v += ri * ri;
    }
    v = block_sum(v);
    if (threadIdx.x == 0) partials[ip * SEG_BLOCKS + blockIdx.y] = v;
}

void seg_update_xr(double *x, double *r, const double *p, const double *q, const PartDesc *parts, int n,
                   SegScalars S, double *partials, cudaStream_t s) {
    k_seg_update_xr<<<dim3(n, SEG_BLOCKS), 256, 0, s>>>(x, r, p, q, parts, S, partials);
    k_seg_final<<<n, SEG_BLOCKS, 0, s>>>(partials, S.rr);
    GL_CUDA(cudaGetLastError());
}

__global__ void __launch_bounds__(256) k_seg_update_p(double *__restrict__ p, const double *__restrict__ z,
                                                      const PartDesc *__restrict__ parts, SegScalars S) {
    const int ip = blockIdx.x;
    const PartDesc pd = parts[ip];
    const double rho = S.rho[ip];
    const double beta = rho != 0.0 ? (S.rho_new[ip] - S.rz_old[ip]) / rho : 0.0;
    for (int64_t i = (int64_t)blockIdx.y * blockDim.x + threadIdx.x; i < pd.n_dof; i += (int64_t)gridDim.y * blockDim.x) {
        const int64_t g = pd.dof_off + i;
        p[g] = z[g] + beta * p[g];
    }
}

__global__ void k_seg_rho(SegScalars S, int n) {
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) S.rho[i] = S.rho_new[i];
}

void seg_update_p(double *p, const double *z, const PartDesc *parts, int n, SegScalars S, cudaStream_t s) {
    k_seg_update_p<<<dim3(n, SEG_BLOCKS), 256, 0, s>>>(p, z, parts, S);
    k_seg_rho<<<(n + 127) / 128, 128, 0, s>>>(S, n);
    GL_CUDA(cudaGetLastError());
}

__global__ void k_seg_check(SegScalars S, int n, double tol2, int max_iter, int *n_active) {
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n || !S.active[i]) return;
    const int it = ++S.iters[i];
    const double rr = S.rr[i];
    int a = 1;
    if (!(rr > tol2 * S.ff[i]) || it >= max_iter) a = 0;   // converged, stalled at max_iter, or NaN
    S.active[i] = a;
    if (a) atomicAdd(n_active, 1);
}

void seg_check(SegScalars S, int n, double tol, int max_iter, int *n_active, cudaStream_t s) {
    GL_CUDA(cudaMemsetAsync(n_active, 0, sizeof(int), s));
    k_seg_check<<<(n + 127) / 128, 128, 0, s>>>(S, n, tol * tol, max_iter, n_active);
    GL_CUDA(cudaGetLastError());
}

__global__ void k_seg_confirm(SegScalars S, int n, double tol2, int max_iter, int *n_active) {
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n || S.active[i] || !(S.ff[i] > 0.0) || S.iters[i] >= max_iter) return;
    const double rr = S.rr[i];
    if (rr > tol2 * S.ff[i] && rr < INFINITY) {
        S.active[i] = 1;
        atomicAdd(n_active, 1);
    }
}

void seg_confirm(SegScalars S, int n, double tol, int max_iter, int *n_active, cudaStream_t s) {
    GL_CUDA(cudaMemsetAsync(n_active, 0, sizeof(int), s));
    k_seg_confirm<<<(n + 127) / 128, 128, 0, s>>>(S, n, tol * tol, max_iter, n_active);
    GL_CUDA(cudaGetLastError());
}

__global__ void k_set_entries(double *__restrict__ y, const int64_t *__restrict__ dof, int64_t n,
                              const double *__restrict__ vals) {
    int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i < n) y[dof[i]] = vals ? vals[i] : 0.0;
}

void set_entries(double *y, const int64_t *dof, int64_t n, const double *vals, cudaStream_t s) {
    if (!n) return;
    k_set_entries<<<(unsigned)((n + 255) / 256), 256, 0, s>>>(y, dof, n, vals);
    GL_CUDA(cudaGetLastError());
}

__global__ void k_sub(double *__restrict__ y, const double *__restrict__ a, const double *__restrict__ b, int64_t n) {
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
        y[i] = a[i] - b[i];
}

void sub(double *y, const double *a, const double *b, int64_t n, cudaStream_t s) {
    k_sub<<<RED_BLOCKS, 256, 0, s>>>(y, a, b, n);
    GL_CUDA(cudaGetLastError());
}

__global__ void k_axpy(double *__restrict__ y, double a, const double *__restrict__ x, int64_t n) {
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
        y[i] += a * x[i];
}

void axpy(double *y, double a, const double *x, int64_t n, cudaStream_t s) {
    k_axpy<<<RED_BLOCKS, 256, 0, s>>>(y, a, x, n);
    GL_CUDA(cudaGetLastError());
}

// The largest v over the masked entries (-1e300 if there are none), in two
// stages: one block took 26 us at 47,104 entries.
__global__ void __launch_bounds__(256) k_max_where(const double *__restrict__ v, const uint8_t *__restrict__ mask,
                                                   int64_t n, double *__restrict__ out) {
    __shared__ double red[256];
    double m = -1e300;
    for (int64_t i = (int64_t)blockIdx.x * 256 + threadIdx.x; i < n; i += (int64_t)gridDim.x * 256)
        if (!mask || mask[i]) m = fmax(m, v[i]);
    red[threadIdx.x] = m;
    __syncthreads();
    for (int o = 128; o > 0; o >>= 1) {
        if (threadIdx.x < o) red[threadIdx.x] = fmax(red[threadIdx.x], red[threadIdx.x + o]);
        __syncthreads();
    }
    if (threadIdx.x == 0) out[blockIdx.x] = red[0];
}

void max_where(const double *v, const uint8_t *mask, int64_t n, double *partials, double *out, cudaStream_t s) {
    const int nb = (int)std::min<int64_t>(RED_BLOCKS, std::max<int64_t>(1, (n + 1023) / 1024));
    k_max_where<<<nb, 256, 0, s>>>(v, mask, n, partials);
    k_max_where<<<1, 256, 0, s>>>(partials, nullptr, nb, out);
    GL_CUDA(cudaGetLastError());
}

}  // namespace gl
