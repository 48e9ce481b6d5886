// FP64 products of the supernodal fronts on the 5th-generation tensor cores
// (tcgen05, FP16 operands, FP32 accumulation in tensor memory).
//
// Section 2.3 solves the overlapping subdomain problems with direct local
// factorisations.  Two products hold nearly all their flops: the trailing
// update of a front's partial Cholesky, F[r, c] -= sum_k P[r, k] P[c, k], and
// W = L21 L11^{-1} of the inverse-form panels.  The FP64 pipe of this part does
// two FMAs per clock and SM, its tensor cores some 3,500 in FP16, so a product
// is formed there from integer slices (the error-free splitting of Ozaki,
// Ogita, Oishi and Rump, Numer. Algorithms 59, 2012, on fixed-point rows):
//   * a row's entries over the summed range are scaled by a power of two to
//     fixed point, 62 bits below the row's largest exponent (entries down to
//     2^-9 of the largest keep all FP64 bits, smaller ones what lies above
//     2^-62 of it);
//   * the fixed-point number is cut into eight signed base-256 digits, each in
//     [-128, 127] and exact in FP16;
//   * the digit products of equal weight i + j = s <= 7 are summed over k <= 128
//     in one FP32 accumulator: an integer of at most 8 x 128 x 2^14 = 2^24, so
//     every addition is exact; the weights s >= 8 (28 of the 64 digit products)
//     are left out: at most 2^-57 of the product of the two rows' largest
//     entries per column, 2^-50 over 128 columns;
//   * the eight sums are put together in two 64-bit integers, converted to
//     FP64 without loss and added to the result by two FMAs.
//
// The inverse of the pivot block (k_trinv_tc) and the eigensolver's sweeps with
// eight vectors (k_fwd_tc, k_bwd_tc) are formed the same way.
//
// One CTA of 256 threads forms a 128 x 32 tile: a thread stages the digits of
// eight columns of a row at a time (K-major core matrices of 8 rows x 16 bytes,
// no swizzle), 32 columns per round.  The eight accumulators take 256 columns
// of tensor memory, so two CTAs share an SM and each works while the other
// waits for its loads or its products.  Every wait is bounded: if a commit does
// not arrive within the limit the kernel raises the error flag, skips the
// write-back, frees its tensor memory and returns (the host reports
// GL_ERR_TIMEOUT).
//
// Measured on the 63k-DOF corner's set-up: trailing updates 50.6 ms on the FP64
// pipe, 13.2 ms here and 7.8 ms inside the panels; W 19.0 ms, 3.8 ms here.  What
// binds it now is the latency of its loads (two CTAs an SM; FP64 pipe 18% and
// tensor pipe 7% active).
//
// Accuracy: better than FP64 sums where the entries of a row are of one size,
// not so where two rows are large in different columns and their products small,
// since the error is relative to the rows' largest entries.  For the Cholesky
// that is the usual bound (a row of L is at most the root of the diagonal entry
// of A), not the entry by entry one.  Residuals of one-subdomain direct solves
// against the same program with FP64 FMAs: 0.75 to 1.0 on laminates and blocks of
// one material (50 to 17,000 DOF), 0.65 to 1.3 with random stiffnesses up to 1e4
// apart, up to 1.7 with a checkerboard 1e4 apart, 60 (2.7e-12 for 4.4e-14) with
// one 1e6 apart; W and L11^{-1} lose that, the trailing updates 0.83 to 1.15
// everywhere.  Solution errors are as large as with FMAs (0.8 to 1.5).  Taking
// the pivots' sizes out of the columns of L21 and the rows of L11^{-1} first (by
// the exponents) gave 44 instead of 60 and made first calls 2% slower; cutting the
// sums to 2^-54 of the largest entries' product instead of converting both halves
// made errors up to 100 times larger.
#include <cuda_fp16.h>

#include <algorithm>

#include "factor.h"

namespace gl {

namespace {

constexpr int OZ_M = 128, OZ_N = 32;        // output tile
constexpr int OZ_KC = 32;                   // summed columns staged per round (2 MMAs of K = 16)
constexpr int OZ_KB = 128;                  // summed columns per exact accumulation
constexpr int OZ_S = 8;                     // digits
constexpr int OZ_THREADS = 256;
constexpr int OZ_TMEM_COLS = OZ_S * OZ_N;   // 256: two CTAs per SM
constexpr int OZ_A_BYTES = OZ_M * OZ_KC * 2, OZ_B_BYTES = OZ_N * OZ_KC * 2;   // one digit of an operand tile
constexpr int OZ_BUF = OZ_S * (OZ_A_BYTES + OZ_B_BYTES);
constexpr int OZ_SMEM = OZ_BUF + 1024;      // + alignment slack
constexpr unsigned OZ_WAIT_LIMIT = 1u << 26;

// Byte offset of element (row m, column k): core matrices are 128 B apart
// along K (leading byte offset) and OZ_KC / 8 x 128 B along M (stride byte offset).
constexpr uint32_t OZ_LBO = 128, OZ_SBO = OZ_KC / 8 * 128;
__device__ __forceinline__ uint32_t oz_off(int m, int k8) {
    return (uint32_t)((m >> 3) * OZ_SBO + k8 * OZ_LBO + (m & 7) * 16);
}

__device__ __forceinline__ uint32_t oz_smem(const void *p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ uint64_t oz_desc(uint32_t addr) {
    return (uint64_t)((addr & 0x3FFFFu) >> 4) | ((uint64_t)(OZ_LBO >> 4) << 16) | ((uint64_t)(OZ_SBO >> 4) << 32) |
           (1ull << 46);
}

// Instruction descriptor of kind::f16: D FP32 (bits 4-5 = 1), A and B FP16 (0),
// both K-major, N >> 3 at bit 17, M >> 4 at bit 24.
constexpr uint32_t OZ_IDESC = (1u << 4) | ((uint32_t)(OZ_N >> 3) << 17) | ((uint32_t)(OZ_M >> 4) << 24);

__device__ __forceinline__ void oz_mma(uint32_t d_tmem, uint64_t a, uint64_t b, uint32_t accumulate,
                                       uint32_t idesc = OZ_IDESC) {
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "setp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}\n" ::"r"(d_tmem),
        "l"(a), "l"(b), "r"(idesc), "r"(accumulate));
}

__device__ __forceinline__ bool oz_wait(uint32_t mbar, uint32_t parity) {
    for (unsigned it = 0; it < OZ_WAIT_LIMIT; ++it) {
        uint32_t done;
        asm volatile(
            "{\n\t.reg .pred P1;\n\t"
            "mbarrier.try_wait.parity.shared::cta.b64 P1, [%1], %2;\n\t"
            "selp.b32 %0, 1, 0, P1;\n\t}\n"
            : "=r"(done)
            : "r"(mbar), "r"(parity)
            : "memory");
        if (done) return true;
    }
    return false;
}

// 8 accumulator columns of this warp's 32 lanes (no wait).
__device__ __forceinline__ void oz_tmem_ld8(uint32_t taddr, uint32_t r[8]) {
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
                 : "r"(taddr));
}

__device__ __forceinline__ void oz_tmem_ld4(uint32_t taddr, uint32_t r[4]) {
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0,%1,%2,%3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
                 : "r"(taddr));
}

// x in fixed point, 2^62 at twice the largest power of two of its row (biased
// exponent e of the row), with 128 added to every base-256 digit.
__device__ __forceinline__ uint64_t oz_fixed(double x, int e) {
    const uint64_t b = (uint64_t)__double_as_longlong(x);
    const int ex = (int)(b >> 52) & 0x7FF;
    int64_t m = (int64_t)((b & 0xFFFFFFFFFFFFFull) | 0x10000000000000ull);
    m = (b >> 63) ? -m : m;
    const int sh = e - ex;                      // >= 0
    int64_t q = m << 9;
    if (sh > 0) q = sh < 63 ? (q + (1ll << (sh - 1))) >> sh : 0;   // to nearest
    if (ex == 0) q = 0;
    return (uint64_t)q + 0x8080808080808080ull;
}

// Digits of eight consecutive summed columns of one row: 16 bytes per digit
// into the digit's tile at `at` (tiles `stride` bytes apart).
__device__ __forceinline__ void oz_stage8(const uint64_t u[8], unsigned char *at, int stride) {
    const __half2 off = __floats2half2_rn(1152.0f, 1152.0f);   // 1024 + 128
#pragma unroll
    for (int i = 0; i < OZ_S; ++i) {
        const int byte = 7 - i, bsel = byte & 3;
        uint32_t w[4];
#pragma unroll
        for (int h = 0; h < 4; ++h) {
            const uint32_t a = (uint32_t)(byte >= 4 ? u[2 * h] >> 32 : u[2 * h]);
            const uint32_t b = (uint32_t)(byte >= 4 ? u[2 * h + 1] >> 32 : u[2 * h + 1]);
            // the digit's bytes as the low bits of 0x64xx = 1024 + byte in FP16
            const uint32_t t = (__byte_perm(a, b, (uint32_t)(bsel | ((4 + bsel) << 8))) & 0x00FF00FFu) | 0x64006400u;
            __half2 v;
            memcpy(&v, &t, 4);
            v = __hsub2(v, off);
            memcpy(&w[h], &v, 4);
        }
        *reinterpret_cast<uint4 *>(at + i * stride) = make_uint4(w[0], w[1], w[2], w[3]);
    }
}

struct OzShared {
    int ea[OZ_M], eb[OZ_N];       // largest biased exponent of each row over the summed range
    uint32_t tmem;
    __align__(8) uint64_t mbar;
    int failed;
};

// Sums over k in [k0, k1) (at most OZ_KB) of A(i, k) B(j, k) for the tile: this
// thread's row 32 (warp % 4) + lane and columns 16 (warp / 4) + c through
// put(c, hi, lo, x): the sum is (hi 2^32 + lo) 2^x (x OZ_NONE: zero, OZ_NOT: not
// a number).
// PART: rows from `used` on (whole warps of them) are left out; a row of the
// result needs no other row of A.  (Always testing it cost the trailing updates
// 15%.)  A and B return 0 out of range; before_wait() runs while the products are
// still being formed.  Returns false if a wait gave up.
constexpr int OZ_NONE = -100000, OZ_NOT = 100000;

template <bool PART, class FA, class FB, class Pre, class Put>
__device__ bool oz_block(OzShared &S, unsigned char *sm, uint32_t &phase, int used, FA A, FB B, int k0, int k1,
                         Pre before_wait, Put put) {
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
    const int ra = t & (OZ_M - 1), ha = t >> 7;      // A: two threads per row, 16 columns each
    const bool live = !PART || (ra & ~31) < used;
    const int rb = t & (OZ_N - 1), hb = t >> 5;      // B: four threads per row, 8 columns each (warps 0-3)
    if (t < OZ_M) S.ea[t] = 0;
    if (t < OZ_N) S.eb[t] = 0;
    __syncthreads();
    {
        int ma = 0, mb = 0;
#pragma unroll 2
        for (int kc = k0; kc < k1; kc += OZ_KC) {
#pragma unroll
            for (int j = 0; j < 16; ++j)
                if (live) ma = max(ma, (int)((uint64_t)__double_as_longlong(A(ra, kc + 16 * ha + j)) >> 52) & 0x7FF);
            if (warp < 4)
#pragma unroll
                for (int j = 0; j < 8; ++j)
                    mb = max(mb, (int)((uint64_t)__double_as_longlong(B(rb, kc + 8 * hb + j)) >> 52) & 0x7FF);
        }
        atomicMax(&S.ea[ra], ma);
        if (warp < 4) atomicMax(&S.eb[rb], mb);
    }
    __syncthreads();
    const int ea = S.ea[ra], eb = S.eb[rb];
    unsigned char *pa = sm, *pb = sm + OZ_S * OZ_A_BYTES;
    for (int kc = k0; kc < k1; kc += OZ_KC) {
        if (kc > k0) {              // until the tensor cores have read the last round's digits
            if (!oz_wait(oz_smem(&S.mbar), phase)) S.failed = 1;
            phase ^= 1u;
            __syncthreads();
            if (S.failed) break;
        }
#pragma unroll
        for (int g = 0; g < 2; ++g) {
            if (!live) break;
            uint64_t u[8];
#pragma unroll
            for (int j = 0; j < 8; ++j) u[j] = oz_fixed(A(ra, kc + 16 * ha + 8 * g + j), ea);
            oz_stage8(u, pa + oz_off(ra, 2 * ha + g), OZ_A_BYTES);
        }
        if (warp < 4) {
            uint64_t u[8];
#pragma unroll
            for (int j = 0; j < 8; ++j) u[j] = oz_fixed(B(rb, kc + 8 * hb + j), eb);
            oz_stage8(u, pb + oz_off(rb, hb), OZ_B_BYTES);
        }
        // generic-proxy stores -> visible to the tensor cores (async proxy)
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        __syncthreads();
        if (t == 0) {
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            const uint32_t a0 = oz_smem(pa), b0 = oz_smem(pb);
#pragma unroll 1
            for (int s = 0; s < OZ_KC / 16; ++s) {
                const uint32_t ko = (uint32_t)(2 * s) * OZ_LBO;    // K = 16 halves = two core matrices
#pragma unroll 1
                for (int i = 0; i < OZ_S; ++i)
#pragma unroll 1
                    for (int j = 0; i + j < OZ_S; ++j)
                        oz_mma(S.tmem + OZ_N * (i + j), oz_desc(a0 + i * OZ_A_BYTES + ko),
                               oz_desc(b0 + j * OZ_B_BYTES + ko), kc > k0 || s > 0 || i > 0 ? 1u : 0u);
            }
            asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(
                             oz_smem(&S.mbar))
                         : "memory");
        }
    }
    before_wait();
    if (!S.failed) {
        if (!oz_wait(oz_smem(&S.mbar), phase)) S.failed = 1;
        phase ^= 1u;
    }
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    __syncthreads();
    if (S.failed) return false;
    // a = q_a 2^(ea - 1084), ea biased by 1023; q_a q_b = 2^56 (hi 2^32 + lo), |hi|, |lo| < 2^50
    const int er = S.ea[32 * (warp & 3) + lane];
    const int col0 = 16 * (warp >> 2);
    const uint32_t tm = S.tmem + ((uint32_t)(32 * (warp & 3)) << 16) + (uint32_t)col0;
#pragma unroll
    for (int cb = 0; cb < 16; cb += 8) {
        if (PART && 32 * (warp & 3) >= used) break;
        uint32_t r[OZ_S][8];
#pragma unroll
        for (int s = 0; s < OZ_S; ++s) oz_tmem_ld8(tm + OZ_N * s + cb, r[s]);
        asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
        for (int j = 0; j < 8; ++j) {
            int64_t hi = 0, lo = 0;
#pragma unroll
            for (int s = 0; s < 4; ++s) {
                hi = (hi << 8) + __float2int_rn(__uint_as_float(r[s][j]));
                lo = (lo << 8) + __float2int_rn(__uint_as_float(r[s + 4][j]));
            }
            const int ec = S.eb[col0 + cb + j];
            const int x = er == 0x7FF || ec == 0x7FF ? OZ_NOT : (er == 0 || ec == 0 ? OZ_NONE : er + ec - 2112);
            put(cb + j, hi, lo, x);
        }
    }
    // the next block's products overwrite the accumulators
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    return true;
}

// 2^x as oz_block gives it: 0 below the normal numbers, NaN for OZ_NOT.
__device__ __forceinline__ double oz_pow2(int x) {
    if (x >= OZ_NOT) return __longlong_as_double(0x7FF8000000000000ll);
    return x > -1023 ? __longlong_as_double((int64_t)(min(x, 1023) + 1023) << 52) : 0.0;
}

template <int COLS, class Sh>
__device__ __forceinline__ unsigned char *oz_begin(Sh &S, unsigned char *raw) {
    if (threadIdx.x < 32) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(oz_smem(&S.tmem)),
                     "r"(COLS));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
    }
    if (threadIdx.x == 0) {
        S.failed = 0;
        asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(oz_smem(&S.mbar)), "r"(1));
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    return reinterpret_cast<unsigned char *>((reinterpret_cast<uintptr_t>(raw) + 1023) & ~static_cast<uintptr_t>(1023));
}

template <int COLS, class Sh>
__device__ __forceinline__ void oz_end(Sh &S, bool ok, int *err) {
    if (!ok && threadIdx.x == 0) atomicExch(err, 2);
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    if (threadIdx.x < 32) {
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(S.tmem), "r"(COLS));
    }
}

// F[r, c] -= sum over the kw = min(panel, p - k0) columns k from k0 of
// F[r, k] F[c, k], k0 + kw <= c <= r < f: one CTA per (front, tile that meets
// the lower triangle).
__global__ void __launch_bounds__(OZ_THREADS, 2) k_syrk64_tc(const int *__restrict__ fronts,
                                                             const FrontDesc *__restrict__ D, double *ws, int k0,
                                                             int panel, int *__restrict__ err) {
    const FrontDesc &d = D[fronts[blockIdx.x]];
    const int p = d.p, f = d.p + d.q;
    if (k0 >= p) return;
    const int base = min(k0 + panel, p), m = f - base;
    constexpr int R = OZ_M / OZ_N;                            // tile columns per tile row: R (ti + 1) in row ti
    const int t = blockIdx.y;
    int ti = (int)((sqrtf(8.0f / R * t + 1.0f) - 1.0f) * 0.5f);
    while (R * (ti + 1) * (ti + 2) / 2 <= t) ++ti;
    while (R * ti * (ti + 1) / 2 > t) --ti;
    const int tj = t - R * ti * (ti + 1) / 2;
    if (ti * OZ_M >= m || tj * OZ_N >= m) return;
    const int r0 = base + ti * OZ_M, c0 = base + tj * OZ_N;
    double *F = ws + d.front_off;
    extern __shared__ unsigned char oz_raw[];
    __shared__ OzShared S;
    unsigned char *sm = oz_begin<OZ_TMEM_COLS>(S, oz_raw);
    uint32_t phase = 0u;
    const int r = r0 + 32 * ((threadIdx.x >> 5) & 3) + (threadIdx.x & 31), cw = c0 + 16 * (threadIdx.x >> 7);
    double e[16];   // the thread's entries of F, loaded while the products are formed
    const bool ok = oz_block<false>(
        S, sm, phase, OZ_M, [&](int i, int k) { return r0 + i < f && k < base ? F[r0 + i + (int64_t)k * f] : 0.0; },
        [&](int i, int k) { return c0 + i < f && k < base ? F[c0 + i + (int64_t)k * f] : 0.0; }, k0, base,
        [&]() {
#pragma unroll
            for (int c = 0; c < 16; ++c) e[c] = r < f && cw + c <= r ? F[r + (int64_t)(cw + c) * f] : 0.0;
        },
        [&](int c, int64_t hi, int64_t lo, int x) {
            if (r < f && cw + c <= r)
                F[r + (int64_t)(cw + c) * f] = fma((double)hi, -oz_pow2(x + 32), fma((double)lo, -oz_pow2(x), e[c]));
        });
    oz_end<OZ_TMEM_COLS>(S, ok, err);
}

// W = L21 L11^{-1}: rows p .. f of the panel, from L21 in the front and the
// inverse in the panel's pivot rows; tile column c0 needs the pivots from c0 on.
__global__ void __launch_bounds__(OZ_THREADS, 2) k_wpanel_tc(const int *__restrict__ fronts,
                                                             const FrontDesc *__restrict__ D, const double *ws,
                                                             double *out, int *__restrict__ err) {
    const FrontDesc &d = D[fronts[blockIdx.x]];
    const int p = d.p, f = d.p + d.q;
    const int ntr = (d.q + OZ_M - 1) / OZ_M;
    if (ntr == 0) return;
    const int ti = blockIdx.y % ntr, tj = blockIdx.y / ntr;
    const int r0 = p + ti * OZ_M, c0 = tj * OZ_N;
    if (c0 >= p) return;
    const double *F = ws + d.front_off;
    double *O = out + d.l_off;
    extern __shared__ unsigned char oz_raw[];
    __shared__ OzShared S;
    unsigned char *sm = oz_begin<OZ_TMEM_COLS>(S, oz_raw);
    uint32_t phase = 0u;
    const int r = r0 + 32 * ((threadIdx.x >> 5) & 3) + (threadIdx.x & 31), cw = c0 + 16 * (threadIdx.x >> 7);
    double acc[16];
#pragma unroll
    for (int j = 0; j < 16; ++j) acc[j] = 0.0;
    bool ok = true;
    for (int kb = c0; kb < p && ok; kb += OZ_KB) {
        const int ke = min(p, kb + OZ_KB);
        ok = oz_block<false>(
            S, sm, phase, OZ_M, [&](int i, int k) { return r0 + i < f && k < ke ? F[r0 + i + (int64_t)k * f] : 0.0; },
            [&](int i, int k) { return c0 + i < p && k < ke ? O[k + (int64_t)(c0 + i) * f] : 0.0; }, kb, ke, []() {},
            [&](int c, int64_t hi, int64_t lo, int x) {
                acc[c] = fma((double)hi, oz_pow2(x + 32), fma((double)lo, oz_pow2(x), acc[c]));
            });
    }
    if (ok && r < f) {
#pragma unroll
        for (int j = 0; j < 16; ++j)
            if (cw + j < p) O[r + (int64_t)(cw + j) * f] = acc[j];
    }
    oz_end<OZ_TMEM_COLS>(S, ok, err);
}

// L11^{-1} from its inverted 32 x 32 diagonal blocks by doubling: with the
// inverses X11, X22 of two neighbouring blocks of b pivots in place, the block
// below the diagonal is X21 = -X22 (L21 X11).  STEP 0 forms the bracket, kept
// transposed in the front's unused upper triangle, STEP 1 the product; one CTA
// per (front, pair, 128 x 32 tile), two launches per doubling.  Block column by
// block column in one CTA each, the FP64 pipe of one SM held a chain of up to
// (p / 32)^2 / 2 block products: 443 us a level on the 63k-DOF corner, 294 us
// in this form (about six launches), which the latency of a tile binds.
template <int STEP>
__global__ void __launch_bounds__(OZ_THREADS, 2) k_trinv_tc(const int *__restrict__ fronts,
                                                            const FrontDesc *__restrict__ D, double *ws, double *out,
                                                            int b, int *__restrict__ err) {
    const FrontDesc &d = D[fronts[blockIdx.x]];
    const int p = d.p, f = d.p + d.q;
    const int ct = b / OZ_N, tiles = ct * ((b + OZ_M - 1) / OZ_M), pair = blockIdx.y / tiles, t = blockIdx.y % tiles;
    const int base = 2 * b * pair, mid = base + b, end = min(p, mid + b);
    const int r0 = mid + OZ_M * (t / ct), c0 = base + OZ_N * (t % ct);
    if (r0 >= end) return;
    double *F = ws + d.front_off, *O = out + d.l_off;
    extern __shared__ unsigned char oz_raw[];
    __shared__ OzShared S;
    unsigned char *sm = oz_begin<OZ_TMEM_COLS>(S, oz_raw);
    uint32_t phase = 0u;
    const int r = r0 + 32 * ((threadIdx.x >> 5) & 3) + (threadIdx.x & 31), cw = c0 + 16 * (threadIdx.x >> 7);
    double acc[16];
#pragma unroll
    for (int j = 0; j < 16; ++j) acc[j] = 0.0;
    bool ok = true;
    // summed pivots: block 1 from the tile's columns on, block 2 up to the tile's rows
    const int k0 = STEP == 0 ? c0 : mid, k1 = STEP == 0 ? mid : min(end, r0 + OZ_M);
    for (int kb = k0; kb < k1 && ok; kb += OZ_KB) {
        const int ke = min(k1, kb + OZ_KB);
        ok = oz_block<true>(
            S, sm, phase, end - r0,
            [&](int i, int k) {
                if (r0 + i >= end || k >= ke) return 0.0;
                if (STEP == 0) return F[r0 + i + (int64_t)k * f];
                return k <= r0 + i ? O[r0 + i + (int64_t)k * f] : 0.0;
            },
            [&](int i, int k) {
                if (k >= ke) return 0.0;
                if (STEP == 0) return k >= c0 + i ? O[k + (int64_t)(c0 + i) * f] : 0.0;
                return F[c0 + i + (int64_t)k * f];
            },
            kb, ke, []() {},
            [&](int c, int64_t hi, int64_t lo, int x) {
                acc[c] = fma((double)hi, oz_pow2(x + 32), fma((double)lo, oz_pow2(x), acc[c]));
            });
    }
    if (ok && r < end) {
        double *up = (STEP == 0 ? F : O) + (int64_t)r * f;      // the mirror entries: the bracket; zeros
#pragma unroll
        for (int j = 0; j < 16; ++j) {
            up[cw + j] = STEP == 0 ? acc[j] : 0.0;
            if (STEP == 1) O[r + (int64_t)(cw + j) * f] = -acc[j];
        }
    }
    oz_end<OZ_TMEM_COLS>(S, ok, err);
}

// ---------------------------------------------------------------- sweeps with eight right-hand sides

// The panel times OZ_V vectors: the digits of the vectors are the columns of
// one operand (row 8 j + v: digit j of vector v), so that digit i of the panel
// times its digit groups, added 8 i columns further in tensor memory, collects
// every weight i + j <= 7 of a vector in one column.  (The columns of D and N
// stay multiples of 16: odd digits have accumulators of their own.)  A CTA takes
// 128 panel rows (forward) or columns (backward) and a chunk of the summed ones,
// 64 at a time, held in registers while their largest exponents are found.
// With eight accumulators a lane on the FP64 pipe (8 of its FMAs an entry, 512
// pipe clocks a warp and 32 entries) a launch took 138 us forward and 131 us
// backward on the 63k-DOF corner's eigensolver, this form 73 and 94 us, about
// 50 integer instructions an entry for its digits, which now bind it together
// with reading the panel; backward its 64-byte lane stride costs the rest.  The
// small levels gain too (20k-DOF plate: 42 to 23 and 44 to 27 us), so there is
// no second form.
constexpr int OZ_V = 8;
constexpr int OZ_VK = 64;                   // summed entries held in registers per accumulation
constexpr int OZ_MV_CTAS = 152 * 16;        // wanted per level (4 and 8 an SM: 3% and 2% slower over a sweep)
constexpr int OZ_MV_COLS = 128;             // of tensor memory
constexpr int OZ_MV_SMEM = OZ_S * OZ_A_BYTES + OZ_S * OZ_V * OZ_KC * 2 + 1024;

struct OzMvShared {
    int ea[2][OZ_M], eb[2][OZ_V];           // largest exponents, alternating between accumulations
    uint32_t tmem;
    __align__(8) uint64_t mbar;
    int failed;
};

// out[v] = sum over k in [k0, k1) of A(i, k) X(k, 4 (warp / 4) + v), v < 4, for
// row i = 32 (warp % 4) + lane of the tile.  unit(pass) = the (row, group of
// eight columns) this thread stages, 2 passes per round; rows from `used` on are
// left out.  A and X return 0 out of range.  Returns false if a wait gave up.
template <class FA, class FX, class Unit>
__device__ bool oz_mv(OzMvShared &S, unsigned char *sm, FA A, FX X, Unit unit, int used, int k0, int k1,
                      double out[4]) {
    constexpr int R = OZ_VK / OZ_KC;
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
    const int xv = lane & 7, xg = lane >> 3;          // warps 0 .. R-1, a round each: vector, group of eight
    int row[2], grp[2];
    unit(0, row[0], grp[0]);
    unit(1, row[1], grp[1]);
    double a[R][2][8], xr[8];
    auto load = [&](int kb) {
#pragma unroll
        for (int h = 0; h < R; ++h)
#pragma unroll
            for (int q = 0; q < 2; ++q)
#pragma unroll
                for (int j = 0; j < 8; ++j)
                    a[h][q][j] = row[q] < used ? A(row[q], kb + OZ_KC * h + 8 * grp[q] + j) : 0.0;
        if (warp < R)
#pragma unroll
            for (int j = 0; j < 8; ++j) xr[j] = X(kb + OZ_KC * warp + 8 * xg + j, xv);
    };
    auto expo = [](double x) { return (int)((uint64_t)__double_as_longlong(x) >> 52) & 0x7FF; };
#pragma unroll
    for (int j = 0; j < 4; ++j) out[j] = 0.0;
    for (int i = t; i < 2 * OZ_M; i += OZ_THREADS) S.ea[i / OZ_M][i % OZ_M] = 0;
    if (t < 2 * OZ_V) S.eb[t / OZ_V][t % OZ_V] = 0;
    load(k0);
    __syncthreads();
    unsigned char *pa = sm, *pb = sm + OZ_S * OZ_A_BYTES;
    uint32_t phase = 0u;
    int w = 0;
    for (int kb = k0; kb < k1; kb += OZ_VK, w ^= 1) {
#pragma unroll
        for (int q = 0; q < 2; ++q) {
            int e = 0;
#pragma unroll
            for (int h = 0; h < R; ++h)
#pragma unroll
                for (int j = 0; j < 8; ++j) e = max(e, expo(a[h][q][j]));
            if (e) atomicMax(&S.ea[w][row[q]], e);
        }
        if (warp < R) {
            int e = 0;
#pragma unroll
            for (int j = 0; j < 8; ++j) e = max(e, expo(xr[j]));
            if (e) atomicMax(&S.eb[w][xv], e);
        }
        __syncthreads();
        if (t < OZ_M) S.ea[w ^ 1][t] = 0;
        if (t < OZ_V) S.eb[w ^ 1][t] = 0;
#pragma unroll
        for (int h = 0; h < R; ++h) {
            if (kb + OZ_KC * h >= k1) break;
            if (h > 0) {            // until the tensor cores have read the last round's digits
                if (!oz_wait(oz_smem(&S.mbar), phase)) S.failed = 1;
                phase ^= 1u;
                __syncthreads();
                if (S.failed) return false;
            }
#pragma unroll
            for (int q = 0; q < 2; ++q)
                if (row[q] < used) {
                    const int e = S.ea[w][row[q]];
                    uint64_t u[8];
#pragma unroll
                    for (int j = 0; j < 8; ++j) u[j] = oz_fixed(a[h][q][j], e);
                    oz_stage8(u, pa + oz_off(row[q], grp[q]), OZ_A_BYTES);
                }
            if (warp == h) {
                const int e = S.eb[w][xv];
                uint64_t u[8];
#pragma unroll
                for (int j = 0; j < 8; ++j) u[j] = oz_fixed(xr[j], e);
                oz_stage8(u, pb + oz_off(xv, xg), OZ_SBO);
            }
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            __syncthreads();
            if (t == 0) {
                asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                const uint32_t a0 = oz_smem(pa), b0 = oz_smem(pb);
#pragma unroll 1
                for (int s = 0; s < OZ_KC / 16; ++s) {
                    const uint32_t ko = (uint32_t)(2 * s) * OZ_LBO;
#pragma unroll 1
                    for (int i = 0; i < OZ_S; ++i) {
                        // even digits into columns 0-63, odd ones, one weight lower, into 64-127
                        const int n = OZ_S * OZ_V - OZ_V * (i & ~1);
                        const uint32_t idesc = (1u << 4) | ((uint32_t)(n >> 3) << 17) | ((uint32_t)(OZ_M >> 4) << 24);
                        oz_mma(S.tmem + (i & 1) * OZ_S * OZ_V + OZ_V * (i & ~1), oz_desc(a0 + i * OZ_A_BYTES + ko),
                               oz_desc(b0 + ko), h > 0 || s > 0 || i > 1 ? 1u : 0u, idesc);
                    }
                }
                asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(
                                 oz_smem(&S.mbar))
                             : "memory");
            }
        }
        if (kb + OZ_VK < k1) load(kb + OZ_VK);
        if (!oz_wait(oz_smem(&S.mbar), phase)) S.failed = 1;
        phase ^= 1u;
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        __syncthreads();
        if (S.failed) return false;
        const int er = S.ea[w][32 * (warp & 3) + lane], v0 = 4 * (warp >> 2);
        const uint32_t tm = S.tmem + ((uint32_t)(32 * (warp & 3)) << 16) + (uint32_t)v0;
        int64_t hi[4] = {0, 0, 0, 0}, lo[4] = {0, 0, 0, 0};
#pragma unroll
        for (int s4 = 0; s4 < 2; ++s4) {
            uint32_t r[4][4], o[4][4];
#pragma unroll
            for (int s = 0; s < 4; ++s) {
                oz_tmem_ld4(tm + OZ_V * (4 * s4 + s), r[s]);
                if (s4 + s > 0) oz_tmem_ld4(tm + OZ_V * (OZ_S + 4 * s4 + s - 1), o[s]);
                else o[s][0] = o[s][1] = o[s][2] = o[s][3] = 0u;
            }
            asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
            for (int s = 0; s < 4; ++s)
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    int64_t &z = s4 ? lo[j] : hi[j];
                    z = (z << 8) + __float2int_rn(__uint_as_float(r[s][j])) + __float2int_rn(__uint_as_float(o[s][j]));
                }
        }
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const int ec = S.eb[w][v0 + j];
            const int x = er == 0x7FF || ec == 0x7FF ? OZ_NOT : (er == 0 || ec == 0 ? OZ_NONE : er + ec - 2112);
            out[j] = fma((double)hi[j], oz_pow2(x + 32), fma((double)lo[j], oz_pow2(x), out[j]));
        }
        asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");   // the next products overwrite them
    }
    return true;
}

// Forward step (k_fwd of the single sweep) with eight vectors: panel rows
// [128 blockIdx.y, ...), pivots [chunk blockIdx.z, ...).
__global__ void __launch_bounds__(OZ_THREADS, 2) k_fwd_tc(const int *__restrict__ fronts,
                                                          const FrontDesc *__restrict__ D,
                                                          const double *__restrict__ L, const int *__restrict__ rows,
                                                          double *b, double *y, int chunk, int *__restrict__ err) {
    const FrontDesc &d = D[fronts[blockIdx.x]];
    const int p = d.p, f = p + d.q, n = d.vlen;
    const int r0 = blockIdx.y * OZ_M, k0 = blockIdx.z * chunk;
    // pivot rows need the pivots up to their own tile, structure rows all
    const int k1 = min(k0 + chunk, r0 + OZ_M <= p ? r0 + OZ_M : p);
    if (r0 >= f || k0 >= k1) return;
    extern __shared__ unsigned char oz_raw[];
    __shared__ OzMvShared S;
    unsigned char *sm = oz_begin<OZ_MV_COLS>(S, oz_raw);
    const double *Lr = L + d.l_off + r0;
    const int64_t vo = d.vec_off * OZ_V;
    const double *b1 = b + vo + d.first;
    const int used = min(OZ_M, f - r0), t = threadIdx.x;
    double out[4];
    const bool ok = oz_mv(
        S, sm, [&](int i, int k) { return k < k1 && k <= r0 + i ? Lr[i + (int64_t)k * f] : 0.0; },
        [&](int k, int v) { return k < k1 ? b1[k + (int64_t)v * n] : 0.0; },
        [&](int pass, int &row, int &grp) {
            row = t & (OZ_M - 1);
            grp = (t >> 7) + 2 * pass;
        },
        used, k0, k1, out);
    const int i = 32 * ((t >> 5) & 3) + (t & 31), row = r0 + i, v0 = 4 * (t >> 7);
    if (ok && i < used) {
        double *o = row < p ? y + vo + d.first + row : b + vo + rows[d.row_off + row];
#pragma unroll
        for (int j = 0; j < 4; ++j) atomicAdd(o + (int64_t)(v0 + j) * n, row < p ? out[j] : -out[j]);
    }
    oz_end<OZ_MV_COLS>(S, ok, err);
}

// Backward step with eight vectors: panel columns [128 blockIdx.y, ...), panel
// rows [chunk blockIdx.z, ...).
__global__ void __launch_bounds__(OZ_THREADS, 2) k_bwd_tc(const int *__restrict__ fronts,
                                                          const FrontDesc *__restrict__ D,
                                                          const double *__restrict__ L, const int *__restrict__ rows,
                                                          const double *__restrict__ y, double *x,
                                                          int chunk, int *__restrict__ err) {
    const FrontDesc &d = D[fronts[blockIdx.x]];
    const int p = d.p, f = p + d.q, n = d.vlen;
    const int j0 = blockIdx.y * OZ_M, k1 = min((int)(blockIdx.z + 1) * chunk, f);
    const int k0 = max((int)blockIdx.z * chunk, j0);   // zeros above the diagonal
    if (j0 >= p || k0 >= k1) return;
    extern __shared__ unsigned char oz_raw[];
    __shared__ OzMvShared S;
    unsigned char *sm = oz_begin<OZ_MV_COLS>(S, oz_raw);
    const double *Lt = L + d.l_off + (int64_t)j0 * f;
    const int64_t vo = d.vec_off * OZ_V;
    const double *y1 = y + vo + d.first, *xo = x + vo;
    const int *rw = rows + d.row_off;
    const int used = min(OZ_M, p - j0), t = threadIdx.x;
    double out[4];
    const bool ok = oz_mv(
        S, sm, [&](int i, int k) { return k < k1 && k >= j0 + i ? Lt[k + (int64_t)i * f] : 0.0; },
        [&](int k, int v) {
            if (k >= k1) return 0.0;
            return k < p ? y1[k + (int64_t)v * n] : -xo[rw[k] + (int64_t)v * n];
        },
        [&](int pass, int &row, int &grp) {   // four threads a column: 256 contiguous bytes
            row = (t >> 2) + 64 * pass;
            grp = t & 3;
        },
        used, k0, k1, out);
    const int i = 32 * ((t >> 5) & 3) + (t & 31), v0 = 4 * (t >> 7);
    if (ok && i < used) {
        double *o = x + vo + d.first + j0 + i;
#pragma unroll
        for (int j = 0; j < 4; ++j) atomicAdd(o + (int64_t)(v0 + j) * n, out[j]);
    }
    oz_end<OZ_MV_COLS>(S, ok, err);
}

void oz_smem_limit() {
    static SmemLimit lim;
    lim.ensure(OZ_SMEM, [](size_t v) {
        GL_CUDA(cudaFuncSetAttribute(k_syrk64_tc, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)v));
        GL_CUDA(cudaFuncSetAttribute(k_wpanel_tc, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)v));
        GL_CUDA(cudaFuncSetAttribute(k_trinv_tc<0>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)v));
        GL_CUDA(cudaFuncSetAttribute(k_trinv_tc<1>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)v));
        GL_CUDA(cudaFuncSetAttribute(k_fwd_tc, cudaFuncAttributeMaxDynamicSharedMemorySize, OZ_MV_SMEM));
        GL_CUDA(cudaFuncSetAttribute(k_bwd_tc, cudaFuncAttributeMaxDynamicSharedMemorySize, OZ_MV_SMEM));
    });
}

}  // namespace

void syrk64_tc_level(const int *d_fronts, int n_fronts, const FrontDesc *d_fr, int k0, int panel, int max_f, double *ws,
                     int *d_err, cudaStream_t s) {
    oz_smem_limit();
    const int m = max_f - k0;   // upper bound of the trailing size over the level's fronts
    if (m <= 0) return;
    const int nt = (m + OZ_M - 1) / OZ_M;
    k_syrk64_tc<<<dim3(n_fronts, OZ_M / OZ_N * nt * (nt + 1) / 2), OZ_THREADS, OZ_SMEM, s>>>(d_fronts, d_fr, ws, k0, panel, d_err);
    GL_CUDA(cudaGetLastError());
}

void trinv_tc_level(const int *d_fronts, int n_fronts, const FrontDesc *d_fr, int max_p, double *ws, double *out,
                    int *d_err, cudaStream_t s) {
    oz_smem_limit();
    for (int b = 32; b < max_p; b *= 2) {
        const int pairs = (max_p - b + 2 * b - 1) / (2 * b);     // pairs with a second block
        const dim3 g(n_fronts, pairs * (b / OZ_N) * ((b + OZ_M - 1) / OZ_M));
        k_trinv_tc<0><<<g, OZ_THREADS, OZ_SMEM, s>>>(d_fronts, d_fr, ws, out, b, d_err);
        k_trinv_tc<1><<<g, OZ_THREADS, OZ_SMEM, s>>>(d_fronts, d_fr, ws, out, b, d_err);
    }
    GL_CUDA(cudaGetLastError());
}

void wpanel_tc_level(const int *d_fronts, int n_fronts, const FrontDesc *d_fr, int max_p, int max_f, const double *ws,
                     double *out, int *d_err, cudaStream_t s) {
    oz_smem_limit();
    const int tiles = ((max_f + OZ_M - 1) / OZ_M) * ((max_p + OZ_N - 1) / OZ_N);
    if (tiles <= 0) return;
    k_wpanel_tc<<<dim3(n_fronts, tiles), OZ_THREADS, OZ_SMEM, s>>>(d_fronts, d_fr, ws, out, d_err);
    GL_CUDA(cudaGetLastError());
}

// Summed entries per CTA: whole accumulations, cut finer while the level has too few CTAs.
static int oz_chunk(int64_t ctas, int n) {
    const int blocks = (n + OZ_VK - 1) / OZ_VK;
    const int split = (int)std::min<int64_t>(blocks, std::max<int64_t>(1, OZ_MV_CTAS / ctas));
    return OZ_VK * ((blocks + split - 1) / split);
}

void fwd_tc_level(const int *d_fronts, int n_fronts, const FrontDesc *d_fr, int max_p, int max_f, const double *L,
                  const int *rows, double *b, double *y, int *d_err, cudaStream_t s) {
    if (n_fronts == 0 || max_p == 0) return;
    oz_smem_limit();
    const int tiles = (max_f + OZ_M - 1) / OZ_M, chunk = oz_chunk((int64_t)n_fronts * tiles, max_p);
    k_fwd_tc<<<dim3(n_fronts, tiles, (max_p + chunk - 1) / chunk), OZ_THREADS, OZ_MV_SMEM, s>>>(d_fronts, d_fr, L, rows,
                                                                                              b, y, chunk, d_err);
    GL_CUDA(cudaGetLastError());
}

void bwd_tc_level(const int *d_fronts, int n_fronts, const FrontDesc *d_fr, int max_p, int max_f, const double *L,
                  const int *rows, const double *y, double *x, int *d_err, cudaStream_t s) {
    if (n_fronts == 0 || max_p == 0) return;
    oz_smem_limit();
    const int tiles = (max_p + OZ_M - 1) / OZ_M, chunk = oz_chunk((int64_t)n_fronts * tiles, max_f);
    k_bwd_tc<<<dim3(n_fronts, tiles, (max_f + chunk - 1) / chunk), OZ_THREADS, OZ_MV_SMEM, s>>>(d_fronts, d_fr, L, rows,
                                                                                              y, x, chunk, d_err);
    GL_CUDA(cudaGetLastError());
}

}  // namespace gl
