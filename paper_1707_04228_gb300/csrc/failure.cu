// Quadratic damage-onset criterion of Section 3.2 (Eq. eq-Camanho):
//   F = sqrt((sigma_r^+ / s33)^2 + (tau_rs / s13)^2 + (tau_rl / s13)^2),
// sigma_r^+ = max(sigma_rr, 0), applied in the isotropic resin interfaces only
// (zero elsewhere), with the stresses recovered at the element centre and
// rotated into the local (s, l, r) frame.  One thread per element; the peak and
// its element come from a block reduction and a 64-bit atomic max on the
// (F, element) pair packed so that larger F wins.
#include "centre_stress.cuh"
#include "gl_internal.h"

namespace gl {

__global__ void __launch_bounds__(128) k_failure(int64_t n_elem, int nx, int ny, int NX, int NY,
                                                 const double *__restrict__ X, const double *__restrict__ C,
                                                 const double *__restrict__ psi_x, const uint8_t *__restrict__ resin,
                                                 const double *__restrict__ u, double s33a, double s13a,
                                                 double *__restrict__ F, unsigned long long *__restrict__ best) {
    const int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    double fval = 0.0;
    if (e < n_elem && resin[e]) {
        double srr, srs, srl;
        centre_stress<true>(e, nx, ny, NX, NY, X, C, psi_x, u, srr, srs, srl);
        const double a = fmax(srr, 0.0) / s33a, b = srs / s13a, c = srl / s13a;
        fval = sqrt(a * a + b * b + c * c);
    }
    if (e < n_elem) F[e] = fval;
    // block max of (F, element), then one atomic per block
    __shared__ double bf[128];
    __shared__ long long be[128];
    bf[threadIdx.x] = e < n_elem ? fval : -1.0;
    be[threadIdx.x] = e;
    __syncthreads();
    for (int o = 64; o > 0; o >>= 1) {
        if (threadIdx.x < o && bf[threadIdx.x + o] > bf[threadIdx.x]) {
            bf[threadIdx.x] = bf[threadIdx.x + o];
            be[threadIdx.x] = be[threadIdx.x + o];
        }
        __syncthreads();
    }
    if (threadIdx.x == 0 && bf[0] >= 0.0) {
        // F >= 0: its bit pattern orders like the value; keep 40 bits of it and 24 of the element id
        unsigned long long key = ((unsigned long long)__double_as_longlong(bf[0]) >> 24) << 24;
        key |= (unsigned long long)(be[0] & 0xFFFFFF);
        atomicMax(best, key);
    }
}

// out[0] = the packed key, out[1] = the untruncated F of its element: one read for the host.
__global__ void k_failure_peak(const double *__restrict__ F, double *__restrict__ out) {
    out[1] = F[__double_as_longlong(out[0]) & 0xFFFFFF];
}

void launch_failure(const MeshHost &m, const double *X, const double *C, const double *psi_x, const uint8_t *resin,
                    const double *u, double s33a, double s13a, double *F, double *peak, cudaStream_t s) {
    GL_CUDA(cudaMemsetAsync(peak, 0, sizeof(double), s));
    k_failure<<<(unsigned)((m.n_elem + 127) / 128), 128, 0, s>>>(m.n_elem, m.nx, m.ny, m.NX, m.NY, X, C, psi_x, resin, u,
                                                                s33a, s13a, F,
                                                                reinterpret_cast<unsigned long long *>(peak));
    k_failure_peak<<<1, 1, 0, s>>>(F, peak);
    GL_CUDA(cudaGetLastError());
}

}  // namespace gl
