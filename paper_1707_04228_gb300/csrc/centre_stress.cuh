// Element-centre strain and stress in the local frame, shared by the stress
// recovery and the failure index.
#pragma once

#include <cstdint>

#include "gl_internal.h"

namespace gl {

// Local components of sigma = C_e eps(u) at the centre of element e: rr, rs, rl
// (frame R_l(psi): e_r = (sin psi, 0, cos psi), e_s = (cos psi, 0, -sin psi)).
// At the centre only the six face-centre nodes have a gradient, +-1/2 along
// their own axis, so J and du/dxi are half differences of opposite nodes.
// RL false leaves rl alone, and with it two rows of C_e.
template <bool RL>
__device__ __forceinline__ void centre_stress(int64_t e, int nx, int ny, int NX, int NY, const double *__restrict__ X,
                                              const double *__restrict__ C, const double *__restrict__ psi_x,
                                              const double *__restrict__ u, double &rr, double &rs, double &rl) {
    const int ex = (int)(e % nx), ey = (int)((e / nx) % ny), ez = (int)(e / ((int64_t)nx * ny));
    const int64_t mid = (int64_t)(2 * ex + 1) + (int64_t)NX * ((2 * ey + 1) + (int64_t)NY * (2 * ez + 1));
    const int64_t step[3] = {1, NX, (int64_t)NX * NY};
    double J[3][3], G[3][3];   // dx_r/dxi_d, du_r/dxi_d
#pragma unroll
    for (int d = 0; d < 3; ++d)
#pragma unroll
        for (int r = 0; r < 3; ++r) {
            const int64_t a = 3 * (mid + step[d]) + r, b = 3 * (mid - step[d]) + r;
            J[r][d] = 0.5 * (X[a] - X[b]);
            G[r][d] = 0.5 * (u[a] - u[b]);
        }
    double A[3][3];            // adj(J) = det(J) J^{-1}
    A[0][0] = J[1][1] * J[2][2] - J[1][2] * J[2][1];
    A[0][1] = J[0][2] * J[2][1] - J[0][1] * J[2][2];
    A[0][2] = J[0][1] * J[1][2] - J[0][2] * J[1][1];
    A[1][0] = J[1][2] * J[2][0] - J[1][0] * J[2][2];
    A[1][1] = J[0][0] * J[2][2] - J[0][2] * J[2][0];
    A[1][2] = J[0][2] * J[1][0] - J[0][0] * J[1][2];
    A[2][0] = J[1][0] * J[2][1] - J[1][1] * J[2][0];
    A[2][1] = J[0][1] * J[2][0] - J[0][0] * J[2][1];
    A[2][2] = J[0][0] * J[1][1] - J[0][1] * J[1][0];
    const double id = 1.0 / (J[0][0] * A[0][0] + J[0][1] * A[1][0] + J[0][2] * A[2][0]);
    double H[3][3];            // det(J) du_r/dx_d
#pragma unroll
    for (int r = 0; r < 3; ++r)
#pragma unroll
        for (int d = 0; d < 3; ++d) H[r][d] = G[r][0] * A[0][d] + G[r][1] * A[1][d] + G[r][2] * A[2][d];
    const double eps[6] = {H[0][0] * id, H[1][1] * id, H[2][2] * id, (H[1][2] + H[2][1]) * id, (H[0][2] + H[2][0]) * id,
                           (H[0][1] + H[1][0]) * id};
    const double *Ce = C + 36 * e;
    auto row = [&](int i) {
        double v = 0.0;
#pragma unroll
        for (int j = 0; j < 6; ++j) v += Ce[6 * i + j] * eps[j];
        return v;
    };
    double s, c;
    sincos(psi_x[ex], &s, &c);
    const double xx = row(0), zz = row(2), xz = row(4);
    const double tx = xx * s + xz * c, tz = xz * s + zz * c;   // sigma e_r
    rr = s * tx + c * tz;
    rs = c * tx - s * tz;
    if (RL) rl = row(5) * s + row(3) * c;
}

}  // namespace gl
