// Warp-level reductions shared by the kernels.
#pragma once

namespace gl {

// Sums N (a power of two) values over the lanes of a warp, about one add per
// value against five of a shuffle tree each: every step halves the values a
// lane holds.  N >= 32: value i comes back as v[i % PL] of lane i / PL, PL =
// N / 32; N < 32: as v[0] of the 32 / N lanes from i 32 / N on.
template <class T, int N>
__device__ __forceinline__ void warp_sum_many(T (&v)[N], int lane) {
    int n = N;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        if (n == 1) {
            v[0] += __shfl_xor_sync(0xffffffffu, v[0], o);
            continue;
        }
        n >>= 1;
        const bool up = lane & o;
#pragma unroll
        for (int k = 0; k < N / 2; ++k)
            if (k < n) {
                const T send = up ? v[k] : v[k + n], keep = up ? v[k + n] : v[k];
                v[k] = keep + __shfl_xor_sync(0xffffffffu, send, o);
            }
    }
}

}  // namespace gl
