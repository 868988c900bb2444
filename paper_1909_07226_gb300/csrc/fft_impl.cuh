// Centred 2D transform of the four polarisation planes of one subgrid held in
// shared memory as s[pol][y][x] (row pitch L + 1, which keeps both passes free
// of bank conflicts).  Rows, then columns, each a length-L FFT in registers,
// spread over the nt threads of the CTA.  The caller applies the (-1)^(x+y)
// centring factors and the 1/L^2 scale.  Ends with a barrier.
#pragma once

#include "device_common.cuh"

namespace idg {
namespace dev {

template <int L, int SIGN>
__device__ __forceinline__ void fft2_planar(float2 *s, int tid, int nt) {
    constexpr int P = L + 1;
    for (int line = tid; line < 4 * L; line += nt) {
        float2 v[L];
        float2 *row = s + line * P;
#pragma unroll
        for (int x = 0; x < L; ++x) v[x] = row[x];
        RegFFT<L, SIGN>::run(v);
#pragma unroll
        for (int x = 0; x < L; ++x) row[x] = v[x];
    }
    __syncthreads();
    for (int line = tid; line < 4 * L; line += nt) {
        const int pol = line / L, x = line - (line / L) * L;
        float2 v[L];
        float2 *col = s + pol * L * P + x;
#pragma unroll
        for (int y = 0; y < L; ++y) v[y] = col[y * P];
        RegFFT<L, SIGN>::run(v);
#pragma unroll
        for (int y = 0; y < L; ++y) col[y * P] = v[y];
    }
    __syncthreads();
}

// Centred transform of one line held in registers, X[k] = sum_n x[n] exp(SIGN 2 pi i (n - L/2)
// (k - L/2) / L): both centrings are index shifts by L / 2, which cost nothing at compile-time
// indices.  load(n) gives sample n, store(k, X) takes sample k.  One thread per line: a
// 32-point line needs 64 registers, no shuffles and 40 % fewer instructions than the
// two-threads-per-line form; in the fused separable kernels, whose second CTA fills the
// issue slots that four busy warps leave, that is the faster one.
template <int L, int SIGN, typename Load, typename Store>
__device__ __forceinline__ void fft_line(Load load, Store store) {
    float2 v[L];
#pragma unroll
    for (int n = 0; n < L; ++n) v[(n + L / 2) % L] = load(n);
    RegFFT<L, SIGN>::run(v);
#pragma unroll
    for (int k = 0; k < L; ++k) store(k, v[(k + L / 2) % L]);
}

// Plane stride (in float2) of four polarisation planes [L][L + 1] for threads (line, pol) with
// the polarisation fastest: 4 mod 16, so that the 4 lines x 4 planes of a half-warp fall into
// different banks both along rows and along columns
template <int L>
struct PolPlanes {
    static constexpr int P = L + 1, N0 = L * P, STRIDE = N0 + (20 - N0 % 16) % 16;
    static_assert(STRIDE % 16 == 4, "plane stride");
};

}  // namespace dev
}  // namespace idg
