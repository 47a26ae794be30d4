// Periodic 3x3 convolution of float32 activations on the CUDA cores, the inner
// product of the float32 forward and of the input gradient.
//
// Activations are position-major, [position][CP] with CP = C + 4 floats, so
// that the 16-byte loads of consecutive positions fall on different banks. A
// thread owns ST positions and OT output channels: four input channels of one
// tap cost ST loads of activations and OT broadcast loads of weights for
// ST * OT * 4 multiply-adds, issued as packed pairs (fma.rn.f32x2) over output
// channels: 16 wavefronts against 16.5 cycles of the FMA pipe at ST = 2,
// OT = 8, where one position and eight channels a thread (the earlier layout)
// took three wavefronts for every eight FMAs and was bound by them. Every
// output sums bias, then taps in order, then input channels in order, each by
// one fused multiply-add.
#pragma once

#include "common.cuh"

namespace nqs {

template <int C> constexpr int kConvPitch = C + 4;   // floats between positions

// Table of neighbour rows for `copies` lattices side by side: nbr[k * npos + p]
// is the position at p + d_k in p's own lattice (npos = copies * N).
__device__ inline void conv_neighbours(uint16_t *nbr, int L, int copies) {
    const int N = L * L, npos = copies * N;
    for (int p = threadIdx.x; p < npos; p += blockDim.x) {
        const int g = p / N, s = p - g * N, y = s / L, x = s - y * L;
        for (int k = 0; k < 9; ++k) {
            const int dy = k / 3 - 1, dx = k % 3 - 1;
            const int yy = y + dy < 0 ? L - 1 : (y + dy == L ? 0 : y + dy);
            const int xx = x + dx < 0 ? L - 1 : (x + dx == L ? 0 : x + dx);
            nbr[k * npos + p] = (uint16_t)(g * N + yy * L + xx);
        }
    }
}

// acc[j][q] += sum over taps k and input channels c < CI of
// w[k][c][o0 + 2 q, + 1] in_j[nbr_k(p_j)][c], with the tap's neighbours from row
// k of nbr (8 - k if FLIP: positions p - d_k). w: [9][CI][C].
template <int CI, int C, int OT, int ST, bool FLIP>
__device__ __forceinline__ void conv_accumulate(const float *const (&in)[ST], const float *w, const uint16_t *nbr,
                                                int npos, const int (&p)[ST], int o0, float2 (&acc)[ST][OT / 2]) {
    constexpr int CP = kConvPitch<C>;
#pragma unroll 1
    for (int k = 0; k < 9; ++k) {
        const float *row[ST];
#pragma unroll
        for (int j = 0; j < ST; ++j) row[j] = in[j] + (int)nbr[(FLIP ? 8 - k : k) * npos + p[j]] * CP;
        const float *wk = w + k * CI * C + o0;
#pragma unroll
        for (int c4 = 0; c4 < CI; c4 += 4) {
            float h[ST][4];
#pragma unroll
            for (int j = 0; j < ST; ++j) {
                const float4 v = *reinterpret_cast<const float4 *>(row[j] + c4);
                h[j][0] = v.x, h[j][1] = v.y, h[j][2] = v.z, h[j][3] = v.w;
            }
#pragma unroll
            for (int cc = 0; cc < (CI - c4 < 4 ? CI - c4 : 4); ++cc) {
                const float *wc = wk + (c4 + cc) * C;
#pragma unroll
                for (int q = 0; q < OT / 4; ++q) {
                    const float4 wv = *reinterpret_cast<const float4 *>(wc + 4 * q);
#pragma unroll
                    for (int j = 0; j < ST; ++j) {
                        const float2 hh = make_float2(h[j][cc], h[j][cc]);
                        acc[j][2 * q] = __ffma2_rn(make_float2(wv.x, wv.y), hh, acc[j][2 * q]);
                        acc[j][2 * q + 1] = __ffma2_rn(make_float2(wv.z, wv.w), hh, acc[j][2 * q + 1]);
                    }
                }
            }
        }
    }
}

// Stage one layer's weights W[o][c][9] of the flat parameters as w[k][c][o]
// (TRANS: w[k][o][c], for the input gradient), its bias after them.
template <int C, bool TRANS>
__device__ __forceinline__ void conv_stage(const float *__restrict__ prm, int cin, float *w) {
    for (int e = threadIdx.x; e < C * cin; e += blockDim.x) {
        // lanes over the index that is contiguous in w
        const int fast = TRANS ? cin : C;
        const int a = e / fast, b = e - a * fast;
        const int o = TRANS ? a : b, c = TRANS ? b : a;
        const float *src = prm + (o * cin + c) * 9;
#pragma unroll
        for (int k = 0; k < 9; ++k) w[k * cin * C + e] = __ldg(src + k);
    }
    for (int o = threadIdx.x; o < C; o += blockDim.x) w[9 * cin * C + o] = __ldg(prm + 9 * cin * C + o);
}

}  // namespace nqs
