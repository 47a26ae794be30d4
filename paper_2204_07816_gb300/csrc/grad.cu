// Per-sample local derivatives O_k = d log W / d theta_k (Sec. 3.2: the
// backward of the network gives O_loc) with float32 internals, for the
// FP32 and tensor-core precisions. A block takes S samples at a time:
//   forward   z_l = conv(h_{l-1}) + b_l, h_l = silu(z_l); h_l and
//             s_l = sigmoid(z_l) go to this block's (L2-resident) scratch
//   head      d a / d w_a = d phi / d w_phi = sum over sites of h_n
//   backward  for l = n_l - 1 .. 0, both outputs (a and phi) at once:
//             gz = g * silu'(z) with silu'(z) = s + h (1 - s)
//             dW[o][c][k] = sum_site gz[o][site] h_{l-1}[c][site + d_k]
//             db[o] = sum_site gz[o][site]
//             g_{l-1}[c][site] = sum_{o,k} W[o][c][k] gz[o][site - d_k],
//             multiplied by silu'(z_{l-1}) as it is written
// The three contractions run on register tiles of packed float32 pairs
// (conv_f32.cuh; the weight gradient: two output channels, one input channel,
// nine taps and both outputs a thread, the 3 x 3 input window in registers),
// so that shared-memory wavefronts stay below the FMA pipe's cycles. Bound:
// the FMA pipe (5 dense forwards a sample) at the tiles' thread use, 78 % at
// 10x10. Measured (GB300, before: one position and eight channels a thread, one
// sample a block): O of 8,192 samples, 10x10, 16 channels, 6 layers 4.88 ->
// 3.23 ms; of 1,024 samples, 16x16, 32 channels, 8 layers 8.92 -> 4.61 ms;
// vector-Jacobian product of 2,048 samples there 13.24 -> 6.96 ms. Every sum
// keeps its order, so the results are bitwise the same.
//
// Vector-Jacobian form (VJP = true): given per-sample output gradients
// (g_a, g_phi), one backward stream seeded with g_a w_a + g_phi w_phi gives
// g_a d a / d theta + g_phi d phi / d theta for every parameter, and the
// samples' vectors are summed per chunk of consecutive samples (each of a
// block's S slots owns one chunk at a time, samples in order) into chunk
// partials; a second kernel sums the partials in chunk order. No per-sample
// row is stored.
#include <algorithm>

#include "conv_f32.cuh"
#include "internal.h"

namespace nqs {

namespace {

constexpr int kGradThreads = 512;
constexpr int kGradMaxSamples = 16;   // samples a block takes at a time, at most

__host__ __device__ inline size_t a16(size_t v) { return (v + 15) & ~size_t(15); }

// Shared memory of a block with S samples and R backward streams.
struct GradLayout {
    size_t w, nbr, h, g0, g1, hbar, turn, total;
};

__host__ __device__ inline GradLayout grad_layout(const Problem &p, int S, int R, bool turn) {
    const size_t act = 4 * (size_t)S * p.N * (p.C + 4);
    GradLayout g;
    size_t o = 0;
    g.w = o; o = a16(o + 4 * (size_t)(9 * p.C * p.C + p.C));
    g.h = o; o = a16(o + act);
    g.g0 = o; o = a16(o + R * act);
    g.g1 = o; o = a16(o + R * act);
    g.nbr = o; o = a16(o + 2 * (size_t)9 * S * p.N);
    g.hbar = o; o = a16(o + 4 * (size_t)S * p.C);
    g.turn = o;   // per warp: grad_store's transposition
    if (turn) o = a16(o + 4 * (size_t)(kGradThreads / 32) * 9 * 32);
    g.total = o;
    return g;
}

// Input encoding of the samples into h.
template <int C>
__device__ __forceinline__ void grad_encode(const Problem &p, const int8_t *const *cfg, int S, float *h) {
    constexpr int CP = kConvPitch<C>;
    for (int q = threadIdx.x; q < S * p.N; q += blockDim.x) {
        const int j = q / p.N, v = cfg[j][q - j * p.N];
        *reinterpret_cast<float4 *>(h + q * CP) =
            p.c_in == 1 ? make_float4((float)v, 0.f, 0.f, 0.f)
                        : make_float4((float)(v == 0), (float)(v == 1), (float)(v == -1), 0.f);
    }
}

__device__ __forceinline__ void store8(float *dst, const float (&v)[8]) {
    *reinterpret_cast<float4 *>(dst) = make_float4(v[0], v[1], v[2], v[3]);
    *reinterpret_cast<float4 *>(dst + 4) = make_float4(v[4], v[5], v[6], v[7]);
}

// Where a sample's derivatives go: rows of O (VJP = false) or its chunk's
// partial, written by the chunk's first sample and added to by the others.
template <bool VJP>
struct GradOut {
    double *a, *phi;   // VJP: a = the chunk's partial; a = null: an idle slot, nothing is stored
    bool first;
    __device__ __forceinline__ void put(int k, float va, float vphi) const {
        if (!a) return;
        if (VJP) {
            a[k] = first ? 0.0 + (double)va : a[k] + (double)va;
        } else {
            a[k] = (double)va;
            phi[k] = (double)vphi;
        }
    }
    __device__ __forceinline__ void put(int k, int stream, float v) const {   // one stream's value
        if (VJP) put(k, v, 0.f);
        else if (a) (stream == 0 ? a : phi)[k] = (double)v;
    }
};

// Weight gradient of one thread: output channels o, o + 1, input channel c,
// nine taps, R streams; sites in row-major order, the 3 x 3 input window (as
// pairs of equal floats) in registers, three new values a site.
template <int C, int R>
__device__ __forceinline__ void grad_weights(const float *h, const float *g, size_t stream, int L, float2 (&acc)[R][9]) {
    constexpr int CP = kConvPitch<C>;
#pragma unroll
    for (int r = 0; r < R; ++r)
#pragma unroll
        for (int k = 0; k < 9; ++k) acc[r][k] = make_float2(0.f, 0.f);
    for (int y = 0; y < L; ++y) {
        const float *row[3] = {h + (y == 0 ? L - 1 : y - 1) * L * CP, h + y * L * CP, h + (y == L - 1 ? 0 : y + 1) * L * CP};
        const float *gy = g + y * L * CP;
        float2 win[3][3];   // [column mod 3][row]
#pragma unroll
        for (int d = 0; d < 3; ++d) {
            const float a = row[d][(L - 1) * CP], b = row[d][0];
            win[2][d] = make_float2(a, a);   // column -1
            win[0][d] = make_float2(b, b);   // column 0
        }
        auto step = [&](int x, float2 (&left)[3], float2 (&mid)[3], float2 (&right)[3]) {
            const int xn = x + 1 == L ? 0 : x + 1;
#pragma unroll
            for (int d = 0; d < 3; ++d) {
                const float v = row[d][xn * CP];
                right[d] = make_float2(v, v);
            }
#pragma unroll
            for (int r = 0; r < R; ++r) {
                const float2 gv = *reinterpret_cast<const float2 *>(gy + r * stream + x * CP);
#pragma unroll
                for (int d = 0; d < 3; ++d) {
                    acc[r][3 * d] = __ffma2_rn(gv, left[d], acc[r][3 * d]);
                    acc[r][3 * d + 1] = __ffma2_rn(gv, mid[d], acc[r][3 * d + 1]);
                    acc[r][3 * d + 2] = __ffma2_rn(gv, right[d], acc[r][3 * d + 2]);
                }
            }
        };
        int x = 0;
        for (; x + 2 < L; x += 3) {   // the window's columns rotate through three register sets
            step(x, win[2], win[0], win[1]);
            step(x + 1, win[0], win[1], win[2]);
            step(x + 2, win[1], win[2], win[0]);
        }
        if (x < L) step(x, win[2], win[0], win[1]);
        if (x + 1 < L) step(x + 1, win[0], win[1], win[2]);
    }
}

// Nine taps of input channel c for one output channel, one value a lane in the
// thread's registers, into nine coalesced stores: the C lanes of an output
// channel hold 9 C consecutive parameters, turned round in shared memory (a
// store per tap touched a sector a lane: 0.7 of 4.0 ms at 10x10).
template <int C, typename Put>
__device__ __forceinline__ void grad_store(float *turn, const float (&v)[9], Put put) {
    const int lane = threadIdx.x & 31, c = lane & (C - 1);
    if (!turn) {   // no room for the transposition
#pragma unroll
        for (int k = 0; k < 9; ++k) put(c * 9 + k, v[k]);
        return;
    }
    float *t = turn + (lane - c) * 9;
    __syncwarp();
#pragma unroll
    for (int k = 0; k < 9; ++k) t[c * 9 + k] = v[k];
    __syncwarp();
#pragma unroll
    for (int k = 0; k < 9; ++k) put(k * C + c, t[k * C + c]);
}

// Sums over the N sites of four channels at v (lane k takes sites k, k + 32,
// ..., then the xor-shuffle tree); the result in every lane.
template <int CP>
__device__ __forceinline__ float4 grad_site_sum(const float *v, int N) {
    float4 a = make_float4(0.f, 0.f, 0.f, 0.f);
    for (int s = threadIdx.x & 31; s < N; s += 32) {
        const float4 x = *reinterpret_cast<const float4 *>(v + s * CP);
        a.x += x.x, a.y += x.y, a.z += x.z, a.w += x.w;
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        a.x += __shfl_xor_sync(0xffffffffu, a.x, o);
        a.y += __shfl_xor_sync(0xffffffffu, a.y, o);
        a.z += __shfl_xor_sync(0xffffffffu, a.z, o);
        a.w += __shfl_xor_sync(0xffffffffu, a.w, o);
    }
    return a;
}

// Backward of S samples. R: streams carried at once; VJP = false with R = 1
// (lattices whose two streams do not fit) runs the backward once per stream.
template <int C, int R, bool VJP>
__device__ void grad_samples(const Problem &p, unsigned char *smem, const GradLayout &gl, const float *__restrict__ prm,
                             const double *__restrict__ p64, int S, bool has_turn, const int8_t *const *cfg, const GradOut<VJP> *out,
                             const double *ga, const double *gp, float *Hs) {
    constexpr int CP = kConvPitch<C>, OT = 8, ST = 2, OG = C / OT;
    const int N = p.N, L = p.L, nl = p.n_layers, npos = S * N;
    float *w = reinterpret_cast<float *>(smem + gl.w), *h = reinterpret_cast<float *>(smem + gl.h);
    float *g0 = reinterpret_cast<float *>(smem + gl.g0), *g1 = reinterpret_cast<float *>(smem + gl.g1);
    float *hbar = reinterpret_cast<float *>(smem + gl.hbar);
    float *turn = has_turn ? reinterpret_cast<float *>(smem + gl.turn) + (threadIdx.x >> 5) * 9 * 32 : nullptr;
    const uint16_t *nbr = reinterpret_cast<const uint16_t *>(smem + gl.nbr);
    float *Ss = Hs + (size_t)nl * npos * C;   // Hs, Ss: [nl][npos][C] h, sigmoid(z)
    const size_t stream = (size_t)npos * CP;  // floats between the streams of a gradient buffer
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
    const int ho = head_offset(p);
    // output gradient of the head for channel c of sample j, stream r
    auto seed = [&](int j, int r, int c) {
        return VJP ? (float)(ga[j] * p64[ho + c] + gp[j] * p64[ho + C + c]) : (float)p64[ho + r * C + c];
    };
    grad_encode<C>(p, cfg, S, h);
    // ---------------- forward: h and g1 in turn; the last layer's gradient into g0
    for (int l = 0; l < nl; ++l) {
        const int cin = layer_cin(p, l);
        conv_stage<C, false>(prm + layer_offset(p, l), cin, w);
        __syncthreads();
        const float *src = l & 1 ? g1 : h, *const in[ST] = {src, src};
        float *hout = l & 1 ? h : g1;
        const int np = (npos + ST - 1) / ST;
        for (int it = threadIdx.x; it < OG * np; it += blockDim.x) {
            const int o0 = it / np * OT, q0 = it % np;
            int q[ST];
            float2 acc[ST][OT / 2];
#pragma unroll
            for (int j = 0; j < ST; ++j) {
                q[j] = min(q0 + j * np, npos - 1);
#pragma unroll
                for (int c = 0; c < OT / 2; ++c)
                    acc[j][c] = *reinterpret_cast<const float2 *>(w + 9 * cin * C + o0 + 2 * c);
            }
            if (l > 0) conv_accumulate<C, C, OT, ST, false>(in, w, nbr, npos, q, o0, acc);
            else if (cin == 1) conv_accumulate<1, C, OT, ST, false>(in, w, nbr, npos, q, o0, acc);
            else conv_accumulate<3, C, OT, ST, false>(in, w, nbr, npos, q, o0, acc);
#pragma unroll
            for (int j = 0; j < ST; ++j) {
                if (q0 + j * np >= npos) continue;
                float hv[OT], sv[OT];
#pragma unroll
                for (int c = 0; c < OT; ++c) {
                    const float z = c & 1 ? acc[j][c / 2].y : acc[j][c / 2].x;
                    sv[c] = 1.0f / (1.0f + expf(-z));
                    hv[c] = z * sv[c];
                }
                store8(hout + q[j] * CP + o0, hv);
                const size_t at = ((size_t)l * npos + q[j]) * C + o0;
                store8(Hs + at, hv);
                store8(Ss + at, sv);
                if (l == nl - 1 && (VJP || R == 2)) {
                    const int js = q[j] / N;
#pragma unroll
                    for (int r = 0; r < R; ++r) {
                        float gv[OT];
#pragma unroll
                        for (int c = 0; c < OT; ++c) gv[c] = seed(js, r, o0 + c) * (sv[c] + hv[c] * (1.0f - sv[c]));
                        store8(g0 + r * stream + q[j] * CP + o0, gv);
                    }
                }
            }
        }
        __syncthreads();
    }
    // ---------------- head
    const float *hn = nl & 1 ? g1 : h;
    for (int t = warp; t < S * (C / 4); t += nw) {
        const int j = t / (C / 4), c = t % (C / 4) * 4;
        const float4 v = grad_site_sum<CP>(hn + (size_t)j * N * CP + c, N);
        if (lane == 0) *reinterpret_cast<float4 *>(hbar + j * C + c) = v;
    }
    __syncthreads();
    for (int t = threadIdx.x; t < S * C; t += blockDim.x) {
        const int j = t / C, c = t - j * C;
        const GradOut<VJP> &o = out[j];
        const double hb = (double)hbar[t];
        if (!o.a) continue;
        if (VJP) {
            o.a[ho + c] = (o.first ? 0.0 : o.a[ho + c]) + ga[j] * hb;
            o.a[ho + C + c] = (o.first ? 0.0 : o.a[ho + C + c]) + gp[j] * hb;
        } else {
            o.a[ho + c] = hb;
            o.a[ho + C + c] = 0.0;
            o.phi[ho + c] = 0.0;
            o.phi[ho + C + c] = hb;
        }
    }
    // ---------------- backward
    constexpr int kPasses = !VJP && R == 1 ? 2 : 1;   // streams one after the other
    for (int pass = 0; pass < kPasses; ++pass) {
        if (kPasses == 2) {   // this stream's gradient at the last layer
            for (int e = threadIdx.x; e < npos * C; e += blockDim.x) {
                const int q = e / C, c = e - q * C;
                const size_t at = ((size_t)(nl - 1) * npos + q) * C + c;
                const float sg = Ss[at], hv = Hs[at];
                g0[q * CP + c] = seed(q / N, pass, c) * (sg + hv * (1.0f - sg));
            }
        }
        float *gc = g0, *gn = g1;
        for (int l = nl - 1; l >= 0; --l) {
            const int cin = layer_cin(p, l), off = layer_offset(p, l);
            __syncthreads();
            // layer input h_{l-1} and the weights as w[k][o][c]
            if (l == 0) {
                grad_encode<C>(p, cfg, S, h);
            } else {
                const float *Hp = Hs + (size_t)(l - 1) * npos * C;
                for (int e = threadIdx.x; e < npos * (C / 4); e += blockDim.x) {
                    const int q = e / (C / 4), c4 = e - q * (C / 4);
                    *reinterpret_cast<float4 *>(h + q * CP + 4 * c4) = *reinterpret_cast<const float4 *>(Hp + (size_t)e * 4);
                }
                conv_stage<C, true>(prm + off, cin, w);
            }
            __syncthreads();
            // weight gradient
            if (l > 0) {
                for (int t = threadIdx.x; t < S * (C / 2) * C; t += blockDim.x) {
                    const int j = t / (C / 2 * C), o = t / C % (C / 2) * 2, c = t % C;
                    float2 acc[R][9];
                    grad_weights<C, R>(h + (size_t)j * N * CP + c, gc + (size_t)j * N * CP + o, stream, L, acc);
                    const GradOut<VJP> ot = out[j];
#pragma unroll
                    for (int u = 0; u < 2; ++u)   // output channels o, o + 1
#pragma unroll
                        for (int r = 0; r < R; ++r) {
                            float v[9];
#pragma unroll
                            for (int k = 0; k < 9; ++k) v[k] = u ? acc[r][k].y : acc[r][k].x;
                            grad_store<C>(turn, v, [&](int k, float x) {
                                ot.put(off + (o + u) * C * 9 + k, kPasses == 2 ? pass : r, x);
                            });
                        }
                }
            } else {
                // one or three input channels: a thread per tap as well
                for (int t = threadIdx.x; t < S * C * cin * 9; t += blockDim.x) {
                    const int j = t / (C * cin * 9), rem = t - j * (C * cin * 9), k = rem / (C * cin), oc = rem - k * C * cin;
                    const int o = oc / cin, c = oc - o * cin;
                    float a[R];
#pragma unroll
                    for (int r = 0; r < R; ++r) a[r] = 0.f;
                    const uint16_t *nk = nbr + k * npos + j * N;
                    for (int s = 0; s < N; ++s) {
                        const float hv = h[(int)nk[s] * CP + c];
#pragma unroll
                        for (int r = 0; r < R; ++r) a[r] = fmaf(gc[r * stream + (j * N + s) * CP + o], hv, a[r]);
                    }
                    const int k0 = off + (o * cin + c) * 9 + k;
                    if (kPasses == 2) out[j].put(k0, pass, a[0]);
                    else out[j].put(k0, a[0], a[R - 1]);
                }
            }
            // bias gradient
            for (int t = warp; t < R * S * (C / 4); t += nw) {
                const int r = t / (S * (C / 4)), j = t / (C / 4) % S, o = t % (C / 4) * 4;
                const float4 v = grad_site_sum<CP>(gc + r * stream + (size_t)j * N * CP + o, N);
                if (lane < 4)
                    out[j].put(off + 9 * cin * C + o + lane, kPasses == 2 ? pass : r,
                               lane < 2 ? (lane == 0 ? v.x : v.y) : (lane == 2 ? v.z : v.w));
            }
            if (l == 0) break;
            // gradient of the layer's input times silu'(z_{l-1}), into the other buffer
            // a thread's two positions: the same site in both streams, or two sites of the one stream
            const int np = R == 2 ? npos : (npos + 1) / 2;
            const float *Hp = Hs + (size_t)(l - 1) * npos * C, *Sp = Ss + (size_t)(l - 1) * npos * C;
            for (int it = threadIdx.x; it < OG * np; it += blockDim.x) {
                const int o0 = it / np * OT, q0 = it % np;
                const int q[ST] = {q0, R == 2 ? q0 : min(q0 + np, npos - 1)};
                const float *const in[ST] = {gc, R == 2 ? gc + stream : gc};
                float2 acc[ST][OT / 2];
#pragma unroll
                for (int j = 0; j < ST; ++j)
#pragma unroll
                    for (int c = 0; c < OT / 2; ++c) acc[j][c] = make_float2(0.f, 0.f);
                conv_accumulate<C, C, OT, ST, true>(in, w, nbr, npos, q, o0, acc);
#pragma unroll
                for (int j = 0; j < ST; ++j) {
                    if (R == 1 && q0 + j * np >= npos) continue;
                    const size_t at = (size_t)q[j] * C + o0;
                    float gv[OT];
#pragma unroll
                    for (int c4 = 0; c4 < OT; c4 += 4) {
                        const float4 hv = *reinterpret_cast<const float4 *>(Hp + at + c4);
                        const float4 sv = *reinterpret_cast<const float4 *>(Sp + at + c4);
                        gv[c4] = acc[j][c4 / 2].x * (sv.x + hv.x * (1.0f - sv.x));
                        gv[c4 + 1] = acc[j][c4 / 2].y * (sv.y + hv.y * (1.0f - sv.y));
                        gv[c4 + 2] = acc[j][c4 / 2 + 1].x * (sv.z + hv.z * (1.0f - sv.z));
                        gv[c4 + 3] = acc[j][c4 / 2 + 1].y * (sv.w + hv.w * (1.0f - sv.w));
                    }
                    store8(gn + (R == 2 ? j * stream : 0) + q[j] * CP + o0, gv);
                }
            }
            float *t = gc;
            gc = gn;
            gn = t;
        }
        __syncthreads();
    }
}

// A block's S slots: sample (VJP = false) or chunk (VJP) number
// blockIdx.x S + j, then gridDim.x S further; every slot's chunk takes one
// sample at a time. grad [n][2] = (g_a, g_phi), part [ceil(n / K)][P].
template <int C, int R, bool VJP>
__global__ void __launch_bounds__(kGradThreads, 1)
    grad_fast_kernel(Problem p, int S, bool turn, const float *__restrict__ prm, const double *__restrict__ p64,
                     const int8_t *__restrict__ configs, int64_t n, double *__restrict__ O,
                     const double *__restrict__ grad, int64_t K, double *__restrict__ part, float *scratch) {
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ const int8_t *cfg[kGradMaxSamples];
    __shared__ GradOut<VJP> out[kGradMaxSamples];
    __shared__ double ga[kGradMaxSamples], gp[kGradMaxSamples];
    const GradLayout gl = grad_layout(p, S, R, turn);
    conv_neighbours(reinterpret_cast<uint16_t *>(smem + gl.nbr), p.L, S);
    float *Hs = scratch + (size_t)2 * p.n_layers * S * p.N * C * blockIdx.x;
    const int64_t slots = VJP ? (n + K - 1) / K : n, steps = VJP ? K : 1;
    for (int64_t b = (int64_t)blockIdx.x * S; b < slots; b += (int64_t)gridDim.x * S)
        for (int64_t i = 0; i < steps; ++i) {
            __syncthreads();
            if ((int)threadIdx.x < S) {
                const int64_t q = b + threadIdx.x, s = VJP ? q * K + i : q;
                const bool busy = q < slots && s < n;
                const int64_t sc = busy ? s : n - 1;   // an idle slot repeats a sample and stores nothing
                cfg[threadIdx.x] = configs + sc * p.N;
                GradOut<VJP> o;
                o.first = i == 0;
                o.a = !busy ? nullptr : (VJP ? part + (size_t)q * p.P : O + (size_t)s * p.P);
                o.phi = VJP || !busy ? nullptr : O + (size_t)(n + s) * p.P;
                out[threadIdx.x] = o;
                ga[threadIdx.x] = VJP ? grad[2 * sc] : 0.0;
                gp[threadIdx.x] = VJP ? grad[2 * sc + 1] : 0.0;
            }
            __syncthreads();
            grad_samples<C, R, VJP>(p, smem, gl, prm, p64, S, turn, cfg, out, ga, gp, Hs);
        }
}

// out[k] = sum over chunks q = 0 .. nq - 1 (in order) of part[q][k]. Sixteen
// loads are in flight before their additions: one at a time, the loop was a
// chain of memory latencies (product at 4x4, 1,024 chunks: 0.335 -> 0.286 ms).
__global__ void __launch_bounds__(128) vjp_reduce_kernel(const double *__restrict__ part, int64_t nq, int P,
                                                         double *__restrict__ out) {
    constexpr int U = 16;
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= P) return;
    double v = 0.0;
    int64_t q = 0;
    for (; q + U <= nq; q += U) {
        double x[U];
#pragma unroll
        for (int u = 0; u < U; ++u) x[u] = __ldcs(part + (size_t)(q + u) * P + k);
#pragma unroll
        for (int u = 0; u < U; ++u) v += x[u];
    }
    for (; q < nq; ++q) v += part[(size_t)q * P + k];
    out[k] = v;
}

// Streams a block carries at once, and samples S: as many as shared memory
// holds, counted in rounds of the block's threads (a forward or input-gradient
// tile is 72 C packed multiply-adds, a weight-gradient tile 9 N R), the
// cheapest per sample; fewer if the call has fewer samples than SMs times S.
// Lattices whose two streams do not fit (24x24 and 25x25 with 16 channels,
// 17x17 with 32) run the backward once a stream, which is still shorter than
// the kernel before, which carried both (three layers, 400 samples, us: 839 ->
// 515, 951 -> 550, 1,375 -> 834).
int grad_streams(const Problem &p, bool vjp, size_t max_smem) {
    return !vjp && grad_layout(p, 1, 2, false).total + 1024 <= max_smem ? 2 : 1;
}

// The transposition buffer, unless it would cost the second stream (32 channels at 16x16).
bool grad_turn(const Problem &p, int R, size_t max_smem) { return grad_layout(p, 1, R, true).total + 1024 <= max_smem; }

int grad_samples_per_block(const Problem &p, bool vjp, int64_t n, int num_sms, size_t max_smem) {
    const int R = grad_streams(p, vjp, max_smem), T = kGradThreads, OG = p.C / 8;
    const int64_t most = std::min<int64_t>(kGradMaxSamples, std::max<int64_t>(1, (n + num_sms - 1) / num_sms));
    int best = 1;
    double cost = 0.0;
    const bool turn = grad_turn(p, R, max_smem);
    for (int S = 1; S <= most && grad_layout(p, S, R, turn).total + 1024 <= max_smem; ++S) {
        const int half = (S * p.N + 1) / 2, full = R == 2 ? S * p.N : half;
        const double tiles = (OG * half + T - 1) / T + (OG * full + T - 1) / T;
        const double c = (tiles * 72.0 * p.C + (S * p.C * p.C / 2 + T - 1) / T * 9.0 * p.N * R) / S;
        if (S == 1 || c < cost) { cost = c; best = S; }
    }
    return best;
}

// Shared memory of the layout this kernel replaced: it decides which problems
// take this path (the others keep the plain kernels).
size_t grad_support_bytes(const Problem &p) {
    const int cmax = p.C > p.c_in ? p.C : p.c_in;
    size_t o = a16(4 * (size_t)(9 * p.C * cmax + p.C));
    o = a16(o + 2 * (size_t)9 * p.N);
    o = a16(o + 4 * (size_t)cmax * (p.N + 1));
    o = a16(o + 4 * (size_t)2 * p.C * (p.N + 1));
    o = a16(o + 4 * (size_t)2 * p.C * (p.N + 1));
    return a16(o + 4 * (size_t)p.C);
}

template <int C, int R, bool VJP>
int launch_grad_t(const Problem &p, int S, int blocks, const float *p32, const double *p64, const int8_t *configs,
                  int64_t n, double *O, const double *grad, int64_t K, double *part, float *scratch,
                  const LaunchEnv &env) {
    auto k = grad_fast_kernel<C, R, VJP>;
    const bool turn = grad_turn(p, R, env.max_smem);
    const size_t bytes = grad_layout(p, S, R, turn).total;
    if (int rc = allow_dynamic_smem(k, bytes, env)) return rc;
    k<<<blocks, kGradThreads, bytes, env.stream>>>(p, S, turn, p32, p64, configs, n, O, grad, K, part, scratch);
    const cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) {
        *env.msg = std::string("grad_fast_kernel: ") + cudaGetErrorString(e);
        return NQS_ERR_CUDA;
    }
    ++*env.launches;
    return NQS_OK;
}

// The scratch decides how many samples are in flight (the allocation-free
// entry point has a fixed array): fewer samples a block, then fewer blocks.
template <bool VJP>
int launch_grad_any(const Problem &p, const float *p32, const double *p64, const int8_t *configs, int64_t n, double *O,
                    const double *grad, double *part, void *scratch, size_t scratch_bytes, const LaunchEnv &env) {
    if (n == 0) return NQS_OK;
    const int64_t K = VJP ? vjp_chunk_samples(n) : 1, slots = (n + K - 1) / K;
    const int64_t fit = std::max<int64_t>(1, (int64_t)(scratch_bytes / grad_fast_scratch_bytes(p, 1)));
    int S = grad_samples_per_block(p, VJP, slots, env.num_sms, env.max_smem);
    if (fit < std::min<int64_t>((slots + S - 1) / S, env.num_sms) * S)
        S = (int)std::max<int64_t>(1, std::min<int64_t>(S, fit / env.num_sms));
    const int blocks = (int)std::min<int64_t>(std::min<int64_t>((slots + S - 1) / S, env.num_sms), std::max<int64_t>(1, fit / S));
    const int R = grad_streams(p, VJP, env.max_smem);
    float *ws = (float *)scratch;
    if constexpr (!VJP)
        if (R == 2)
            return p.C == 16 ? launch_grad_t<16, 2, false>(p, S, blocks, p32, p64, configs, n, O, grad, K, part, ws, env)
                             : launch_grad_t<32, 2, false>(p, S, blocks, p32, p64, configs, n, O, grad, K, part, ws, env);
    return p.C == 16 ? launch_grad_t<16, 1, VJP>(p, S, blocks, p32, p64, configs, n, O, grad, K, part, ws, env)
                     : launch_grad_t<32, 1, VJP>(p, S, blocks, p32, p64, configs, n, O, grad, K, part, ws, env);
}

}  // namespace

int64_t vjp_chunk_samples(int64_t n) { return std::max<int64_t>(1, (n + 1023) / 1024); }

int launch_vjp_reduce(const Problem &p, const double *part, int64_t n, double *out, const LaunchEnv &env) {
    const int64_t nq = (n + vjp_chunk_samples(n) - 1) / vjp_chunk_samples(n);
    vjp_reduce_kernel<<<(p.P + 127) / 128, 128, 0, env.stream>>>(part, nq, p.P, out);
    const cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) {
        *env.msg = std::string("vjp_reduce_kernel: ") + cudaGetErrorString(e);
        return NQS_ERR_CUDA;
    }
    ++*env.launches;
    return NQS_OK;
}

int launch_vjp_fast(const Problem &p, const float *p32, const double *p64, const int8_t *configs, int64_t n,
                    const double *grad, double *part, void *scratch, size_t scratch_bytes, const LaunchEnv &env) {
    return launch_grad_any<true>(p, p32, p64, configs, n, nullptr, grad, part, scratch, scratch_bytes, env);
}

int launch_grad_fast(const Problem &p, const float *p32, const double *p64, const int8_t *configs, int64_t n,
                     double *O, void *scratch, size_t scratch_bytes, const LaunchEnv &env) {
    return launch_grad_any<false>(p, p32, p64, configs, n, O, nullptr, nullptr, scratch, scratch_bytes, env);
}

int64_t grad_fast_samples(const Problem &p, bool vjp, int64_t n, int num_sms, size_t max_smem) {
    const int64_t S = grad_samples_per_block(p, vjp, n, num_sms, max_smem);
    return std::min<int64_t>((n + S - 1) / S, num_sms) * S;
}

bool grad_fast_supported(const Problem &p, size_t max_smem) {
    return p.net == NQS_NET_SILU && (p.C == 16 || p.C == 32) && grad_support_bytes(p) <= max_smem;
}

size_t grad_fast_scratch_bytes(const Problem &p, int64_t samples) {
    return (size_t)2 * p.n_layers * p.C * p.N * sizeof(float) * (size_t)samples;
}

}  // namespace nqs
