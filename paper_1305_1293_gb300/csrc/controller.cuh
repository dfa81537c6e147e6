// Learned selection controller: device-side features and inference.
//
// The paper controls each iteration with a fixed window count k (Section 4.2, Step 1;
// the trade-off of Section 5.2, Fig. `fig:parameter`).  This controller replaces the
// fixed k by a 3 x 64 hidden-layer fp32 MLP that maps the frontier statistics of one
// instance to log2 of the number of windows to select, divided by 24.  Any window order
// gives the same distances (Section 4.3, Remark 2), so the controller can change speed,
// never results; an output outside 2^12 to 2^24 windows is clamped, and only one that is not
// finite falls back to the plain k.
#pragma once
#include "pch_common.cuh"

namespace pch {

// Parameter layout: W1[64][24] b1[64] W2[64][64] b2[64] W3[64][64] b3[64] W4[64] b4[1].
constexpr int kMlpW1 = 0;
constexpr int kMlpB1 = kMlpW1 + kHidden * kFeatures;
constexpr int kMlpW2 = kMlpB1 + kHidden;
constexpr int kMlpB2 = kMlpW2 + kHidden * kHidden;
constexpr int kMlpW3 = kMlpB2 + kHidden;
constexpr int kMlpB3 = kMlpW3 + kHidden * kHidden;
constexpr int kMlpW4 = kMlpB3 + kHidden;
constexpr int kMlpB4 = kMlpW4 + kHidden;
constexpr int kMlpParams = kMlpB4 + 1;

// Frontier statistics of one instance at the start of an iteration (row a8):
//  f0      log2(1 + pending) / 20
//  f1..16  cumulative fraction of pending windows within 2^j/4 mean edge lengths of the
//          reference (the nearest pending key), j = 0..15 (octave-coarsened histogram)
//  f17     log2(faces) / 24
//  f18     log2(mean edge length) / 8
//  f19     log2(1 + iteration) / 16
//  f20     windows created (before their filters) per selected one in the previous iteration / 4
//  f21     log2(1 + front distance / mean edge length) / 16
//  f22     log2(1 + pending / faces) / 8
//  f23     1
// `prefix`: inclusive sums of the 256-bin histogram.  Called by the first kFeatures threads
// of a block.
__device__ __forceinline__ void controller_features(const InstCtl& c, const Inst& I, const unsigned* prefix, int np,
                                                    int it, float* f) {
    const int j = threadIdx.x;
    const float faces = (float)(I.nh / 3);
    float v = 1.f;
    if (j == 0) v = log2f(1.f + (float)np) / 20.f;
    else if (j <= 16) v = np > 0 ? (float)prefix[16 * j - 1] / (float)np : 0.f;
    else if (j == 17) v = log2f(faces) / 24.f;
    else if (j == 18) v = log2f((float)I.lbar) / 8.f;
    else if (j == 19) v = log2f(1.f + (float)it) / 16.f;
    else if (j == 20) v = c.last_ratio / 4.f;
    else if (j == 21) v = log2f(1.f + (float)(c.ref * I.ilbar)) / 16.f;
    else if (j == 22) v = log2f(1.f + (float)np / faces) / 8.f;
    f[j] = v;
}

// Block-cooperative forward pass, four threads a neuron (4 * kHidden threads).  The
// control kernel is one block that waits for memory: a thread's weights of all layers are
// loaded together by `load`, before the features are made, so that their latency is paid
// once (with one thread a neuron, layer by layer, a 1M-face torus took 21.26 ms, with this
// 20.92).  `x` (kFeatures) and `h` (kHidden, every layer's values in turn) live in shared
// memory; every thread of the block calls both.
struct MlpRows {
    float w1[kFeatures / 4], w2[kHidden / 4], w3[kHidden / 4], w4, b1, b2, b3, b4;

    __device__ __forceinline__ void load(const float* __restrict__ p) {
        const int n = threadIdx.x >> 2, q = threadIdx.x & 3;
        if (n >= kHidden) return;
#pragma unroll
        for (int j = 0; j < kFeatures / 4; ++j) w1[j] = p[kMlpW1 + n * kFeatures + 4 * j + q];
#pragma unroll
        for (int j = 0; j < kHidden / 4; ++j) w2[j] = p[kMlpW2 + n * kHidden + 4 * j + q];
#pragma unroll
        for (int j = 0; j < kHidden / 4; ++j) w3[j] = p[kMlpW3 + n * kHidden + 4 * j + q];
        b1 = p[kMlpB1 + n];
        b2 = p[kMlpB2 + n];
        b3 = p[kMlpB3 + n];
        w4 = p[kMlpW4 + n];
        b4 = p[kMlpB4];
    }
    // The output, for thread 0.
    __device__ __forceinline__ float forward(const float* x, float* h) {
        const int n = threadIdx.x >> 2, q = threadIdx.x & 3;
        const unsigned full = 0xffffffffu;
        float s = 0.f;
#pragma unroll
        for (int j = 0; j < kFeatures / 4; ++j) s = fmaf(w1[j], x[4 * j + q], s);
        s += __shfl_xor_sync(full, s, 1);
        s += __shfl_xor_sync(full, s, 2);
        if (q == 0) h[n] = fmaxf(s + b1, 0.f);
        __syncthreads();
        s = 0.f;
#pragma unroll
        for (int j = 0; j < kHidden / 4; ++j) s = fmaf(w2[j], h[4 * j + q], s);
        s += __shfl_xor_sync(full, s, 1);
        s += __shfl_xor_sync(full, s, 2);
        __syncthreads();
        if (q == 0) h[n] = fmaxf(s + b2, 0.f);
        __syncthreads();
        s = 0.f;
#pragma unroll
        for (int j = 0; j < kHidden / 4; ++j) s = fmaf(w3[j], h[4 * j + q], s);
        s += __shfl_xor_sync(full, s, 1);
        s += __shfl_xor_sync(full, s, 2);
        __syncthreads();
        if (q == 0) h[n] = fmaxf(s + b3, 0.f) * w4;
        __syncthreads();
        s = 0.f;
        if (threadIdx.x < 32) {
            s = h[threadIdx.x] + h[threadIdx.x + 32];
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(full, s, o);
        }
        return s + b4;
    }
};
static_assert(kFeatures % 4 == 0 && kHidden == 64, "four threads a neuron, the output by one warp");

}  // namespace pch
