// Learned selection controller: parameters, training kernels (forward, backward, Adam)
// and the FP64 peak microbenchmark.  The network and its role are described in
// controller.cuh; none of this has a counterpart in the paper, which fixes k by hand
// (Section 5.2).
#include <algorithm>
#include <climits>
#include <cmath>
#include <cstddef>
#include <cstdlib>
#include <mutex>
#include <vector>

#include "pch_host.h"
#include "solver.cuh"

namespace pch {

// Installed controller weights, one device buffer per device, each valid only in the
// context it was allocated in (a reset device loses its weights).
constexpr int kMaxDevices = 64;
struct DevPtrSlot {
    unsigned long long ctx = 0;   // current_context_id() when ptr was obtained; 0 = empty
    float* ptr = nullptr;
};
static DevPtrSlot g_mlp_slot[kMaxDevices];
static std::mutex g_mlp_mu;

// The current device's weights, or nullptr when none were installed in its current
// context: PCH_CONTROL_LEARNED then runs the plain control.
const float* mlp_device_params() {
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices) return nullptr;
    const unsigned long long ctx = current_context_id();
    std::lock_guard<std::mutex> lk(g_mlp_mu);
    const DevPtrSlot& sl = g_mlp_slot[dev];
    return (ctx != 0 && sl.ctx == ctx) ? sl.ptr : nullptr;
}

long long default_k() {
    const char* e = std::getenv("PCH_DEFAULT_K");
    if (e) {
        long long v = std::atoll(e);
        if (v > 0) return v;
    }
    return 24576;   // the paper's tuned range 16*2^10 .. 24*2^10 (Section 5.2)
}

int default_hops() {
    const char* e = std::getenv("PCH_DEFAULT_HOPS");
    if (e) {
        int v = std::atoi(e);
        if (v > 0) return v;
    }
    return 32;
}

int default_take_min() {
    const char* e = std::getenv("PCH_TAKE_MIN");
    if (e) {
        int v = std::atoi(e);
        if (v >= 1 && v <= 32) return v;
    }
    return 1;
}

int default_tail_cut() {
    const char* e = std::getenv("PCH_TAIL_CUT");
    if (e) {
        int v = std::atoi(e);
        if (v >= 0) return v;
    }
    return 0;
}

// Resident propagation blocks per SM: 512 threads per SM (16 warps of up to 128
// registers a thread fill the register file), unless PCH_PROP_BLOCKS_PER_SM says otherwise.
int default_prop_blocks_per_sm(int block) {
    const char* e = std::getenv("PCH_PROP_BLOCKS_PER_SM");
    if (e) {
        int v = std::atoi(e);
        if (v > 0 && v <= 32) return v;
    }
    return block >= 512 ? 1 : 512 / block;
}

// ---------------------------------------------------------------- training kernels
// Forward, backward and weight gradients of a batch in one pass over it.
//
// A block takes tiles of kTile samples: the three hidden layers are 64 x 64 x 64 products
// (FP32 FMA: the controller's arithmetic is FP32 throughout) of the weights, resident in shared
// memory, with activations that never leave it, 4 x 4 outputs a thread; the deltas replace
// the activations they belong to once these are used up, and each thread keeps the same
// 41 of the 9,985 weight gradients in registers over all tiles of its block.  Every sum
// over a layer's inputs keeps the order bias, input 0, 1, ...; the sums over samples are
// per block, and k_mlp_reduce adds the blocks in a fixed order (deterministic).
// What bounds it: shared memory (three wavefronts for every 16 FMA instructions of a warp) and
// the last, partly filled round of tiles (31,722 samples = 3.3 tiles an SM).  Two tiles at
// once on an SM, by two groups of threads with the weights in common, hide each other's
// barriers; the products use packed pairs of FMAs, so that their issue slots do not compete with
// the loads.  Before, one 64-thread block a sample re-read all weights from L2, and
// one thread a weight summed over all samples in turn: 31,722 samples took 2.41 ms and
// take 86 us (with the Adam step).
constexpr int kTile = 64;                // samples per tile
constexpr int kTilePad = kTile + 4;      // row stride of activations [neuron][sample]
constexpr int kMlpThreads = 256;         // 16 x 16 threads, 4 x 4 outputs each
constexpr int kGrid = 16;
// Tiles of n samples (n up to INT_MAX: the sum n + kTile - 1 would not hold).
__host__ __device__ constexpr int mlp_tile_count(int n) { return n / kTile + (n % kTile ? 1 : 0); }
static_assert(mlp_tile_count(1) == 1 && mlp_tile_count(kTile) == 1 && mlp_tile_count(kTile + 1) == 2, "tiles");
static_assert(mlp_tile_count(INT_MAX) == 1 << 25, "no overflow at the largest n");
static_assert(kHidden == 4 * kGrid && kTile == 4 * kGrid && kFeatures <= 2 * kGrid, "tile layout");

struct MlpTile {
    float x[kFeatures][kTilePad];
    float h0[kHidden][kTilePad], h1[kHidden][kTilePad], h2[kHidden][kTilePad];
    float dy[kTile];
};
struct MlpShared {
    // [input][4 (o mod 16) + o / 16]: the four outputs of a thread (o = tx + 16 q) are adjacent
    float w1[kFeatures][kHidden], w2[kHidden][kHidden], w3[kHidden][kHidden];
    float b1[kHidden], b2[kHidden], b3[kHidden], w4[kHidden];
    MlpTile tile0;
    // TRAIN only: [output][4 (i mod 16) + i / 16]; the second group's tile
    float t2[kHidden][kHidden], t3[kHidden][kHidden];
    MlpTile tile1;
};
static_assert(sizeof(MlpTile) >= sizeof(float) * kMlpParams, "the second group's gradients take its tile's place");
constexpr size_t kMlpForwardBytes = offsetof(MlpShared, t2);

__device__ __forceinline__ int mlp_perm(int o) { return 4 * (o & (kGrid - 1)) + o / kGrid; }

// Two FP32 multiply-adds an instruction (each rounded as by fmaf): half the issue slots.
__device__ __forceinline__ unsigned long long pair_f32(float a, float b) {
    unsigned long long r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
    return r;
}
__device__ __forceinline__ void fma_f32x2(unsigned long long& acc, unsigned long long a, unsigned long long b) {
    asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(acc) : "l"(a), "l"(b));
}

// acc[q][r] += sum over rows i in order of w[i][tx + 16 q] * in[i][4 ty + r]
// (PACKED: two samples an instruction; worth it where two groups of threads share the SM, with one
// group the latency counts: 512 samples 38.5 and 39.2 us)
template <int K, bool PACKED>
__device__ __forceinline__ void mlp_product(const float (*w)[kHidden], const float (*in)[kTilePad], float acc[4][4], int tx,
                                            int ty) {
    if constexpr (!PACKED) {
#pragma unroll 4
        for (int i = 0; i < K; ++i) {
            const float4 a = *reinterpret_cast<const float4*>(&in[i][4 * ty]);
            const float4 v = *reinterpret_cast<const float4*>(&w[i][4 * tx]);
            const float av[4] = {a.x, a.y, a.z, a.w}, wv[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
            for (int q = 0; q < 4; ++q)
#pragma unroll
                for (int r = 0; r < 4; ++r) acc[q][r] = fmaf(wv[q], av[r], acc[q][r]);
        }
        return;
    }
    unsigned long long sum[4][2];
#pragma unroll
    for (int q = 0; q < 4; ++q)
#pragma unroll
        for (int r = 0; r < 2; ++r) sum[q][r] = pair_f32(acc[q][2 * r], acc[q][2 * r + 1]);
#pragma unroll 4
    for (int i = 0; i < K; ++i) {
        const ulonglong2 a = *reinterpret_cast<const ulonglong2*>(&in[i][4 * ty]);
        const float4 v = *reinterpret_cast<const float4*>(&w[i][4 * tx]);
        const float wv[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const unsigned long long ww = pair_f32(wv[q], wv[q]);
            fma_f32x2(sum[q][0], ww, a.x);
            fma_f32x2(sum[q][1], ww, a.y);
        }
    }
#pragma unroll
    for (int q = 0; q < 4; ++q)
#pragma unroll
        for (int r = 0; r < 2; ++r)
            asm("mov.b64 {%0, %1}, %2;" : "=f"(acc[q][2 * r]), "=f"(acc[q][2 * r + 1]) : "l"(sum[q][r]));
}

// out = relu(w in + b); samples past `valid` get 0
template <int K, bool PACKED>
__device__ __forceinline__ void mlp_layer(const float (*w)[kHidden], const float* b, const float (*in)[kTilePad],
                                          float (*out)[kTilePad], int valid, int tx, int ty) {
    float acc[4][4];
#pragma unroll
    for (int q = 0; q < 4; ++q)
#pragma unroll
        for (int r = 0; r < 4; ++r) acc[q][r] = b[tx + kGrid * q];
    mlp_product<K, PACKED>(w, in, acc, tx, ty);
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        float v[4];
#pragma unroll
        for (int r = 0; r < 4; ++r) v[r] = 4 * ty + r < valid ? fmaxf(acc[q][r], 0.f) : 0.f;
        *reinterpret_cast<float4*>(&out[tx + kGrid * q][4 * ty]) = make_float4(v[0], v[1], v[2], v[3]);
    }
}

// grad[q][p] += sum over the tile's samples of d[tx + 16 q] * in[ty + 16 p]
template <int P>
__device__ __forceinline__ void mlp_outer(const float (*d)[kTilePad], const float (*in)[kTilePad], float grad[4][P], int rows,
                                          int tx, int ty) {
#pragma unroll 2
    for (int s = 0; s < kTile; s += 4) {
        float4 dv[4], iv[P];
#pragma unroll
        for (int q = 0; q < 4; ++q) dv[q] = *reinterpret_cast<const float4*>(&d[tx + kGrid * q][s]);
#pragma unroll
        for (int p = 0; p < P; ++p)
            iv[p] = *reinterpret_cast<const float4*>(&in[min(ty + kGrid * p, rows - 1)][s]);
#pragma unroll
        for (int q = 0; q < 4; ++q)
#pragma unroll
            for (int p = 0; p < P; ++p) {
                float g = grad[q][p];
                g = fmaf(dv[q].x, iv[p].x, g);
                g = fmaf(dv[q].y, iv[p].y, g);
                g = fmaf(dv[q].z, iv[p].z, g);
                grad[q][p] = fmaf(dv[q].w, iv[p].w, g);
            }
    }
}

// TRAIN: loss L = 0.5 mean((y - target)^2); part [gridDim.x][kMlpParams] gets the blocks'
// gradient sums, part_loss their sums of (y - target)^2.  Else y [n] gets the outputs.
// GROUPS: tiles that the block works on at once, each by kMlpThreads threads of its own.
template <bool TRAIN, int GROUPS>
__global__ void __launch_bounds__(GROUPS * kMlpThreads)
    k_mlp_tiles(const float* __restrict__ p, const float* __restrict__ x, const float* __restrict__ target, int n,
                float* __restrict__ y, float* __restrict__ part, double* __restrict__ part_loss) {
    extern __shared__ __align__(16) unsigned char mlp_smem[];
    MlpShared& S = *reinterpret_cast<MlpShared*>(mlp_smem);
    const int group = GROUPS > 1 ? threadIdx.x / kMlpThreads : 0, t = threadIdx.x % kMlpThreads;
    const int tx = t & (kGrid - 1), ty = t / kGrid;
    for (int j = threadIdx.x; j < kHidden * kFeatures; j += GROUPS * kMlpThreads)
        S.w1[j % kFeatures][mlp_perm(j / kFeatures)] = p[kMlpW1 + j];
    for (int j = threadIdx.x; j < kHidden * kHidden; j += GROUPS * kMlpThreads) {
        const int o = j / kHidden, i = j % kHidden;
        const float w2 = p[kMlpW2 + j], w3 = p[kMlpW3 + j];
        S.w2[i][mlp_perm(o)] = w2;
        S.w3[i][mlp_perm(o)] = w3;
        if (TRAIN) {
            S.t2[o][mlp_perm(i)] = w2;
            S.t3[o][mlp_perm(i)] = w3;
        }
    }
    if (threadIdx.x < kHidden) {
        S.b1[t] = p[kMlpB1 + t];
        S.b2[t] = p[kMlpB2 + t];
        S.b3[t] = p[kMlpB3 + t];
        S.w4[t] = p[kMlpW4 + t];
    }
    const float b4 = p[kMlpB4];
    float g3[4][4] = {}, g2[4][4] = {}, g1[4][2] = {};
    float gv = 0.f, gb4 = 0.f;      // one of W4, b3, b2, b1 (by thread / 64); b4
    double loss = 0.0;
    const int tiles = mlp_tile_count(n);
    MlpTile& T = group ? S.tile1 : S.tile0;
    auto sync = [&] {                // the group's barrier
        if (GROUPS == 1) __syncthreads();
        else asm volatile("bar.sync %0, %1;" ::"r"(1 + group), "n"(kMlpThreads) : "memory");
    };
    if (GROUPS > 1) __syncthreads(); // weights are loaded
    for (int tile = blockIdx.x + group * gridDim.x; tile < tiles; tile += GROUPS * gridDim.x) {
        const int s0 = tile * kTile, valid = min(kTile, n - s0);
        sync();                      // weights are loaded / the group's last tile is done
        for (int j = t; j < kTile * kFeatures; j += kMlpThreads)
            T.x[j % kFeatures][j / kFeatures] = j / kFeatures < valid ? x[(size_t)s0 * kFeatures + j] : 0.f;
        sync();
        mlp_layer<kFeatures, (GROUPS > 1)>(S.w1, S.b1, T.x, T.h0, valid, tx, ty);
        sync();
        mlp_layer<kHidden, (GROUPS > 1)>(S.w2, S.b2, T.h0, T.h1, valid, tx, ty);
        sync();
        mlp_layer<kHidden, (GROUPS > 1)>(S.w3, S.b3, T.h1, T.h2, valid, tx, ty);
        sync();
        if (t < kTile) {
            float o = b4;
#pragma unroll 8
            for (int i = 0; i < kHidden; ++i) o = fmaf(S.w4[i], T.h2[i][t], o);
            if (TRAIN) {
                const float want = t < valid ? target[s0 + t] : 0.f;
                const double e = t < valid ? (double)o - (double)want : 0.0;
                loss += e * e;
                T.dy[t] = t < valid ? (o - want) / (float)n : 0.f;
            } else if (t < valid) {
                y[s0 + t] = o;
            }
        }
        if (!TRAIN) continue;
        sync();
        const int row = t & (kHidden - 1), role = t / kHidden;
        if (role == 0) {
            for (int s = 0; s < kTile; ++s) gv = fmaf(T.dy[s], T.h2[row][s], gv);
        } else if (t == kHidden) {
            for (int s = 0; s < kTile; ++s) gb4 += T.dy[s];
        }
        sync();
        // d2 = dL/dz of the last hidden layer, in place of its activations
#pragma unroll
        for (int q = 0; q < 4; ++q)
#pragma unroll
            for (int r = 0; r < 4; ++r) {
                float& a = T.h2[tx + kGrid * q][4 * ty + r];
                a = a > 0.f ? T.dy[4 * ty + r] * S.w4[tx + kGrid * q] : 0.f;
            }
        sync();
        auto back = [&](const float (*w)[kHidden], const float (*d)[kTilePad], float (*h)[kTilePad], float grad[4][4],
                        int bias_role) {
            mlp_outer<4>(d, h, grad, kHidden, tx, ty);
            if (role == bias_role)
                for (int s = 0; s < kTile; ++s) gv += d[row][s];
            float acc[4][4] = {};
            mlp_product<kHidden, (GROUPS > 1)>(w, d, acc, tx, ty);
            sync();         // every thread has read h
#pragma unroll
            for (int q = 0; q < 4; ++q)
#pragma unroll
                for (int r = 0; r < 4; ++r) {
                    float& a = h[tx + kGrid * q][4 * ty + r];
                    a = a > 0.f ? acc[q][r] : 0.f;
                }
            sync();
        };
        back(S.t3, T.h2, T.h1, g3, 1);
        back(S.t2, T.h1, T.h0, g2, 2);
        mlp_outer<2>(T.h0, T.x, g1, kFeatures, tx, ty);
        if (role == 3)
            for (int s = 0; s < kTile; ++s) gv += T.h0[row][s];
    }
    if (!TRAIN) return;
    // the second group's sums to shared memory (its tile is done), the first adds them to its own
    __shared__ double sl[GROUPS][kMlpThreads / 32];
    float* other = reinterpret_cast<float*>(&S.tile1);
    float* out = part + (size_t)blockIdx.x * kMlpParams;
    auto put = [&](int at, float v) {
        if (group) other[at] = v;
        else out[at] = GROUPS > 1 ? v + other[at] : v;
    };
    auto put_all = [&] {
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const int o = tx + kGrid * q;
#pragma unroll
            for (int r = 0; r < 4; ++r) {
                put(kMlpW3 + o * kHidden + ty + kGrid * r, g3[q][r]);
                put(kMlpW2 + o * kHidden + ty + kGrid * r, g2[q][r]);
            }
#pragma unroll
            for (int r = 0; r < 2; ++r)
                if (ty + kGrid * r < kFeatures) put(kMlpW1 + o * kFeatures + ty + kGrid * r, g1[q][r]);
        }
        const int at[4] = {kMlpW4, kMlpB3, kMlpB2, kMlpB1};
        put(at[t / kHidden] + (t & (kHidden - 1)), gv);
        if (t == kHidden) put(kMlpB4, gb4);
    };
    if (GROUPS == 1) put_all();
    for (int o = 16; o > 0; o >>= 1) loss += __shfl_xor_sync(0xffffffffu, loss, o);
    if ((t & 31) == 0) sl[group][t / 32] = loss;     // (the first two warps of a group hold it)
    __syncthreads();
    if (GROUPS > 1) {
        if (group) put_all();
        __syncthreads();
        if (!group) put_all();
    }
    if (threadIdx.x == 0) {
        double sum = sl[0][0] + sl[0][1];
        if (GROUPS > 1) sum += sl[GROUPS - 1][0] + sl[GROUPS - 1][1];
        part_loss[blockIdx.x] = sum;
    }
}

// Adds the blocks' partial gradients (and losses) in a fixed order: four threads a weight,
// each every fourth block.
__global__ void __launch_bounds__(256) k_mlp_reduce(const float* __restrict__ part, const double* __restrict__ part_loss,
                                                    int blocks, int n, float* __restrict__ grad, float* __restrict__ loss) {
    __shared__ float sh[4][64];
    const int c = threadIdx.x & 63, seg = threadIdx.x / 64, q = blockIdx.x * 64 + c;
    float s = 0.f;
    if (q < kMlpParams) {
#pragma unroll 8
        for (int b = seg; b < blocks; b += 4) s += part[(size_t)b * kMlpParams + q];
    }
    sh[seg][c] = s;
    __syncthreads();
    if (seg == 0 && q < kMlpParams) grad[q] = (sh[0][c] + sh[1][c]) + (sh[2][c] + sh[3][c]);
    if (blockIdx.x == 0 && threadIdx.x >= 64 && threadIdx.x < 96) {
        double l = 0.0;
        for (int b = threadIdx.x - 64; b < blocks; b += 32) l += part_loss[b];
        for (int o = 16; o > 0; o >>= 1) l += __shfl_xor_sync(0xffffffffu, l, o);
        if (threadIdx.x == 64) *loss = (float)(0.5 * l / n);
    }
}

// Blocks of a training pass over n samples: one an SM at most.
static int mlp_blocks(int n) { return std::min(mlp_tile_count(n), sm_count()); }

// Launches the pass with `scratch` for mlp_blocks(n) partial results of kMlpParams floats, the
// losses (doubles) first.
static cudaError_t launch_backward(const float* params, const float* x, const float* target, int n, float* grad, float* loss,
                                   void* scratch, cudaStream_t s) {
    const int blocks = mlp_blocks(n);
    double* part_loss = static_cast<double*>(scratch);
    float* part = reinterpret_cast<float*>(part_loss + blocks);
    // Two tiles at once on an SM as soon as some SM has two: 31,722 samples 96.4 -> 86.2 us; with
    // one tile an SM at most the second group is only more threads to start (512 samples: 39.1
    // and 41.1 us).
    const bool two = mlp_tile_count(n) > blocks;
    const auto kernel = two ? k_mlp_tiles<true, 2> : k_mlp_tiles<true, 1>;
    const size_t smem = two ? sizeof(MlpShared) : offsetof(MlpShared, tile1);
    cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e) return e;
    kernel<<<blocks, (two ? 2 : 1) * kMlpThreads, smem, s>>>(params, x, target, n, nullptr, part, part_loss);
    k_mlp_reduce<<<(kMlpParams + 63) / 64, 256, 0, s>>>(part, part_loss, blocks, n, grad, loss);
    return cudaGetLastError();
}
static size_t backward_bytes(int blocks) { return (size_t)blocks * (sizeof(double) + sizeof(float) * kMlpParams); }

__global__ void k_mlp_adam(float* p, const float* __restrict__ g, float* m, float* v, int t, float lr) {
    const float b1 = 0.9f, b2 = 0.999f, eps = 1e-8f;
    const float c1 = 1.f - powf(b1, (float)t), c2 = 1.f - powf(b2, (float)t);
    for (int q = blockIdx.x * blockDim.x + threadIdx.x; q < kMlpParams; q += gridDim.x * blockDim.x) {
        float gq = g[q];
        float mq = b1 * m[q] + (1.f - b1) * gq;
        float vq = b2 * v[q] + (1.f - b2) * gq * gq;
        m[q] = mq;
        v[q] = vq;
        p[q] -= lr * (mq / c1) / (sqrtf(vq / c2) + eps);
    }
}

// ---------------------------------------------------------------- FP64 peak
__global__ void k_dfma_peak(double* out, int iters) {
    double a0 = threadIdx.x * 1e-9, a1 = a0 + 1e-3, a2 = a0 + 2e-3, a3 = a0 + 3e-3;
    double a4 = a0 + 4e-3, a5 = a0 + 5e-3, a6 = a0 + 6e-3, a7 = a0 + 7e-3;
    const double m = 0.999999, c = 1e-7;
    for (int i = 0; i < iters; ++i) {
        a0 = fma(a0, m, c); a1 = fma(a1, m, c); a2 = fma(a2, m, c); a3 = fma(a3, m, c);
        a4 = fma(a4, m, c); a5 = fma(a5, m, c); a6 = fma(a6, m, c); a7 = fma(a7, m, c);
    }
    double s = a0 + a1 + a2 + a3 + a4 + a5 + a6 + a7;
    if (s == 12345.678) out[0] = s;   // keep the chains alive
}

}  // namespace pch

using namespace pch;

extern "C" int32_t pch_mlp_num_features(void) { return kFeatures; }
extern "C" int32_t pch_mlp_num_params(void) { return kMlpParams; }

extern "C" pch_status pch_mlp_set_weights(const float* params, int32_t n_params) {
    clear_error();
    if (!params || n_params != kMlpParams) return set_error(PCH_ERR_INVALID_ARG, "expected %d parameters", kMlpParams);
    for (int i = 0; i < n_params; ++i)
        if (!std::isfinite(params[i])) return set_error(PCH_ERR_INVALID_ARG, "non-finite weight %d", i);
    int dev = 0;
    PCH_CUDA(cudaGetDevice(&dev));
    if (dev < 0 || dev >= kMaxDevices) return set_error(PCH_ERR_INVALID_ARG, "device id %d out of range", dev);
    std::lock_guard<std::mutex> lk(g_mlp_mu);
    DevPtrSlot& sl = g_mlp_slot[dev];
    unsigned long long ctx = current_context_id();
    if (ctx == 0 || sl.ctx != ctx) {
        // first weights in this device's current context (a buffer of an earlier, destroyed
        // context is gone with it and is not freed)
        float* p = nullptr;
        PCH_CUDA(cudaMalloc(&p, sizeof(float) * kMlpParams));
        sl.ptr = p;
        sl.ctx = current_context_id();   // the allocation made the context current
    }
    PCH_CUDA(cudaMemcpy(sl.ptr, params, sizeof(float) * kMlpParams, cudaMemcpyHostToDevice));
    return PCH_OK;
}

extern "C" pch_status pch_mlp_forward(const float* params_dev, const float* x_dev, int32_t n, float* y_dev,
                                      void* stream) {
    clear_error();
    if (!params_dev || !x_dev || !y_dev || n <= 0) return set_error(PCH_ERR_INVALID_ARG, "bad arguments");
    cudaStream_t s = (cudaStream_t)stream;
    PCH_CUDA(cudaFuncSetAttribute(k_mlp_tiles<false, 1>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kMlpForwardBytes));
    const int blocks = std::min(mlp_tile_count(n), 2 * sm_count());
    k_mlp_tiles<false, 1><<<blocks, kMlpThreads, kMlpForwardBytes, s>>>(params_dev, x_dev, nullptr, n, y_dev, nullptr, nullptr);
    PCH_CUDA(cudaGetLastError());
    return PCH_OK;
}

extern "C" pch_status pch_mlp_backward(const float* params_dev, const float* x_dev, const float* target_dev, int32_t n,
                                       float* grad_dev, float* loss_dev, void* stream) {
    clear_error();
    if (!params_dev || !x_dev || !target_dev || !grad_dev || !loss_dev || n <= 0)
        return set_error(PCH_ERR_INVALID_ARG, "bad arguments");
    cudaStream_t s = (cudaStream_t)stream;
    void* scratch = nullptr;
    PCH_CUDA(tmp_alloc(&scratch, backward_bytes(mlp_blocks(n)), s));
    cudaError_t e = launch_backward(params_dev, x_dev, target_dev, n, grad_dev, loss_dev, scratch, s);
    cudaFreeAsync(scratch, s);
    PCH_CUDA(e);
    return PCH_OK;
}

extern "C" pch_status pch_mlp_adam(float* params_dev, const float* grad_dev, float* m_dev, float* v_dev, int32_t t,
                                   float lr, void* stream) {
    clear_error();
    if (!params_dev || !grad_dev || !m_dev || !v_dev || t < 1) return set_error(PCH_ERR_INVALID_ARG, "bad arguments");
    k_mlp_adam<<<(kMlpParams + 255) / 256, 256, 0, (cudaStream_t)stream>>>(params_dev, grad_dev, m_dev, v_dev, t, lr);
    PCH_CUDA(cudaGetLastError());
    return PCH_OK;
}

extern "C" pch_status pch_measure_fp64_peak(double* tflops) {
    clear_error();
    if (!tflops) return set_error(PCH_ERR_INVALID_ARG, "null output");
    double* out = nullptr;
    PCH_CUDA(cudaMalloc(&out, sizeof(double)));
    const int blocks = sm_count() * 8, threads = 256, iters = 1 << 14;
    cudaEvent_t a, b;
    cudaEventCreate(&a);
    cudaEventCreate(&b);
    k_dfma_peak<<<blocks, threads>>>(out, 256);   // warm-up
    cudaEventRecord(a);
    k_dfma_peak<<<blocks, threads>>>(out, iters);
    cudaEventRecord(b);
    cudaError_t e = cudaEventSynchronize(b);
    float ms = 0.f;
    cudaEventElapsedTime(&ms, a, b);
    cudaEventDestroy(a);
    cudaEventDestroy(b);
    cudaFree(out);
    PCH_CUDA(e);
    double flops = 2.0 * 8.0 * (double)iters * blocks * threads;
    *tflops = flops / (ms * 1e-3) / 1e12;
    return PCH_OK;
}

// ---------------------------------------------------------------- allocation-free backward
// Scratch of pch_mlp_backward_noalloc, in a file-scope device array instead of a
// stream-ordered allocation: the partial results of the blocks of at most
// kNoAllocMaxSamples samples (2.6 MB).  Every GPU that loads the library holds this array
// until the process exits.
namespace pch {
constexpr int kNoAllocMaxSamples = 4096;
constexpr size_t kNoAllocBlocks = mlp_tile_count(kNoAllocMaxSamples);
static __device__ __align__(256) unsigned char g_noalloc_scratch[kNoAllocBlocks * (sizeof(double) + sizeof(float) * kMlpParams)];
// Host side: the array's device address, resolved once per device and context (a reset
// device gets a new context, and the array a new address).  The symbol itself is only a
// host-side stand-in and must never be handed to a kernel.
static DevPtrSlot g_noalloc_slot[kMaxDevices];
static std::mutex g_noalloc_mu;
}  // namespace pch

extern "C" pch_status pch_mlp_backward_noalloc(const float* params_dev, const float* x_dev, const float* target_dev,
                                               int32_t n, float* grad_dev, float* loss_dev, void* stream) {
    clear_error();
    if (!params_dev || !x_dev || !target_dev || !grad_dev || !loss_dev || n <= 0)
        return set_error(PCH_ERR_INVALID_ARG, "bad arguments");
    if (n > kNoAllocMaxSamples)
        return set_error(PCH_ERR_CAPACITY, "pch_mlp_backward_noalloc takes at most %d samples (got %d)",
                         kNoAllocMaxSamples, n);
    int dev = 0;
    PCH_CUDA(cudaGetDevice(&dev));
    if (dev < 0 || dev >= kMaxDevices) return set_error(PCH_ERR_INVALID_ARG, "device id %d out of range", dev);
    void* scratch = nullptr;
    {
        std::lock_guard<std::mutex> lk(g_noalloc_mu);
        DevPtrSlot& sl = g_noalloc_slot[dev];
        const unsigned long long ctx = current_context_id();
        if (ctx != 0 && sl.ctx == ctx) {
            scratch = sl.ptr;
        } else {
            // first call on this device in its current context (the device is current):
            // look the array up
            void* p = nullptr;
            cudaError_t e = cudaGetSymbolAddress(&p, g_noalloc_scratch);
            if (e != cudaSuccess || p == nullptr)
                return set_error(PCH_ERR_CUDA, "cudaGetSymbolAddress of the scratch array failed: %s",
                                 cudaGetErrorString(e));
            scratch = p;
            sl.ptr = static_cast<float*>(p);
            sl.ctx = current_context_id();
        }
    }
    cudaStream_t s = (cudaStream_t)stream;
    // every scratch element read is written first by the same call: nothing to clear
    PCH_CUDA(launch_backward(params_dev, x_dev, target_dev, n, grad_dev, loss_dev, scratch, s));
    return PCH_OK;
}
