// Iso-contours of a distance field on the mesh (the iso-contours of the exact geodesic
// field that Section 2 cites as a use of exact distances, built from the field PCH
// computes).  On each face the field is taken as the linear interpolation of its three
// vertex distances; the contour at level L then crosses every edge whose ends lie on
// different sides of L (a vertex is inside when its distance is below L) at the
// interpolated point, and is one straight segment per crossed face and level.
// Entry point pch_iso_contours.
#include <algorithm>
#include <climits>
#include <cmath>
#include <cstring>
#include <vector>

#include "pch_host.h"

namespace pch {

// Order tests run on signed 64-bit images of the doubles (FP64 compares would run on the
// FP64 unit, at a 64th of the integer rate): images order as the values do, -0 counts as +0.
__host__ __device__ __forceinline__ long long order_image(long long bits) {
    return bits >= 0 ? bits : (bits == (long long)0x8000000000000000ull ? 0 : bits ^ 0x7fffffffffffffffll);
}
constexpr long long kImageMax = 0x7fefffffffffffffll;                            // the largest finite double
constexpr long long kImageMin = (long long)0xfff0000000000000ull ^ 0x7fffffffffffffffll;   // -infinity

// A face's corner images; false for a face with a corner that is not finite (no segment).
struct FaceImage {
    long long d[3], lo, hi;
};
__device__ __forceinline__ bool face_image(const int* __restrict__ tri, const double* __restrict__ dist, int f, FaceImage& I) {
#pragma unroll
    for (int i = 0; i < 3; ++i) I.d[i] = order_image(__double_as_longlong(dist[tri[3 * (size_t)f + i]]));
    I.lo = min(I.d[0], min(I.d[1], I.d[2]));
    I.hi = max(I.d[0], max(I.d[1], I.d[2]));
    return I.lo >= kImageMin && I.hi <= kImageMax;
}
// A level crosses the face when a corner is below it and another is not.
__device__ __forceinline__ bool crosses(const FaceImage& I, long long L) { return I.lo < L && I.hi >= L; }
__device__ __forceinline__ int crossed_levels(const int* __restrict__ tri, const double* __restrict__ dist,
                                              const long long* __restrict__ image, int n_levels, int f, FaceImage& I) {
    int c = 0;
    if (face_image(tri, dist, f, I))
        for (int l = 0; l < n_levels; ++l) c += crosses(I, image[l]) ? 1 : 0;
    return c;
}

// Both kernels give block b the faces [b C, (b + 1) C), C = ceil(nf / gridDim.x), 256 at a
// time.  Bound by memory: 12 bytes of vertex ids and three distance gathers (L2) a face,
// 32 bytes a segment.  With the order tests on the FP64 unit a call for 32 levels of
// 1,310,720 faces (62,860 segments to the host) took 1.54 ms; it takes 0.13.

// Segments of every block's faces, and of all.
__global__ void __launch_bounds__(256) k_contour_count(const int* __restrict__ tri, int nf, const double* __restrict__ dist,
                                                       const long long* __restrict__ image, int n_levels,
                                                       unsigned long long* __restrict__ block_count,
                                                       unsigned long long* total) {
    const long long C = ((long long)nf + gridDim.x - 1) / gridDim.x;
    const int f0 = (int)min((long long)nf, C * blockIdx.x), f1 = (int)min((long long)nf, C * (blockIdx.x + 1));
    unsigned long long t = 0;
    for (int f = f0 + threadIdx.x; f < f1; f += blockDim.x) {
        FaceImage I;
        t += (unsigned long long)crossed_levels(tri, dist, image, n_levels, f, I);
    }
    __shared__ unsigned long long sh[8];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
    if ((threadIdx.x & 31) == 0) sh[threadIdx.x / 32] = t;
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int q = 1; q < 8; ++q) t += sh[q];
        block_count[blockIdx.x] = t;
        if (t) atomicAdd(total, t);
    }
}

// One segment: from the crossing on the edge whose start corner is inside to the crossing on
// the edge whose start corner is outside, so that the inside (distance below L) lies to the
// left of the segment seen from the face's front side (corners counter-clockwise).
__device__ __forceinline__ pch_contour_segment segment(const int* __restrict__ tri, const double* __restrict__ dist,
                                                       const double* __restrict__ levels,
                                                       const long long* __restrict__ image, int f, int l) {
    double d[3];
    bool in[3];
    const long long Li = image[l];
    const double L = levels[l];
#pragma unroll
    for (int i = 0; i < 3; ++i) {
        d[i] = dist[tri[3 * (size_t)f + i]];
        in[i] = order_image(__double_as_longlong(d[i])) < Li;
    }
    pch_contour_segment sgm;
    sgm.level = l;
    sgm.face = f;
#pragma unroll
    for (int k = 0; k < 2; ++k) {
        const int i = in[0] == (k == 0) && in[1] != in[0] ? 0 : (in[1] == (k == 0) && in[2] != in[1] ? 1 : 2);
        const double a = i == 0 ? d[0] : (i == 1 ? d[1] : d[2]), b = i == 0 ? d[1] : (i == 1 ? d[2] : d[0]);
        sgm.half_edge[k] = 3 * f + i;
        sgm.t[k] = (L - a) / (b - a);
    }
    return sgm;
}

// Writes the segments in face order.  A block adds up the counts of the blocks before it
// and scans its own faces, so that no array of per-face offsets is written and scanned
// between the two kernels.  The faces of a tile first list their (face, level) pairs in
// shared memory; the divisions then run with every lane on a segment.  Nothing is written
// when all blocks together have more than 2^31 - 1 segments: the host refuses such a call,
// and the 32-bit offsets within a tile hold no more.
constexpr int kTileSegments = 2048;
__global__ void __launch_bounds__(256) k_contour_write(const int* __restrict__ tri, int nf, const double* __restrict__ dist,
                                                       const double* __restrict__ levels,
                                                       const long long* __restrict__ image, int n_levels,
                                                       const unsigned long long* __restrict__ block_count,
                                                       const unsigned long long* __restrict__ total,
                                                       long long capacity, pch_contour_segment* __restrict__ out) {
    if (*total > (unsigned long long)INT_MAX) return;
    const long long C = ((long long)nf + gridDim.x - 1) / gridDim.x;
    const int f0 = (int)min((long long)nf, C * blockIdx.x), f1 = (int)min((long long)nf, C * (blockIdx.x + 1));
    const int lane = threadIdx.x & 31, warp = threadIdx.x / 32;
    __shared__ unsigned long long sh[8];
    __shared__ int wsum[8];
    __shared__ int2 list[kTileSegments];
    unsigned long long before = 0;
    for (int b = threadIdx.x; b < (int)blockIdx.x; b += blockDim.x) before += block_count[b];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) before += __shfl_xor_sync(0xffffffffu, before, o);
    if (lane == 0) sh[warp] = before;
    __syncthreads();
    long long base = 0;
    for (int q = 0; q < 8; ++q) base += (long long)sh[q];
    for (int tile = f0; tile < f1 && base < capacity; tile += blockDim.x) {
        const int f = tile + threadIdx.x;
        FaceImage I;
        const int c = f < f1 ? crossed_levels(tri, dist, image, n_levels, f, I) : 0;
        int incl = c;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int t = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += t;
        }
        if (lane == 31) wsum[warp] = incl;
        __syncthreads();
        int at = incl - c, n = 0;
        for (int q = 0; q < 8; ++q) {
            if (q < warp) at += wsum[q];
            n += wsum[q];
        }
        const bool listed = n <= kTileSegments;
        if (c)
            for (int l = 0; l < n_levels; ++l) {
                if (!crosses(I, image[l])) continue;
                if (listed) list[at] = make_int2(f, l);
                else if (base + at < capacity) out[base + at] = segment(tri, dist, levels, image, f, l);
                ++at;
            }
        __syncthreads();
        if (listed)
            for (int j = threadIdx.x; j < n; j += blockDim.x)
                if (base + j < capacity) out[base + j] = segment(tri, dist, levels, image, list[j].x, list[j].y);
        base += n;
        __syncthreads();           // the list and the warps' sums are read
    }
}

}  // namespace pch

using namespace pch;

extern "C" pch_status pch_iso_contours(const pch_mesh* m, const double* dist, int32_t dist_on_device,
                                       const double* levels, int32_t n_levels, pch_contour_segment* segments,
                                       int64_t capacity, int64_t* n_segments) {
    clear_error();
    if (!m || !dist || !levels || n_levels <= 0 || !n_segments || capacity < 0 || (capacity > 0 && !segments))
        return set_error(PCH_ERR_INVALID_ARG, "null argument, no level or negative capacity");
    for (int l = 0; l < n_levels; ++l)
        if (!std::isfinite(levels[l])) return set_error(PCH_ERR_INVALID_ARG, "level %d is not finite", l);
    const int nf = m->dm.nf, nv = m->dm.nv;
    // one temporary: levels, block counts, total, the distances (host fields) and, when the
    // bound on their number is small, the segments; else these are allocated once counted
    struct {
        double *dist, *lev;
        long long* image;
        unsigned long long *count, *total;
        pch_contour_segment* seg;
    } t{};
    const cudaStream_t s = 0;
    const int grid = sm_count() * 8;
    const long long most = std::min<long long>(capacity, (long long)nf * n_levels);
    const bool at_once = most <= (64ll << 20) / (long long)sizeof(pch_contour_segment);
    auto carve = [&](Carver& c) {
        c.take(&t.lev, n_levels);
        c.take(&t.image, n_levels);
        c.take(&t.count, grid);
        c.take(&t.total, 1);
        if (!dist_on_device) c.take(&t.dist, nv);
        if (at_once) c.take(&t.seg, most);
    };
    std::vector<long long> image(n_levels);
    for (int l = 0; l < n_levels; ++l) {
        long long bits;
        std::memcpy(&bits, levels + l, sizeof bits);
        image[l] = order_image(bits);
    }
    Carver c;
    carve(c);
    void *tmp = nullptr, *seg_tmp = nullptr;
    unsigned long long total = 0;
    pch_status st = PCH_OK;
    cudaError_t e = tmp_alloc(&tmp, c.off, s);
    if (!e) {
        c = Carver{static_cast<char*>(tmp), 0};
        carve(c);
        e = cudaMemcpyAsync(t.lev, levels, sizeof(double) * (size_t)n_levels, cudaMemcpyHostToDevice, s);
        if (!e) e = cudaMemcpyAsync(t.image, image.data(), sizeof(long long) * (size_t)n_levels, cudaMemcpyHostToDevice, s);
        if (!e && !dist_on_device) e = cudaMemcpyAsync(t.dist, dist, sizeof(double) * (size_t)nv, cudaMemcpyHostToDevice, s);
        if (!e) e = cudaMemsetAsync(t.total, 0, sizeof(unsigned long long), s);
    }
    const double* dd = dist_on_device ? dist : t.dist;
    auto write = [&](long long room, pch_contour_segment* seg) {
        k_contour_write<<<grid, 256, 0, s>>>(m->dm.tri, nf, dd, t.lev, t.image, n_levels, t.count, t.total, room,
                                               seg);
        return cudaGetLastError();
    };
    if (!e) {
        k_contour_count<<<grid, 256, 0, s>>>(m->dm.tri, nf, dd, t.image, n_levels, t.count, t.total);
        e = cudaGetLastError();
        if (!e && at_once && most > 0) e = write(most, t.seg);
    }
    if (!e) e = cudaMemcpyAsync(&total, t.total, sizeof(unsigned long long), cudaMemcpyDeviceToHost, s);
    if (!e) e = cudaStreamSynchronize(s);
    if (!e && total > (unsigned long long)INT_MAX) {
        st = set_error(PCH_ERR_CAPACITY, "%llu contour segments exceed 2^31 - 1", total);
    } else if (!e) {
        const long long keep = std::min<long long>(capacity, (long long)total);
        if (!at_once && keep > 0) {
            e = tmp_alloc(&seg_tmp, sizeof(pch_contour_segment) * (size_t)keep, s);
            t.seg = static_cast<pch_contour_segment*>(seg_tmp);
            if (!e) e = write(keep, t.seg);
        }
        if (!e && keep > 0)
            e = cudaMemcpyAsync(segments, t.seg, sizeof(pch_contour_segment) * (size_t)keep, cudaMemcpyDeviceToHost, s);
        if (!e) e = cudaStreamSynchronize(s);
    }
    if (e) cudaStreamSynchronize(s);       // a call that fails leaves nothing in flight
    if (tmp) cudaFreeAsync(tmp, s);
    if (seg_tmp) cudaFreeAsync(seg_tmp, s);
    if (e) return set_error(e == cudaErrorMemoryAllocation ? PCH_ERR_OOM : PCH_ERR_CUDA, "iso-contours: %s",
                            cudaGetErrorString(e));
    if (st != PCH_OK) return st;
    *n_segments = (int64_t)total;
    return PCH_OK;
}
