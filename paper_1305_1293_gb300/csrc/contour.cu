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
#include <vector>

#include "pch_host.h"

namespace pch {

__device__ __forceinline__ bool finite_d(double x) { return x <= 1.7976931348623157e308; }

// Crossing mask of face f at level L: bit i set when half-edge 3f+i (corner i -> corner
// i+1) has its ends on different sides.  A face with a non-finite distance has none.
__device__ __forceinline__ int face_mask(const double d[3], double L) {
    if (!(finite_d(d[0]) && finite_d(d[1]) && finite_d(d[2]))) return 0;
    int m = 0;
#pragma unroll
    for (int i = 0; i < 3; ++i)
        if ((d[i] < L) != (d[(i + 1) % 3] < L)) m |= 1 << i;
    return m;
}

__device__ __forceinline__ void face_dist(const int* __restrict__ tri, const double* __restrict__ dist, int f,
                                          double d[3]) {
#pragma unroll
    for (int i = 0; i < 3; ++i) d[i] = dist[tri[3 * f + i]];
}

// Both kernels give block b the faces [b C, (b + 1) C), C = ceil(nf / gridDim.x), 256 at a
// time.  Bound by memory: 12 bytes of vertex ids and three distance gathers (L2) a face,
// 32 bytes a segment.
__device__ __forceinline__ int crossed_levels(const int* __restrict__ tri, const double* __restrict__ dist,
                                              const double* __restrict__ levels, int n_levels, int f, double d[3]) {
    face_dist(tri, dist, f, d);
    int c = 0;
    for (int l = 0; l < n_levels; ++l) c += face_mask(d, levels[l]) != 0;
    return c;
}

// Segments of every block's faces, and of all.
__global__ void __launch_bounds__(256) k_contour_count(const int* __restrict__ tri, int nf, const double* __restrict__ dist,
                                                       const double* __restrict__ levels, int n_levels,
                                                       unsigned long long* __restrict__ block_count,
                                                       unsigned long long* total) {
    const long long C = ((long long)nf + gridDim.x - 1) / gridDim.x;
    const int f0 = (int)min((long long)nf, C * blockIdx.x), f1 = (int)min((long long)nf, C * (blockIdx.x + 1));
    unsigned long long t = 0;
    for (int f = f0 + threadIdx.x; f < f1; f += blockDim.x) {
        double d[3];
        t += (unsigned long long)crossed_levels(tri, dist, levels, n_levels, f, d);
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

// Segment endpoints: from the crossing on the edge whose start corner is inside to the
// crossing on the edge whose start corner is outside, so that the inside (distance
// below L) lies to the left of the segment seen from the face's front side (corners
// counter-clockwise).
//
// A block adds up the counts of the blocks before it and scans its own faces, so that no
// array of per-face offsets is written and scanned between the two kernels.
__global__ void __launch_bounds__(256) k_contour_write(const int* __restrict__ tri, int nf, const double* __restrict__ dist,
                                                       const double* __restrict__ levels, int n_levels,
                                                       const unsigned long long* __restrict__ block_count,
                                                       long long capacity, pch_contour_segment* __restrict__ out) {
    const long long C = ((long long)nf + gridDim.x - 1) / gridDim.x;
    const int f0 = (int)min((long long)nf, C * blockIdx.x), f1 = (int)min((long long)nf, C * (blockIdx.x + 1));
    const int lane = threadIdx.x & 31, warp = threadIdx.x / 32;
    __shared__ unsigned long long sh[8];
    __shared__ int wsum[8];
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
        double d[3] = {0.0, 0.0, 0.0};
        const int c = f < f1 ? crossed_levels(tri, dist, levels, n_levels, f, d) : 0;
        int incl = c;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int t = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += t;
        }
        if (lane == 31) wsum[warp] = incl;
        __syncthreads();
        long long o = base + incl - c;
        for (int q = 0; q < 8; ++q) {
            if (q < warp) o += wsum[q];
            base += wsum[q];
        }
        __syncthreads();
        if (c == 0) continue;
        for (int l = 0; l < n_levels; ++l) {
            const double L = levels[l];
            const int m = face_mask(d, L);
            if (!m) continue;
            if (o < capacity) {
                pch_contour_segment sgm;
                sgm.level = l;
                sgm.face = f;
                int k = 0;
                // first the edge leaving the inside, then the edge entering it
                for (int pass = 0; pass < 2; ++pass)
                    for (int i = 0; i < 3; ++i) {
                        if (!(m >> i & 1)) continue;
                        const bool start_inside = d[i] < L;
                        if (start_inside != (pass == 0)) continue;
                        const double a = d[i], b = d[(i + 1) % 3];
                        sgm.half_edge[k] = 3 * f + i;
                        sgm.t[k] = (L - a) / (b - a);
                        ++k;
                    }
                out[o] = sgm;
            }
            ++o;
        }
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
        unsigned long long *count, *total;
        pch_contour_segment* seg;
    } t{};
    const cudaStream_t s = 0;
    const int grid = sm_count() * 8;
    const long long most = std::min<long long>(capacity, (long long)nf * n_levels);
    const bool at_once = most <= (64ll << 20) / (long long)sizeof(pch_contour_segment);
    auto carve = [&](Carver& c) {
        c.take(&t.lev, n_levels);
        c.take(&t.count, grid);
        c.take(&t.total, 1);
        if (!dist_on_device) c.take(&t.dist, nv);
        if (at_once) c.take(&t.seg, most);
    };
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
        if (!e && !dist_on_device) e = cudaMemcpyAsync(t.dist, dist, sizeof(double) * (size_t)nv, cudaMemcpyHostToDevice, s);
        if (!e) e = cudaMemsetAsync(t.total, 0, sizeof(unsigned long long), s);
    }
    const double* dd = dist_on_device ? dist : t.dist;
    auto write = [&](long long room, pch_contour_segment* seg) {
        k_contour_write<<<grid, 256, 0, s>>>(m->dm.tri, nf, dd, t.lev, n_levels, t.count, room, seg);
        return cudaGetLastError();
    };
    if (!e) {
        k_contour_count<<<grid, 256, 0, s>>>(m->dm.tri, nf, dd, t.lev, n_levels, t.count, t.total);
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
    if (tmp) cudaFreeAsync(tmp, s);
    if (seg_tmp) cudaFreeAsync(seg_tmp, s);
    if (e) return set_error(e == cudaErrorMemoryAllocation ? PCH_ERR_OOM : PCH_ERR_CUDA, "iso-contours: %s",
                            cudaGetErrorString(e));
    if (st != PCH_OK) return st;
    *n_segments = (int64_t)total;
    return PCH_OK;
}
