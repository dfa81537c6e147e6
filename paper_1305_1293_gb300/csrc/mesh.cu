// Mesh preparation on the device (Section 4.1): half-edge table, edge lengths,
// per-half-edge unfolding frames, one-ring order, total angles and the saddle /
// boundary classification of Section 3.  Entry points pch_create_mesh, pch_mesh_info,
// pch_destroy, pch_last_error.
#include <algorithm>
#include <cmath>
#include <cstring>
#include <mutex>
#include <string>
#include <vector>

#include "pch_host.h"
#include "radix.cuh"

namespace pch {

static thread_local std::string g_err;

pch_status set_error(pch_status st, const char* fmt, ...) {
    char buf[512];
    va_list ap;
    va_start(ap, fmt);
    vsnprintf(buf, sizeof buf, fmt, ap);
    va_end(ap);
    g_err = buf;
    return st;
}
void clear_error() { g_err.clear(); }

int sm_count() {
    static int cached = -1;
    static int cached_dev = -1;
    int dev = 0;
    cudaGetDevice(&dev);
    if (cached < 0 || dev != cached_dev) {
        cudaDeviceGetAttribute(&cached, cudaDevAttrMultiProcessorCount, dev);
        cached_dev = dev;
    }
    return cached;
}

// The driver's cuCtxGetCurrent / cuCtxGetId, reached through the runtime so that the
// library does not link libcuda (it must load on a machine without a GPU driver).
typedef int (*CtxGetCurrentFn)(void**);
typedef int (*CtxGetIdFn)(void*, unsigned long long*);

unsigned long long current_context_id() {
    static CtxGetCurrentFn get_current = nullptr;
    static CtxGetIdFn get_id = nullptr;
    static std::once_flag once;
    std::call_once(once, [] {
        void* f = nullptr;
        cudaDriverEntryPointQueryResult q = cudaDriverEntryPointSymbolNotFound;
        if (cudaGetDriverEntryPointByVersion("cuCtxGetCurrent", &f, 12000, cudaEnableDefault, &q) == cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            get_current = reinterpret_cast<CtxGetCurrentFn>(f);
        f = nullptr;
        if (cudaGetDriverEntryPointByVersion("cuCtxGetId", &f, 12000, cudaEnableDefault, &q) == cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            get_id = reinterpret_cast<CtxGetIdFn>(f);
    });
    if (!get_current || !get_id) return 0;
    void* ctx = nullptr;
    if (get_current(&ctx) != 0 || !ctx) return 0;
    unsigned long long id = 0;
    return get_id(ctx, &id) == 0 ? id : 0;
}

// ---------------------------------------------------------------- device memory
struct PoolSlot {
    unsigned long long ctx = 0;       // current_context_id() when the pool was made
    cudaMemPool_t pool = nullptr;
    cudaStream_t stream = nullptr;    // orders the allocations of blocks that any stream uses
    int blocks = 0;                   // dev_alloc blocks that live in it
};
constexpr int kMaxPoolDevices = 64;
// the pools of each device, one a context (those of a destroyed context are gone with it);
// never destroyed, as a mesh may be released while the process exits
static std::vector<PoolSlot>* const g_pools = new std::vector<PoolSlot>[kMaxPoolDevices];
static std::mutex g_pool_mu;

// The current device's pool in its current context.  Call with g_pool_mu held; the slot is
// valid until it is released.
static cudaError_t current_pool(PoolSlot** out) {
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e) return e;
    if (dev < 0 || dev >= kMaxPoolDevices) return cudaErrorInvalidDevice;
    unsigned long long ctx = current_context_id();
    if (ctx == 0) {                   // make the device's primary context current
        if ((e = cudaFree(nullptr))) return e;
        ctx = current_context_id();
    }
    if (ctx != 0)
        for (PoolSlot& sl : g_pools[dev])
            if (sl.ctx == ctx) {
                *out = &sl;
                return cudaSuccess;
            }
    PoolSlot fresh;
    cudaMemPoolProps props{};
    props.allocType = cudaMemAllocationTypePinned;
    props.location.type = cudaMemLocationTypeDevice;
    props.location.id = dev;
    if ((e = cudaMemPoolCreate(&fresh.pool, &props))) return e;
    unsigned long long keep = kPoolKeep;
    e = cudaMemPoolSetAttribute(fresh.pool, cudaMemPoolAttrReleaseThreshold, &keep);
    if (!e) e = cudaStreamCreateWithFlags(&fresh.stream, cudaStreamNonBlocking);
    if (e) {
        cudaMemPoolDestroy(fresh.pool);
        return e;
    }
    fresh.ctx = ctx;
    g_pools[dev].push_back(fresh);
    *out = &g_pools[dev].back();
    return cudaSuccess;
}

// Memory that the pool keeps, back to the driver (what is in use stays).  Done when the last
// block is freed: a mesh loaded, solved and destroyed with no other alive takes 3.61 ms with
// it and 3.37 without (81,920 faces), and the memory is another program's to use.
static void trim(const PoolSlot& ps) {
    cudaStreamSynchronize(ps.stream);
    cudaMemPoolTrimTo(ps.pool, 0);
}

cudaError_t dev_alloc(DevMem& m, size_t bytes) {
    m.bytes = bytes ? bytes : 1;
    m.pooled = m.bytes <= kPoolKeep / 2;
    std::lock_guard<std::mutex> lk(g_pool_mu);
    PoolSlot* ps = nullptr;
    cudaError_t e = current_pool(&ps);
    for (int attempt = 0; attempt < 2 && !e; ++attempt) {
        if (m.pooled) {
            e = cudaMallocFromPoolAsync(&m.p, m.bytes, ps->pool, ps->stream);
            if (!e) e = cudaStreamSynchronize(ps->stream);
        } else {
            e = cudaMalloc(&m.p, m.bytes);
        }
        if (e != cudaErrorMemoryAllocation || attempt) break;
        cudaGetLastError();           // once more without what the pool keeps
        trim(*ps);
        e = cudaSuccess;
    }
    if (e) {
        cudaGetLastError();           // (reported by the caller, not by the next launch)
        m = DevMem{};
        return e;
    }
    cudaGetDevice(&m.dev);
    m.ctx = ps->ctx;
    if (m.pooled) ++ps->blocks;
    return e;
}

void dev_free(DevMem& m) {
    if (m.p) {
        int cur = 0;
        cudaGetDevice(&cur);
        if (cur != m.dev) cudaSetDevice(m.dev);
        {
            std::lock_guard<std::mutex> lk(g_pool_mu);
            PoolSlot* ps = nullptr;
            if (current_pool(&ps) == cudaSuccess && ps->ctx == m.ctx) {   // else: gone with its context
                if (m.pooled) {
                    cudaFreeAsync(m.p, ps->stream);
                    if (--ps->blocks == 0) trim(*ps);
                } else {
                    cudaFree(m.p);
                }
            }
        }
        if (cur != m.dev) cudaSetDevice(cur);
    }
    m = DevMem{};
}

cudaError_t tmp_alloc(void** p, size_t bytes, cudaStream_t s) {
    // a captured allocation belongs to the graph, and a pool cannot be made while a stream is
    // captured (the legacy stream never is)
    cudaStreamCaptureStatus capture = cudaStreamCaptureStatusNone;
    if (s && s != cudaStreamLegacy && cudaStreamIsCapturing(s, &capture) == cudaSuccess &&
        capture == cudaStreamCaptureStatusActive)
        return cudaMallocAsync(p, bytes ? bytes : 1, s);
    std::lock_guard<std::mutex> lk(g_pool_mu);
    PoolSlot* ps = nullptr;
    cudaError_t e = current_pool(&ps);
    if (!e) e = cudaMallocFromPoolAsync(p, bytes ? bytes : 1, ps->pool, s);
    if (e != cudaErrorMemoryAllocation) return e;
    cudaGetLastError();
    trim(*ps);
    e = cudaMallocFromPoolAsync(p, bytes ? bytes : 1, ps->pool, s);
    if (e) cudaGetLastError();
    return e;
}

// ---------------------------------------------------------------- exclusive scan
constexpr int kScanBlock = 1024;

__global__ void k_scan_block(const int* in, int* out, int n, int* block_sums) {
    __shared__ int sh[kScanBlock];
    int i = blockIdx.x * kScanBlock + threadIdx.x;
    int x = i < n ? in[i] : 0;
    sh[threadIdx.x] = x;
    __syncthreads();
    for (int off = 1; off < kScanBlock; off <<= 1) {
        int t = threadIdx.x >= off ? sh[threadIdx.x - off] : 0;
        __syncthreads();
        sh[threadIdx.x] += t;
        __syncthreads();
    }
    if (i < n) out[i] = sh[threadIdx.x] - x;
    if (threadIdx.x == kScanBlock - 1) block_sums[blockIdx.x] = sh[threadIdx.x];
}

__global__ void k_scan_sums(int* sums, int nb) {
    // single block: sequential chunks, deterministic
    __shared__ int carry;
    if (threadIdx.x == 0) carry = 0;
    __syncthreads();
    __shared__ int sh[kScanBlock];
    for (int base = 0; base < nb; base += kScanBlock) {
        int i = base + threadIdx.x;
        int x = i < nb ? sums[i] : 0;
        sh[threadIdx.x] = x;
        __syncthreads();
        for (int off = 1; off < kScanBlock; off <<= 1) {
            int t = threadIdx.x >= off ? sh[threadIdx.x - off] : 0;
            __syncthreads();
            sh[threadIdx.x] += t;
            __syncthreads();
        }
        if (i < nb) sums[i] = carry + sh[threadIdx.x] - x;
        __syncthreads();
        if (threadIdx.x == kScanBlock - 1) carry += sh[threadIdx.x];
        __syncthreads();
    }
}

__global__ void k_scan_add(int* out, int n, const int* sums) {
    int i = blockIdx.x * kScanBlock + threadIdx.x;
    if (i < n) out[i] += sums[blockIdx.x];
}

size_t scan_tmp_ints(int n) { return (size_t)(n + kScanBlock - 1) / kScanBlock + 1; }

cudaError_t exclusive_scan(const int* in, int* out, int n, int* tmp, cudaStream_t s) {
    if (n <= 0) return cudaSuccess;
    int nb = (n + kScanBlock - 1) / kScanBlock;
    k_scan_block<<<nb, kScanBlock, 0, s>>>(in, out, n, tmp);
    k_scan_sums<<<1, kScanBlock, 0, s>>>(tmp, nb);
    k_scan_add<<<nb, kScanBlock, 0, s>>>(out, n, tmp);
    return cudaGetLastError();
}

// ---------------------------------------------------------------- mesh kernels
enum : int { kMeshErrDegenerate = 1, kMeshErrDup = 2, kMeshErrFan = 4, kMeshErrProbe = 8 };

__device__ __forceinline__ int he_next(int h) { return 3 * (h / 3) + (h % 3 + 1) % 3; }
__device__ __forceinline__ int he_prev(int h) { return 3 * (h / 3) + (h % 3 + 2) % 3; }

__device__ __forceinline__ double dist3(const double* x, int a, int b) {
    double dx = x[3 * a] - x[3 * b], dy = x[3 * a + 1] - x[3 * b + 1], dz = x[3 * a + 2] - x[3 * b + 2];
    return sqrt(dx * dx + dy * dy + dz * dz);
}

// Edge lengths and the apex frame of every half-edge (the metric is all the method
// needs, Section 4.1).
__global__ void k_frames(int nh, const double* __restrict__ xyz, const int* __restrict__ tri, HERec* rec,
                         double* hang, int* err) {
    for (int h = blockIdx.x * blockDim.x + threadIdx.x; h < nh; h += gridDim.x * blockDim.x) {
        int a = tri[h], b = tri[he_next(h)], c = tri[he_prev(h)];
        double L = dist3(xyz, a, b), L1 = dist3(xyz, b, c), L2 = dist3(xyz, c, a);
        double xc = ((L2 - L1) * (L2 + L1) + L * L) / (2.0 * L);
        double t = (L2 - xc) * (L2 + xc);
        double yc = sqrt(t > 0.0 ? t : 0.0);
        HERec r;
        r.L = L; r.xc = xc; r.yc = yc; r.L1 = L1; r.L2 = L2;
        r.u1x = (L - xc) / L1; r.u1y = -yc / L1; r.u2x = xc / L2; r.u2y = yc / L2;
        r.tw1 = r.tw2 = r.twin = -1;
        r.v0 = a; r.v1 = b; r.v2 = c;
        rec[h] = r;
        hang[h] = atan2(yc, xc);
        if (a == b || b == c || c == a || !(yc > 1e-12 * L) || !(L > 1e-250)) atomicOr(err, kMeshErrDegenerate);
    }
}

__device__ __forceinline__ unsigned long long mix64(unsigned long long z) {
    z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
    z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
    return z ^ (z >> 31);
}

__global__ void k_hash_insert(int nh, const int* __restrict__ tri, unsigned long long* keys, int* vals,
                              unsigned long long mask, int* err) {
    for (int h = blockIdx.x * blockDim.x + threadIdx.x; h < nh; h += gridDim.x * blockDim.x) {
        unsigned long long k = (unsigned long long)(unsigned)tri[h] << 32 | (unsigned)tri[he_next(h)];
        unsigned long long s = mix64(k) & mask;
        for (unsigned long long probe = 0; probe <= mask; ++probe) {
            unsigned long long prev = atomicCAS(&keys[s], ~0ull, k);
            if (prev == ~0ull) { vals[s] = h; break; }
            if (prev == k) { atomicOr(err, kMeshErrDup); break; }
            s = (s + 1) & mask;
            if (probe == mask) atomicOr(err, kMeshErrProbe);
        }
    }
}

__global__ void k_twins(int nh, const int* __restrict__ tri, const unsigned long long* keys, const int* vals,
                        unsigned long long mask, int* twin, int* vcount, int* vout) {
    for (int h = blockIdx.x * blockDim.x + threadIdx.x; h < nh; h += gridDim.x * blockDim.x) {
        int a = tri[h], b = tri[he_next(h)];
        unsigned long long k = (unsigned long long)(unsigned)b << 32 | (unsigned)a;
        unsigned long long s = mix64(k) & mask;
        int t = -1;
        for (unsigned long long probe = 0; probe <= mask; ++probe) {
            unsigned long long kk = keys[s];
            if (kk == k) { t = vals[s]; break; }
            if (kk == ~0ull) break;
            s = (s + 1) & mask;
        }
        twin[h] = t;
        atomicAdd(&vcount[a], 1);
        atomicMin(&vout[a], h);
    }
}

// One thread per vertex: walk its one-ring (clockwise to a boundary, then
// counter-clockwise), record the ring order, angular positions and total angle.
__global__ void k_rings(int nv, const int* __restrict__ twin, const int* __restrict__ vout,
                        const int* __restrict__ vstart, const double* __restrict__ hang, int* vlist,
                        float* vphi, float* vtheta, float* hang_f, double2* vrot, double2* vtrot,
                        unsigned char* vflag, int* err) {
    const double kTwoPi = 6.283185307179586476925286766559;
    for (int v = blockIdx.x * blockDim.x + threadIdx.x; v < nv; v += gridDim.x * blockDim.x) {
        int cnt = vstart[v + 1] - vstart[v];
        if (cnt == 0) { vtheta[v] = 0; vtrot[v] = make_double2(1.0, 0.0); vflag[v] = 0; continue; }
        int h0 = vout[v];
        int start = h0;
        bool boundary = false;
        for (int s = 0; s <= cnt; ++s) {   // clockwise: h -> next(twin(h))
            int t = twin[start];
            if (t < 0) { boundary = true; break; }
            int hn = he_next(t);
            if (hn == h0) break;
            start = hn;
        }
        if (!boundary) start = h0;
        int h = start, k = 0;
        double phi = 0.0;
        while (k < cnt) {
            vlist[vstart[v] + k] = h;
            vphi[h] = (float)phi;
            hang_f[h] = (float)hang[h];
            double sp, cp;
            sincos(phi, &sp, &cp);
            vrot[h] = make_double2(cp, sp);
            phi += hang[h];
            ++k;
            int t = twin[he_prev(h)];           // counter-clockwise: h -> twin(prev(h))
            if (t < 0 || t == start) break;
            h = t;
        }
        if (k != cnt) atomicOr(err, kMeshErrFan);
        vtheta[v] = (float)phi;
        {
            double sp, cp;
            sincos(phi, &sp, &cp);
            vtrot[v] = make_double2(cp, sp);
        }
        unsigned char f = boundary ? 1 : 0;
        // Saddle (total angle above 2 pi, Section 3) or boundary vertex: a pseudo-source
        // candidate.  The 1e-9 band keeps flat vertices in the candidate set (superset).
        if (boundary || phi > kTwoPi - 1e-9) f |= 2;
        vflag[v] = f;
    }
}

__global__ void k_rec_ids(int nh, const int* __restrict__ twin, const unsigned char* __restrict__ vflag, HERec* rec) {
    for (int h = blockIdx.x * blockDim.x + threadIdx.x; h < nh; h += gridDim.x * blockDim.x) {
        HERec r = rec[h];
        r.twin = twin[h];
        r.tw1 = twin[he_next(h)];
        r.tw2 = twin[he_prev(h)];
        r.v0 |= (vflag[r.v0] & 2) ? kPseudoBit : 0u;
        r.v1 |= (vflag[r.v1] & 2) ? kPseudoBit : 0u;
        r.v2 |= (vflag[r.v2] & 2) ? kPseudoBit : 0u;
        rec[h] = r;
    }
}

// ---------------------------------------------------------------- face order
// Faces are kept in the order of the Morton codes of their centroids (the Z-order curve
// of G. M. Morton, 1966): neighbours on the surface are then neighbours in memory, whatever
// order the caller's list has.  A window reads the 96-byte records of a band of the
// surface; scattered over the 1.5 GB of a 5.2M-face sphere (whose subdivision puts the four
// children of a face a quarter of the list apart) those reads were bound by address
// translation and L2 misses: a field took 647 ms, in this order 335 (327 by now).  A mesh of
// fewer than kReorderFaces faces (its records fit L2 and the TLBs) gains nothing and
// keeps its order: 8.4 ms either way at 327,680 faces, 46 against 39 at 1,310,720.
constexpr int kReorderFaces = 1 << 19;
constexpr int kMortonBits = 24;

// Signed 64-bit image of a double whose integer order is the doubles' order.
__device__ __forceinline__ long long ordered(double x) {
    const long long b = __double_as_longlong(x);
    return b < 0 ? b ^ 0x7fffffffffffffffll : b;
}
__device__ __forceinline__ double unordered(long long b) {
    return __longlong_as_double(b < 0 ? b ^ 0x7fffffffffffffffll : b);
}

// box[0..2]: minimum, box[3..5]: minimum of the negated coordinates.
__global__ void __launch_bounds__(256) k_bounds(int nv, const double* __restrict__ xyz, long long* box) {
    long long m[6];
#pragma unroll
    for (int j = 0; j < 6; ++j) m[j] = 0x7fffffffffffffffll;
    for (int v = blockIdx.x * blockDim.x + threadIdx.x; v < nv; v += gridDim.x * blockDim.x) {
#pragma unroll
        for (int j = 0; j < 3; ++j) {
            const double x = xyz[3 * (size_t)v + j];
            m[j] = min(m[j], ordered(x));
            m[j + 3] = min(m[j + 3], ordered(-x));
        }
    }
#pragma unroll
    for (int j = 0; j < 6; ++j) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) m[j] = min(m[j], __shfl_xor_sync(0xffffffffu, m[j], o));
        if ((threadIdx.x & 31) == 0) atomicMin(box + j, m[j]);
    }
}

__device__ __forceinline__ unsigned spread3(unsigned x) {   // 8 bits, two zeros between
    x = (x | x << 8) & 0x00f00fu;
    x = (x | x << 4) & 0x0c30c3u;
    return (x | x << 2) & 0x249249u;
}

__global__ void k_morton(int nf, const double* __restrict__ xyz, const int* __restrict__ tri, const long long* box,
                         unsigned* key) {
    double lo[3], ext = 0.0;
    for (int j = 0; j < 3; ++j) {
        lo[j] = unordered(box[j]);
        ext = fmax(ext, -unordered(box[j + 3]) - lo[j]);
    }
    const double scale = 256.0 / (3.0 * ext);
    for (int f = blockIdx.x * blockDim.x + threadIdx.x; f < nf; f += gridDim.x * blockDim.x) {
        unsigned code = 0;
        for (int j = 0; j < 3; ++j) {
            double s = 0.0;
            for (int c = 0; c < 3; ++c) s += xyz[3 * (size_t)tri[3 * f + c] + j] - lo[j];
            const double q = s * scale;
            code |= spread3(q > 0.0 ? (unsigned)fmin(q, 255.0) : 0u) << j;   // (a NaN: 0)
        }
        key[f] = code;
    }
}

__global__ void k_permute_faces(int nf, const int* __restrict__ tri, const int* __restrict__ perm, int* tri_out,
                                int* fperm, int* finv) {
    for (int f = blockIdx.x * blockDim.x + threadIdx.x; f < nf; f += gridDim.x * blockDim.x) {
        const int o = perm[f];
        fperm[f] = o;
        finv[o] = f;
        for (int c = 0; c < 3; ++c) tri_out[3 * f + c] = tri[3 * o + c];
    }
}

// Deterministic mean edge length and counts: block b reduces a fixed contiguous range of
// half-edges and vertices in a fixed order, then k_stats_final adds the kStatBlocks
// partial results in a fixed tree, so the sum does not depend on scheduling.
constexpr int kStatBlocks = 256;

__device__ __forceinline__ void block_sum3(double& s, int& a, int& b) {
    __shared__ double sh[256];
    __shared__ int sa[256], sb[256];
    sh[threadIdx.x] = s; sa[threadIdx.x] = a; sb[threadIdx.x] = b;
    __syncthreads();
    for (int off = 128; off > 0; off >>= 1) {
        if (threadIdx.x < off) {
            sh[threadIdx.x] += sh[threadIdx.x + off];
            sa[threadIdx.x] += sa[threadIdx.x + off];
            sb[threadIdx.x] += sb[threadIdx.x + off];
        }
        __syncthreads();
    }
    s = sh[0]; a = sa[0]; b = sb[0];
}

__global__ void __launch_bounds__(256) k_stats(int nh, int nv, const HERec* rec, const int* twin,
                                               const unsigned char* vflag, double* part_l, int* part_c) {
    const long long h0 = (long long)nh * blockIdx.x / gridDim.x, h1 = (long long)nh * (blockIdx.x + 1) / gridDim.x;
    const long long v0 = (long long)nv * blockIdx.x / gridDim.x, v1 = (long long)nv * (blockIdx.x + 1) / gridDim.x;
    double s = 0.0;
    int nb = 0, np = 0;
    for (long long h = h0 + threadIdx.x; h < h1; h += blockDim.x) {
        s += rec[h].L;
        nb += twin[h] < 0;
    }
    for (long long v = v0 + threadIdx.x; v < v1; v += blockDim.x) np += (vflag[v] & 2) ? 1 : 0;
    block_sum3(s, nb, np);
    if (threadIdx.x == 0) { part_l[blockIdx.x] = s; part_c[2 * blockIdx.x] = nb; part_c[2 * blockIdx.x + 1] = np; }
}

__global__ void __launch_bounds__(256) k_stats_final(const double* part_l, const int* part_c, double* out_lsum,
                                                     int* out_counts) {
    double s = part_l[threadIdx.x];
    int nb = part_c[2 * threadIdx.x], np = part_c[2 * threadIdx.x + 1];
    block_sum3(s, nb, np);
    if (threadIdx.x == 0) { *out_lsum = s; out_counts[0] = nb; out_counts[1] = np; }
}

// Lays out the arrays of a mesh.
static void carve_mesh(Carver& c, DevMesh& d, bool reorder) {
    c.take(&d.rec, d.nh);
    c.take(&d.vrot, d.nh);
    c.take(&d.vtrot, d.nv);
    c.take(&d.tri, d.nh);
    c.take(&d.vlist, d.nh);
    c.take(&d.hang, d.nh);
    c.take(&d.vphi, d.nh);
    c.take(&d.vstart, d.nv + 1);
    c.take(&d.vtheta, d.nv);
    c.take(&d.vflag, d.nv);
    if (reorder) {
        c.take(&d.fperm, d.nf);
        c.take(&d.finv, d.nf);
    }
}

// Temporaries of the mesh preparation.
struct MeshTmp {
    double *xyz, *hang64, *lsum;
    unsigned long long* hkeys;
    long long* box;
    int *twin, *vcount, *vout, *hvals, *counts, *scan_tmp, *tri_sorted, *fval[2], *fhist;
    unsigned* fkey[2];
    int* err;               // kMeshErr* flags
};
static void carve_tmp(Carver& c, MeshTmp& t, int nv, int nf, unsigned long long cap, bool reorder, int sort_blocks) {
    const int nh = 3 * nf;
    c.take(&t.xyz, 3 * (size_t)nv);
    c.take(&t.hang64, nh);
    c.take(&t.lsum, 1 + kStatBlocks);
    c.take(&t.hkeys, cap);
    c.take(&t.hvals, cap);
    c.take(&t.twin, nh);
    c.take(&t.vcount, nv + 1);
    c.take(&t.vout, nv);
    c.take(&t.counts, 2 + 2 * kStatBlocks);
    c.take(&t.scan_tmp, scan_tmp_ints(nv + 1));
    c.take(&t.err, 1);
    if (reorder) {
        c.take(&t.tri_sorted, nh);
        for (int j = 0; j < 2; ++j) {
            c.take(&t.fkey[j], nf);
            c.take(&t.fval[j], nf);
        }
        c.take(&t.fhist, kRsDigits * sort_blocks + 1);
        c.take(&t.box, 6);
    }
}

// Input checks (before any device work): one branch-free pass over each array, the index of
// the first offender only when there is one.
static bool all_finite(const double* x, long long n) {
    unsigned long long bad = 0;
    for (long long i = 0; i < n; ++i) {
        unsigned long long b;
        std::memcpy(&b, x + i, sizeof b);
        bad |= ((b & 0x7fffffffffffffffull) + 0x0010000000000000ull) & 0x8000000000000000ull;   // exponent all ones
    }
    return bad == 0;
}
static bool all_below(const int32_t* x, long long n, int32_t limit) {
    unsigned most = 0;
    for (long long i = 0; i < n; ++i) most = std::max(most, (unsigned)x[i]);
    return most < (unsigned)limit;
}

void destroy_workspace(Workspace* w);   // solver.cu

}  // namespace pch

using namespace pch;

extern "C" const char* pch_last_error(void) { return pch::g_err.c_str(); }

extern "C" pch_status pch_create_mesh(const double* vertices, int32_t n_vertices, const int32_t* faces,
                                      int32_t n_faces, pch_mesh** out) {
    clear_error();
    if (!vertices || !faces || !out) return set_error(PCH_ERR_INVALID_ARG, "null pointer argument");
    if (n_vertices < 3 || n_faces < 1) return set_error(PCH_ERR_INVALID_ARG, "need >= 3 vertices and >= 1 face");
    if ((long long)n_faces * 3 >= (1LL << 31) - 1) return set_error(PCH_ERR_CAPACITY, "too many faces");
    if (!all_finite(vertices, 3LL * n_vertices))
        for (long long i = 0; i < 3LL * n_vertices; ++i)
            if (!std::isfinite(vertices[i])) return set_error(PCH_ERR_INVALID_ARG, "non-finite coordinate at vertex %lld", i / 3);
    if (!all_below(faces, 3LL * n_faces, n_vertices))
        for (long long i = 0; i < 3LL * n_faces; ++i)
            if (faces[i] < 0 || faces[i] >= n_vertices)
                return set_error(PCH_ERR_INVALID_ARG, "face %lld references vertex %d out of range", i / 3, faces[i]);

    const int nv = n_vertices, nf = n_faces, nh = 3 * n_faces;
    const bool reorder = nf >= kReorderFaces;
    const int sort_blocks = 2 * sm_count();
    const cudaStream_t s = 0;         // the legacy default stream, as the callers' copies
    unsigned long long cap = 1;
    while (cap < 2ull * (unsigned long long)nh) cap <<= 1;
    DevMesh d{};
    d.nv = nv; d.nf = nf; d.nh = nh;
    DevMem mem;
    MeshTmp t{};
    void* tmp = nullptr;
    pch_status st = PCH_OK;
    int herr = 0;
    double hl = 0.0;
    int hc[2] = {0, 0};
    auto fail = [&](pch_status s) { st = s; };
#define MCHK(call)                                                                              \
    do {                                                                                        \
        cudaError_t e_ = (call);                                                                \
        if (e_ != cudaSuccess) {                                                                \
            fail(set_error(e_ == cudaErrorMemoryAllocation ? PCH_ERR_OOM : PCH_ERR_CUDA, "%s: %s", #call, \
                           cudaGetErrorString(e_)));                                            \
            goto cleanup;                                                                       \
        }                                                                                       \
    } while (0)
    {
        Carver cm, ct;
        carve_mesh(cm, d, reorder);
        MCHK(dev_alloc(mem, cm.off));
        cm = Carver{static_cast<char*>(mem.p), 0};
        carve_mesh(cm, d, reorder);
        carve_tmp(ct, t, nv, nf, cap, reorder, sort_blocks);
        MCHK(tmp_alloc(&tmp, ct.off, s));
        ct = Carver{static_cast<char*>(tmp), 0};
        carve_tmp(ct, t, nv, nf, cap, reorder, sort_blocks);
        MCHK(cudaMemcpyAsync(t.xyz, vertices, sizeof(double) * 3 * nv, cudaMemcpyHostToDevice, s));
        MCHK(cudaMemcpyAsync(d.tri, faces, sizeof(int) * nh, cudaMemcpyHostToDevice, s));
        MCHK(cudaMemsetAsync(t.err, 0, sizeof(int), s));
        MCHK(cudaMemsetAsync(t.vcount, 0, sizeof(int) * (nv + 1), s));
        MCHK(cudaMemsetAsync(t.vout, 0x7f, sizeof(int) * nv, s));
        MCHK(cudaMemsetAsync(t.hkeys, 0xff, sizeof(unsigned long long) * cap, s));
        const int tb = 256;
        const int gb = std::max(1, std::min((nh + tb - 1) / tb, sm_count() * 8));
        const int gv = std::max(1, std::min((nv + tb - 1) / tb, sm_count() * 8));
        const int* tri = d.tri;
        if (reorder) {
            MCHK(cudaMemsetAsync(t.box, 0x7f, sizeof(long long) * 6, s));
            MCHK(cudaMemcpyAsync(t.fhist + kRsDigits * sort_blocks, &nf, sizeof(int), cudaMemcpyHostToDevice, s));
            k_bounds<<<gv, tb, 0, s>>>(nv, t.xyz, t.box);
            k_morton<<<gb, tb, 0, s>>>(nf, t.xyz, tri, t.box, t.fkey[0]);
            const int r = launch_sort_keys(t.fhist + kRsDigits * sort_blocks, nf, kMortonBits, t.fkey, t.fval, t.fhist,
                                           sort_blocks, s);
            k_permute_faces<<<gb, tb, 0, s>>>(nf, tri, t.fval[r], t.tri_sorted, d.fperm, d.finv);
            MCHK(cudaGetLastError());
            tri = t.tri_sorted;
        }
        k_frames<<<gb, tb, 0, s>>>(nh, t.xyz, tri, d.rec, t.hang64, t.err);
        k_hash_insert<<<gb, tb, 0, s>>>(nh, tri, t.hkeys, t.hvals, cap - 1, t.err);
        k_twins<<<gb, tb, 0, s>>>(nh, tri, t.hkeys, t.hvals, cap - 1, t.twin, t.vcount, t.vout);
        MCHK(cudaGetLastError());
        MCHK(exclusive_scan(t.vcount, d.vstart, nv + 1, t.scan_tmp, s));
        k_rings<<<gv, tb, 0, s>>>(nv, t.twin, t.vout, d.vstart, t.hang64, d.vlist, d.vphi, d.vtheta, d.hang, d.vrot, d.vtrot,
                                  d.vflag, t.err);
        k_rec_ids<<<gb, tb, 0, s>>>(nh, t.twin, d.vflag, d.rec);
        k_stats<<<kStatBlocks, 256, 0, s>>>(nh, nv, d.rec, t.twin, d.vflag, t.lsum + 1, t.counts + 2);
        k_stats_final<<<1, kStatBlocks, 0, s>>>(t.lsum + 1, t.counts + 2, t.lsum, t.counts);
        MCHK(cudaGetLastError());
        MCHK(cudaMemcpyAsync(&herr, t.err, sizeof(int), cudaMemcpyDeviceToHost, s));
        MCHK(cudaMemcpyAsync(&hl, t.lsum, sizeof(double), cudaMemcpyDeviceToHost, s));
        MCHK(cudaMemcpyAsync(hc, t.counts, sizeof(int) * 2, cudaMemcpyDeviceToHost, s));
        MCHK(cudaStreamSynchronize(s));
        if (herr & kMeshErrDup) { fail(set_error(PCH_ERR_NONMANIFOLD, "an oriented edge appears in two faces (non-manifold or inconsistent orientation)")); goto cleanup; }
        if (herr & kMeshErrDegenerate) { fail(set_error(PCH_ERR_DEGENERATE, "a face has a repeated vertex or (near) zero area")); goto cleanup; }
        if (herr & kMeshErrFan) { fail(set_error(PCH_ERR_NONMANIFOLD, "a vertex whose faces do not form a single fan")); goto cleanup; }
        if (herr & kMeshErrProbe) { fail(set_error(PCH_ERR_CUDA, "edge hash table overflow")); goto cleanup; }
        d.lbar = hl / nh;
        pch_mesh* m = new pch_mesh();
        m->dm = d;
        m->mem = mem;
        cudaGetDevice(&m->device);
        m->n_boundary_he = hc[0];
        m->n_pseudo = hc[1];
        m->ws = nullptr;
        *out = m;
    }
cleanup:
#undef MCHK
    if (st != PCH_OK) cudaStreamSynchronize(s);   // nothing is in flight on what is freed below
    if (tmp) cudaFreeAsync(tmp, s);
    if (st != PCH_OK) dev_free(mem);
    return st;
}

extern "C" pch_status pch_mesh_info(const pch_mesh* m, int32_t* n_vertices, int32_t* n_faces,
                                    int32_t* n_boundary_half_edges, int32_t* n_pseudo_vertices) {
    if (!m) return set_error(PCH_ERR_INVALID_ARG, "null mesh");
    if (n_vertices) *n_vertices = m->dm.nv;
    if (n_faces) *n_faces = m->dm.nf;
    if (n_boundary_half_edges) *n_boundary_half_edges = m->n_boundary_he;
    if (n_pseudo_vertices) *n_pseudo_vertices = m->n_pseudo;
    return PCH_OK;
}

extern "C" void pch_destroy(pch_mesh* m) {
    if (!m) return;
    int cur = 0;
    cudaGetDevice(&cur);
    cudaSetDevice(m->device);
    if (m->ws) destroy_workspace(m->ws);   // (waits for the mesh's last call)
    dev_free(m->mem);
    cudaSetDevice(cur);
    delete m;
}
