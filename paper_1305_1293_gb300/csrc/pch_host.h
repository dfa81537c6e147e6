// Host-side internals shared by the library's translation units.
#pragma once

#include <cuda_runtime.h>

#include <cstdarg>
#include <cstdio>
#include <string>

#include "pch_common.cuh"

namespace pch {

pch_status set_error(pch_status st, const char* fmt, ...);
void clear_error();

struct Workspace;   // solver.cu

}  // namespace pch

namespace pch {

// ---- device memory -------------------------------------------------------------------
// The library's own stream-ordered pools, one per device and context (safe for several
// threads and streams, as the driver's pools are): while a mesh is alive, up to kPoolKeep bytes
// of freed memory stay for the next mesh, workspace or temporary and the rest goes back to the
// driver at the next synchronisation; when the last mesh is destroyed, or an allocation
// fails, all of it does.  (cudaMalloc / cudaFree of a mesh and its workspace took 4 ms a
// mesh, and temporaries of the default pool, which keeps nothing, were mapped anew after
// every synchronising call.)
constexpr unsigned long long kPoolKeep = 512ull << 20;

// A block of memory that any stream may use once dev_alloc returns.  Blocks above half of
// kPoolKeep come from cudaMalloc.
struct DevMem {
    void* p = nullptr;
    size_t bytes = 0;
    unsigned long long ctx = 0;       // context and device it was allocated in
    int dev = 0;
    bool pooled = false;
};
cudaError_t dev_alloc(DevMem& m, size_t bytes);
// The caller has made sure that no work on the device uses the block any more (cudaFree, for
// the large ones, waits for the device itself).
void dev_free(DevMem& m);

// Stream-ordered temporaries; released with cudaFreeAsync.
cudaError_t tmp_alloc(void** p, size_t bytes, cudaStream_t s);

// Lays arrays out in one block: a first pass over the take() calls with base = nullptr
// gives the size.
struct Carver {
    char* base = nullptr;
    size_t off = 0;
    template <class T>
    void take(T** p, size_t n) {
        off = (off + 255) & ~(size_t)255;
        *p = base ? reinterpret_cast<T*>(base + off) : nullptr;
        off += sizeof(T) * n;
    }
};

}  // namespace pch

struct pch_mesh {
    pch::DevMesh dm;
    pch::DevMem mem;        // every array of dm
    int device;
    int n_boundary_he;
    int n_pseudo;
    pch::Workspace* ws;
};

#define PCH_CUDA(call)                                                                    \
    do {                                                                                  \
        cudaError_t e_ = (call);                                                          \
        if (e_ != cudaSuccess) {                                                          \
            return pch::set_error(e_ == cudaErrorMemoryAllocation ? PCH_ERR_OOM : PCH_ERR_CUDA, \
                                  "%s failed: %s (%s:%d)", #call, cudaGetErrorString(e_), \
                                  __FILE__, __LINE__);                                    \
        }                                                                                 \
    } while (0)

namespace pch {

// Exclusive scan of n ints (device), out may alias in.  Uses tmp of scan_tmp_ints(n).
size_t scan_tmp_ints(int n);
cudaError_t exclusive_scan(const int* in, int* out, int n, int* tmp, cudaStream_t s);

// Number of SMs of the current device (cached).
int sm_count();

// Unique id of the calling thread's current CUDA context, 0 if there is none (or the
// driver cannot tell).  Device pointers the library caches across calls are keyed on it,
// so that a pointer from a context that has since been destroyed (cudaDeviceReset, a new
// primary context) is never used again.
unsigned long long current_context_id();

}  // namespace pch
