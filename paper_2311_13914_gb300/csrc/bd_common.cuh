// bd_common.cuh -- internal declarations shared by the CUDA translation units
// of the Bidomain SA-AMG-PCG library (not part of the public ABI).
#pragma once

#include <cuda_runtime.h>

#include <cstdint>
#include <cstdio>
#include <utility>
#include <vector>

#include "bidomain.h"

namespace bd {

// ------------------------------------------------------------------ launch counter
// Every kernel launch of the library calls note_launch(); bd_launch_count()
// reports the running total (host-side, atomic).
void note_launch();
void note_launches(long long n);  // adds n (may be negative: undo capture-time counts)
// SpGEMM calls of the setup by path (hash: warp per row; dense: block per row),
// counted process-wide for bd_spgemm_path_counts().
void note_spgemm_path(bool dense);
long long spgemm_path_count(bool dense);
long long launch_count();

// ------------------------------------------------------------------ errors
void record_cuda_error(cudaError_t e, const char *what, const char *file, int line);

#define BD_CUDA(x)                                                                   \
    do {                                                                             \
        cudaError_t e_ = (x);                                                        \
        if (e_ != cudaSuccess) {                                                     \
            ::bd::record_cuda_error(e_, #x, __FILE__, __LINE__);                     \
            return e_ == cudaErrorMemoryAllocation ? BD_ENOMEM : BD_ECUDA;           \
        }                                                                            \
    } while (0)

#define BD_LAUNCH_CHECK() BD_CUDA(cudaGetLastError())

#define BD_TRY(x)                                                                    \
    do {                                                                             \
        int s_ = (x);                                                                \
        if (s_ != BD_OK) return s_;                                                  \
    } while (0)

// ------------------------------------------------------------------ device buffers
// Memory pool of the scratch buffers of one setup call, current on the calling
// thread while it lives: a setup allocates and frees some two hundred of them,
// and cudaMalloc and cudaFree cost 2 us for pages and 15 to 700 us for
// megabytes to gigabytes (cudaFree waits for the device, too), a pool allocation
// one.  Scratch is allocated and freed in the order of the call's stream, and
// everything goes back when the call returns, or earlier if an allocation finds
// no room (trim).  Without a current pool (or if none can be made) scratch comes
// from cudaMalloc.  Setup of 48x48x12 elements 10.8 -> 9.2 ms; six setups
// and 28 time steps between them 90 -> 77 ms.
class ScratchPool {
public:
    ScratchPool();
    ~ScratchPool();
    ScratchPool(const ScratchPool &) = delete;
    ScratchPool &operator=(const ScratchPool &) = delete;
    static cudaMemPool_t current();
    // an allocation failed: hand back what the current pool keeps free; false if
    // there is none, or the failure was another one
    static bool trim(cudaError_t e);

private:
    cudaMemPool_t pool_ = nullptr, outer_ = nullptr;
};

// Owning, move-only device allocation.  Every allocation of the library goes
// through here so that the destructors of the handles release everything.
template <class T>
struct DBuf {
    T *p = nullptr;
    size_t n = 0;
    DBuf() = default;
    DBuf(const DBuf &) = delete;
    DBuf &operator=(const DBuf &) = delete;
    DBuf(DBuf &&o) noexcept : p(o.p), n(o.n), kind_(o.kind_), s_(o.s_) { o.p = nullptr; o.n = 0; }
    DBuf &operator=(DBuf &&o) noexcept {
        if (this != &o) {
            release();
            p = o.p; n = o.n; kind_ = o.kind_; s_ = o.s_;
            o.p = nullptr; o.n = 0;
        }
        return *this;
    }
    ~DBuf() { release(); }
    int alloc(size_t count) {
        release();
        if (count == 0) count = 1;
        cudaError_t e = cudaMalloc((void **)&p, count * sizeof(T));
        if (ScratchPool::trim(e)) e = cudaMalloc((void **)&p, count * sizeof(T));
        if (e != cudaSuccess) {
            p = nullptr;
            record_cuda_error(e, "cudaMalloc", __FILE__, __LINE__);
            return BD_ENOMEM;
        }
        kind_ = kOwned;
        n = count;
        return BD_OK;
    }
    // scratch used in the order of stream s only, from the current pool
    int scratch(size_t count, cudaStream_t s) {
        cudaMemPool_t pool = ScratchPool::current();
        if (!pool) return alloc(count);
        release();
        if (count == 0) count = 1;
        cudaError_t e = cudaMallocFromPoolAsync((void **)&p, count * sizeof(T), pool, s);
        if (ScratchPool::trim(e)) e = cudaMallocFromPoolAsync((void **)&p, count * sizeof(T), pool, s);
        if (e != cudaSuccess) {
            p = nullptr;
            record_cuda_error(e, "cudaMallocFromPoolAsync", __FILE__, __LINE__);
            cudaGetLastError();
            return BD_ENOMEM;
        }
        kind_ = kScratch;
        s_ = s;
        n = count;
        return BD_OK;
    }
    // part of another buffer, which must outlive this one
    void view(T *part, size_t count) {
        release();
        p = part;
        n = count;
        kind_ = kView;
    }
    void release() {
        if (p && kind_ == kOwned) cudaFree(p);
        if (p && kind_ == kScratch) cudaFreeAsync(p, s_);
        p = nullptr;
        n = 0;
    }
    size_t bytes() const { return n * sizeof(T); }

private:
    enum Kind { kOwned, kScratch, kView };
    Kind kind_ = kOwned;
    cudaStream_t s_ = nullptr;
};

// 2x2-block CSR: block row i holds blocks (i, ci[t]) for t in [rp[i], rp[i+1]),
// columns ascending; the block values are v[4t..4t+3] = [a00 a01 a10 a11].
struct BSR {
    int nbr = 0, nbc = 0;  // block rows / block columns
    long long nb = 0;      // blocks
    DBuf<int> rp, ci;
    DBuf<double> v;
};

// scalar CSR with int32 indices (node graphs)
struct CSR {
    int nr = 0, nc = 0;
    long long nnz = 0;
    DBuf<int> rp, ci;
    DBuf<double> v;
};

// Doubles of a raw stencil row (bd_assemble.cu): 27 (Ki, Ke) pairs, c M, M.
constexpr int kFineRaw = 56;

// ------------------------------------------------------------------ utilities
constexpr int kSM = 152;  // GB300 streaming multiprocessors (grid sizing)

// Dynamic shared memory above the default 48 KB for a kernel's launches.  The limit
// is an attribute of the function that every thread of the process shares: set to
// each launch's size, one thread's smaller size between another's setting and its
// launch made that launch fail.  One value for all sizes instead (the launch's own
// size decides what a block takes).
constexpr size_t kDynamicSmem = 200u << 10;
template <class K> int allow_smem(K kernel)
{
    BD_CUDA(cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kDynamicSmem));
    return BD_OK;
}

inline int grid_for(long long work, int block, int per_sm_cap = 8) {
    long long g = (work + block - 1) / block;
    long long cap = (long long)kSM * per_sm_cap * 4;
    if (g > cap) g = cap;
    if (g < 1) g = 1;
    return (int)g;
}

// out[0..n] = exclusive prefix sum of in[0..n) (out[n] = total); *total gets the
// total on the host (stream synchronised).  BD_ERANGE if the total exceeds 2^31-1.
int exclusive_scan(const int *in, int *out, int n, long long *total, cudaStream_t s);

// *slot = max(0, a[0..n)) on the device, stream-ordered (slot: one device int;
// the caller reads it back after its next synchronisation).
int device_max(const int *a, int n, int *slot, cudaStream_t s);

// Sort the keys of every segment [seg[i], seg[i+1]) ascending (keys unique
// within a segment), permuting `payload` alongside when it is not NULL.
// BD_ERANGE if a segment is longer than kMaxSortSeg.
constexpr int kMaxSortSeg = 8192;
int sort_segments(int *keys, int *payload, const int *seg, int nseg, int max_len,
                  cudaStream_t s);

// Correctly rounded dot product sum_i x[i]*y[i] (each product rounded, then an
// exact long accumulator and one rounding to nearest-even), written to *out on
// the device.  Order-independent, hence bit-reproducible.  `acc` must hold
// kExactScratch long longs: the limbs, the flags of infinities and NaNs, and the
// blocks' arrival counter.
constexpr int kExactLimbs = 68;
constexpr int kExactScratch = kExactLimbs + 2;
int exact_dot(const double *x, const double *y, int n, double *out, long long *acc, cudaStream_t s,
              bool clean = false);
// r -= (*num / *den) q, z = r / diag (entry by entry), out = r . z, with a clean
// accumulator; one launch less for vectors of one product per thread (up to
// kDotUpdateMax), where longer ones would take their divisions on few warps
constexpr int kDotUpdateMax = 2 * kSM * 512;
int exact_dot_update(const double *num, const double *den, const double *q, const double *diag, double *r, double *z,
                     int n, double *out, long long *acc, cudaStream_t s);

// Copy helpers between caller arrays (host or device) and device buffers.
int copy_in(void *dst_dev, const void *src, size_t bytes, int src_on_device, cudaStream_t s);
int copy_out(void *dst, const void *src_dev, size_t bytes, int dst_on_device, cudaStream_t s);

// Scalar CSR (2N x 2M, full 2x2 node blocks) <-> BSR conversion on the device.
int bsr_from_scalar_csr(int n, const int *rp, const int *ci, const double *v, BSR &out,
                        cudaStream_t s);
int bsr_to_scalar_csr_host(const BSR &a, int *rp, int *ci, double *v, cudaStream_t s);

}  // namespace bd

// ------------------------------------------------------------------ handles
struct bd_system {
    bd_mesh mesh{};
    bd_params params{};
    int N = 0;              // nodes
    bd::BSR A;              // block operator, 2x2 blocks per node pair
    bd::DBuf<double> M;     // lumped mass (N)
    bd::DBuf<double> Ki;    // node-pattern stiffness values (shared pattern with A)
    bd::DBuf<double> Ke;
    bd::DBuf<double> raw;   // rows per plane and row type: (nz + 1) x 9 x kFineRaw
    bool sym = false;       // the symmetric stencil form holds for every row (bd_assemble.cu)
};
