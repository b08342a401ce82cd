// bd_runtime.cu -- status codes, option defaults, device utilities (prefix
// scan, segmented sort, correctly rounded dot product), copies and format
// conversion used by the other translation units.
#include <algorithm>
#include <atomic>
#include <climits>
#include <cstring>
#include <mutex>

#include "bd_common.cuh"

namespace bd {

static thread_local char g_last_err[256];
static std::atomic<long long> g_launches{0};

void note_launch() { g_launches.fetch_add(1, std::memory_order_relaxed); }
void note_launches(long long n) { g_launches.fetch_add(n, std::memory_order_relaxed); }
long long launch_count() { return g_launches.load(std::memory_order_relaxed); }
static std::atomic<long long> g_spgemm_paths[2]{{0}, {0}};
void note_spgemm_path(bool dense) { g_spgemm_paths[dense ? 1 : 0].fetch_add(1, std::memory_order_relaxed); }
long long spgemm_path_count(bool dense) { return g_spgemm_paths[dense ? 1 : 0].load(std::memory_order_relaxed); }

void record_cuda_error(cudaError_t e, const char *what, const char *file, int line)
{
    snprintf(g_last_err, sizeof(g_last_err), "%s failed: %s (%s:%d)", what,
             cudaGetErrorString(e), file, line);
}

// ------------------------------------------------------------------ scratch pool
static thread_local cudaMemPool_t g_scratch = nullptr;

ScratchPool::ScratchPool() : outer_(g_scratch)
{
    int dev = 0;
    cudaMemPoolProps props = {};
    props.allocType = cudaMemAllocationTypePinned;
    props.location.type = cudaMemLocationTypeDevice;
    if (cudaGetDevice(&dev) != cudaSuccess) return;
    props.location.id = dev;
    unsigned long long keep = ~0ULL;  // nothing goes back before the pool does
    if (cudaMemPoolCreate(&pool_, &props) != cudaSuccess) {
        pool_ = nullptr;
        cudaGetLastError();
        return;
    }
    cudaMemPoolSetAttribute(pool_, cudaMemPoolAttrReleaseThreshold, &keep);
    g_scratch = pool_;
}

ScratchPool::~ScratchPool()
{
    g_scratch = outer_;
    if (pool_) cudaMemPoolDestroy(pool_);
}

cudaMemPool_t ScratchPool::current() { return g_scratch; }

bool ScratchPool::trim(cudaError_t e)
{
    if (e != cudaErrorMemoryAllocation || !g_scratch) return false;
    cudaGetLastError();
    return cudaDeviceSynchronize() == cudaSuccess && cudaMemPoolTrimTo(g_scratch, 0) == cudaSuccess;
}

// ------------------------------------------------------------------ prefix scan
constexpr int kScanThreads = 1024;
constexpr int kScanTile = 2 * kScanThreads;

__device__ __forceinline__ long long block_exclusive_scan(long long v, long long *warp_tot,
                                                           long long *block_total)
{
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    long long inc = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        long long t = __shfl_up_sync(0xffffffffu, inc, o);
        if (lane >= o) inc += t;
    }
    if (lane == 31) warp_tot[wid] = inc;
    __syncthreads();
    if (wid == 0) {
        long long w = (lane < (int)(blockDim.x >> 5)) ? warp_tot[lane] : 0;
        long long wi = w;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            long long t = __shfl_up_sync(0xffffffffu, wi, o);
            if (lane >= o) wi += t;
        }
        warp_tot[lane] = wi - w;
        if (lane == 31) *block_total = wi;
    }
    __syncthreads();
    long long r = warp_tot[wid] + inc - v;
    __syncthreads();
    return r;
}

__global__ void k_scan_tiles(const int *__restrict__ in, int *__restrict__ out, int n,
                             long long *__restrict__ tile_sums)
{
    __shared__ long long wt[32];
    __shared__ long long tot;
    long long base = (long long)blockIdx.x * kScanTile;
    long long i0 = base + 2 * threadIdx.x;
    int a = i0 < n ? in[i0] : 0;
    int b = i0 + 1 < n ? in[i0 + 1] : 0;
    long long ex = block_exclusive_scan((long long)a + b, wt, &tot);
    if (i0 < n) out[i0] = (int)ex;  // tile-local, fits: tile sum checked below
    if (i0 + 1 < n) out[i0 + 1] = (int)(ex + a);
    if (threadIdx.x == 0) tile_sums[blockIdx.x] = tot;
}

__global__ void k_scan_sums(long long *sums, int ntiles, long long *total)
{
    __shared__ long long wt[32];
    __shared__ long long tot;
    long long carry = 0;
    for (int base = 0; base < ntiles; base += blockDim.x) {
        int i = base + threadIdx.x;
        long long v = i < ntiles ? sums[i] : 0;
        long long ex = block_exclusive_scan(v, wt, &tot);
        if (i < ntiles) sums[i] = carry + ex;
        carry += tot;
        __syncthreads();
    }
    if (threadIdx.x == 0) *total = carry;
}

// Adds a tile's offset: the sum of the tiles before it, which every block forms
// itself (scanned: sums already holds the offsets).
__global__ void k_scan_add(int *out, int n, const long long *sums, bool scanned, long long *total)
{
    __shared__ long long wt[32];
    __shared__ long long tot;
    const int b = blockIdx.x;
    long long off = 0;
    if (scanned) {
        off = sums[b];
    } else {
        for (int i = threadIdx.x; i < b; i += blockDim.x) off += sums[i];
        block_exclusive_scan(off, wt, &tot);
        off = tot;
    }
    const long long base = (long long)b * kScanTile;
    for (int k = 0; k < 2; k++) {
        const long long i = base + 2 * threadIdx.x + k;
        if (i < n) out[i] = (int)(off + out[i]);
    }
    if (b == (int)gridDim.x - 1 && threadIdx.x == 0) {
        const long long t = scanned ? *total : off + sums[b];
        *total = t;
        out[n] = (int)(t > INT_MAX ? INT_MAX : t);
    }
}

constexpr int kScanDirect = 4096;  // tiles up to which every block adds up its own offset

int exclusive_scan(const int *in, int *out, int n, long long *total, cudaStream_t s)
{
    int ntiles = (n + kScanTile - 1) / kScanTile;
    if (ntiles < 1) ntiles = 1;
    DBuf<long long> sums;
    BD_TRY(sums.scratch((size_t)ntiles + 1, s));
    k_scan_tiles<<<ntiles, kScanThreads, 0, s>>>(in, out, n, sums.p); ::bd::note_launch();
    BD_LAUNCH_CHECK();
    const bool scanned = ntiles > kScanDirect;
    if (scanned) {
        k_scan_sums<<<1, kScanThreads, 0, s>>>(sums.p, ntiles, sums.p + ntiles); ::bd::note_launch();
        BD_LAUNCH_CHECK();
    }
    k_scan_add<<<ntiles, kScanThreads, 0, s>>>(out, n, sums.p, scanned, sums.p + ntiles); ::bd::note_launch();
    BD_LAUNCH_CHECK();
    long long t = 0;
    BD_CUDA(cudaMemcpyAsync(&t, sums.p + ntiles, sizeof(t), cudaMemcpyDeviceToHost, s));
    BD_CUDA(cudaStreamSynchronize(s));
    if (t > INT_MAX) return BD_ERANGE;  // (counts are not negative, so no offset exceeds the total)
    if (total) *total = t;
    return BD_OK;
}

// ------------------------------------------------------------------ maximum
// Warp maxima combined by atomicMax: the result does not depend on the order.
__global__ void k_max_int(const int *__restrict__ a, int n, int *out)
{
    int m = 0;
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n;
         i += (long long)gridDim.x * blockDim.x)
        m = max(m, a[i]);
    m = __reduce_max_sync(0xffffffffu, m);
    if ((threadIdx.x & 31) == 0 && m > 0) atomicMax(out, m);
}

int device_max(const int *a, int n, int *slot, cudaStream_t s)
{
    BD_CUDA(cudaMemsetAsync(slot, 0, sizeof(int), s));
    if (n <= 0) return BD_OK;
    k_max_int<<<grid_for(n, 256), 256, 0, s>>>(a, n, slot); ::bd::note_launch();
    BD_LAUNCH_CHECK();
    return BD_OK;
}

// ------------------------------------------------------------------ segmented sort
// One block per segment, bitonic sort in shared memory (padded to a power of 2).
__global__ void k_sort_segments(int *keys, int *payload, const int *seg, int nseg, int P)
{
    extern __shared__ int sm[];
    int *sk = sm, *sp = sm + P;
    for (int g = blockIdx.x; g < nseg; g += gridDim.x) {
        int b = seg[g], len = seg[g + 1] - b;
        if (len <= 1) continue;
        int p2 = 1;
        while (p2 < len) p2 <<= 1;
        for (int i = threadIdx.x; i < p2; i += blockDim.x) {
            sk[i] = i < len ? keys[b + i] : INT_MAX;
            if (payload) sp[i] = i < len ? payload[b + i] : 0;
        }
        __syncthreads();
        for (int k = 2; k <= p2; k <<= 1)
            for (int j = k >> 1; j > 0; j >>= 1) {
                for (int i = threadIdx.x; i < p2; i += blockDim.x) {
                    int ixj = i ^ j;
                    if (ixj > i) {
                        bool up = (i & k) == 0;
                        int ki = sk[i], kj = sk[ixj];
                        if ((ki > kj) == up) {
                            sk[i] = kj;
                            sk[ixj] = ki;
                            if (payload) {
                                int t = sp[i];
                                sp[i] = sp[ixj];
                                sp[ixj] = t;
                            }
                        }
                    }
                }
                __syncthreads();
            }
        for (int i = threadIdx.x; i < len; i += blockDim.x) {
            keys[b + i] = sk[i];
            if (payload) payload[b + i] = sp[i];
        }
        __syncthreads();
    }
}

int sort_segments(int *keys, int *payload, const int *seg, int nseg, int max_len, cudaStream_t s)
{
    if (nseg <= 0 || max_len <= 1) return BD_OK;
    if (max_len > kMaxSortSeg) return BD_ERANGE;
    int P = 1;
    while (P < max_len) P <<= 1;
    size_t smem = 2 * (size_t)P * sizeof(int);
    BD_TRY(allow_smem(k_sort_segments));
    int threads = P >= 256 ? 256 : (P < 32 ? 32 : P);
    int grid = nseg < kSM * 16 ? nseg : kSM * 16;
    k_sort_segments<<<grid, threads, smem, s>>>(keys, payload, seg, nseg, P); ::bd::note_launch();
    BD_LAUNCH_CHECK();
    return BD_OK;
}

// ------------------------------------------------------------------ exact dot
// Long accumulator: limb i holds a signed count of units 2^(32 i - 1074).
// Each rounded product is split into three 32-bit digits and added with
// 64-bit integer atomics (associative, so the result does not depend on the
// order of the additions).

// Digits of a finite double: limb index li and three signed 32-bit digits
// (two's complement in 64 bits) such that x = sum_k d_k 2^(32 (li + k) - 1074).
// Returns false for an infinity or NaN (flag bits in *nf: 1 NaN, 2 +inf, 4 -inf).
__device__ __forceinline__ bool exact_digits(double x, int &li, unsigned long long &d0, unsigned long long &d1,
                                             unsigned long long &d2, int &nf)
{
    unsigned long long b = (unsigned long long)__double_as_longlong(x);
    int neg = (int)(b >> 63);
    int E = (int)((b >> 52) & 0x7ff);
    unsigned long long m = b & 0xFFFFFFFFFFFFFULL;
    li = 0;
    d0 = d1 = d2 = 0;
    nf = 0;
    if (E == 0x7ff) {
        nf = m ? 1 : (neg ? 4 : 2);
        return false;
    }
    int off = 0;
    if (E != 0) {
        m |= (1ULL << 52);
        off = E - 1;
    }
    if (m == 0) return true;
    li = off >> 5;
    const int sh = off & 31;
    unsigned long long t0 = (m & 0xffffffffULL) << sh;
    unsigned long long t1 = (m >> 32) << sh;
    d0 = t0 & 0xffffffffULL;
    unsigned long long u1 = (t0 >> 32) + (t1 & 0xffffffffULL);
    d1 = u1 & 0xffffffffULL;
    d2 = (u1 >> 32) + (t1 >> 32);
    if (neg) {
        d0 = 0ULL - d0;
        d1 = 0ULL - d1;
        d2 = 0ULL - d2;
    }
    return true;
}

__device__ __forceinline__ void exact_acc_digits(long long *acc, int li, unsigned long long d0,
                                                 unsigned long long d1, unsigned long long d2)
{
    unsigned long long *a = (unsigned long long *)acc;
    if (d0) atomicAdd(a + li, d0);
    if (d1) atomicAdd(a + li + 1, d1);
    if (d2) atomicAdd(a + li + 2, d2);
}

// A thread's window: a 256-bit two's complement integer in units of
// 2^(b0 - 1074), b0 a multiple of 32 that the warp's threads share.
struct ExactWindow {
    unsigned long long w[4] = {0, 0, 0, 0};
    __device__ __forceinline__ void add(unsigned long long v0, unsigned long long v1, unsigned long long v2,
                                        unsigned long long v3)
    {
        asm("add.cc.u64 %0, %0, %4;\n\t"
            "addc.cc.u64 %1, %1, %5;\n\t"
            "addc.cc.u64 %2, %2, %6;\n\t"
            "addc.u64 %3, %3, %7;"
            : "+l"(w[0]), "+l"(w[1]), "+l"(w[2]), "+l"(w[3])
            : "l"(v0), "l"(v1), "l"(v2), "l"(v3));
    }
    // p, finite, zero or with its last bit in the window
    __device__ __forceinline__ void add(double p, int b0)
    {
        const unsigned long long bits = (unsigned long long)__double_as_longlong(p);
        const int E = (int)((bits >> 52) & 0x7ff);
        const unsigned long long m = (bits & 0xFFFFFFFFFFFFFULL) | (E ? 1ULL << 52 : 0);
        const int s = max(E, 1) - 1 - b0, r = s & 63, k = s >> 6;
        const unsigned long long neg = (unsigned long long)((long long)bits >> 63);
        // (m << s) negated where the sign is set: xor and add one
        const unsigned long long a = m << r, c = r ? m >> (64 - r) : 0;
        const unsigned long long v0 = k == 0 ? a : 0, v1 = k == 1 ? a : (k == 0 ? c : 0);
        const unsigned long long v2 = k == 2 ? a : (k == 1 ? c : 0), v3 = k == 2 ? c : 0;
        add(v0 ^ neg, v1 ^ neg, v2 ^ neg, v3 ^ neg);
        add(neg & 1, 0, 0, 0);
    }
    // the whole warp's sum to the limbs acc
    __device__ __forceinline__ void flush(int b0, long long *acc)
    {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            unsigned long long v[4];
#pragma unroll
            for (int k = 0; k < 4; k++) v[k] = __shfl_xor_sync(0xffffffffu, w[k], o);
            add(v[0], v[1], v[2], v[3]);
        }
        const int lane = threadIdx.x & 31;
        if (lane < 8) {  // every lane holds the total: lane d adds digit d, the top one signed
            const int q = lane >> 1;
            const unsigned long long x = q == 0 ? w[0] : (q == 1 ? w[1] : (q == 2 ? w[2] : w[3]));
            const long long d = lane == 7 ? (long long)x >> 32 : (long long)((lane & 1) ? x >> 32 : x & 0xffffffffULL);
            if (d) atomicAdd((unsigned long long *)&acc[(b0 >> 5) + lane], (unsigned long long)d);
        }
        w[0] = w[1] = w[2] = w[3] = 0;
    }
};
// Highest position of a product's last bit in the window: 53 bits above it and
// 2^31 of them stay below 2^255.
constexpr int kWindowTop = 169;
constexpr int kNoWindow = 1 << 12;

// Biased exponents of a warp's products (subnormals 1): the largest and the
// smallest of those that are not zero, hi beyond every window for an infinity or NaN.
struct ExactRange {
    int hi = 0, lo = 0x7ff;
    __device__ __forceinline__ void note(double p)
    {
        const unsigned long long b = (unsigned long long)__double_as_longlong(p) << 1;
        const int E = (int)(b >> 53), e = b ? max(E, 1) : 0;
        hi = max(hi, E == 0x7ff ? 1 << 16 : e);
        lo = min(lo, b ? e : 0x7ff);
    }
    __device__ __forceinline__ void of_warp()
    {
        hi = __reduce_max_sync(0xffffffffu, hi);
        lo = __reduce_min_sync(0xffffffffu, lo);
    }
    __device__ __forceinline__ bool in(int b0) const { return hi - 1 - b0 <= kWindowTop && lo - 1 >= b0; }
    // base of a window with the largest 128 to 159 bits above it
    __device__ __forceinline__ int base() const { return max(0, hi - 1 - 128) & ~31; }
};

// The exact total of gacc's limbs rounded to the nearest double (ties to even).
// Called by one whole warp with the limbs in shared memory.
__device__ double exact_round(long long *l, int flags)
{
    const int lane = threadIdx.x & 31;
    int lo = kExactLimbs, hi = -1;
    for (int i0 = 0; i0 < kExactLimbs; i0 += 32) {
        const int i = i0 + lane;
        const unsigned m = __ballot_sync(0xffffffffu, i < kExactLimbs && l[i] != 0);
        if (m) {
            if (lo == kExactLimbs) lo = i0 + __ffs(m) - 1;
            hi = i0 + 31 - __clz(m);
        }
    }
    if (lane != 0) return 0.0;
    if (flags) {
        if ((flags & 1) || ((flags & 2) && (flags & 4))) return __longlong_as_double(0x7ff8000000000000LL);
        return __longlong_as_double((flags & 2) ? 0x7ff0000000000000LL : (long long)0xfff0000000000000ULL);
    }
    if (hi < 0) return 0.0;
    // carries into 32-bit digits; the limb above the highest nonzero one takes the
    // last carry and the sign
    const int end = hi < kExactLimbs - 1 ? hi + 1 : hi;
    bool negative = false;
    for (int pass = 0; pass < 2; pass++) {
        for (int i = lo; i < end; i++) {
            const long long d = l[i] & 0xffffffffLL;
            l[i + 1] += (l[i] - d) >> 32;  // exact: l[i] - d is a multiple of 2^32
            l[i] = d;
        }
        if (pass || l[end] >= 0) break;
        negative = true;
        for (int i = lo; i <= end; i++) l[i] = -l[i];
    }
    int top = end;
    while (top > lo && l[top] == 0) top--;
    double r;
    if (l[top] == 0) return 0.0;
    if (l[top] >= (1LL << 32)) {
        r = __longlong_as_double(0x7ff0000000000000LL);
    } else {
        auto limb = [&](int i) -> unsigned long long { return i >= lo ? (unsigned long long)l[i] : 0ULL; };
        const int H = 32 * top + 31 - __clz((unsigned)l[top]);  // the highest bit
        const unsigned long long u = (limb(top) << 32) | limb(top - 1), v = (limb(top - 2) << 32) | limb(top - 3);
        if (H < 53) {
            r = scalbn((double)(top == 0 ? u >> 32 : u), -1074);
        } else {
            // 128 bits from limb top down; bit H sits at position P
            const int P = 96 + (H & 31), sh = P - 52;  // 44 .. 75
            unsigned long long mant = sh < 64 ? (u << (64 - sh)) | (v >> sh) : u >> (sh - 64);
            const int rb = sh - 1;
            const bool round = rb < 64 ? (v >> rb) & 1 : (u >> (rb - 64)) & 1;
            bool sticky = rb < 64 ? (v & ((1ULL << rb) - 1)) != 0 : v != 0 || (u & ((1ULL << (rb - 64)) - 1)) != 0;
            for (int i = top - 4; i >= lo && !sticky; i--) sticky = l[i] != 0;
            int e = H;
            if (round && (sticky || (mant & 1)) && ++mant == (1ULL << 53)) {
                mant >>= 1;
                e++;
            }
            r = scalbn((double)mant, e - 52 - 1074);
        }
    }
    return negative ? -r : r;
}

// Every thread sums its products in a register window, about 45 integer
// instructions a product.  A warp's threads share the window's place: where their
// next products do not all fit it but would fit another, the window is folded by
// shuffles into the block's limbs and moves there (vectors whose magnitude changes
// along the way, zeros before the first entries).  Products too far apart for one
// window are taken 32 at a time: one window more for those outside the warp's,
// or, if that does not hold them either, the limbs one by one (four copies of
// them, or the block's warps hold each other up).  The blocks add their limbs to the
// global accumulator, and the last block to arrive rounds it.  One launch and a clear.
// Host-timed, 1.1 M and 10 M products, against digit-wise sums per warp step in
// three launches: N(0,1) 70 -> 31 and 323 -> 70 us; the first two thirds zero 51 ->
// 30 and 155 -> 58; falling or rising by e^600 90 -> 36 and 345 -> 71; every second
// product 2^-400 104 -> 41 and 635 -> 151; exponents +-400 at random 48 -> 41 and
// 201 -> 152 (277 with one copy of the limbs).  With windows that stay where a block's first
// products put them the same five took 31, 130, 138, 138, 54 and 70, 731, 1140, 931, 261.
constexpr int kDotThreads = 512, kDotUnroll = 4, kDotCopies = 4;
// Products of two vectors.
struct DotProducts {
    const double *__restrict__ x;
    const double *__restrict__ y;
    __device__ __forceinline__ void start() {}
    __device__ __forceinline__ double operator()(long long j) const { return __dmul_rn(x[j], y[j]); }
};
// Products r_j z_j of the vectors it forms in passing: r -= (num / den) q, z = r / diag.
struct DotUpdate {
    const double *num, *den;
    const double *__restrict__ q;
    const double *__restrict__ diag;
    double *__restrict__ r;
    double *__restrict__ z;
    double alpha;
    __device__ __forceinline__ void start() { alpha = __ddiv_rn(*num, *den); }
    __device__ __forceinline__ double operator()(long long j) const
    {
        const double rj = __dsub_rn(r[j], __dmul_rn(alpha, q[j])), zj = __ddiv_rn(rj, diag[j]);
        r[j] = rj;
        z[j] = zj;
        return __dmul_rn(rj, zj);
    }
};
// clean: the accumulator is zero and is left so (no clear between the calls of a
// sequence).
template <class F>
__global__ void __launch_bounds__(kDotThreads) k_exact_dot(F product, int n, long long *gacc, double *__restrict__ out,
                                                           int clean)
{
    product.start();
    __shared__ long long limbs[kDotCopies][kExactLimbs];
    __shared__ int flags;
    __shared__ bool last;
    for (int i = threadIdx.x; i < kDotCopies * kExactLimbs; i += blockDim.x) (&limbs[0][0])[i] = 0;
    long long *acc = limbs[(threadIdx.x >> 5) % kDotCopies];
    if (threadIdx.x == 0) flags = 0;
    __syncthreads();
    const long long stride = (long long)gridDim.x * blockDim.x;
    const int lane = threadIdx.x & 31;
    ExactWindow W;
    int b0 = kNoWindow;
    auto move = [&](int to) {
        if (b0 != kNoWindow) W.flush(b0, acc);
        b0 = to;
    };
    // the warp's next 32 products, of a step too wide for one window
    auto chunk = [&](double p) {
        ExactRange r;
        r.note(p);
        const ExactRange own = r;
        r.of_warp();
        if (r.hi == 0) return;
        const bool some = __any_sync(0xffffffffu, own.hi && own.in(b0));
        if (!r.in(b0) && (r.in(r.base()) || (!some && r.hi <= 0x7ff))) move(r.base());
        const bool here = own.in(b0);
        ExactRange o;
        if (!here) o = own;
        o.of_warp();
        if (o.hi == 0) {
            W.add(p, b0);
        } else if (o.in(o.base())) {
            ExactWindow T;
            if (here) W.add(p, b0);
            else T.add(p, o.base());
            T.flush(o.base(), acc);
        } else {
            int li, nf;
            unsigned long long d0, d1, d2;
            if (!exact_digits(p, li, d0, d1, d2, nf)) atomicOr(&flags, nf);
            else exact_acc_digits(acc, li, d0, d1, d2);
        }
    };
    for (long long i = blockIdx.x * (long long)blockDim.x + (threadIdx.x & ~31); i < n; i += kDotUnroll * stride) {
        double p[kDotUnroll];
        ExactRange r;
#pragma unroll
        for (int k = 0; k < kDotUnroll; k++) {
            const long long j = i + lane + k * stride;
            p[k] = j < n ? product(j) : 0.0;
        }
#pragma unroll
        for (int k = 0; k < kDotUnroll; k++) r.note(p[k]);
        r.of_warp();
        if (r.hi == 0) continue;
        if (!r.in(b0) && r.in(r.base())) move(r.base());
        if (r.in(b0)) {
#pragma unroll
            for (int k = 0; k < kDotUnroll; k++) W.add(p[k], b0);
        } else {
            static_assert(kDotUnroll == 4, "the steps below");
#pragma unroll 1
            for (int k = 0; k < kDotUnroll; k++) chunk(k == 0 ? p[0] : (k == 1 ? p[1] : (k == 2 ? p[2] : p[3])));
        }
    }
    if (b0 != kNoWindow) W.flush(b0, acc);
    __syncthreads();
    for (int i = threadIdx.x; i < kExactLimbs; i += blockDim.x) {
        long long t = 0;
#pragma unroll
        for (int k = 0; k < kDotCopies; k++) t += limbs[k][i];
        if (t) atomicAdd((unsigned long long *)&gacc[i], (unsigned long long)t);
    }
    if (threadIdx.x == 0 && flags) atomicOr((int *)&gacc[kExactLimbs], flags);
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) last = atomicAdd((unsigned int *)&gacc[kExactLimbs + 1], 1u) == gridDim.x - 1;
    __syncthreads();
    if (!last || threadIdx.x >= 32) return;
    __threadfence();
    for (int i = threadIdx.x; i < kExactLimbs; i += 32) limbs[0][i] = __ldcg(gacc + i);
    __syncwarp();
    const double r = exact_round(limbs[0], (int)__ldcg(gacc + kExactLimbs));
    if (threadIdx.x == 0) *out = r;
    __syncwarp();
    if (clean)
        for (int i = threadIdx.x; i < kExactScratch; i += 32) gacc[i] = 0;
}

// Two blocks per SM at most; a product per thread before a second one (62426
// products in 31 blocks of four 9.2 us, in 122 blocks 8.4).
static int dot_blocks(int n)
{
    return (int)std::max<long long>(1, std::min<long long>(2 * kSM, ((long long)n + kDotThreads - 1) / kDotThreads));
}

int exact_dot(const double *x, const double *y, int n, double *out, long long *acc, cudaStream_t s, bool clean)
{
    if (!clean) BD_CUDA(cudaMemsetAsync(acc, 0, sizeof(long long) * kExactScratch, s));
    k_exact_dot<<<dot_blocks(n), kDotThreads, 0, s>>>(DotProducts{x, y}, n, acc, out, clean); ::bd::note_launch();
    BD_LAUNCH_CHECK();
    return BD_OK;
}

int exact_dot_update(const double *num, const double *den, const double *q, const double *diag, double *r, double *z,
                     int n, double *out, long long *acc, cudaStream_t s)
{
    k_exact_dot<<<dot_blocks(n), kDotThreads, 0, s>>>(DotUpdate{num, den, q, diag, r, z, 0.0}, n, acc, out, 1);
    ::bd::note_launch();
    BD_LAUNCH_CHECK();
    return BD_OK;
}

// ------------------------------------------------------------------ copies
int copy_in(void *dst_dev, const void *src, size_t bytes, int src_on_device, cudaStream_t s)
{
    if (bytes == 0) return BD_OK;
    BD_CUDA(cudaMemcpyAsync(dst_dev, src, bytes,
                            src_on_device ? cudaMemcpyDeviceToDevice : cudaMemcpyHostToDevice, s));
    return BD_OK;
}

int copy_out(void *dst, const void *src_dev, size_t bytes, int dst_on_device, cudaStream_t s)
{
    if (bytes == 0) return BD_OK;
    BD_CUDA(cudaMemcpyAsync(dst, src_dev, bytes,
                            dst_on_device ? cudaMemcpyDeviceToDevice : cudaMemcpyDeviceToHost, s));
    return BD_OK;
}

// ------------------------------------------------------------------ format conversion
__global__ void k_bsr_count(int N, const int *__restrict__ rp, const int *__restrict__ ci,
                            int *cnt, int *bad)
{
    int p = blockIdx.x * blockDim.x + threadIdx.x;
    if (p >= N) return;
    int a = rp[2 * p], b = rp[2 * p + 1], c = rp[2 * p + 2];
    int l0 = b - a, l1 = c - b;
    if (l0 != l1 || (l0 & 1) || l0 < 0) {
        *bad = 1;
        cnt[p] = 0;
        return;
    }
    int prev = -1;
    for (int t = 0; t < l0; t += 2) {
        int c0 = ci[a + t], c1 = ci[a + t + 1], e0 = ci[b + t], e1 = ci[b + t + 1];
        if ((c0 & 1) || c1 != c0 + 1 || e0 != c0 || e1 != c1 || c0 < 0 || c0 / 2 <= prev ||
            c0 / 2 >= N) {
            *bad = 1;
            break;
        }
        prev = c0 / 2;
    }
    cnt[p] = l0 / 2;
}

__global__ void k_bsr_fill(int N, const int *__restrict__ rp, const int *__restrict__ ci,
                           const double *__restrict__ v, const int *__restrict__ brp,
                           int *__restrict__ bci, double *__restrict__ bv)
{
    int p = blockIdx.x * blockDim.x + threadIdx.x;
    if (p >= N) return;
    int a = rp[2 * p], b = rp[2 * p + 1];
    int o = brp[p];
    for (int t = 0, k = 0; t < b - a; t += 2, k++) {
        bci[o + k] = ci[a + t] / 2;
        bv[4 * (size_t)(o + k) + 0] = v[a + t];
        bv[4 * (size_t)(o + k) + 1] = v[a + t + 1];
        bv[4 * (size_t)(o + k) + 2] = v[b + t];
        bv[4 * (size_t)(o + k) + 3] = v[b + t + 1];
    }
}

int bsr_from_scalar_csr(int n, const int *rp, const int *ci, const double *v, BSR &out,
                        cudaStream_t s)
{
    if (n < 2 || (n & 1)) return BD_EINVAL;
    int N = n / 2;
    DBuf<int> cnt, bad;
    BD_TRY(cnt.alloc((size_t)N + 1));
    BD_TRY(bad.alloc(1));
    BD_CUDA(cudaMemsetAsync(bad.p, 0, sizeof(int), s));
    out.nbr = out.nbc = N;
    BD_TRY(out.rp.alloc((size_t)N + 1));
    k_bsr_count<<<(N + 255) / 256, 256, 0, s>>>(N, rp, ci, cnt.p, bad.p); ::bd::note_launch();
    BD_LAUNCH_CHECK();
    int hbad = 0;
    BD_CUDA(cudaMemcpyAsync(&hbad, bad.p, sizeof(int), cudaMemcpyDeviceToHost, s));
    BD_CUDA(cudaStreamSynchronize(s));
    if (hbad) return BD_EINVAL;
    long long nb = 0;
    BD_TRY(exclusive_scan(cnt.p, out.rp.p, N, &nb, s));
    out.nb = nb;
    BD_TRY(out.ci.alloc((size_t)nb));
    BD_TRY(out.v.alloc(4 * (size_t)nb));
    k_bsr_fill<<<(N + 255) / 256, 256, 0, s>>>(N, rp, ci, v, out.rp.p, out.ci.p, out.v.p); ::bd::note_launch();
    BD_LAUNCH_CHECK();
    return BD_OK;
}

int bsr_to_scalar_csr_host(const BSR &a, int *rp, int *ci, double *v, cudaStream_t s)
{
    std::vector<int> brp((size_t)a.nbr + 1), bci((size_t)a.nb);
    std::vector<double> bv(4 * (size_t)a.nb);
    BD_CUDA(cudaMemcpyAsync(brp.data(), a.rp.p, brp.size() * sizeof(int), cudaMemcpyDeviceToHost, s));
    if (a.nb) {
        BD_CUDA(cudaMemcpyAsync(bci.data(), a.ci.p, bci.size() * sizeof(int), cudaMemcpyDeviceToHost, s));
        BD_CUDA(cudaMemcpyAsync(bv.data(), a.v.p, bv.size() * sizeof(double), cudaMemcpyDeviceToHost, s));
    }
    BD_CUDA(cudaStreamSynchronize(s));
    long long pos = 0;
    for (int p = 0; p < a.nbr; p++)
        for (int f = 0; f < 2; f++) {
            if (rp) rp[2 * p + f] = (int)pos;
            for (int t = brp[p]; t < brp[p + 1]; t++)
                for (int g = 0; g < 2; g++) {
                    if (ci) ci[pos] = 2 * bci[t] + g;
                    if (v) v[pos] = bv[4 * (size_t)t + 2 * f + g];
                    pos++;
                }
        }
    if (rp) rp[2 * a.nbr] = (int)pos;
    return BD_OK;
}

// ------------------------------------------------------------------ allocation-free dot
// Scratch of bd_dot_exact_noalloc: one long accumulator (kExactLimbs limbs and
// two words, 560 bytes) in device memory that every GPU loading the library
// holds until the process exits.  Host code must not use the array's name as a
// device address: the address is looked up once per device below.
static __device__ __align__(256) long long g_noalloc_dot_acc[kExactScratch];

constexpr int kNoallocMaxDevices = 64;
static std::mutex g_noalloc_mu;
static long long *g_noalloc_acc[kNoallocMaxDevices];

// Device address of g_noalloc_dot_acc for the current device (first use on a
// device performs the lookup).
static int noalloc_scratch(long long **out)
{
    int dev = 0;
    BD_CUDA(cudaGetDevice(&dev));
    if (dev < 0 || dev >= kNoallocMaxDevices) return BD_ERANGE;
    std::lock_guard<std::mutex> lock(g_noalloc_mu);
    if (!g_noalloc_acc[dev]) {
        void *p = nullptr;
        BD_CUDA(cudaGetSymbolAddress(&p, g_noalloc_dot_acc));
        g_noalloc_acc[dev] = (long long *)p;
    }
    *out = g_noalloc_acc[dev];
    return BD_OK;
}

}  // namespace bd

// ------------------------------------------------------------------ public: misc
extern "C" const char *bd_strerror(int st)
{
    switch (st) {
    case BD_OK: return "ok";
    case BD_EINVAL: return "invalid argument";
    case BD_ENOMEM: return "out of memory";
    case BD_ENOTCONV: return "PCG did not converge within max_it";
    case BD_EBREAKDOWN: return "PCG breakdown (p^T A p <= 0, NaN or Inf)";
    case BD_ETIMEOUT: return "bounded device loop timed out";
    case BD_ECUDA: return "CUDA runtime error";
    case BD_EINCONSISTENT: return "right-hand side not orthogonal to the null space";
    case BD_ERANGE: return "size exceeds a documented maximum";
    case BD_ESTATE: return "handle in the wrong state";
    default: return "unknown status";
    }
}

extern "C" long long bd_launch_count(void) { return bd::g_launches.load(); }

extern "C" int bd_spgemm_path_counts(long long *hash_calls, long long *dense_calls)
{
    if (!hash_calls || !dense_calls) return BD_EINVAL;
    *hash_calls = bd::spgemm_path_count(false);
    *dense_calls = bd::spgemm_path_count(true);
    return BD_OK;
}

extern "C" int bd_dot_exact(const double *x, const double *y, long long n, int on_device,
                            double *out, void *stream)
{
    if (!x || !y || !out || n < 0) return BD_EINVAL;
    if (n > 2147483647LL) return BD_ERANGE;
    cudaStream_t s = (cudaStream_t)stream;
    bd::DBuf<long long> acc;
    bd::DBuf<double> res, dx, dy;
    BD_TRY(acc.alloc(bd::kExactScratch));
    BD_TRY(res.alloc(1));
    const double *px = x, *py = y;
    if (!on_device && n > 0) {
        BD_TRY(dx.alloc((size_t)n));
        BD_TRY(dy.alloc((size_t)n));
        BD_TRY(bd::copy_in(dx.p, x, sizeof(double) * (size_t)n, 0, s));
        BD_TRY(bd::copy_in(dy.p, y, sizeof(double) * (size_t)n, 0, s));
        px = dx.p;
        py = dy.p;
    }
    BD_TRY(bd::exact_dot(px, py, (int)n, res.p, acc.p, s));
    BD_CUDA(cudaMemcpyAsync(out, res.p, sizeof(double), cudaMemcpyDeviceToHost, s));
    BD_CUDA(cudaStreamSynchronize(s));
    return BD_OK;
}

extern "C" int bd_dot_exact_noalloc(const double *x, const double *y, long long n, double *out,
                                    void *stream)
{
    if (!x || !y || !out || n < 0) return BD_EINVAL;
    if (n > 2147483647LL) return BD_ERANGE;
    long long *acc = nullptr;
    BD_TRY(bd::noalloc_scratch(&acc));
    // exact_dot clears the accumulator on `stream`, then launches one kernel whose
    // last block rounds; nothing is allocated.
    return bd::exact_dot(x, y, (int)n, out, acc, (cudaStream_t)stream);
}

extern "C" void amg_options_default(amg_options *o)
{
    if (!o) return;
    o->theta = 0.06;
    o->coarse_eq_limit = 100;
    o->max_levels = 10;
    o->cheb_degree = 2;
    o->esteig_steps = 10;
    o->square_levels = 16;  /* every level (App. A squares the first only) */
    o->eig_lo = 0.05;
    o->eig_hi = 1.05;
    o->seed = 0;
    o->precision = 0;
    o->autotune = 0;
}

extern "C" void solve_options_default(solve_options *o)
{
    if (!o) return;
    o->rtol = 1e-8;
    o->max_it = 500;
    o->warm_start = 0;
    o->strict = 0;
}

extern "C" void bd_rm_params_default(bd_rm_params *p)
{
    if (!p) return;
    p->G = 1.5;
    p->vth = 13.0;
    p->vp = 100.0;
    p->eta1 = 4.4;
    p->eta2 = 0.012;
    p->eta3 = 1.0;
}
