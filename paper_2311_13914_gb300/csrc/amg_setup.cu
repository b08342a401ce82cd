// amg_setup.cu -- a1..a9: smoothed-aggregation hierarchy setup on the device
// (Algorithm 1; Section 4 for the strength graph, MIS, cluster rule and
// tentative prolongator; Appendix A for the squared graph, one prolongator
// smoothing step, the 10-step CG eigen-estimate and the coarse limit).
//
// Compiled with -fmad=false.  Every floating-point value that decides an
// integer (strength, aggregate choice) or enters the next level is formed by
// the documented sequence of rounded operations: sums over the middle index in
// ascending order, correctly rounded dot products, IEEE sqrt and division.
// Aggregates and sparsity patterns are therefore bit-identical to any
// implementation that follows the same order, whatever the thread schedule.
#include <algorithm>
#include <new>
#include <climits>
#include <cmath>

#include "amg_internal.cuh"
#include "grid_index.h"
#include "scalar.cuh"

namespace bd {

// ------------------------------------------------------------------ hashing
__host__ __device__ __forceinline__ unsigned long long mix64(unsigned long long z)
{
    z = (z ^ (z >> 30)) * 0xbf58476d1ce4e5b9ULL;
    z = (z ^ (z >> 27)) * 0x94d049bb133111ebULL;
    return z ^ (z >> 31);
}

static unsigned long long level_key(unsigned long long seed, int level, int stream)
{
    return mix64(seed + 0x9E3779B97F4A7C15ULL * (unsigned long long)(2 * level + stream + 1));
}

__device__ __forceinline__ int find_block(const int *__restrict__ rp, const int *__restrict__ ci,
                                          int row, int col)
{
    int lo = rp[row], hi = rp[row + 1] - 1;
    while (lo <= hi) {
        int mid = (lo + hi) >> 1;
        int c = ci[mid];
        if (c == col) return mid;
        if (c < col) lo = mid + 1;
        else hi = mid - 1;
    }
    return -1;
}

// ------------------------------------------------------------------ diagonal
__global__ void k_diag(int N, const int *__restrict__ rp, const int *__restrict__ ci,
                       const double *__restrict__ v, double *__restrict__ diag, int *bad)
{
    int p = blockIdx.x * blockDim.x + threadIdx.x;
    if (p >= N) return;
    int t = find_block(rp, ci, p, p);
    double d0 = t >= 0 ? v[4 * (size_t)t] : 0.0, d1 = t >= 0 ? v[4 * (size_t)t + 3] : 0.0;
    if (!(d0 > 0.0) || !(d1 > 0.0)) *bad = 1;
    diag[2 * p] = d0;
    diag[2 * p + 1] = d1;
}

// ------------------------------------------------------------------ a1 strength
// w_pq = 0.5 (|A_u(p,q)| + |A_u(q,p)|) / sqrt(A_u(p,p) A_u(q,q)), kept if >= theta,
// A_u = the (u_e, u_e) entry of the 2x2 node block.
__device__ __forceinline__ bool strength_w(const int *rp, const int *ci, const double *v,
                                           const double *diag, int p, int t, double theta,
                                           double *w_out)
{
    int q = ci[t];
    if (q == p) return false;
    int tt = find_block(rp, ci, q, p);
    double apq = fabs(v[4 * (size_t)t + 3]);
    double aqp = tt >= 0 ? fabs(v[4 * (size_t)tt + 3]) : 0.0;
    double num = 0.5 * (apq + aqp);
    double den = sqrt(diag[2 * p + 1] * diag[2 * q + 1]);
    if (!(den > 0.0)) return false;
    double w = num / den;
    *w_out = w;
    return w >= theta;
}

// One pass forms every entry's weight (a square root and a division, costly
// on the FP64 pipe) and counts the strong ones; wt[t] keeps the weight of a
// strong entry and -1 otherwise (weights are >= 0), so the fill only compacts.
// A warp per row: entries are independent, and each looks its transpose up by a
// chain of dependent loads (with a thread per row, 2718 rows of 223 blocks took
// 1250 us).
__global__ void k_strength_count(int N, const int *__restrict__ rp, const int *__restrict__ ci,
                                 const double *__restrict__ v, const double *__restrict__ diag,
                                 double theta, int *cnt, double *__restrict__ wt)
{
    const int lane = threadIdx.x & 31, p = grid_row<5>(blockIdx.x, blockDim.x, threadIdx.x);
    if (p >= N) return;
    int c = 0;
    for (int t = rp[p] + lane; t < rp[p + 1]; t += 32) {
        double w = 0.0;
        const bool strong = strength_w(rp, ci, v, diag, p, t, theta, &w);
        wt[t] = strong ? w : -1.0;
        c += strong;
    }
    c = __reduce_add_sync(0xffffffffu, c);
    if (lane == 0) cnt[p] = c;
}

__global__ void k_strength_fill(int N, const int *__restrict__ rp, const int *__restrict__ ci,
                                const double *__restrict__ wt, const int *__restrict__ srp,
                                int *__restrict__ sci, double *__restrict__ sw)
{
    const int lane = threadIdx.x & 31, p = grid_row<5>(blockIdx.x, blockDim.x, threadIdx.x);
    if (p >= N) return;
    int pos = srp[p];
    for (int t0 = rp[p]; t0 < rp[p + 1]; t0 += 32) {
        const int t = t0 + lane;
        const double w = t < rp[p + 1] ? wt[t] : -1.0;
        const unsigned m = __ballot_sync(0xffffffffu, w >= 0.0);
        if (w >= 0.0) {
            const int o = pos + __popc(m & ((1u << lane) - 1u));
            sci[o] = ci[t];
            sw[o] = w;
        }
        pos += __popc(m);
    }
}

// ------------------------------------------------------------------ deterministic SpGEMM
// C = A B for BS x BS block CSR (BS = 1 scalar, 2 node blocks).  One thread
// block per output row; a dense accumulator indexed by output column lives in
// global scratch (one slice per resident block); touched columns are listed
// in shared memory, sorted, and emitted ascending.  Every entry is
// accumulated as acc = acc + a*b over the scalar middle index in ascending
// order (for BS = 2: middle block k ascending, then its two scalar columns).
template <int BS>
__global__ void k_spgemm_count(int nrows, const int *__restrict__ arp, const int *__restrict__ aci,
                               const int *__restrict__ brp, const int *__restrict__ bci, int ncols,
                               int *__restrict__ mark_all, int *__restrict__ cnt, int *longest)
{
    __shared__ int count;
    int most = 0;
    int *mark = mark_all + (size_t)blockIdx.x * ncols;
    for (int i = blockIdx.x; i < nrows; i += gridDim.x) {
        if (threadIdx.x == 0) count = 0;
        __syncthreads();
        for (int t = arp[i]; t < arp[i + 1]; t++) {
            int k = aci[t];
            for (int s = brp[k] + threadIdx.x; s < brp[k + 1]; s += blockDim.x) {
                int j = bci[s];
                if (atomicExch(&mark[j], i) != i) atomicAdd(&count, 1);
            }
        }
        __syncthreads();
        if (threadIdx.x == 0) cnt[i] = count;
        most = max(most, count);
        __syncthreads();
    }
    if (threadIdx.x == 0 && most > 0) atomicMax(longest, most);
}

template <int BS>
__global__ void k_spgemm_fill(int nrows, const int *__restrict__ arp, const int *__restrict__ aci,
                              const double *__restrict__ av, const int *__restrict__ brp,
                              const int *__restrict__ bci, const double *__restrict__ bv, int ncols,
                              int *__restrict__ mark_all, double *__restrict__ acc_all,
                              const int *__restrict__ crp, int *__restrict__ cci,
                              double *__restrict__ cv, int P2)
{
    extern __shared__ int cols[];
    __shared__ int count;
    constexpr int BB = BS * BS;
    int *mark = mark_all + (size_t)blockIdx.x * ncols;
    double *acc = acc_all + (size_t)blockIdx.x * ncols * BB;
    for (int i = blockIdx.x; i < nrows; i += gridDim.x) {
        if (threadIdx.x == 0) count = 0;
        __syncthreads();
        for (int t = arp[i]; t < arp[i + 1]; t++) {
            int k = aci[t];
            double a[BB];
#pragma unroll
            for (int e = 0; e < BB; e++) a[e] = av[(size_t)t * BB + e];
            for (int s = brp[k] + threadIdx.x; s < brp[k + 1]; s += blockDim.x) {
                int j = bci[s];
                double *c = acc + (size_t)j * BB;
                if (mark[j] != i) {
                    mark[j] = i;
#pragma unroll
                    for (int e = 0; e < BB; e++) c[e] = 0.0;
                    cols[atomicAdd(&count, 1)] = j;
                }
                const double *b = bv + (size_t)s * BB;
                if (BS == 1) {
                    c[0] = c[0] + a[0] * b[0];
                } else {
                    // scalar middle index 2k then 2k+1
                    c[0] = c[0] + a[0] * b[0];
                    c[0] = c[0] + a[1] * b[2];
                    c[1] = c[1] + a[0] * b[1];
                    c[1] = c[1] + a[1] * b[3];
                    c[2] = c[2] + a[2] * b[0];
                    c[2] = c[2] + a[3] * b[2];
                    c[3] = c[3] + a[2] * b[1];
                    c[3] = c[3] + a[3] * b[3];
                }
            }
            __syncthreads();
        }
        int n = count;
        int p2 = 1;
        while (p2 < n) p2 <<= 1;
        for (int x = n + threadIdx.x; x < p2; x += blockDim.x) cols[x] = INT_MAX;
        __syncthreads();
        for (int kk = 2; kk <= p2; kk <<= 1)
            for (int jj = kk >> 1; jj > 0; jj >>= 1) {
                for (int x = threadIdx.x; x < p2; x += blockDim.x) {
                    int y = x ^ jj;
                    if (y > x) {
                        bool up = (x & kk) == 0;
                        int cx = cols[x], cy = cols[y];
                        if ((cx > cy) == up) {
                            cols[x] = cy;
                            cols[y] = cx;
                        }
                    }
                }
                __syncthreads();
            }
        int base = crp[i];
        for (int x = threadIdx.x; x < n; x += blockDim.x) {
            int j = cols[x];
            cci[base + x] = j;
#pragma unroll
            for (int e = 0; e < BB; e++) cv[(size_t)(base + x) * BB + e] = acc[(size_t)j * BB + e];
        }
        __syncthreads();
    }
    (void)P2;
}

// The middles [t, te) of an output row, one at a time: the block a of A and the
// entry of B's row that a thread of offset `off` takes first, with the loads of
// the following middles in flight (column of the third, range of the second,
// entry of the next): three dependent loads from L2 would otherwise stand between
// a middle's products and the next's.
template <int BS> struct MidWalk {
    static constexpr int BB = BS * BS;
    const int *__restrict__ aci;
    const double *__restrict__ av;
    const int *__restrict__ brp;
    const int *__restrict__ bci;
    const double *__restrict__ bv;
    int t, te, off;
    int s0, s1, j;          // this middle
    double a[BB], b[BB];
    int n0, n1, jn;         // the next one
    double an[BB], bn[BB];
    int m0, m1, k3;         // range of the second, column of the third

    static __device__ __forceinline__ void load(const double *__restrict__ v, size_t at, double (&o)[BB])
    {
        if constexpr (BS == 2) {
            const double2 x = ((const double2 *)v)[2 * at], y = ((const double2 *)v)[2 * at + 1];
            o[0] = x.x;
            o[1] = x.y;
            o[2] = y.x;
            o[3] = y.y;
        } else {
            o[0] = v[at];
        }
    }
    __device__ __forceinline__ int column(int q) const { return q < te ? aci[q] : -1; }
    __device__ __forceinline__ void range(int k, int &b0, int &b1) const
    {
        b0 = k >= 0 ? brp[k] : 0;
        b1 = k >= 0 ? brp[k + 1] : 0;
    }
    __device__ __forceinline__ void entry(int q, int b0, int b1, int &jj, double (&aa)[BB], double (&bb)[BB]) const
    {
        if (q < te) load(av, (size_t)q, aa);
        if (b0 + off < b1) {
            jj = bci[b0 + off];
            load(bv, (size_t)(b0 + off), bb);
        }
    }
    __device__ __forceinline__ void start(int t_, int te_, int off_)
    {
        t = t_;
        te = te_;
        off = off_;
        const int k0 = column(t), k1 = column(t + 1), k2 = column(t + 2);
        k3 = column(t + 3);
        range(k0, s0, s1);
        range(k1, n0, n1);
        range(k2, m0, m1);
        j = jn = 0;
        entry(t, s0, s1, j, a, b);
        entry(t + 1, n0, n1, jn, an, bn);
    }
    __device__ __forceinline__ void next()
    {
        t++;
        s0 = n0;
        s1 = n1;
        j = jn;
#pragma unroll
        for (int e = 0; e < BB; e++) {
            a[e] = an[e];
            b[e] = bn[e];
        }
        n0 = m0;
        n1 = m1;
        range(k3, m0, m1);
        k3 = column(t + 3);
        entry(t + 1, n0, n1, jn, an, bn);
    }
    // f(column, block of B) for this middle's entries off, off + stride, ...
    template <class F> __device__ __forceinline__ void entries(int stride, F &&f) const
    {
        int q = s0 + off, jc = j;
        if (q >= s1) return;
        double bc[BB];
#pragma unroll
        for (int e = 0; e < BB; e++) bc[e] = b[e];
        for (;;) {
            const int q2 = q + stride;
            const bool more = q2 < s1;
            int j2 = 0;
            double b2[BB];
            if (more) {
                j2 = bci[q2];
                load(bv, (size_t)q2, b2);
            }
            f(jc, bc);
            if (!more) break;
            jc = j2;
#pragma unroll
            for (int e = 0; e < BB; e++) bc[e] = b2[e];
            q = q2;
        }
    }
};

// The same for 2x2 blocks by groups of four lanes, lane e of a group forming element e
// of its entry's product: group `grp` of the row's G takes entries grp, grp + G, ...
struct MidWalkElem {
    const int *__restrict__ aci;
    const double *__restrict__ av;
    const int *__restrict__ brp;
    const int *__restrict__ bci;
    const double *__restrict__ bv;
    int t, te, grp, e;
    int s0, s1, j;
    double2 a;              // the row of a that element e needs
    double b0, b1;          // and the column of b
    int n0, n1, jn;
    double2 an;
    double bn0, bn1;
    int m0, m1, k3;

    __device__ __forceinline__ int column(int q) const { return q < te ? aci[q] : -1; }
    __device__ __forceinline__ void range(int k, int &r0, int &r1) const
    {
        r0 = k >= 0 ? brp[k] : 0;
        r1 = k >= 0 ? brp[k + 1] : 0;
    }
    __device__ __forceinline__ void block(int q, int &jj, double &x, double &y) const
    {
        jj = bci[q];
        const double *b = bv + 4 * (size_t)q + (e & 1);
        x = b[0];
        y = b[2];
    }
    __device__ __forceinline__ void entry(int q, int r0, int r1, int &jj, double2 &aa, double &x, double &y) const
    {
        if (q < te) aa = ((const double2 *)av)[2 * (size_t)q + (e >> 1)];
        if (r0 + grp < r1) block(r0 + grp, jj, x, y);
    }
    __device__ __forceinline__ void start(int t_, int te_, int grp_, int e_)
    {
        t = t_;
        te = te_;
        grp = grp_;
        e = e_;
        const int k0 = column(t), k1 = column(t + 1), k2 = column(t + 2);
        k3 = column(t + 3);
        range(k0, s0, s1);
        range(k1, n0, n1);
        range(k2, m0, m1);
        j = jn = 0;
        a = an = make_double2(0.0, 0.0);
        b0 = b1 = bn0 = bn1 = 0.0;
        entry(t, s0, s1, j, a, b0, b1);
        entry(t + 1, n0, n1, jn, an, bn0, bn1);
    }
    __device__ __forceinline__ void next()
    {
        t++;
        s0 = n0;
        s1 = n1;
        j = jn;
        a = an;
        b0 = bn0;
        b1 = bn1;
        n0 = m0;
        n1 = m1;
        range(k3, m0, m1);
        k3 = column(t + 3);
        entry(t + 1, n0, n1, jn, an, bn0, bn1);
    }
    // f(has an entry, column, b) by all lanes together
    template <class F> __device__ __forceinline__ void entries(int G, F &&f) const
    {
        int q = s0 + grp, jc = j;
        double x = b0, y = b1;
        for (int base = s0; base < s1; base += G) {
            const int q2 = q + G;
            int j2 = 0;
            double x2 = 0.0, y2 = 0.0;
            if (q2 < s1) block(q2, j2, x2, y2);
            f(q < s1, jc, x, y);
            q = q2;
            jc = j2;
            x = x2;
            y = y2;
        }
    }
    // element e of c + a b, or of a b (fresh), in the order of block_mac
    __device__ __forceinline__ double mac(double c, bool fresh, double x, double y) const
    {
        double v = fresh ? 0.0 : c;
        v = v + a.x * x;
        v = v + a.y * y;
        return v;
    }
};

// c (+)= a b in the order of the scalar middle index (2k, then 2k + 1); fresh:
// from zero.  c's elements are `plane` apart.
template <int BS>
__device__ __forceinline__ void block_mac(double *c, int plane, const double (&a)[BS * BS], const double (&b)[BS * BS],
                                          bool fresh)
{
    constexpr int BB = BS * BS;
    double v[BB];
#pragma unroll
    for (int e = 0; e < BB; e++) v[e] = fresh ? 0.0 : c[(size_t)e * plane];
    if (BS == 1) {
        v[0] = v[0] + a[0] * b[0];
    } else {
        v[0] = v[0] + a[0] * b[0];
        v[1] = v[1] + a[0] * b[1];
        v[2] = v[2] + a[2] * b[0];
        v[3] = v[3] + a[2] * b[1];
        v[0] = v[0] + a[1] * b[2];
        v[1] = v[1] + a[1] * b[3];
        v[2] = v[2] + a[3] * b[2];
        v[3] = v[3] + a[3] * b[3];
    }
#pragma unroll
    for (int e = 0; e < BB; e++) c[(size_t)e * plane] = v[e];
}

// Dense path with the row's accumulators and column marks in shared memory
// (coarse levels: few columns), otherwise identical to k_spgemm_count /
// k_spgemm_fill: a block per output row, every entry accumulated in ascending
// middle index.  Shared memory: marks (ncols ints) for the count; marks,
// accumulators (ncols x BB doubles) and the row's column list (P2 ints) for
// the fill.
__global__ void k_spgemm_count_smem(int nrows, const int *__restrict__ arp, const int *__restrict__ aci,
                                    const int *__restrict__ brp, const int *__restrict__ bci, int ncols,
                                    int *__restrict__ cnt, int *longest)
{
    int most = 0;
    extern __shared__ int smark[];
    __shared__ int count;
    for (int j = threadIdx.x; j < ncols; j += blockDim.x) smark[j] = -1;
    __syncthreads();
    for (int i = blockIdx.x; i < nrows; i += gridDim.x) {
        if (threadIdx.x == 0) count = 0;
        __syncthreads();
        for (int t = arp[i]; t < arp[i + 1]; t++) {
            int k = aci[t];
            for (int s2 = brp[k] + threadIdx.x; s2 < brp[k + 1]; s2 += blockDim.x) {
                int j = bci[s2];
                if (atomicExch(&smark[j], i) != i) atomicAdd(&count, 1);
            }
        }
        __syncthreads();
        if (threadIdx.x == 0) cnt[i] = count;
        most = max(most, count);
        __syncthreads();
    }
    if (threadIdx.x == 0 && most > 0) atomicMax(longest, most);
}

template <int BS>
__global__ void k_spgemm_fill_smem(int nrows, const int *__restrict__ arp, const int *__restrict__ aci,
                                   const double *__restrict__ av, const int *__restrict__ brp,
                                   const int *__restrict__ bci, const double *__restrict__ bv, int ncols,
                                   const int *__restrict__ crp, int *__restrict__ cci, double *__restrict__ cv)
{
    constexpr int BB = BS * BS;
    extern __shared__ double sacc[];
    int *mark = (int *)(sacc + (size_t)ncols * BB);
    int *cols = mark + ncols;
    __shared__ int count;
    for (int j = threadIdx.x; j < ncols; j += blockDim.x) mark[j] = -1;
    __syncthreads();
    for (int i = blockIdx.x; i < nrows; i += gridDim.x) {
        if (threadIdx.x == 0) count = 0;
        __syncthreads();
        if constexpr (BS == 2) {
            MidWalkElem w{aci, av, brp, bci, bv};
            const int lane = threadIdx.x & 31, e = threadIdx.x & 3;
            for (w.start(arp[i], arp[i + 1], threadIdx.x >> 2, e); w.t < w.te; w.next()) {
                w.entries(blockDim.x >> 2, [&](bool on, int j, double x, double y) {
                    bool fresh = false;
                    if (on && e == 0) {
                        fresh = mark[j] != i;
                        if (fresh) {
                            mark[j] = i;
                            cols[atomicAdd(&count, 1)] = j;
                        }
                    }
                    fresh = __shfl_sync(0xffffffffu, (int)fresh, lane & ~3);
                    double *c = sacc + 4 * (size_t)j + e;
                    if (on) *c = w.mac(*c, fresh, x, y);
                });
                __syncthreads();
            }
        } else {
            MidWalk<BS> w{aci, av, brp, bci, bv};
            for (w.start(arp[i], arp[i + 1], threadIdx.x); w.t < w.te; w.next()) {
                w.entries(blockDim.x, [&](int j, const double (&b)[BB]) {
                    const bool fresh = mark[j] != i;
                    if (fresh) {
                        mark[j] = i;
                        cols[atomicAdd(&count, 1)] = j;
                    }
                    block_mac<BS>(sacc + j, 1, w.a, b, fresh);
                });
                __syncthreads();
            }
        }
        int n = count;
        int p2 = 1;
        while (p2 < n) p2 <<= 1;
        for (int x = n + threadIdx.x; x < p2; x += blockDim.x) cols[x] = INT_MAX;
        __syncthreads();
        for (int kk = 2; kk <= p2; kk <<= 1)
            for (int jj = kk >> 1; jj > 0; jj >>= 1) {
                for (int x = threadIdx.x; x < p2; x += blockDim.x) {
                    int y = x ^ jj;
                    if (y > x) {
                        bool up = (x & kk) == 0;
                        int cx = cols[x], cy = cols[y];
                        if ((cx > cy) == up) {
                            cols[x] = cy;
                            cols[y] = cx;
                        }
                    }
                }
                __syncthreads();
            }
        int base = crp[i];
        for (int x = threadIdx.x; x < n; x += blockDim.x) {
            int j = cols[x];
            cci[base + x] = j;
#pragma unroll
            for (int e = 0; e < BB; e++) cv[(size_t)(base + x) * BB + e] = sacc[(size_t)j * BB + e];
        }
        __syncthreads();
    }
}

// Hash path for products with very many columns and short rows (the squared
// strength graph of a large fine level): one warp per output row, open
// addressing in shared memory, the same accumulation order.
__device__ __forceinline__ int hslot(int key, int mask) { return (int)(((unsigned)key * 2654435761u) & (unsigned)mask); }

// Largest number of products of a row; eight lanes per row (rows of hundreds of
// blocks: a thread's chain of loads).
__global__ void k_spgemm_bound(int nrows, const int *__restrict__ arp, const int *__restrict__ aci,
                               const int *__restrict__ brp, int *__restrict__ ub)
{
    const int i = grid_row<3>(blockIdx.x, blockDim.x, threadIdx.x), l = threadIdx.x & 7;
    long long u = 0;
    if (i < nrows)
        for (int t = arp[i] + l; t < arp[i + 1]; t += 8) u += brp[aci[t] + 1] - brp[aci[t]];
    for (int o = 4; o; o >>= 1) u += __shfl_xor_sync(0xffffffffu, u, o);
    const int m = __reduce_max_sync(0xffffffffu, u > INT_MAX ? INT_MAX : (int)u);
    if ((threadIdx.x & 31) == 0 && m > 0) atomicMax(ub, m);
}

// Hash-path SpGEMM: L lanes per output row, 32/L rows per warp (L from the
// average row length of B, so that short rows of B -- a tentative
// prolongator has one block per row -- do not leave most lanes idle: every
// FP64 instruction costs the pipe a full warp slot however few lanes are on).
// Each row has its own hash table in shared memory.
template <int L>
__device__ __forceinline__ unsigned sub_mask(int lane)
{
    return L == 32 ? 0xffffffffu : (((1u << L) - 1u) << (lane & ~(L - 1)));
}

template <int L>
__global__ void k_spgemm_count_hash(int nrows, const int *__restrict__ arp, const int *__restrict__ aci,
                                    const int *__restrict__ brp, const int *__restrict__ bci, int HC,
                                    int *__restrict__ cnt, int *overflow, int *longest)
{
    constexpr int R = 32 / L;
    extern __shared__ int hk[];
    const int warps = blockDim.x >> 5, wid = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int sub = lane / L, sl = lane % L;
    int most = 0;
    int *keys = hk + ((size_t)wid * R + sub) * HC;
    for (int base = (blockIdx.x * warps + wid) * R; base < nrows; base += gridDim.x * warps * R) {
        const int i = base + sub;
        for (int x = sl; x < HC; x += L) keys[x] = -1;
        __syncwarp();
        int c = 0;
        bool full = false;
        if (i < nrows) {
            // the columns of the middles after this one, as MidWalk
            const int te = arp[i + 1];
            int t = arp[i];
            auto column = [&](int q) { return q < te ? aci[q] : -1; };
            auto first = [&](int b0, int b1) { return b0 + sl < b1 ? bci[b0 + sl] : 0; };
            const int k0 = column(t), k1 = column(t + 1), k2 = column(t + 2);
            int k3 = column(t + 3);
            int s0 = k0 >= 0 ? brp[k0] : 0, s1 = k0 >= 0 ? brp[k0 + 1] : 0;
            int n0 = k1 >= 0 ? brp[k1] : 0, n1 = k1 >= 0 ? brp[k1 + 1] : 0;
            int m0 = k2 >= 0 ? brp[k2] : 0, m1 = k2 >= 0 ? brp[k2 + 1] : 0;
            int j = first(s0, s1), jn = first(n0, n1);
            for (; t < te; t++) {
                for (int q = s0 + sl; q < s1 && !full; q += L) {
                    const int j2 = q + L < s1 ? bci[q + L] : 0;
                    int h = hslot(j, HC - 1), probe = 0;
                    for (; probe < HC; probe++) {
                        int old = atomicCAS(&keys[h], -1, j);
                        if (old == -1) { c++; break; }
                        if (old == j) break;
                        h = (h + 1) & (HC - 1);
                    }
                    full = probe == HC;
                    j = j2;
                }
                s0 = n0;
                s1 = n1;
                j = jn;
                n0 = m0;
                n1 = m1;
                m0 = k3 >= 0 ? brp[k3] : 0;
                m1 = k3 >= 0 ? brp[k3 + 1] : 0;
                k3 = column(t + 4);
                jn = first(n0, n1);
            }
            if (full) atomicOr(overflow, 1);
        }
#pragma unroll
        for (int o = L / 2; o; o >>= 1) c += __shfl_xor_sync(0xffffffffu, c, o, L);
        if (i < nrows && sl == 0) cnt[i] = c;
        most = max(most, c);
        __syncwarp();
    }
    most = __reduce_max_sync(0xffffffffu, most);
    if (lane == 0 && most > 0) atomicMax(longest, most);
}

template <int BS, int L>
__global__ void k_spgemm_fill_hash(int nrows, const int *__restrict__ arp, const int *__restrict__ aci,
                                   const double *__restrict__ av, const int *__restrict__ brp,
                                   const int *__restrict__ bci, const double *__restrict__ bv, int HC,
                                   const int *__restrict__ crp, int *__restrict__ cci,
                                   double *__restrict__ cv)
{
    constexpr int BB = BS * BS;
    constexpr int R = 32 / L;
    extern __shared__ double hs[];
    const int warps = blockDim.x >> 5, wid = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int sub = lane / L, sl = lane % L;
    const size_t per = (size_t)HC * BB + (size_t)(3 * HC + 1) / 2;  // in doubles
    double *acc = hs + ((size_t)wid * R + sub) * per;
    int *keys = (int *)(acc + (size_t)HC * BB);
    int *sk = keys + HC, *sp = sk + HC;
    for (int base = (blockIdx.x * warps + wid) * R; base < nrows; base += gridDim.x * warps * R) {
        const int i = base + sub;
        const bool act = i < nrows;
        for (int x = sl; x < HC; x += L) keys[x] = -1;
        __syncwarp();
        // middle indices in ascending order, all rows of the warp in step (a
        // barrier per middle index keeps each entry's additions in that order)
        const int t0 = act ? arp[i] : 0, tn = act ? arp[i + 1] - t0 : 0;
        int tmax = tn;
#pragma unroll
        for (int o = 16; o; o >>= 1) tmax = max(tmax, __shfl_xor_sync(0xffffffffu, tmax, o));
        MidWalk<BS> w{aci, av, brp, bci, bv};
        w.start(t0, t0 + tn, sl);
        for (int tt = 0; tt < tmax; tt++, w.next()) {
            w.entries(L, [&](int j, const double (&b)[BB]) {
                int h = hslot(j, HC - 1);
                bool fresh = false;
                for (int probe = 0; probe < HC; probe++) {
                    const int old = atomicCAS(&keys[h], -1, j);
                    fresh = old == -1;
                    if (fresh || old == j) break;
                    h = (h + 1) & (HC - 1);
                }
                block_mac<BS>(acc + h, HC, w.a, b, fresh);
            });
            __syncwarp();
        }
        // compact the occupied slots, sort them by column, emit
        const unsigned smask = sub_mask<L>(lane);
        int n = 0;
        for (int x0 = 0; x0 < HC; x0 += L) {
            const int x = x0 + sl;
            const bool has = keys[x] != -1;
            const unsigned m = __ballot_sync(0xffffffffu, has) & smask;
            if (has) {
                const int pos = n + __popc(m & ((1u << lane) - 1u));
                sk[pos] = keys[x];
                sp[pos] = x;
            }
            n += __popc(m);
        }
        int p2 = 1;
        while (p2 < n) p2 <<= 1;
        int p2max = p2;
#pragma unroll
        for (int o = 16; o; o >>= 1) p2max = max(p2max, __shfl_xor_sync(0xffffffffu, p2max, o));
        for (int x = n + sl; x < p2max; x += L) {
            sk[x] = INT_MAX;
            sp[x] = 0;
        }
        __syncwarp();
        for (int kk = 2; kk <= p2max; kk <<= 1)
            for (int jj = kk >> 1; jj > 0; jj >>= 1) {
                for (int x = sl; x < p2max; x += L) {
                    int y = x ^ jj;
                    if (y > x) {
                        bool up = (x & kk) == 0;
                        int cx = sk[x], cy = sk[y];
                        if ((cx > cy) == up) {
                            sk[x] = cy;
                            sk[y] = cx;
                            int tp = sp[x];
                            sp[x] = sp[y];
                            sp[y] = tp;
                        }
                    }
                }
                __syncwarp();
            }
        if (act) {
            const int cb = crp[i];
            for (int x = sl; x < n; x += L) {
                cci[cb + x] = sk[x];
#pragma unroll
                for (int e = 0; e < BB; e++) cv[(size_t)(cb + x) * BB + e] = acc[(size_t)e * HC + sp[x]];
            }
        }
        __syncwarp();
    }
}

// Hash path with a warp per row and four lanes per product (MidWalkElem): eight
// products at a time in four FP64 instructions, where a lane per product takes
// sixteen for up to 32 and leaves most lanes idle on rows of B of 7 to 20 blocks, and
// half of one row's chain of middles.  128x128x32: the finest A P (rows of B of 6.8
// blocks) 6.6 -> 5.2 ms, R (A P) 4.9 -> 4.0, the next level's 3.1 -> 2.4 (the FP64
// operations at full lanes take 2.5, 2.0 and 1.2); 48x48x12, 1463 rows of 120
// middles: 0.76 -> 0.48.  A thread block per row gains the same way (39.5 M products of
// 2718 rows 2.6 -> 2.1).
__global__ void __launch_bounds__(256, 3) k_spgemm_fill_elem(int nrows, const int *__restrict__ arp,
                                                          const int *__restrict__ aci, const double *__restrict__ av,
                                                          const int *__restrict__ brp, const int *__restrict__ bci,
                                                          const double *__restrict__ bv, int HC,
                                                          const int *__restrict__ crp, int *__restrict__ cci,
                                                          double *__restrict__ cv)
{
    extern __shared__ double hs[];
    const int warps = blockDim.x >> 5, wid = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int grp = lane >> 2, e = lane & 3;
    const size_t per = (size_t)HC * 4 + (size_t)(3 * HC + 1) / 2;  // in doubles
    double *acc = hs + (size_t)wid * per;
    int *keys = (int *)(acc + (size_t)HC * 4);
    int *sk = keys + HC, *sp = sk + HC;
    for (int i = blockIdx.x * warps + wid; i < nrows; i += gridDim.x * warps) {
        for (int x = lane; x < HC; x += 32) keys[x] = -1;
        __syncwarp();
        MidWalkElem w{aci, av, brp, bci, bv};
        for (w.start(arp[i], arp[i + 1], grp, e); w.t < w.te; w.next()) {
            w.entries(8, [&](bool on, int j, double x, double y) {
                int h = 0;
                if (on && e == 0) {
                    h = hslot(j, HC - 1);
                    for (int probe = 0; probe < HC; probe++) {
                        const int old = atomicCAS(&keys[h], -1, j);
                        if (old == -1) {
                            h |= 1 << 30;
                            break;
                        }
                        if (old == j) break;
                        h = (h + 1) & (HC - 1);
                    }
                }
                h = __shfl_sync(0xffffffffu, h, lane & ~3);
                const bool fresh = h >> 30;
                double *c = acc + 4 * (size_t)(h & (HC - 1)) + e;
                if (on) *c = w.mac(*c, fresh, x, y);
            });
            __syncwarp();
        }
        // compact the occupied slots, sort them by column, emit
        int n = 0;
        for (int x0 = 0; x0 < HC; x0 += 32) {
            const int x = x0 + lane;
            const bool has = x < HC && keys[x] != -1;
            const unsigned m = __ballot_sync(0xffffffffu, has);
            if (has) {
                const int pos = n + __popc(m & ((1u << lane) - 1u));
                sk[pos] = keys[x];
                sp[pos] = x;
            }
            n += __popc(m);
        }
        int p2 = 1;
        while (p2 < n) p2 <<= 1;
        for (int x = n + lane; x < p2; x += 32) {
            sk[x] = INT_MAX;
            sp[x] = 0;
        }
        __syncwarp();
        for (int kk = 2; kk <= p2; kk <<= 1)
            for (int jj = kk >> 1; jj > 0; jj >>= 1) {
                for (int x = lane; x < p2; x += 32) {
                    const int y = x ^ jj;
                    if (y > x) {
                        const int cx = sk[x], cy = sk[y];
                        if ((cx > cy) == ((x & kk) == 0)) {
                            sk[x] = cy;
                            sk[y] = cx;
                            const int tp = sp[x];
                            sp[x] = sp[y];
                            sp[y] = tp;
                        }
                    }
                }
                __syncwarp();
            }
        const int cb = crp[i];
        for (int x = lane; x < n; x += 32) cci[cb + x] = sk[x];
        for (int x = lane; x < 4 * n; x += 32) cv[4 * (size_t)cb + x] = acc[4 * (size_t)sp[x >> 2] + (x & 3)];
        __syncwarp();
    }
}

// Dense path by warps: a warp per output row with its own accumulators for all
// ncols columns and a bit per column that is in use, no barrier between middles and
// no sort.  For products of many rows onto few columns: two rows and more for every
// warp the SMs hold, or the slowest row's chain of middles sets the time and a
// thread block per row is faster (128x128x32's levels: 2718 rows by 971 columns, 402
// blocks a row, 4.0 ms by blocks, 2.9 by warps; 971 by 971 5.3 by blocks, 7.1 by
// warps; the FP64 operations take 1.8 and 3.3).
template <int BS>
__global__ void k_spgemm_fill_warp(int nrows, const int *__restrict__ arp, const int *__restrict__ aci,
                                   const double *__restrict__ av, const int *__restrict__ brp,
                                   const int *__restrict__ bci, const double *__restrict__ bv, int ncols,
                                   const int *__restrict__ crp, int *__restrict__ cci, double *__restrict__ cv)
{
    constexpr int BB = BS * BS;
    extern __shared__ double wacc[];
    const int lane = threadIdx.x;
    const int words = (ncols + 31) >> 5;
    unsigned *used = (unsigned *)(wacc + (size_t)ncols * BB);
    for (int x = lane; x < words; x += 32) used[x] = 0u;
    __syncwarp();
    for (int i = blockIdx.x; i < nrows; i += gridDim.x) {
        MidWalk<BS> w{aci, av, brp, bci, bv};
        for (w.start(arp[i], arp[i + 1], lane); w.t < w.te; w.next()) {
            w.entries(32, [&](int j, const double (&b)[BB]) {
                const unsigned bit = 1u << (j & 31);
                const bool fresh = !(atomicOr(&used[j >> 5], bit) & bit);
                block_mac<BS>(wacc + j, ncols, w.a, b, fresh);
            });
            __syncwarp();
        }
        int at = crp[i];
        for (int x = 0; x < words; x++) {
            const unsigned m = used[x];
            __syncwarp();
            if (m >> lane & 1u) {
                const int pos = at + __popc(m & ((1u << lane) - 1u)), j = 32 * x + lane;
                cci[pos] = j;
#pragma unroll
                for (int e = 0; e < BB; e++) cv[(size_t)pos * BB + e] = wacc[(size_t)e * ncols + j];
            }
            if (lane == 0) used[x] = 0u;
            at += __popc(m);
        }
        __syncwarp();
    }
}

static int pow2_at_least(long long v)
{
    int p = 1;
    while (p < v) p <<= 1;
    return p;
}

// Shared memory of an SM, and how much of it a warp's rows may take: four warps, one
// per scheduler, keep the FP64 pipe about two thirds busy.
constexpr size_t kSmemSM = 227u << 10, kWarpRowBytes = 55u << 10;
constexpr long long kHashProducts = 4096;  // products per row up to which the hash path is used

// Lanes per output row of the hash path: the power of two nearest above the
// average row length of B (at most 32).
static int hash_lanes(double b_per_row)
{
    int L = 1;
    while (L < 32 && L < b_per_row) L <<= 1;
    return L;
}

// Warps of a block: as many as fit, unless the rows would then leave SMs without a
// block (all products of a 48x48x12 slab, 1463 rows on the second level: setup 9.2 -> 8.7 ms,
// with the launches saved in the scans and maxima).
static int hash_warps(int nrows, int rows_per_warp, size_t fit)
{
    const long long spread = ((long long)nrows + rows_per_warp * kSM - 1) / (rows_per_warp * kSM);
    return (int)std::max<long long>(1, std::min<long long>({8, (long long)fit, spread}));
}

template <int L>
static int launch_count_hash(int nrows, int HCs, const int *arp, const int *aci, const int *brp, const int *bci,
                             int *cnt, int *flag, cudaStream_t s)
{
    constexpr int R = 32 / L;
    const size_t per_warp = (size_t)R * HCs * 4;
    const int warps = hash_warps(nrows, R, (192u << 10) / per_warp);
    const size_t smem = (size_t)warps * per_warp;
    if (smem > kDynamicSmem) return BD_ERANGE;
    BD_TRY(allow_smem(k_spgemm_count_hash<L>));
    const long long rows_per_block = (long long)warps * R;
    const int gb = (int)std::min<long long>(kSM * 8, std::max<long long>(1, (nrows + rows_per_block - 1) / rows_per_block));
    k_spgemm_count_hash<L><<<gb, 32 * warps, smem, s>>>(nrows, arp, aci, brp, bci, HCs, cnt, flag, flag + 2);
    ::bd::note_launch();
    BD_LAUNCH_CHECK();
    return BD_OK;
}

// Table of the count pass: half full at most for rows of n columns.
static int count_table(long long n)
{
    return std::max(32, pow2_at_least(2 * std::min<long long>(n, kMaxSortSeg)));
}

// Row lengths by hashing.  The bound on a row's products is several times its length
// (the products of A P meet four to a column, those of R (A P) tens), and tables of
// that size leave room for a few rows per SM only, so the first attempt takes
// tables for a quarter of it; flag[0] tells that some row did not fit.
static int count_hash_rows(int nrows, int HCs, int lanes, const int *arp, const int *aci, const int *brp,
                           const int *bci, int *cnt, int *flag, cudaStream_t s)
{
    // rows whose tables do not fit 32/lanes to a warp take more lanes each
    int Lc = lanes;
    while (Lc < 32 && (size_t)(32 / Lc) * HCs * 4 > (192u << 10)) Lc <<= 1;
    switch (Lc) {
    case 1: return launch_count_hash<1>(nrows, HCs, arp, aci, brp, bci, cnt, flag, s);
    case 2: return launch_count_hash<2>(nrows, HCs, arp, aci, brp, bci, cnt, flag, s);
    case 4: return launch_count_hash<4>(nrows, HCs, arp, aci, brp, bci, cnt, flag, s);
    case 8: return launch_count_hash<8>(nrows, HCs, arp, aci, brp, bci, cnt, flag, s);
    case 16: return launch_count_hash<16>(nrows, HCs, arp, aci, brp, bci, cnt, flag, s);
    default: return launch_count_hash<32>(nrows, HCs, arp, aci, brp, bci, cnt, flag, s);
    }
}

template <int BS, int L>
static int launch_fill_hash(int nrows, int HCn, const int *arp, const int *aci, const double *av, const int *brp,
                            const int *bci, const double *bv, const int *crp, int *cci, double *cv, cudaStream_t s)
{
    constexpr int R = 32 / L;
    const size_t per = ((size_t)HCn * BS * BS + (size_t)(3 * HCn + 1) / 2) * sizeof(double);
    const size_t per_warp = (size_t)R * per;
    if (per_warp > kDynamicSmem) return BD_ERANGE;
    const int warps = hash_warps(nrows, R, kDynamicSmem / per_warp);
    const size_t smem = per_warp * warps;
    BD_TRY(allow_smem(k_spgemm_fill_hash<BS, L>));
    const long long rows_per_block = (long long)warps * R;
    const int gb = (int)std::min<long long>(kSM * 8, std::max<long long>(1, (nrows + rows_per_block - 1) / rows_per_block));
    k_spgemm_fill_hash<BS, L><<<gb, 32 * warps, smem, s>>>(nrows, arp, aci, av, brp, bci, bv, HCn, crp, cci, cv);
    ::bd::note_launch();
    BD_LAUNCH_CHECK();
    return BD_OK;
}

// 2x2 blocks: rows of B of one or two blocks (a tentative prolongator) keep a lane or two
// per row, which fills every FP64 instruction (549153 rows 1.8 ms; four lanes per
// product would take 3.0 for the FP64 operations alone), unless that leaves
// schedulers without a warp (1463 rows: 0.21 -> 0.08 ms by elements).
constexpr int kLaneRows = 32 * 4 * kSM;

static int launch_fill_elem(int nrows, int HCn, const int *arp, const int *aci, const double *av, const int *brp,
                            const int *bci, const double *bv, const int *crp, int *cci, double *cv, cudaStream_t s)
{
    const size_t per_warp = ((size_t)HCn * 4 + (size_t)(3 * HCn + 1) / 2) * sizeof(double);
    if (per_warp > kDynamicSmem) return BD_ERANGE;
    const int warps = hash_warps(nrows, 1, kDynamicSmem / per_warp);
    const size_t smem = per_warp * warps;
    BD_TRY(allow_smem(k_spgemm_fill_elem));
    const int gb = (int)std::min<long long>(kSM * 32, std::max<long long>(1, (nrows + warps - 1) / warps));
    k_spgemm_fill_elem<<<gb, 32 * warps, smem, s>>>(nrows, arp, aci, av, brp, bci, bv, HCn, crp, cci, cv);
    ::bd::note_launch();
    BD_LAUNCH_CHECK();
    return BD_OK;
}

// b_per_row: average blocks per row of B (sets the lanes per row of the hash path);
// scratch: C is scratch of the setup call
template <int BS>
static int spgemm(int nrows, int ncols, const int *arp, const int *aci, const double *av,
                  const int *brp, const int *bci, const double *bv, DBuf<int> &crp, DBuf<int> &cci,
                  DBuf<double> &cv, long long *cnnz, cudaStream_t s, double b_per_row, bool scratch)
{
    constexpr int BB = BS * BS;
    BD_TRY(scratch ? crp.scratch((size_t)nrows + 1, s) : crp.alloc((size_t)nrows + 1));
    DBuf<int> cnt;
    BD_TRY(cnt.scratch((size_t)nrows + 1, s));
    size_t per_block = (size_t)ncols * (sizeof(int) + BB * sizeof(double));
    long long g = kSM * 4;
    long long cap = (2LL << 30) / (long long)(per_block ? per_block : 1);
    if (g > cap) g = cap;
    bool dense = g >= kSM || g >= nrows;
    if (g > nrows) g = nrows > 0 ? nrows : 1;
    if (g < 1) g = 1;
    int grid = (int)g;
    DBuf<int> mark;
    DBuf<double> acc;
    DBuf<int> flag;  // [0] hash-table overflow, [1] largest product bound, [2] longest output row
    BD_TRY(flag.scratch(3, s));
    BD_CUDA(cudaMemsetAsync(flag.p, 0, 3 * sizeof(int), s));
    // Rows with few products (the fine levels' many short rows) go to the
    // warp-per-row hash path: the dense path's thread block per row then idles
    // most of its threads and synchronises once per middle index.  Both paths
    // accumulate every entry in the same order, so the choice changes no bit.
    long long mub = 1;
    if (nrows > 0) {
        k_spgemm_bound<<<(nrows + 31) / 32, 256, 0, s>>>(nrows, arp, aci, brp, flag.p + 1); ::bd::note_launch();
        BD_LAUNCH_CHECK();
        int hb = 0;
        BD_CUDA(cudaMemcpyAsync(&hb, flag.p + 1, sizeof(int), cudaMemcpyDeviceToHost, s));
        BD_CUDA(cudaStreamSynchronize(s));
        mub = std::max<long long>(mub, hb);
        if (mub <= kHashProducts) dense = false;
    }
    const int lanes = hash_lanes(b_per_row);
    ::bd::note_spgemm_path(dense);
    // the dense path keeps a row's accumulators in shared memory when they
    // fit (with the largest column list a row can have)
    const size_t dense_smem = (size_t)ncols * (BB * sizeof(double) + sizeof(int)) +
                              (size_t)pow2_at_least(std::max(ncols, 1)) * sizeof(int);
    const bool dense_in_smem = dense && dense_smem <= kDynamicSmem;
    if (dense_in_smem) {
        const size_t cs = (size_t)ncols * sizeof(int);
        BD_TRY(allow_smem(k_spgemm_count_smem));
        const int gc = (int)std::min<long long>(nrows, (long long)kSM * 8);
        k_spgemm_count_smem<<<std::max(gc, 1), 128, std::max<size_t>(cs, 4), s>>>(nrows, arp, aci, brp, bci, ncols,
                                                                                   cnt.p, flag.p + 2);
        ::bd::note_launch();
        BD_LAUNCH_CHECK();
    } else if (dense) {
        BD_TRY(mark.scratch((size_t)grid * ncols, s));
        BD_TRY(acc.scratch((size_t)grid * ncols * BB, s));
        BD_CUDA(cudaMemsetAsync(mark.p, 0xff, mark.bytes(), s));
        k_spgemm_count<BS><<<grid, 128, 0, s>>>(nrows, arp, aci, brp, bci, ncols, mark.p, cnt.p, flag.p + 2);
        ::bd::note_launch();
        BD_LAUNCH_CHECK();
    } else {
        BD_TRY(count_hash_rows(nrows, count_table(mub / 4), lanes, arp, aci, brp, bci, cnt.p, flag.p, s));
    }
    long long total = 0;
    BD_TRY(exclusive_scan(cnt.p, crp.p, nrows, &total, s));
    int hf[3] = {0, 0, 0};
    BD_CUDA(cudaMemcpyAsync(hf, flag.p, sizeof(hf), cudaMemcpyDeviceToHost, s));
    BD_CUDA(cudaStreamSynchronize(s));
    if (hf[0]) {  // a row outgrew the count's first table: once more with one that holds all products
        BD_CUDA(cudaMemsetAsync(flag.p, 0, 3 * sizeof(int), s));
        BD_TRY(count_hash_rows(nrows, count_table(mub), lanes, arp, aci, brp, bci, cnt.p, flag.p, s));
        BD_TRY(exclusive_scan(cnt.p, crp.p, nrows, &total, s));
        BD_CUDA(cudaMemcpyAsync(hf, flag.p, sizeof(hf), cudaMemcpyDeviceToHost, s));
        BD_CUDA(cudaStreamSynchronize(s));
    }
    if (hf[0]) return BD_ERANGE;
    const int maxrow = hf[2];
    if (maxrow > kMaxSortSeg) return BD_ERANGE;
    BD_TRY(scratch ? cci.scratch((size_t)total, s) : cci.alloc((size_t)total));
    BD_TRY(scratch ? cv.scratch((size_t)total * BB, s) : cv.alloc((size_t)total * BB));
    // tables at most three quarters full
    const int HCn = pow2_at_least(std::max(16LL, 4LL * maxrow / 3 + 1));
    const size_t hash_row = ((size_t)HCn * BB + (size_t)(3 * HCn + 1) / 2) * sizeof(double);
    const size_t warp_row = (size_t)ncols * BB * sizeof(double) + (size_t)((ncols + 31) / 32) * sizeof(int);
    if (dense && warp_row <= kWarpRowBytes && nrows >= 2 * kSM * (long long)(kSmemSM / (warp_row + 1024))) {
        BD_TRY(allow_smem(k_spgemm_fill_warp<BS>));
        const int gw = (int)std::min<long long>(nrows, kSM * 32LL);
        k_spgemm_fill_warp<BS><<<gw, 32, warp_row, s>>>(nrows, arp, aci, av, brp, bci, bv, ncols, crp.p, cci.p, cv.p);
        ::bd::note_launch();
        BD_LAUNCH_CHECK();
    } else if (dense_in_smem) {
        BD_TRY(allow_smem(k_spgemm_fill_smem<BS>));
        const int per_sm = std::max(1, (int)((227u << 10) / (dense_smem + 1024)));
        const int gf = (int)std::min<long long>(nrows, (long long)kSM * per_sm);
        k_spgemm_fill_smem<BS><<<std::max(gf, 1), 256, dense_smem, s>>>(nrows, arp, aci, av, brp, bci, bv, ncols,
                                                                         crp.p, cci.p, cv.p);
        ::bd::note_launch();
        BD_LAUNCH_CHECK();
    } else if (dense) {
        int P2 = pow2_at_least(maxrow);
        BD_CUDA(cudaMemsetAsync(mark.p, 0xff, mark.bytes(), s));
        size_t smem = (size_t)P2 * sizeof(int);
        BD_TRY(allow_smem(k_spgemm_fill<BS>));
        k_spgemm_fill<BS><<<grid, 128, smem, s>>>(nrows, arp, aci, av, brp, bci, bv, ncols, mark.p,
                                                  acc.p, crp.p, cci.p, cv.p, P2); ::bd::note_launch();
        BD_LAUNCH_CHECK();
    } else {
        bool done = false;
        if constexpr (BS == 2) {
            if (lanes >= 4 || nrows < kLaneRows) {
                BD_TRY(launch_fill_elem(nrows, HCn, arp, aci, av, brp, bci, bv, crp.p, cci.p, cv.p, s));
                done = true;
            }
        }
        // rows whose tables do not fit 32/lanes to a warp take more lanes each
        int Lf = lanes;
        while (Lf < 32 && (size_t)(32 / Lf) * hash_row > kWarpRowBytes) Lf <<= 1;
        if (!done) switch (Lf) {
        case 1: BD_TRY((launch_fill_hash<BS, 1>(nrows, HCn, arp, aci, av, brp, bci, bv, crp.p, cci.p, cv.p, s))); break;
        case 2: BD_TRY((launch_fill_hash<BS, 2>(nrows, HCn, arp, aci, av, brp, bci, bv, crp.p, cci.p, cv.p, s))); break;
        case 4: BD_TRY((launch_fill_hash<BS, 4>(nrows, HCn, arp, aci, av, brp, bci, bv, crp.p, cci.p, cv.p, s))); break;
        case 8: BD_TRY((launch_fill_hash<BS, 8>(nrows, HCn, arp, aci, av, brp, bci, bv, crp.p, cci.p, cv.p, s))); break;
        case 16: BD_TRY((launch_fill_hash<BS, 16>(nrows, HCn, arp, aci, av, brp, bci, bv, crp.p, cci.p, cv.p, s))); break;
        default: BD_TRY((launch_fill_hash<BS, 32>(nrows, HCn, arp, aci, av, brp, bci, bv, crp.p, cci.p, cv.p, s))); break;
        }
    }
    *cnnz = total;
    return BD_OK;
}

// ------------------------------------------------------------------ squared graph
// Wh = I + W (unit diagonal inserted in order), S2 = Wh*Wh without diagonal.
__global__ void k_insert_diag(int N, const int *__restrict__ srp, const int *__restrict__ sci,
                              const double *__restrict__ sw, int *__restrict__ wrp,
                              int *__restrict__ wci, double *__restrict__ wv)
{
    int p = blockIdx.x * blockDim.x + threadIdx.x;
    if (p > N) return;
    wrp[p] = srp[p] + p;
    if (p == N) return;
    int pos = srp[p] + p;
    bool done = false;
    for (int t = srp[p]; t < srp[p + 1]; t++) {
        if (!done && sci[t] > p) {
            wci[pos] = p;
            wv[pos++] = 1.0;
            done = true;
        }
        wci[pos] = sci[t];
        wv[pos++] = sw[t];
    }
    if (!done) {
        wci[pos] = p;
        wv[pos] = 1.0;
    }
}

// (every row of Wh*Wh holds its diagonal: entries before it move up by the p
// diagonals of earlier rows, entries behind it by one more)
__global__ void k_drop_diag(int N, const int *__restrict__ qrp, const int *__restrict__ qci,
                            const double *__restrict__ qv, int *__restrict__ orp,
                            int *__restrict__ oci, double *__restrict__ ov)
{
    const int lane = threadIdx.x & 31, p = grid_row<5>(blockIdx.x, blockDim.x, threadIdx.x);
    if (p > N) return;
    if (lane == 0) orp[p] = qrp[p] - p;
    if (p == N) return;
    for (int t = qrp[p] + lane; t < qrp[p + 1]; t += 32) {
        const int q = qci[t];
        if (q == p) continue;
        const int o = t - p - (q > p ? 1 : 0);
        oci[o] = q;
        ov[o] = qv[t];
    }
}

// ------------------------------------------------------------------ a2 MIS (Luby rounds)
// state: 0 undecided, 1 in the set, 2 out.  Node p beats q when its priority
// (mix64(p ^ key), -p) is larger.  With fixed priorities the rounds return the
// set the sequential greedy pass builds in decreasing priority.
__device__ __forceinline__ bool beats(unsigned long long hp, int p, unsigned long long hq, int q)
{
    return hp > hq || (hp == hq && p < q);
}

// Eight lanes per node here and in k_assign (rows of the squared graph hold some 125
// entries; a thread's walk is a chain of loads: 31213 nodes, select 16.5 -> 6.7 us,
// exclude 10.6 -> 7.2, assign 28 -> 8).
struct NodeLanes {
    int p, l;           // node, lane of the node's eight
    unsigned mask;      // the node's lanes in the warp
    __device__ __forceinline__ NodeLanes()
        : p(grid_row<3>(blockIdx.x, blockDim.x, threadIdx.x)), l(threadIdx.x & 7),
          mask(0xffu << (threadIdx.x & 24)) {}
    // whether f(t) holds for an entry t of [b, e), by all lanes of the warp together
    template <class F> __device__ __forceinline__ bool any(int b, int e, F &&f) const
    {
        bool found = false;
        for (int t = b + l;; t += 8) {
            const bool go = !found && t < e;
            if (!__any_sync(0xffffffffu, go)) break;
            found = (__ballot_sync(0xffffffffu, go ? f(t) : found) & mask) != 0;
        }
        return found;
    }
};

__global__ void k_mis_select(int N, const int *__restrict__ srp, const int *__restrict__ sci,
                             unsigned char *state, unsigned long long key)
{
    const NodeLanes n;
    const bool act = n.p < N && state[n.p] == 0;
    const unsigned long long hp = mix64((unsigned long long)n.p ^ key);
    const bool lost = n.any(act ? srp[n.p] : 0, act ? srp[n.p + 1] : 0, [&](int t) {
        const int q = sci[t];
        const unsigned char sq = ((volatile unsigned char *)state)[q];
        return sq == 1 || (sq == 0 && beats(mix64((unsigned long long)q ^ key), q, hp, n.p));
    });
    if (act && n.l == 0 && !lost) state[n.p] = 1;
}

__global__ void k_mis_exclude(int N, const int *__restrict__ srp, const int *__restrict__ sci,
                              unsigned char *state, int *undecided)
{
    const NodeLanes n;
    const bool act = n.p < N && state[n.p] == 0;
    const bool out = n.any(act ? srp[n.p] : 0, act ? srp[n.p + 1] : 0,
                           [&](int t) { return ((volatile unsigned char *)state)[sci[t]] == 1; });
    const bool left = act && n.l == 0 && !out;
    if (act && n.l == 0 && out) state[n.p] = 2;
    const unsigned m = __ballot_sync(0xffffffffu, left);
    if ((threadIdx.x & 31) == 0 && m) atomicAdd(undecided, __popc(m));
}

// ------------------------------------------------------------------ a3 aggregation
__global__ void k_root_flags(int N, const unsigned char *state, unsigned char *mis, int *flag)
{
    int p = blockIdx.x * blockDim.x + threadIdx.x;
    if (p >= N) return;
    int r = state[p] == 1;
    mis[p] = (unsigned char)r;
    flag[p] = r;
}

__global__ void k_assign(int N, const int *__restrict__ srp, const int *__restrict__ sci,
                         const double *__restrict__ sw, const unsigned char *__restrict__ mis,
                         const int *__restrict__ root_id, int *__restrict__ agg, int *bad)
{
    const NodeLanes n;
    const int p = n.p;
    const bool act = p < N, root = act && mis[p];
    int best = -1;  // the first entry of the largest weight
    double bw = -1.0;
    for (int t = act && !root ? srp[p] + n.l : 0, e = act && !root ? srp[p + 1] : 0; t < e; t += 8)
        if (mis[sci[t]] && sw[t] > bw) {
            bw = sw[t];
            best = t;
        }
    for (int o = 4; o; o >>= 1) {
        const double w2 = __shfl_xor_sync(0xffffffffu, bw, o);
        const int t2 = __shfl_xor_sync(0xffffffffu, best, o);
        if (t2 >= 0 && (best < 0 || w2 > bw || (w2 == bw && t2 < best))) {
            bw = w2;
            best = t2;
        }
    }
    if (!act || n.l) return;
    if (root) {
        agg[p] = root_id[p];
    } else if (best < 0) {
        *bad = 1;
        agg[p] = 0;
    } else {
        agg[p] = root_id[sci[best]];
    }
}

// ------------------------------------------------------------------ a4 tentative prolongator
__global__ void k_count_members(int N, const int *agg, int *cnt)
{
    int p = blockIdx.x * blockDim.x + threadIdx.x;
    if (p < N) atomicAdd(&cnt[agg[p]], 1);
}

__global__ void k_scatter_members(int N, const int *agg, const int *off, int *fill, int *members)
{
    int p = blockIdx.x * blockDim.x + threadIdx.x;
    if (p < N) {
        int J = agg[p];
        members[off[J] + atomicAdd(&fill[J], 1)] = p;
    }
}

// Bc(2J+f) = sqrt(sum over members k ascending of B(2k+f)^2)
__global__ void k_coarse_B(int nagg, const int *__restrict__ off, const int *__restrict__ members,
                           const double *__restrict__ B, double *__restrict__ Bc)
{
    int J = blockIdx.x * blockDim.x + threadIdx.x;
    if (J >= nagg) return;
    double s0 = 0.0, s1 = 0.0;
    for (int t = off[J]; t < off[J + 1]; t++) {
        int k = members[t];
        double b0 = B[2 * k], b1 = B[2 * k + 1];
        s0 = s0 + b0 * b0;
        s1 = s1 + b1 * b1;
    }
    Bc[2 * J] = sqrt(s0);
    Bc[2 * J + 1] = sqrt(s1);
}

// Pt as 2x2-block CSR: one block per node row, diag(B(2k)/Bc(2J), B(2k+1)/Bc(2J+1)).
__global__ void k_ptent(int N, const int *__restrict__ agg, const double *__restrict__ B,
                        const double *__restrict__ Bc, int *__restrict__ rp, int *__restrict__ ci,
                        double *__restrict__ v, double *__restrict__ ptd)
{
    int p = blockIdx.x * blockDim.x + threadIdx.x;
    if (p > N) return;
    rp[p] = p;
    if (p == N) return;
    int J = agg[p];
    double a = B[2 * p] / Bc[2 * J], b = B[2 * p + 1] / Bc[2 * J + 1];
    ci[p] = J;
    v[4 * (size_t)p + 0] = a;
    v[4 * (size_t)p + 1] = 0.0;
    v[4 * (size_t)p + 2] = 0.0;
    v[4 * (size_t)p + 3] = b;
    ptd[2 * p] = a;
    ptd[2 * p + 1] = b;
}

// ------------------------------------------------------------------ a5 lambda_max (CG-Lanczos)
// The CG scalars of every step; the tridiagonal's coefficients and the step at
// which the recurrence ends (a pq or rz that is not positive) follow from them
// in k_lanczos_finish.  Steps past that end still run and are not read.
struct LanczosState {
    double rz[65], pq[64];
    double lam;
    int bad;
};

__global__ void k_lanczos_init(int n, unsigned long long key, const double *__restrict__ diag,
                               double *r, double *z, double *p)
{
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    unsigned long long h = mix64(key ^ (unsigned long long)i);
    double u = (double)(h >> 11) * (1.0 / 9007199254740992.0);
    double ri = 2.0 * u - 1.0;
    double zi = ri / diag[i];
    r[i] = ri;
    z[i] = zi;
    p[i] = zi;
}

// y = A x, scalar rows in ascending column order, acc = acc + a*x from 0.0: one
// thread per scalar row (its additions are one chain), whose loads run eight
// blocks ahead of the chain.  Bound by the FP64 pipe on large levels (4 rounded
// operations per scalar row and block; 128x128x32 237 us, floor 183), by the
// chain on small ones (2718 rows of 223 blocks: 307 -> 94 us).
__global__ void __launch_bounds__(256, 3) k_spmv_ordered(int n, const int *__restrict__ rp, const int *__restrict__ ci,
                               const double *__restrict__ v, const double *__restrict__ x,
                               double *__restrict__ y)
{
    constexpr int U = 8;
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const double2 *a = (const double2 *)v + (i & 1), *w = (const double2 *)x;
    double s = 0.0;
    const int e = rp[(i >> 1) + 1];
    int t = rp[i >> 1];
    for (; t + U <= e; t += U) {
        double2 av[U], wv[U];
        int q[U];
#pragma unroll
        for (int k = 0; k < U; k++) q[k] = ci[t + k];
#pragma unroll
        for (int k = 0; k < U; k++) {
            av[k] = a[2 * (size_t)(t + k)];
            wv[k] = w[q[k]];
        }
#pragma unroll
        for (int k = 0; k < U; k++) {
            s = s + av[k].x * wv[k].x;
            s = s + av[k].y * wv[k].y;
        }
    }
    for (; t < e; t++) {
        const double2 av = a[2 * (size_t)t], wv = w[ci[t]];
        s = s + av.x * wv.x;
        s = s + av.y * wv.y;
    }
    y[i] = s;
}

__global__ void k_lanczos_update_r(int n, const LanczosState *st, int j, const double *__restrict__ q,
                                   const double *__restrict__ diag, double *r, double *z)
{
    __shared__ double alpha;
    if (threadIdx.x == 0) alpha = st->rz[j] / st->pq[j];
    __syncthreads();
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    double ri = r[i] - alpha * q[i];
    r[i] = ri;
    z[i] = ri / diag[i];
}

__global__ void k_lanczos_update_p(int n, const LanczosState *st, int j, const double *__restrict__ z,
                                   double *p)
{
    __shared__ double beta;
    if (threadIdx.x == 0) beta = st->rz[j + 1] / st->rz[j];
    __syncthreads();
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    p[i] = z[i] + beta * p[i];
}

// eigenvalues of the tridiagonal (diagonal d, squared off-diagonal e2) below x
__device__ int sturm_count_below(int m, const double *d, const double *e2, double x)
{
    int c = 0;
    double q = d[0] - x;
    if (q < 0.0) c++;
    for (int i = 1; i < m; i++) {
        if (q == 0.0) q = -1e-300;
        q = (d[i] - x) - e2[i - 1] / q;
        if (q < 0.0) c++;
    }
    return c;
}

// Largest Ritz value by bisection to the last bit.  One warp runs five bisection
// steps at a time: lane l takes node l of the tree of their midpoints (heap
// order), forms its midpoint by the additions the steps on its path would make,
// and the walk down the tree then reads five answers after one evaluation's
// latency.  The midpoints and answers are those of the sequential bisection, so
// the result is its result (one thread stepping alone: 255 us, now 68).
__global__ void k_lanczos_finish(LanczosState *st, int steps)
{
    __shared__ double d[64], e[64], e2[64];
    const int lane = threadIdx.x;
    int m = 0;
    while (m < steps && st->pq[m] > 0.0 && st->rz[m] > 0.0) {
        m++;
        if (!(st->rz[m] > 0.0)) break;
    }
    if (m == 0) {
        if (lane == 0) {
            st->bad = 1;
            st->lam = 0.0;
        }
        return;
    }
    for (int j = lane; j < m; j += 32) {
        const double al = st->rz[j] / st->pq[j];
        double dj = 1.0 / al;
        if (j > 0) {
            const double alp = st->rz[j - 1] / st->pq[j - 1], bep = st->rz[j] / st->rz[j - 1];
            dj = dj + bep / alp;
        }
        d[j] = dj;
        double ej = 0.0;
        if (j < m - 1) ej = sqrt(st->rz[j + 1] / st->rz[j]) / al;
        e[j] = ej;
        e2[j] = ej * ej;
    }
    __syncwarp();
    double lo = 0.0, hi = 0.0;
    for (int i = 0; i < m; i++) {
        double r = 0.0;
        if (i > 0) r = r + fabs(e[i - 1]);
        if (i < m - 1) r = r + fabs(e[i]);
        double a = d[i] - r, b = d[i] + r;
        if (i == 0 || a < lo) lo = a;
        if (i == 0 || b > hi) hi = b;
    }
    for (int it = 0; it < 4096;) {
        // lane l's midpoint: from the root (1) down to node l
        double nlo = lo, nhi = hi, mid = 0.5 * (nlo + nhi);
        const int node = lane > 0 ? lane : 1;
        for (int bit = 30 - __clz(node); bit >= 0; bit--) {
            if ((node >> bit) & 1) nlo = mid;
            else nhi = mid;
            mid = 0.5 * (nlo + nhi);
        }
        const unsigned open = __ballot_sync(0xffffffffu, mid > nlo && mid < nhi);
        const unsigned all = __ballot_sync(0xffffffffu, sturm_count_below(m, d, e2, mid) == m);
        bool done = false;
        for (int k = 1; k < 32 && it < 4096; it++) {
            if (!((open >> k) & 1)) {
                done = true;
                break;
            }
            const double x = 0.5 * (lo + hi);
            const bool below = (all >> k) & 1;
            if (below) hi = x;
            else lo = x;
            k = 2 * k + (below ? 0 : 1);
        }
        if (done) break;
    }
    if (lane == 0) st->lam = hi;
}

// ------------------------------------------------------------------ a6 smoothed prolongator
// P(i,j) = Pt(i,j) - s_i AP(i,j),  s_i = omega / A(i,i),  omega = 4/(3 lambda)
// (eight lanes per row)
__global__ void k_smooth_p(int N, const int *__restrict__ rp, const int *__restrict__ ci,
                           double *__restrict__ v, const int *__restrict__ agg,
                           const double *__restrict__ ptd, const double *__restrict__ diag,
                           const LanczosState *st)
{
    const int p = grid_row<3>(blockIdx.x, blockDim.x, threadIdx.x), l = threadIdx.x & 7;
    if (p >= N) return;
    double omega = 4.0 / (3.0 * st->lam);
    double s0 = omega / diag[2 * p], s1 = omega / diag[2 * p + 1];
    int J = agg[p];
    for (int t = rp[p] + l; t < rp[p + 1]; t += 8) {
        bool own = ci[t] == J;
        double2 *b = (double2 *)v + 2 * (size_t)t;
        double p00 = own ? ptd[2 * p] : 0.0, p11 = own ? ptd[2 * p + 1] : 0.0;
        const double2 x = b[0], y = b[1];
        b[0] = make_double2(p00 - s0 * x.x, 0.0 - s0 * x.y);
        b[1] = make_double2(0.0 - s1 * y.x, p11 - s1 * y.y);
    }
}

// ------------------------------------------------------------------ a7 transpose
__global__ void k_count_cols(long long nb, const int *ci, int *cnt)
{
    long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    if (t < nb) atomicAdd(&cnt[ci[t]], 1);
}

__global__ void k_scatter_t(int N, const int *__restrict__ rp, const int *__restrict__ ci,
                            const int *__restrict__ off, int *fill, int *tci, int *perm)
{
    int p = blockIdx.x * blockDim.x + threadIdx.x;
    if (p >= N) return;
    for (int t = rp[p]; t < rp[p + 1]; t++) {
        int J = ci[t];
        int pos = off[J] + atomicAdd(&fill[J], 1);
        tci[pos] = p;
        perm[pos] = t;
    }
}

__global__ void k_gather_t(long long nb, const int *__restrict__ perm, const double *__restrict__ v,
                           double *__restrict__ tv)
{
    long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    if (t >= nb) return;
    const double *a = v + 4 * (size_t)perm[t];
    double *b = tv + 4 * (size_t)t;
    b[0] = a[0];
    b[1] = a[2];
    b[2] = a[1];
    b[3] = a[3];
}

static int bsr_transpose(const BSR &a, BSR &t, cudaStream_t s)
{
    t.nbr = a.nbc;
    t.nbc = a.nbr;
    t.nb = a.nb;
    DBuf<int> cnt, fill, perm;
    BD_TRY(cnt.scratch((size_t)a.nbc + 2, s));  // counts, then the largest at [a.nbc + 1]
    BD_TRY(fill.scratch((size_t)a.nbc + 1, s));
    BD_TRY(perm.scratch((size_t)a.nb, s));
    BD_TRY(t.rp.alloc((size_t)a.nbc + 1));
    BD_TRY(t.ci.alloc((size_t)a.nb));
    BD_TRY(t.v.alloc(4 * (size_t)a.nb));
    BD_CUDA(cudaMemsetAsync(cnt.p, 0, cnt.bytes(), s));
    BD_CUDA(cudaMemsetAsync(fill.p, 0, fill.bytes(), s));
    k_count_cols<<<(int)((a.nb + 255) / 256), 256, 0, s>>>(a.nb, a.ci.p, cnt.p); ::bd::note_launch();
    BD_LAUNCH_CHECK();
    BD_TRY(device_max(cnt.p, a.nbc, cnt.p + a.nbc + 1, s));
    long long tot = 0;
    BD_TRY(exclusive_scan(cnt.p, t.rp.p, a.nbc, &tot, s));  // stream synchronised
    int mx = 0;
    BD_CUDA(cudaMemcpyAsync(&mx, cnt.p + a.nbc + 1, sizeof(int), cudaMemcpyDeviceToHost, s));
    BD_CUDA(cudaStreamSynchronize(s));
    k_scatter_t<<<(a.nbr + 255) / 256, 256, 0, s>>>(a.nbr, a.rp.p, a.ci.p, t.rp.p, fill.p, t.ci.p,
                                                    perm.p); ::bd::note_launch();
    BD_LAUNCH_CHECK();
    BD_TRY(sort_segments(t.ci.p, perm.p, t.rp.p, a.nbc, mx, s));
    k_gather_t<<<(int)((a.nb + 255) / 256), 256, 0, s>>>(a.nb, perm.p, a.v.p, t.v.p); ::bd::note_launch();
    BD_LAUNCH_CHECK();
    return BD_OK;
}

// ------------------------------------------------------------------ a9 coarsest level
// a warp per block row; ld: row stride of Ad
__global__ void k_coarse_dense(int N, const int *__restrict__ rp, const int *__restrict__ ci,
                               const double *__restrict__ v, int ld, double *__restrict__ Ad)
{
    const int lane = threadIdx.x & 31, p = grid_row<5>(blockIdx.x, blockDim.x, threadIdx.x);
    if (p >= N) return;
    double2 *r0 = (double2 *)(Ad + (size_t)(2 * p) * ld), *r1 = (double2 *)(Ad + (size_t)(2 * p + 1) * ld);
    for (int t = rp[p] + lane; t < rp[p + 1]; t += 32) {
        const int q = ci[t];
        r0[q] = ((const double2 *)v)[2 * (size_t)t];
        r1[q] = ((const double2 *)v)[2 * (size_t)t + 1];
    }
}

// Single block: rank-one fix, Cholesky (left-looking, sums ascending), then the
// explicit inverse by forward/backward substitution of unit vectors.
__global__ void k_coarse_factor(int n, double *A, const double *__restrict__ z, double *Ainv,
                                double *zz_out, int *bad)
{
    __shared__ double smax_s, zz_s;
    if (threadIdx.x == 0) {
        double smax = 0.0, zz = 0.0;
        for (int i = 0; i < n; i++) {
            double d = A[(size_t)i * n + i];
            if (d > smax) smax = d;
            zz = zz + z[i] * z[i];
        }
        smax_s = smax;
        zz_s = zz;
        *zz_out = zz;
    }
    __syncthreads();
    double smax = smax_s, zz = zz_s;
    for (size_t e = threadIdx.x; e < (size_t)n * n; e += blockDim.x) {
        int i = (int)(e / n), j = (int)(e % n);
        A[e] = A[e] + (smax * z[i]) * z[j] / zz;
    }
    __syncthreads();
    __shared__ double dj;
    for (int j = 0; j < n; j++) {
        if (threadIdx.x == 0) {
            double sdiag = A[(size_t)j * n + j];
            for (int k = 0; k < j; k++) sdiag = sdiag - A[(size_t)j * n + k] * A[(size_t)j * n + k];
            if (!(sdiag > 0.0)) *bad = 1;
            dj = sqrt(sdiag > 0.0 ? sdiag : 1.0);
            A[(size_t)j * n + j] = dj;
        }
        __syncthreads();
        for (int i = j + 1 + threadIdx.x; i < n; i += blockDim.x) {
            double t = A[(size_t)i * n + j];
            for (int k = 0; k < j; k++) t = t - A[(size_t)i * n + k] * A[(size_t)j * n + k];
            A[(size_t)i * n + j] = t / dj;
        }
        __syncthreads();
    }
    // columns of the inverse: L y = e_c, L^T x = y
    for (int c = threadIdx.x; c < n; c += blockDim.x) {
        double *x = Ainv + (size_t)c * n;  // column c stored contiguously (inverse is symmetric)
        for (int i = 0; i < n; i++) {
            double s = (i == c) ? 1.0 : 0.0;
            for (int k = 0; k < i; k++) s = s - A[(size_t)i * n + k] * x[k];
            x[i] = s / A[(size_t)i * n + i];
        }
        for (int i = n - 1; i >= 0; i--) {
            double s = x[i];
            for (int k = i + 1; k < n; k++) s = s - A[(size_t)k * n + i] * x[k];
            x[i] = s / A[(size_t)i * n + i];
        }
    }
}

// Larger coarsest levels: the same rank-one-fixed matrix, inverted in place by
// symmetric block elimination without pivoting (the matrix is symmetric positive
// definite), kGJ pivots at a time on a copy padded to whole blocks.  With M = A at
// first, the step of pivot block P is D = M[P,P]^-1, W = M[:,P] D and
//     M[i,j] -= W[i,:] M[j,P]^T,   M[i,P] = W[i,:],   M[P,P] = -D,
// which keeps M symmetric and ends with M = -A^-1, so only the block-lower half
// is formed: half the FP64 work of Gauss-Jordan, which bounds the update.
__global__ void __launch_bounds__(1024) k_coarse_stats(int n, int ld, const double *__restrict__ A,
                                                       const double *__restrict__ z, double *__restrict__ out)
{
    __shared__ double sm[32], sz[32];
    double smax = 0.0, zz = 0.0;
    for (int i = threadIdx.x; i < n; i += blockDim.x) {
        smax = fmax(smax, A[(size_t)i * ld + i]);
        zz = zz + z[i] * z[i];
    }
    for (int o = 16; o; o >>= 1) {
        smax = fmax(smax, __shfl_xor_sync(0xffffffffu, smax, o));
        zz += __shfl_xor_sync(0xffffffffu, zz, o);
    }
    if ((threadIdx.x & 31) == 0) {
        sm[threadIdx.x >> 5] = smax;
        sz[threadIdx.x >> 5] = zz;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int w = 1; w < (int)(blockDim.x >> 5); w++) {
            smax = fmax(smax, sm[w]);
            zz += sz[w];
        }
        out[0] = smax;
        out[1] = zz;
    }
}

// one thread block per row; rows past n (the padding) get a unit diagonal
__global__ void k_coarse_rank1(int n, int ld, double *__restrict__ A, const double *__restrict__ z,
                               const double *__restrict__ st)
{
    const double smax = st[0], zz = st[1];
    const int i = blockIdx.x;
    if (i >= n) {
        if (threadIdx.x == 0) A[(size_t)i * ld + i] = 1.0;
        return;
    }
    for (int j = threadIdx.x; j < n; j += blockDim.x) {
        const size_t e = (size_t)i * ld + j;
        A[e] = A[e] + (smax * z[i]) * z[j] / zz;
    }
}

constexpr int kGJ = 32;        // pivots per step, and the tile of the update
constexpr int kGJThreads = 64;

// Inverse of the kGJ x kGJ block in S (row stride kGJ + 1) by kGJThreads threads:
// thread t holds half a row in registers; a step costs one barrier (the pivot
// row's owners scale it and publish it) and 16 multiply-adds per thread.
__device__ void gj_invert(const double (*S)[kGJ + 1], double *__restrict__ Dinv, int *__restrict__ bad)
{
    __shared__ double prow[2][kGJ + 1];  // scaled pivot row, its reciprocal pivot
    const int i = threadIdx.x >> 1, half = threadIdx.x & 1;
    double a[kGJ / 2];
#pragma unroll
    for (int c = 0; c < kGJ / 2; c++) a[c] = S[i][half * (kGJ / 2) + c];
#pragma unroll
    for (int k = 0; k < kGJ; k++) {
        constexpr int H = kGJ / 2;
        const int hk = k / H, ck = k % H;
        double *pr = prow[k & 1];
        // the row's entry in the pivot column, from the thread that holds it
        const double f = __shfl_sync(0xffffffffu, a[ck], (threadIdx.x & 30) | hk);
        if (i == k) {
            if (!(f > 0.0)) *bad = 1;
            const double rp = 1.0 / f;
#pragma unroll
            for (int c = 0; c < H; c++) {
                a[c] = half == hk && c == ck ? rp : a[c] * rp;
                pr[half * H + c] = a[c];
            }
            if (half == 0) pr[kGJ] = rp;
        }
        __syncthreads();
        if (i != k) {
            const double rp = pr[kGJ];
#pragma unroll
            for (int c = 0; c < H; c++)
                a[c] = half == hk && c == ck ? -f * rp : fma(-f, pr[half * H + c], a[c]);
        }
    }
#pragma unroll
    for (int c = 0; c < kGJ / 2; c++) Dinv[i * kGJ + half * (kGJ / 2) + c] = a[c];
}

__global__ void __launch_bounds__(kGJThreads) k_gj_first(int ld, const double *__restrict__ M, double *__restrict__ Dinv,
                                                         int *__restrict__ bad)
{
    __shared__ double S[kGJ][kGJ + 1];
    for (int e = threadIdx.x; e < kGJ * kGJ; e += kGJThreads) S[e / kGJ][e % kGJ] = M[(size_t)(e / kGJ) * ld + e % kGJ];
    __syncthreads();
    gj_invert(S, Dinv, bad);
}

// Rows of the panel C = M[:,P] (the block-lower half read by rows below the
// pivots, by columns above them) and of W = C D, eight rows per block.
constexpr int kGJPanelRows = 8;
__global__ void __launch_bounds__(kGJPanelRows * kGJ) k_gj_panel(int ld, int K, const double *__restrict__ M,
                                                                 const double *__restrict__ Dinv,
                                                                 double *__restrict__ C, double *__restrict__ W)
{
    __shared__ double c[kGJPanelRows][kGJ + 1], D[kGJ][kGJ + 1];
    const int i0 = blockIdx.x * kGJPanelRows, t = threadIdx.x;
    for (int e = t; e < kGJ * kGJ; e += kGJPanelRows * kGJ) D[e / kGJ][e % kGJ] = Dinv[e];
    if (i0 >= K) c[t / kGJ][t % kGJ] = M[(size_t)(i0 + t / kGJ) * ld + K + t % kGJ];
    else c[t % kGJPanelRows][t / kGJPanelRows] = M[(size_t)(K + t / kGJPanelRows) * ld + i0 + t % kGJPanelRows];
    __syncthreads();
    const int r = t / kGJ, k = t % kGJ;
    double w = 0.0;
#pragma unroll
    for (int m = 0; m < kGJ; m++) w = fma(c[r][m], D[m][k], w);
    C[(size_t)(i0 + r) * kGJ + k] = c[r][k];
    W[(size_t)(i0 + r) * kGJ + k] = w;
}

// One kGJ x kGJ tile of the block-lower half per block (two thousand of them at
// 1942 unknowns, so the SMs finish within a tile or two of each other), a thread
// 4 x 4 of it.  The next pivot block's tile goes first and its block inverts it
// while the others update.  FP64-bound: n^2 / 2 x 32 multiply-adds a step, 1942
// unknowns 95 us against 148 measured (the full Gauss-Jordan step took 215 us and
// 54 more to invert its pivot block).
__global__ void __launch_bounds__(kGJThreads) k_gj_update(int ld, int K, double *__restrict__ M,
                                                          const double *__restrict__ Dinv,
                                                          const double *__restrict__ C, const double *__restrict__ W,
                                                          double *__restrict__ Dnext, int *__restrict__ bad)
{
    __shared__ double Ws[kGJ][kGJ + 2], Cs[kGJ][kGJ + 2];  // [m][row]
    const int nt = ld / kGJ, kp = K / kGJ, t = threadIdx.x;
    int idx = blockIdx.x;
    if (kp + 1 < nt) {
        const int first = (kp + 1) * (kp + 2) / 2 + kp + 1;  // tile (kp + 1, kp + 1)
        idx = idx == 0 ? first : (idx == first ? 0 : idx);
    }
    int ti = (int)((sqrtf(8.0f * (float)idx + 1.0f) - 1.0f) * 0.5f);
    while (ti * (ti + 1) / 2 > idx) ti--;
    while ((ti + 1) * (ti + 2) / 2 <= idx) ti++;
    const int tj = idx - ti * (ti + 1) / 2;
    double *tile = M + (size_t)ti * kGJ * ld + (size_t)tj * kGJ;
    if (ti == kp || tj == kp) {
        for (int e = t; e < kGJ * kGJ; e += kGJThreads) {
            const int r = e / kGJ, c = e % kGJ;
            double v;
            if (ti == tj) v = -Dinv[e];
            else if (tj == kp) v = W[(size_t)(ti * kGJ + r) * kGJ + c];
            else v = W[(size_t)(tj * kGJ + c) * kGJ + r];
            tile[(size_t)r * ld + c] = v;
        }
        return;
    }
    for (int e = t; e < kGJ * kGJ; e += kGJThreads) {
        Ws[e % kGJ][e / kGJ] = W[(size_t)ti * kGJ * kGJ + e];
        Cs[e % kGJ][e / kGJ] = C[(size_t)tj * kGJ * kGJ + e];
    }
    const int r0 = (t >> 3) * 4, c0 = (t & 7) * 4;
    double a[4][4];
#pragma unroll
    for (int r = 0; r < 4; r++) {
        const double2 x = *(const double2 *)(tile + (size_t)(r0 + r) * ld + c0);
        const double2 y = *(const double2 *)(tile + (size_t)(r0 + r) * ld + c0 + 2);
        a[r][0] = x.x;
        a[r][1] = x.y;
        a[r][2] = y.x;
        a[r][3] = y.y;
    }
    __syncthreads();
#pragma unroll 4
    for (int m = 0; m < kGJ; m++) {
        double w[4], c[4];
#pragma unroll
        for (int k = 0; k < 4; k++) {
            w[k] = -Ws[m][r0 + k];
            c[k] = Cs[m][c0 + k];
        }
#pragma unroll
        for (int r = 0; r < 4; r++)
#pragma unroll
            for (int k = 0; k < 4; k++) a[r][k] = fma(w[r], c[k], a[r][k]);
    }
#pragma unroll
    for (int r = 0; r < 4; r++) {
        *(double2 *)(tile + (size_t)(r0 + r) * ld + c0) = make_double2(a[r][0], a[r][1]);
        *(double2 *)(tile + (size_t)(r0 + r) * ld + c0 + 2) = make_double2(a[r][2], a[r][3]);
    }
    if (ti != kp + 1 || tj != kp + 1) return;
    __syncthreads();
    double (*S)[kGJ + 1] = (double (*)[kGJ + 1])&Ws[0][0];
#pragma unroll
    for (int r = 0; r < 4; r++)
#pragma unroll
        for (int k = 0; k < 4; k++) S[r0 + r][c0 + k] = a[r][k];
    __syncthreads();
    gj_invert(S, Dnext, bad);
}

// the inverse, both halves, from -M's block-lower half
__global__ void k_gj_inverse(int n, int ld, const double *__restrict__ M, double *__restrict__ Cinv)
{
    const int i = blockIdx.x;
    for (int j = threadIdx.x; j < n; j += blockDim.x) {
        const bool low = j / kGJ <= i / kGJ;
        Cinv[(size_t)i * n + j] = -(low ? M[(size_t)i * ld + j] : M[(size_t)j * ld + i]);
    }
}

// C = Cinv (I - z z^T / z.z): the solve's projection of the residual orthogonal
// to the null vector z, folded into the inverse once.  One block per row.
__global__ void __launch_bounds__(128) k_coarse_project(int n, double *__restrict__ C, const double *__restrict__ z,
                                                        const double *__restrict__ zz)
{
    __shared__ double part[4];
    double *row = C + (size_t)blockIdx.x * n;
    double s = 0.0;
    for (int j = threadIdx.x; j < n; j += blockDim.x) s = s + row[j] * z[j];
    for (int o = 16; o; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if ((threadIdx.x & 31) == 0) part[threadIdx.x >> 5] = s;
    __syncthreads();
    s = ((part[0] + part[1]) + part[2]) + part[3];
    if (!(*zz > 0.0)) return;
    const double a = s / *zz;
    for (int j = threadIdx.x; j < n; j += blockDim.x) row[j] = row[j] - a * z[j];
}

__global__ void k_null_vector(int N, const double *__restrict__ B, double *z)
{
    int p = blockIdx.x * blockDim.x + threadIdx.x;
    if (p >= N) return;
    z[2 * p] = 0.0;
    z[2 * p + 1] = B[2 * p + 1];
}

__global__ void k_invdiag(int n, const double *__restrict__ d, double *inv)
{
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) inv[i] = 1.0 / d[i];
}

__global__ void k_fill(int n, double v, double *x)
{
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) x[i] = v;
}

static inline int nblk(long long n, int b = 256) { return (int)((n + b - 1) / b); }

// Thread block size of the one-thread-per-row setup kernels: on coarse levels
// (few, long rows) one warp per block, so the rows spread over as many SMs as
// possible instead of crowding a handful (each row is a sequential sum).
static inline int row_block(long long rows) { return rows < (long long)kSM * 256 ? 32 : 256; }

// ------------------------------------------------------------------ one level of Algorithm 1
static int coarsen_level(amg_hierarchy *h, int l, bool &is_coarsest, cudaStream_t s)
{
    Level &L = h->lev[l];
    const amg_options &o = h->opts;
    int N = L.N, n = 2 * N;
    is_coarsest = false;
    if (n <= o.coarse_eq_limit || l == o.max_levels - 1 || l == kMaxLevels - 1) {
        is_coarsest = true;
        return BD_OK;
    }
    // a1 strength
    DBuf<double> diag;
    BD_TRY(diag.scratch((size_t)n, s));
    DBuf<int> bad;
    BD_TRY(bad.scratch(1, s));
    BD_CUDA(cudaMemsetAsync(bad.p, 0, sizeof(int), s));
    k_diag<<<nblk(N), 256, 0, s>>>(N, L.A.rp.p, L.A.ci.p, L.A.v.p, diag.p, bad.p); ::bd::note_launch();
    BD_LAUNCH_CHECK();
    CSR S;
    S.nr = S.nc = N;
    DBuf<int> cnt;
    DBuf<double> wt;
    BD_TRY(cnt.scratch((size_t)N + 1, s));
    BD_TRY(wt.scratch((size_t)L.A.nb, s));
    BD_TRY(S.rp.scratch((size_t)N + 1, s));
    k_strength_count<<<nblk(32LL * N), 256, 0, s>>>(N, L.A.rp.p, L.A.ci.p, L.A.v.p, diag.p, o.theta,
                                                                   cnt.p, wt.p); ::bd::note_launch();
    BD_LAUNCH_CHECK();
    long long snnz = 0;
    BD_TRY(exclusive_scan(cnt.p, S.rp.p, N, &snnz, s));
    S.nnz = snnz;
    BD_TRY(S.ci.scratch((size_t)snnz, s));
    BD_TRY(S.v.scratch((size_t)snnz, s));
    k_strength_fill<<<nblk(32LL * N), 256, 0, s>>>(N, L.A.rp.p, L.A.ci.p, wt.p, S.rp.p, S.ci.p,
                                                                  S.v.p); ::bd::note_launch();
    BD_LAUNCH_CHECK();
    int hbad = 0;
    BD_CUDA(cudaMemcpyAsync(&hbad, bad.p, sizeof(int), cudaMemcpyDeviceToHost, s));
    BD_CUDA(cudaStreamSynchronize(s));
    if (hbad) return BD_EINVAL;  // non-positive diagonal: not a semi-definite operator
    if (l < o.square_levels) {
        CSR W, Q, S2;
        BD_TRY(W.rp.scratch((size_t)N + 1, s));
        BD_TRY(W.ci.scratch((size_t)snnz + N, s));
        BD_TRY(W.v.scratch((size_t)snnz + N, s));
        k_insert_diag<<<nblk(N + 1), 256, 0, s>>>(N, S.rp.p, S.ci.p, S.v.p, W.rp.p, W.ci.p, W.v.p); ::bd::note_launch();
        BD_LAUNCH_CHECK();
        long long qn = 0;
        BD_TRY(spgemm<1>(N, N, W.rp.p, W.ci.p, W.v.p, W.rp.p, W.ci.p, W.v.p, Q.rp, Q.ci, Q.v, &qn, s,
                         (double)(snnz + N) / std::max(N, 1), true));
        BD_TRY(S2.rp.scratch((size_t)N + 1, s));
        BD_TRY(S2.ci.scratch((size_t)(qn - N), s));
        BD_TRY(S2.v.scratch((size_t)(qn - N), s));
        k_drop_diag<<<nblk(32LL * (N + 1)), 256, 0, s>>>(N, Q.rp.p, Q.ci.p, Q.v.p, S2.rp.p, S2.ci.p, S2.v.p); ::bd::note_launch();
        BD_LAUNCH_CHECK();
        S.rp = std::move(S2.rp);
        S.ci = std::move(S2.ci);
        S.v = std::move(S2.v);
        S.nnz = qn - N;
    }
    // a2 MIS
    DBuf<unsigned char> state;
    BD_TRY(state.scratch((size_t)N, s));
    BD_CUDA(cudaMemsetAsync(state.p, 0, (size_t)N, s));
    DBuf<int> und;
    BD_TRY(und.scratch(1, s));
    unsigned long long key = level_key(o.seed, l, 0);
    int rounds = 0;
    for (;;) {
        BD_CUDA(cudaMemsetAsync(und.p, 0, sizeof(int), s));
        k_mis_select<<<nblk(8LL * N), 256, 0, s>>>(N, S.rp.p, S.ci.p, state.p, key); ::bd::note_launch();
        BD_LAUNCH_CHECK();
        k_mis_exclude<<<nblk(8LL * N), 256, 0, s>>>(N, S.rp.p, S.ci.p, state.p, und.p); ::bd::note_launch();
        BD_LAUNCH_CHECK();
        int hu = 0;
        BD_CUDA(cudaMemcpyAsync(&hu, und.p, sizeof(int), cudaMemcpyDeviceToHost, s));
        BD_CUDA(cudaStreamSynchronize(s));
        if (hu == 0) break;
        if (++rounds > N + 1) return BD_ETIMEOUT;  // each round settles at least one node
    }
    // a3 aggregates
    BD_TRY(L.mis.alloc((size_t)N));
    BD_TRY(L.agg.alloc((size_t)N));
    DBuf<int> flag, rid;
    BD_TRY(flag.scratch((size_t)N + 1, s));
    BD_TRY(rid.scratch((size_t)N + 1, s));
    k_root_flags<<<nblk(N), 256, 0, s>>>(N, state.p, L.mis.p, flag.p); ::bd::note_launch();
    BD_LAUNCH_CHECK();
    long long nagg = 0;
    BD_TRY(exclusive_scan(flag.p, rid.p, N, &nagg, s));
    BD_CUDA(cudaMemsetAsync(bad.p, 0, sizeof(int), s));
    k_assign<<<nblk(8LL * N), 256, 0, s>>>(N, S.rp.p, S.ci.p, S.v.p, L.mis.p, rid.p, L.agg.p, bad.p); ::bd::note_launch();
    BD_LAUNCH_CHECK();
    BD_CUDA(cudaMemcpyAsync(&hbad, bad.p, sizeof(int), cudaMemcpyDeviceToHost, s));
    BD_CUDA(cudaStreamSynchronize(s));
    if (hbad) return BD_ECUDA;  // a non-root without a root neighbour: MIS not maximal
    L.nagg = (int)nagg;
    if (2 * nagg >= n) {  // no coarsening: this level is the coarsest
        L.mis.release();
        L.agg.release();
        L.nagg = 0;
        is_coarsest = true;
        return BD_OK;
    }
    int Nc = (int)nagg;
    // a4 tentative prolongator and coarse near-null coefficients
    DBuf<int> moff, mfill, members;
    BD_TRY(moff.scratch((size_t)Nc + 1, s));
    BD_TRY(mfill.scratch((size_t)Nc + 2, s));  // counts, then the largest at [Nc + 1]
    BD_TRY(members.scratch((size_t)N, s));
    BD_CUDA(cudaMemsetAsync(mfill.p, 0, mfill.bytes(), s));
    k_count_members<<<nblk(N), 256, 0, s>>>(N, L.agg.p, mfill.p); ::bd::note_launch();
    BD_LAUNCH_CHECK();
    BD_TRY(device_max(mfill.p, Nc, mfill.p + Nc + 1, s));
    long long tot = 0;
    BD_TRY(exclusive_scan(mfill.p, moff.p, Nc, &tot, s));  // stream synchronised
    int mx = 0;
    BD_CUDA(cudaMemcpyAsync(&mx, mfill.p + Nc + 1, sizeof(int), cudaMemcpyDeviceToHost, s));
    BD_CUDA(cudaStreamSynchronize(s));
    BD_CUDA(cudaMemsetAsync(mfill.p, 0, mfill.bytes(), s));
    k_scatter_members<<<nblk(N), 256, 0, s>>>(N, L.agg.p, moff.p, mfill.p, members.p); ::bd::note_launch();
    BD_LAUNCH_CHECK();
    BD_TRY(sort_segments(members.p, nullptr, moff.p, Nc, mx, s));
    Level &C = h->lev[l + 1];
    C.N = Nc;
    BD_TRY(C.B.alloc(2 * (size_t)Nc));
    k_coarse_B<<<nblk(Nc), 256, 0, s>>>(Nc, moff.p, members.p, L.B.p, C.B.p); ::bd::note_launch();
    BD_LAUNCH_CHECK();
    BSR Pt;
    Pt.nbr = N;
    Pt.nbc = Nc;
    Pt.nb = N;
    DBuf<double> ptd;
    BD_TRY(Pt.rp.scratch((size_t)N + 1, s));
    BD_TRY(Pt.ci.scratch((size_t)N, s));
    BD_TRY(Pt.v.scratch(4 * (size_t)N, s));
    BD_TRY(ptd.scratch((size_t)n, s));
    k_ptent<<<nblk(N + 1), 256, 0, s>>>(N, L.agg.p, L.B.p, C.B.p, Pt.rp.p, Pt.ci.p, Pt.v.p, ptd.p); ::bd::note_launch();
    BD_LAUNCH_CHECK();
    // a5 lambda_max of D^{-1}A
    DBuf<LanczosState> lst;
    BD_TRY(lst.scratch(1, s));
    BD_CUDA(cudaMemsetAsync(lst.p, 0, sizeof(LanczosState), s));
    DBuf<double> vr, vz, vp, vq;
    BD_TRY(vr.scratch((size_t)n, s));
    BD_TRY(vz.scratch((size_t)n, s));
    BD_TRY(vp.scratch((size_t)n, s));
    BD_TRY(vq.scratch((size_t)n, s));
    k_lanczos_init<<<nblk(n), 256, 0, s>>>(n, level_key(o.seed, l, 1), diag.p, vr.p, vz.p, vp.p); ::bd::note_launch();
    BD_LAUNCH_CHECK();
    long long *acc = h->exact_acc.p;
    BD_CUDA(cudaMemsetAsync(acc, 0, h->exact_acc.bytes(), s));
    BD_TRY(exact_dot(vr.p, vz.p, n, &lst.p->rz[0], acc, s, true));
    for (int j = 0; j < o.esteig_steps; j++) {
        k_spmv_ordered<<<nblk(n, row_block(N)), row_block(N), 0, s>>>(n, L.A.rp.p, L.A.ci.p, L.A.v.p, vp.p, vq.p);
        ::bd::note_launch();
        BD_LAUNCH_CHECK();
        BD_TRY(exact_dot(vp.p, vq.p, n, &lst.p->pq[j], acc, s, true));
        if (n <= kDotUpdateMax) {
            BD_TRY(exact_dot_update(&lst.p->rz[j], &lst.p->pq[j], vq.p, diag.p, vr.p, vz.p, n, &lst.p->rz[j + 1], acc,
                                    s));
        } else {
            k_lanczos_update_r<<<nblk(n), 256, 0, s>>>(n, lst.p, j, vq.p, diag.p, vr.p, vz.p); ::bd::note_launch();
            BD_LAUNCH_CHECK();
            BD_TRY(exact_dot(vr.p, vz.p, n, &lst.p->rz[j + 1], acc, s, true));
        }
        if (j + 1 == o.esteig_steps) break;
        k_lanczos_update_p<<<nblk(n), 256, 0, s>>>(n, lst.p, j, vz.p, vp.p); ::bd::note_launch();
        BD_LAUNCH_CHECK();
    }
    k_lanczos_finish<<<1, 32, 0, s>>>(lst.p, o.esteig_steps); ::bd::note_launch();
    BD_LAUNCH_CHECK();
    LanczosState hst;
    BD_CUDA(cudaMemcpyAsync(&hst, lst.p, sizeof(hst), cudaMemcpyDeviceToHost, s));
    BD_CUDA(cudaStreamSynchronize(s));
    if (hst.bad) return BD_EINVAL;
    L.lam = hst.lam;
    // a6 P = Pt - omega D^{-1} A Pt
    long long pnb = 0;
    L.P.nbr = N;
    L.P.nbc = Nc;
    BD_TRY(spgemm<2>(N, Nc, L.A.rp.p, L.A.ci.p, L.A.v.p, Pt.rp.p, Pt.ci.p, Pt.v.p, L.P.rp, L.P.ci,
                     L.P.v, &pnb, s, 1.0, false));  // one block per row of the tentative prolongator
    L.P.nb = pnb;
    k_smooth_p<<<nblk(8LL * N), 256, 0, s>>>(N, L.P.rp.p, L.P.ci.p, L.P.v.p, L.agg.p, ptd.p, diag.p, lst.p); ::bd::note_launch();
    BD_LAUNCH_CHECK();
    // a7 R = P^T
    BD_TRY(bsr_transpose(L.P, L.R, s));
    // a8 A_c = R (A P)
    BSR AP;
    long long apnb = 0;
    BD_TRY(spgemm<2>(N, Nc, L.A.rp.p, L.A.ci.p, L.A.v.p, L.P.rp.p, L.P.ci.p, L.P.v.p, AP.rp, AP.ci,
                     AP.v, &apnb, s, (double)L.P.nb / std::max(N, 1), true));
    AP.nbr = N;
    AP.nbc = Nc;
    AP.nb = apnb;
    long long cnb = 0;
    C.A.nbr = C.A.nbc = Nc;
    BD_TRY(spgemm<2>(Nc, Nc, L.R.rp.p, L.R.ci.p, L.R.v.p, AP.rp.p, AP.ci.p, AP.v.p, C.A.rp, C.A.ci,
                     C.A.v, &cnb, s, (double)apnb / std::max(N, 1), false));
    C.A.nb = cnb;
    BD_CUDA(cudaStreamSynchronize(s));
    return BD_OK;
}

static int finish_level_common(Level &L, cudaStream_t s)
{
    int n = 2 * L.N;
    DBuf<double> diag;
    DBuf<int> bad;
    BD_TRY(diag.scratch((size_t)n, s));
    BD_TRY(bad.scratch(1, s));
    BD_CUDA(cudaMemsetAsync(bad.p, 0, sizeof(int), s));
    k_diag<<<nblk(L.N), 256, 0, s>>>(L.N, L.A.rp.p, L.A.ci.p, L.A.v.p, diag.p, bad.p); ::bd::note_launch();
    BD_LAUNCH_CHECK();
    BD_TRY(L.invdiag.alloc((size_t)n));
    k_invdiag<<<nblk(n), 256, 0, s>>>(n, diag.p, L.invdiag.p); ::bd::note_launch();
    BD_LAUNCH_CHECK();
    int hbad = 0;
    BD_CUDA(cudaMemcpyAsync(&hbad, bad.p, sizeof(int), cudaMemcpyDeviceToHost, s));
    BD_CUDA(cudaStreamSynchronize(s));
    return hbad ? BD_EINVAL : BD_OK;
}

constexpr int kCoarseSingleBlock = 256;  // coarsest sizes factored by one thread block

static int build_coarsest(amg_hierarchy *h, int l, cudaStream_t s)
{
    Level &L = h->lev[l];
    int n = 2 * L.N;
    if (n > kMaxCoarse) return BD_ERANGE;
    h->nc = n;
    const bool single = n <= kCoarseSingleBlock;
    const int ld = single ? n : (n + kGJ - 1) / kGJ * kGJ;  // padded to whole pivot blocks
    DBuf<double> Ad;
    BD_TRY(Ad.scratch((size_t)ld * ld, s));
    BD_TRY(h->cinv.alloc((size_t)n * n));
    BD_TRY(h->zc.alloc((size_t)n));
    BD_CUDA(cudaMemsetAsync(Ad.p, 0, Ad.bytes(), s));
    k_coarse_dense<<<nblk(32LL * L.N), 256, 0, s>>>(L.N, L.A.rp.p, L.A.ci.p, L.A.v.p, ld, Ad.p); ::bd::note_launch();
    BD_LAUNCH_CHECK();
    k_null_vector<<<nblk(L.N), 256, 0, s>>>(L.N, L.B.p, h->zc.p); ::bd::note_launch();
    BD_LAUNCH_CHECK();
    DBuf<double> zz;
    DBuf<int> bad;
    BD_TRY(zz.scratch(1, s));
    BD_TRY(bad.scratch(1, s));
    BD_CUDA(cudaMemsetAsync(bad.p, 0, sizeof(int), s));
    DBuf<double> st, Dinv, W, C;
    if (single) {
        k_coarse_factor<<<1, 256, 0, s>>>(n, Ad.p, h->zc.p, h->cinv.p, zz.p, bad.p); ::bd::note_launch();
        BD_LAUNCH_CHECK();
    } else {
        BD_TRY(st.scratch(2, s));
        BD_TRY(Dinv.scratch((size_t)2 * kGJ * kGJ, s));
        BD_TRY(W.scratch((size_t)kGJ * ld, s));
        BD_TRY(C.scratch((size_t)kGJ * ld, s));
        k_coarse_stats<<<1, 1024, 0, s>>>(n, ld, Ad.p, h->zc.p, st.p); ::bd::note_launch();
        k_coarse_rank1<<<ld, 256, 0, s>>>(n, ld, Ad.p, h->zc.p, st.p); ::bd::note_launch();
        k_gj_first<<<1, kGJThreads, 0, s>>>(ld, Ad.p, Dinv.p, bad.p); ::bd::note_launch();
        const int nt = ld / kGJ;
        for (int k = 0; k < nt; k++) {
            double *D = Dinv.p + (k & 1) * kGJ * kGJ, *Dn = Dinv.p + (1 - (k & 1)) * kGJ * kGJ;
            k_gj_panel<<<ld / kGJPanelRows, kGJPanelRows * kGJ, 0, s>>>(ld, k * kGJ, Ad.p, D, C.p, W.p);
            ::bd::note_launch();
            k_gj_update<<<nt * (nt + 1) / 2, kGJThreads, 0, s>>>(ld, k * kGJ, Ad.p, D, C.p, W.p, Dn, bad.p);
            ::bd::note_launch();
        }
        k_gj_inverse<<<n, 256, 0, s>>>(n, ld, Ad.p, h->cinv.p); ::bd::note_launch();
        BD_LAUNCH_CHECK();
        BD_CUDA(cudaMemcpyAsync(zz.p, st.p + 1, sizeof(double), cudaMemcpyDeviceToDevice, s));
    }
    k_coarse_project<<<n, 128, 0, s>>>(n, h->cinv.p, h->zc.p, zz.p); ::bd::note_launch();
    BD_LAUNCH_CHECK();
    int hbad = 0;
    BD_CUDA(cudaMemcpyAsync(&hbad, bad.p, sizeof(int), cudaMemcpyDeviceToHost, s));
    BD_CUDA(cudaStreamSynchronize(s));
    return hbad ? BD_EINVAL : BD_OK;
}

static int setup_from_level0(amg_hierarchy *h, cudaStream_t s)
{
    Level &L0 = h->lev[0];
    BD_TRY(h->exact_acc.alloc(kExactScratch));
    BD_TRY(L0.B.alloc(2 * (size_t)L0.N));
    k_fill<<<nblk(2LL * L0.N), 256, 0, s>>>(2 * L0.N, 1.0, L0.B.p); ::bd::note_launch();
    BD_LAUNCH_CHECK();
    int l = 0;
    for (;;) {
        BD_TRY(finish_level_common(h->lev[l], s));
        bool coarsest = false;
        BD_TRY(coarsen_level(h, l, coarsest, s));
        if (coarsest) break;
        l++;
    }
    h->nlev = l + 1;
    BD_TRY(build_coarsest(h, l, s));
    return BD_OK;
}

static int check_opts(const amg_options *o)
{
    if (!(o->theta >= 0.0) || o->coarse_eq_limit < 2 || o->max_levels < 1 ||
        o->max_levels > kMaxLevels || (o->cheb_degree != 1 && o->cheb_degree != 2) ||
        o->esteig_steps < 1 || o->esteig_steps > 64 || o->square_levels < 0 ||
        !(o->eig_lo > 0.0) || !(o->eig_hi > o->eig_lo) || (o->precision != 0 && o->precision != 1) ||
        (o->autotune != 0 && o->autotune != 1))
        return BD_EINVAL;
    return BD_OK;
}

}  // namespace bd

using namespace bd;

extern "C" int amg_setup(const bd_system *sys, const amg_options *opts, void *stream,
                         amg_hierarchy **out)
{
    if (!sys || !out) return BD_EINVAL;
    *out = nullptr;
    amg_options o;
    amg_options_default(&o);
    if (opts) o = *opts;
    BD_TRY(check_opts(&o));
    cudaStream_t s = (cudaStream_t)stream;
    ScratchPool pool;
    amg_hierarchy *h = new (std::nothrow) amg_hierarchy();
    if (!h) return BD_ENOMEM;
    h->opts = o;
    Level &L0 = h->lev[0];
    L0.N = sys->N;
    L0.A.nbr = L0.A.nbc = sys->N;
    L0.A.nb = sys->A.nb;
    int st;
    if ((st = L0.A.rp.alloc((size_t)sys->N + 1)) || (st = L0.A.ci.alloc((size_t)sys->A.nb)) ||
        (st = L0.A.v.alloc(4 * (size_t)sys->A.nb))) {
        delete h;
        return st;
    }
    if (cudaMemcpyAsync(L0.A.rp.p, sys->A.rp.p, L0.A.rp.bytes(), cudaMemcpyDeviceToDevice, s) ||
        cudaMemcpyAsync(L0.A.ci.p, sys->A.ci.p, L0.A.ci.bytes(), cudaMemcpyDeviceToDevice, s) ||
        cudaMemcpyAsync(L0.A.v.p, sys->A.v.p, L0.A.v.bytes(), cudaMemcpyDeviceToDevice, s)) {
        delete h;
        return BD_ECUDA;
    }
    h->prec32 = o.precision == 1;
    if ((st = setup_from_level0(h, s)) || (st = build_fine_stencil(h, sys, s)) ||
        (st = prepare_solve(h, s))) {
        delete h;
        return st;
    }
    *out = h;
    return BD_OK;
}

// The elliptic operator Ai + Ae of the decoupled scheme (Section 2.2, Eq. 6)
// as the block operator [I, 0; 0, Ai + Ae] on the assembled node pattern, so
// that the block hierarchy's u-field is smoothed aggregation on Ai + Ae.
__global__ void k_elliptic_values(int N, const int *__restrict__ rp, const int *__restrict__ ci,
                                  const double *__restrict__ Ki, const double *__restrict__ Ke,
                                  double *__restrict__ v)
{
    for (int p = blockIdx.x * blockDim.x + threadIdx.x; p < N; p += gridDim.x * blockDim.x)
        for (int t = rp[p]; t < rp[p + 1]; t++) {
            v[4 * (size_t)t] = ci[t] == p ? 1.0 : 0.0;
            v[4 * (size_t)t + 1] = 0.0;
            v[4 * (size_t)t + 2] = 0.0;
            v[4 * (size_t)t + 3] = Ki[t] + Ke[t];
        }
}

extern "C" int bd_elliptic_setup(const bd_system *sys, const amg_options *opts, void *stream,
                                 amg_hierarchy **out)
{
    if (!sys || !out) return BD_EINVAL;
    *out = nullptr;
    amg_options o;
    amg_options_default(&o);
    if (opts) o = *opts;
    BD_TRY(check_opts(&o));
    cudaStream_t s = (cudaStream_t)stream;
    ScratchPool pool;
    amg_hierarchy *h = new (std::nothrow) amg_hierarchy();
    if (!h) return BD_ENOMEM;
    h->opts = o;
    h->prec32 = o.precision == 1;
    Level &L0 = h->lev[0];
    L0.N = sys->N;
    L0.A.nbr = L0.A.nbc = sys->N;
    L0.A.nb = sys->A.nb;
    int st;
    if ((st = L0.A.rp.alloc((size_t)sys->N + 1)) || (st = L0.A.ci.alloc((size_t)sys->A.nb)) ||
        (st = L0.A.v.alloc(4 * (size_t)sys->A.nb))) {
        delete h;
        return st;
    }
    if (cudaMemcpyAsync(L0.A.rp.p, sys->A.rp.p, L0.A.rp.bytes(), cudaMemcpyDeviceToDevice, s) ||
        cudaMemcpyAsync(L0.A.ci.p, sys->A.ci.p, L0.A.ci.bytes(), cudaMemcpyDeviceToDevice, s)) {
        delete h;
        return BD_ECUDA;
    }
    k_elliptic_values<<<grid_for(sys->N, 256), 256, 0, s>>>(sys->N, sys->A.rp.p, sys->A.ci.p, sys->Ki.p,
                                                            sys->Ke.p, L0.A.v.p); ::bd::note_launch();
    if (cudaGetLastError() != cudaSuccess) {
        delete h;
        return BD_ECUDA;
    }
    if ((st = setup_from_level0(h, s)) || (st = prepare_solve(h, s)) || (st = scalar_build(h, sys, s))) {
        delete h;
        return st;
    }
    *out = h;
    return BD_OK;
}

extern "C" int amg_setup_from_csr(int n, const int *row_ptr, const int *col, const double *val,
                                  int on_device, const amg_options *opts, void *stream,
                                  amg_hierarchy **out)
{
    if (!row_ptr || !col || !val || !out || n < 2 || (n & 1)) return BD_EINVAL;
    *out = nullptr;
    amg_options o;
    amg_options_default(&o);
    if (opts) o = *opts;
    BD_TRY(check_opts(&o));
    cudaStream_t s = (cudaStream_t)stream;
    ScratchPool pool;
    DBuf<int> drp, dci;
    DBuf<double> dv;
    const int *prp = row_ptr, *pci = col;
    const double *pv = val;
    if (!on_device) {
        int nnz = row_ptr[n];
        if (nnz < 0) return BD_EINVAL;
        BD_TRY(drp.alloc((size_t)n + 1));
        BD_TRY(dci.alloc((size_t)nnz));
        BD_TRY(dv.alloc((size_t)nnz));
        BD_TRY(copy_in(drp.p, row_ptr, sizeof(int) * ((size_t)n + 1), 0, s));
        BD_TRY(copy_in(dci.p, col, sizeof(int) * (size_t)nnz, 0, s));
        BD_TRY(copy_in(dv.p, val, sizeof(double) * (size_t)nnz, 0, s));
        prp = drp.p;
        pci = dci.p;
        pv = dv.p;
    }
    amg_hierarchy *h = new (std::nothrow) amg_hierarchy();
    if (!h) return BD_ENOMEM;
    h->opts = o;
    h->prec32 = o.precision == 1;
    h->lev[0].N = n / 2;
    int st = bsr_from_scalar_csr(n, prp, pci, pv, h->lev[0].A, s);
    if (!st) st = setup_from_level0(h, s);
    if (!st) st = prepare_solve(h, s);
    if (st) {
        delete h;
        return st;
    }
    *out = h;
    return BD_OK;
}

extern "C" int amg_num_levels(const amg_hierarchy *h, int *nlevels)
{
    if (!h || !nlevels) return BD_EINVAL;
    *nlevels = h->nlev;
    return BD_OK;
}

extern "C" int amg_level_info(const amg_hierarchy *h, int level, int *n, long long *nnz, int *n_agg,
                              double *lambda, long long *p_nnz)
{
    if (!h || level < 0 || level >= h->nlev) return BD_EINVAL;
    const Level &L = h->lev[level];
    bool last = level == h->nlev - 1;
    if (n) *n = 2 * L.N;
    if (nnz) *nnz = 4 * L.A.nb;
    if (n_agg) *n_agg = last ? 0 : L.nagg;
    if (lambda) *lambda = last ? 0.0 : L.lam;
    if (p_nnz) *p_nnz = last ? 0 : 4 * L.P.nb;
    return BD_OK;
}

extern "C" int amg_level_lanes(const amg_hierarchy *h, int level, int lanes[3])
{
    if (!h || !lanes || level < 0 || level >= h->nlev) return BD_EINVAL;
    const Level &L = h->lev[level];
    const bool last = level == h->nlev - 1;
    lanes[0] = last || (level == 0 && h->fine.valid) ? 0 : L.lanes[0];
    lanes[1] = last ? 0 : L.lanes[1];
    lanes[2] = last ? 0 : L.lanes[2];
    return BD_OK;
}

extern "C" int amg_export_level(const amg_hierarchy *h, int level, int *a_row_ptr, int *a_col,
                                double *a_val, unsigned char *mis, int *agg, int *p_row_ptr,
                                int *p_col, double *p_val, void *stream)
{
    if (!h || level < 0 || level >= h->nlev) return BD_EINVAL;
    cudaStream_t s = (cudaStream_t)stream;
    const Level &L = h->lev[level];
    bool last = level == h->nlev - 1;
    if (a_row_ptr || a_col || a_val) BD_TRY(bsr_to_scalar_csr_host(L.A, a_row_ptr, a_col, a_val, s));
    if (!last) {
        if (mis) BD_CUDA(cudaMemcpyAsync(mis, L.mis.p, (size_t)L.N, cudaMemcpyDeviceToHost, s));
        if (agg) BD_CUDA(cudaMemcpyAsync(agg, L.agg.p, sizeof(int) * (size_t)L.N, cudaMemcpyDeviceToHost, s));
        if (p_row_ptr || p_col || p_val) BD_TRY(bsr_to_scalar_csr_host(L.P, p_row_ptr, p_col, p_val, s));
    }
    BD_CUDA(cudaStreamSynchronize(s));
    return BD_OK;
}

extern "C" void amg_destroy(amg_hierarchy *h)
{
    if (!h) return;
    if (h->host_scal) cudaFreeHost(h->host_scal);
    delete h;
}
