// amg_bsr.cuh -- 2x2-block CSR operator application shared by the V-cycle of
// one hierarchy (amg_solve.cu) and of a stack of hierarchies (amg_stack.cu):
// scalar traits, block loads, the lane-parallel SpMV kernels with fused
// epilogues, their launcher and the lanes-per-row rule.
#pragma once

#include <algorithm>

#include "amg_internal.cuh"
#include "fp_convert.h"

namespace bd {

// ------------------------------------------------------------------ scalar traits
template <class S> struct V2;
template <> struct V2<double> {
    using T = double2;
    static __device__ __forceinline__ double2 mk(double a, double b) { return make_double2(a, b); }
};
template <> struct V2<float> {
    using T = float2;
    static __device__ __forceinline__ float2 mk(float a, float b) { return make_float2(a, b); }
};
template <class S> using v2 = typename V2<S>::T;

template <class S> struct BlkS {
    S a00, a01, a10, a11;
};
static __device__ __forceinline__ BlkS<double> load_blk(const double *__restrict__ v, size_t t)
{
    const double2 p = ((const double2 *)v)[2 * t], q = ((const double2 *)v)[2 * t + 1];
    return {p.x, p.y, q.x, q.y};
}
static __device__ __forceinline__ BlkS<float> load_blk(const float *__restrict__ v, size_t t)
{
    const float4 p = ((const float4 *)v)[t];
    return {p.x, p.y, p.z, p.w};
}

// ------------------------------------------------------------------ lane sums
// Sums of y0 and y1 over the T lanes of a group, left in the group's first
// lane (the other lanes hold partial values).  The lower half of the group
// reduces y0 and the upper half y1, each in the tree an xor butterfly uses
// (IEEE addition is commutative, so the results carry the butterfly's bits),
// then y1 moves to the first lane: log2(T) adds per lane instead of 2 log2(T),
// and FP64 adds are scarce on this part.
template <int T, class S>
static __device__ __forceinline__ void group_sum2(S &y0, S &y1)
{
    if constexpr (T > 1) {
        const bool hi = (threadIdx.x & (T - 1)) >= T / 2;
        S mine = hi ? y1 : y0;
        mine += __shfl_xor_sync(0xffffffffu, hi ? y0 : y1, T / 2, T);
#pragma unroll
        for (int o = T / 4; o > 0; o >>= 1) mine += __shfl_xor_sync(0xffffffffu, mine, o, T);
        y0 = mine;
        y1 = __shfl_down_sync(0xffffffffu, mine, T / 2, T);
    }
}

// ------------------------------------------------------------------ entries of a block operator
// How one entry of a block operator is stored and applied.  t: position of the
// entry, q: its column as stored, g: the gathered vector.
// Full: a 2x2 block, four multiply-adds.
template <class S> struct MatFull {
    using Sc = S;
    static constexpr bool OWN = false;
    const S *__restrict__ v;
    struct Acc {
        S y0 = 0, y1 = 0;
    };
    template <class G> __device__ __forceinline__ void step(Acc &A, size_t t, int q, const G &g) const
    {
        const BlkS<S> a = load_blk(v, t);
        const v2<S> x = g(q);
        A.y0 = fma(a.a00, x.x, fma(a.a01, x.y, A.y0));
        A.y1 = fma(a.a10, x.x, fma(a.a11, x.y, A.y1));
    }
    __device__ __forceinline__ void finish(const Acc &A, S &y0, S &y1) const
    {
        y0 = A.y0;
        y1 = A.y1;
    }
};
// Pair: the finest level's P and R (PairOp).  A block K [ki + alpha, ki; ki, ki +
// ke] holds two numbers, two multiply-adds on (v + u, u); alpha is nonzero for
// a row's own entries only, which come first with the sign bit of their column
// set, and applies to v.  Half the FP64 work and 20 instead of 36 bytes (FP32: 12
// instead of 20) per block; the kernels are bound by the latency of their gathers
// (FP64 pipe 65-70 % busy while SMs are active): 128x128x32 FP64 R 45.5 -> 35.8 us,
// P 46 -> 39.6; 256x256x64 FP32 R 124 -> 105, P 126 -> 107.
constexpr int kColMask = 0x7fffffff;
template <class S> struct MatPair {
    using Sc = S;
    static constexpr bool OWN = true;
    const v2<S> *__restrict__ v;
    const S *__restrict__ alpha;
    struct Acc {
        S a = 0, b = 0, c = 0;
    };
    template <class G> __device__ __forceinline__ void own(Acc &A, size_t t, int q, const G &g) const
    {
        A.c = fma(alpha[t], g.v(q & kColMask), A.c);
    }
    template <class G> __device__ __forceinline__ void step(Acc &A, size_t t, int q, const G &g) const
    {
        const v2<S> k = v[t], x = g.su(q & kColMask);
        A.a = fma(k.x, x.x, A.a);
        A.b = fma(k.y, x.y, A.b);
    }
    __device__ __forceinline__ void finish(const Acc &A, S &y0, S &y1) const
    {
        y0 = A.a + A.c;
        y1 = A.a + A.b;
    }
};

template <class S> MatPair<S> mat_pair(const PairOp &p);
template <> inline MatPair<double> mat_pair<double>(const PairOp &p) { return {(const double2 *)p.v.p, p.alpha.p}; }
template <> inline MatPair<float> mat_pair<float>(const PairOp &p) { return {(const float2 *)p.v32.p, p.alpha32.p}; }

// A gathered vector of (v, u) pairs, or (SU) of (v + u, u) pairs.
template <class S, bool SU = false> struct GatherVec {
    const v2<S> *__restrict__ x;
    __device__ __forceinline__ v2<S> operator()(int q) const
    {
        const v2<S> a = x[q];
        return SU ? V2<S>::mk(a.x - a.y, a.y) : a;
    }
    __device__ __forceinline__ v2<S> su(int q) const
    {
        const v2<S> a = x[q];
        return SU ? a : V2<S>::mk(a.x + a.y, a.y);
    }
    __device__ __forceinline__ S v(int q) const
    {
        const v2<S> a = x[q];
        return SU ? a.x - a.y : a.x;
    }
};

// Entries [b, e) of a row in steps of T, from lane `lane`.
template <int T, class M, class G>
static __device__ __forceinline__ void row_sum(const M &mat, const int *__restrict__ ci, int b, int e, const G &g,
                                               typename M::Sc &y0, typename M::Sc &y1)
{
    typename M::Acc A;
    if constexpr (M::OWN) {
        for (int t = b; t < e; t += T) {
            const int q = ci[t];
            if (q >= 0) break;
            mat.own(A, (size_t)t, q, g);
        }
    }
#pragma unroll 4
    for (int t = b; t < e; t += T) mat.step(A, (size_t)t, ci[t], g);
    mat.finish(A, y0, y1);
}

// ------------------------------------------------------------------ block-CSR SpMV
// T lanes cooperate on one 2x2 block row (T = 1: one thread per row, no
// reduction).  The row loop is warp-uniform so every lane reaches the shuffles.
template <int T, class M, class G, class E>
static __global__ void __launch_bounds__(256) k_bsr(int N, const int *__restrict__ rp,
                                              const int *__restrict__ ci, M mat, G gather, E epi)
{
    const int lane = threadIdx.x & (T - 1);
    const int groups = (gridDim.x * blockDim.x) / T;
    const int warp_first = ((blockIdx.x * blockDim.x + threadIdx.x) & ~31) / T;
    const int g_in_warp = (threadIdx.x & 31) / T;
    for (int pw = warp_first; pw < N; pw += groups) {
        const int p = pw + g_in_warp;
        const bool act = p < N;
        typename M::Sc y0, y1;
        row_sum<T>(mat, ci, act ? rp[p] + lane : 0, act ? rp[p + 1] : 0, gather, y0, y1);
        group_sum2<T>(y0, y1);
        if (act && lane == 0) epi(p, y0, y1);
    }
}

// The same rows in equal contiguous shares, one thread block per SM (rows
// [N b / G, N (b + 1) / G) for block b of G): for operators whose row groups
// fit one wave, so that no SM runs a block more than the others.
template <int T, class M, class G, class E>
static __global__ void __launch_bounds__(1024, 1) k_bsr_eq(int N, const int *__restrict__ rp,
                                                  const int *__restrict__ ci, M mat, G gather, E epi)
{
    const int r0 = (int)((long long)N * blockIdx.x / gridDim.x);
    const int r1 = (int)((long long)N * (blockIdx.x + 1) / gridDim.x);
    const int lane = threadIdx.x & (T - 1);
    const int groups = blockDim.x / T;
    const int warp_first = (threadIdx.x & ~31) / T;
    const int g_in_warp = (threadIdx.x & 31) / T;
    for (int pw = r0 + warp_first; pw < r1; pw += groups) {
        const int p = pw + g_in_warp;
        const bool act = p < r1;
        typename M::Sc y0, y1;
        row_sum<T>(mat, ci, act ? rp[p] + lane : 0, act ? rp[p + 1] : 0, gather, y0, y1);
        group_sum2<T>(y0, y1);
        if (act && lane == 0) epi(p, y0, y1);
    }
}

// Long rows on small levels (few hundred to a few thousand block rows of
// hundreds of blocks): a whole thread block of TB threads per row, so that each
// thread walks only a few blocks; warp shuffles then shared memory reduce.
// The launch bound asks for 1024 resident threads per SM, not 2048, so that
// the FP64 instantiations get 64 registers (at 32 they spill).
template <int TB, class M, class G, class E>
static __global__ void __launch_bounds__(TB, 1024 / TB) k_bsr_wide(int N, const int *__restrict__ rp,
                                                  const int *__restrict__ ci, M mat, G gather,
                                                  E epi)
{
    __shared__ typename M::Sc red[2][TB / 32];
    for (int p = blockIdx.x; p < N; p += gridDim.x) {
        typename M::Sc y0, y1;
        row_sum<TB>(mat, ci, rp[p] + threadIdx.x, rp[p + 1], gather, y0, y1);
        group_sum2<32>(y0, y1);
        const int w = threadIdx.x >> 5;
        if ((threadIdx.x & 31) == 0) {
            red[0][w] = y0;
            red[1][w] = y1;
        }
        __syncthreads();
        if (threadIdx.x == 0) {
            typename M::Sc a0 = 0, a1 = 0;
#pragma unroll
            for (int i = 0; i < TB / 32; i++) {
                a0 += red[0][i];
                a1 += red[1][i];
            }
            epi(p, a0, a1);
        }
        __syncthreads();
    }
}

// Rows [0, N) of a block-CSR operator given by its arrays (a prefix of the
// rows of a larger operator is a valid argument).
template <class M, class G, class E>
static int launch_bsr_rows(int N, const int *rp, const int *ci, M mat, int T, G g, E e, cudaStream_t s)
{
    if (N <= 0) return BD_OK;
    const int threads = 256;
    long long groups_per_block = T >= 64 ? 1 : threads / T;
    int grid = (int)std::min<long long>((N + groups_per_block - 1) / groups_per_block, (long long)kSM * 16);
    if (T >= 64) {
        int gw = (int)std::min<long long>(N, (long long)kSM * 32);
        switch (T) {
        case 64: k_bsr_wide<64, M><<<gw, 64, 0, s>>>(N, rp, ci, mat, g, e); ::bd::note_launch(); break;
        case 128: k_bsr_wide<128, M><<<gw, 128, 0, s>>>(N, rp, ci, mat, g, e); ::bd::note_launch(); break;
        default: k_bsr_wide<256, M><<<gw, 256, 0, s>>>(N, rp, ci, mat, g, e); ::bd::note_launch(); break;
        }
        BD_LAUNCH_CHECK();
        return BD_OK;
    }
    if ((long long)N * T <= (long long)kSM * 1024) {
        // one block per SM, equal shares of the rows
        const long long per = ((long long)N + kSM - 1) / kSM * T;
        const int tb = (int)std::min<long long>(1024, std::max<long long>(32, (per + 31) / 32 * 32));
        const int gb = (int)std::min<long long>(kSM, N);
        switch (T) {
        case 1: k_bsr_eq<1, M><<<gb, tb, 0, s>>>(N, rp, ci, mat, g, e); break;
        case 2: k_bsr_eq<2, M><<<gb, tb, 0, s>>>(N, rp, ci, mat, g, e); break;
        case 4: k_bsr_eq<4, M><<<gb, tb, 0, s>>>(N, rp, ci, mat, g, e); break;
        case 8: k_bsr_eq<8, M><<<gb, tb, 0, s>>>(N, rp, ci, mat, g, e); break;
        case 16: k_bsr_eq<16, M><<<gb, tb, 0, s>>>(N, rp, ci, mat, g, e); break;
        default: k_bsr_eq<32, M><<<gb, tb, 0, s>>>(N, rp, ci, mat, g, e); break;
        }
        ::bd::note_launch();
        BD_LAUNCH_CHECK();
        return BD_OK;
    }
    switch (T) {
    case 1: k_bsr<1, M><<<grid, threads, 0, s>>>(N, rp, ci, mat, g, e); ::bd::note_launch(); break;
    case 2: k_bsr<2, M><<<grid, threads, 0, s>>>(N, rp, ci, mat, g, e); ::bd::note_launch(); break;
    case 4: k_bsr<4, M><<<grid, threads, 0, s>>>(N, rp, ci, mat, g, e); ::bd::note_launch(); break;
    case 8: k_bsr<8, M><<<grid, threads, 0, s>>>(N, rp, ci, mat, g, e); ::bd::note_launch(); break;
    case 16: k_bsr<16, M><<<grid, threads, 0, s>>>(N, rp, ci, mat, g, e); ::bd::note_launch(); break;
    default: k_bsr<32, M><<<grid, threads, 0, s>>>(N, rp, ci, mat, g, e); ::bd::note_launch(); break;
    }
    BD_LAUNCH_CHECK();
    return BD_OK;
}

template <class S, class G, class E>
static int launch_bsr(const BSR &A, const S *vals, int T, G g, E e, cudaStream_t s)
{
    return launch_bsr_rows(A.nbr, A.rp.p, A.ci.p, MatFull<S>{vals}, T, g, e, s);
}

// Lanes per block row, from per-operator timings inside the V-cycle on the
// 128x128x32 slab's levels.  Every lane-level reduction step costs adds,
// which are scarce in FP64 on this part, so FP64 rows use as few lanes as
// their length allows; FP32 adds are cheap, so FP32 rows use more lanes to
// shorten each thread's chain of dependent loads.  Small levels get more lanes
// so the grid still fills the GPU.  Levels with few, long rows (the dense-ish
// coarse levels): a warp per row in FP64 (a thread block's extra reduction
// steps cost more FP64 adds than its extra lanes save), a thread block per
// row in FP32.
// Rows of 1000 blocks and more (the nearly dense levels of large slabs) take a
// thread block each, however many they are (11501 rows of 2830 blocks, us per
// V-cycle: FP64 sliced 8 1980, 128 threads 1061; FP32 32 lanes 528, 256 threads 403).
constexpr double kLongRow = 1000.0;
static int lanes_for(const BSR &A, bool fp32)
{
    const double avg = A.nbr > 0 ? (double)A.nb / A.nbr : 1.0;
    if (avg >= kLongRow) return fp32 ? 256 : 128;
    int T;
    if (fp32) T = avg <= 3 ? 1 : (avg <= 12 ? 2 : (avg <= 48 ? 4 : (avg <= 100 ? 8 : (avg <= 160 ? 16 : 32))));
    else T = avg <= 40 ? 1 : (avg <= 160 ? 4 : (avg <= 640 ? 8 : 16));
    while (T < 32 && (long long)A.nbr * T < 65536) T <<= 1;
    if ((long long)A.nbr * 32 < 131072 && avg > 96) {  // few long rows
        if (!fp32) return A.nbr >= 2048 ? 32 : (avg <= 600 ? 64 : 128);
        T = 64;
        while (T < 256 && T * 3 < avg) T <<= 1;
    }
    return T;
}

}  // namespace bd
