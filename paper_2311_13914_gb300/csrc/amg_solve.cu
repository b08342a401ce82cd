// amg_solve.cu -- a10/a11: V-cycle (Algorithm 2) with Chebyshev-Jacobi
// smoothing (Appendix A) and the projected PCG of Section 2.2 on the device.
//
// Every operator application is one pass of an SpMV kernel whose epilogue
// fuses the vector work of the step around it (Chebyshev recurrence, residual,
// correction), so each level streams its matrix four times per cycle and its
// vectors a few times.  The V-cycle is written once over the storage scalar S:
// S = double is the plain FP64 form; S = float keeps FP32 copies of every
// level's values and vectors (half the bytes, none of the FP64 pipe) and runs
// inside an FP64 flexible CG, with the coarsest solve, the outer residual, the
// dot products and the null-space projection in FP64.  Reductions are
// deterministic: fixed grid, per-block partial sums, one finishing block.
#include <algorithm>
#include <cmath>
#include <cstdlib>
#include <new>
#include <type_traits>

#include "amg_bsr.cuh"
#include "amg_internal.cuh"
#include "fine_stencil.cuh"
#include "grid_index.h"
#include "pcg_reduce.cuh"
#include "scalar.cuh"

namespace bd {

// ------------------------------------------------------------------ sliced block operator
// FP64 values sit in two planes, (a00, a01) then (a10, a11), so each half of a
// group is one contiguous 512-byte warp load; FP32 values are one float4.
__device__ __forceinline__ BlkS<double> load_sliced(const double *__restrict__ v, size_t idx, size_t plane)
{
    const double2 p = ((const double2 *)v)[idx], q = ((const double2 *)v)[plane + idx];
    return {p.x, p.y, q.x, q.y};
}
__device__ __forceinline__ BlkS<float> load_sliced(const float *__restrict__ v, size_t idx, size_t)
{
    const float4 p = ((const float4 *)v)[idx];
    return {p.x, p.y, p.z, p.w};
}

// One warp per slice of 32/K rows with K lanes each.  Block b owns slices
// [bsl[b], bsl[b+1]), which split the groups evenly over the blocks, and its
// warps take the next slice whenever they finish one: slices differ in length
// (sorted rows: a window's first are its longest), and with a fixed share of
// three or four slices per warp the slowest held its SM for a third of the
// launch.  Lane k of a row sums entries k, k+K, ... and the K partial sums meet
// in the lane-sum tree k_bsr<K> uses (group_sum2), so both forms give the same
// bits.  Rows sorted by length leave few padded positions, and every FP64
// instruction of the loop and the epilogue works on 32 lanes (the FP64 pipe,
// not HBM, bounds the coarse levels in FP64).
constexpr int kSlicedTPB = 512;
template <class S> struct SlicedMinB { static constexpr int v = sizeof(S) == 8 ? 2 : 4; };
template <int K, class M, class G, class E>
__global__ void __launch_bounds__(kSlicedTPB, SlicedMinB<typename M::Sc>::v)
    k_bsell(const int *__restrict__ sptr, const int *__restrict__ bsl, const int *__restrict__ order,
            const int *__restrict__ col, M mat, G gather, E epi)
{
    __shared__ int next;
    if (threadIdx.x == 0) next = bsl[blockIdx.x];
    const int s1 = bsl[blockIdx.x + 1];
    __syncthreads();
    const int lane = threadIdx.x & 31;
    for (;;) {
        int sl = 0;
        if (lane == 0) sl = atomicAdd(&next, 1);
        sl = __shfl_sync(0xffffffffu, sl, 0);
        if (sl >= s1) break;
        const int j0 = sptr[sl], j1 = sptr[sl + 1];
        const int r = order[sl * (32 / K) + lane / K];
        typename M::Acc A;
        typename M::Sc r0 = 0, r1 = 0;
        if constexpr (M::OWN) {
            for (int j = j0; j < j1; j++) {
                const size_t idx = (size_t)j * 32 + lane;
                const int q = col[idx];
                if (q >= 0) break;
                mat.own(A, idx, q, gather);
            }
        }
#pragma unroll 4
        for (int j = j0; j < j1; j++) {
            const size_t idx = (size_t)j * 32 + lane;
            mat.step(A, idx, col[idx], gather);
        }
        mat.finish(A, r0, r1);
        group_sum2<K>(r0, r1);
        if ((lane & (K - 1)) == 0 && r >= 0) epi(r, r0, r1);
    }
}

// Full blocks in the sliced form: two planes of half blocks in FP64.
template <class S> struct MatSliced {
    using Sc = S;
    static constexpr bool OWN = false;
    using Acc = typename MatFull<S>::Acc;
    const S *__restrict__ v;
    size_t plane;
    __device__ __forceinline__ void finish(const Acc &A, S &y0, S &y1) const
    {
        y0 = A.y0;
        y1 = A.y1;
    }
    template <class G> __device__ __forceinline__ void step(Acc &A, size_t t, int q, const G &g) const
    {
        const BlkS<S> a = load_sliced(v, t, plane);
        const v2<S> x = g(q);
        A.y0 = fma(a.a00, x.x, fma(a.a01, x.y, A.y0));
        A.y1 = fma(a.a10, x.x, fma(a.a11, x.y, A.y1));
    }
};

// Sorted position of every row of a window: by block count, descending, ties
// by row (a stable, deterministic order).  One thread block per window.
__global__ void k_slice_order(int rows, const int *__restrict__ rp, int *__restrict__ order)
{
    __shared__ int len[kSliceWindow];
    const int w0 = blockIdx.x * kSliceWindow;
    const int n = min(kSliceWindow, rows - w0);
    for (int i = threadIdx.x; i < n; i += blockDim.x) len[i] = rp[w0 + i + 1] - rp[w0 + i];
    __syncthreads();
    for (int i = threadIdx.x; i < n; i += blockDim.x) {
        const int li = len[i];
        int rank = 0;
        for (int j = 0; j < n; j++) {
            const int lj = len[j];
            rank += (lj > li) || (lj == li && j < i);
        }
        order[w0 + rank] = w0 + i;
    }
}

// groups of slice sl: its longest row's block count over K, rounded up
__global__ void k_slice_groups(int nsl, int K, const int *__restrict__ rp, const int *__restrict__ order,
                               int *__restrict__ cnt)
{
    const int sl = blockIdx.x * blockDim.x + threadIdx.x;
    if (sl >= nsl) return;
    const int H = 32 / K;
    int mx = 0;
    for (int i = 0; i < H; i++) {
        const int r = order[sl * H + i];
        if (r >= 0) mx = max(mx, rp[r + 1] - rp[r]);
    }
    cnt[sl] = (mx + K - 1) / K;
}

__device__ __forceinline__ void store_sliced(double *v, size_t idx, size_t plane, const double *a, bool in)
{
    ((double2 *)v)[idx] = in ? make_double2(a[0], a[1]) : make_double2(0.0, 0.0);
    ((double2 *)v)[plane + idx] = in ? make_double2(a[2], a[3]) : make_double2(0.0, 0.0);
}
__device__ __forceinline__ void store_sliced(float *v, size_t idx, size_t, const double *a, bool in)
{
    ((float4 *)v)[idx] = in ? make_float4((float)a[0], (float)a[1], (float)a[2], (float)a[3])
                            : make_float4(0.0f, 0.0f, 0.0f, 0.0f);
}

// one thread per (slice, lane): the entries of its row it owns, group by group
template <class S>
__global__ void k_slice_fill(int nsl, int K, const int *__restrict__ rp, const int *__restrict__ ci,
                             const double *__restrict__ bv, const int *__restrict__ order,
                             const int *__restrict__ sptr, int *__restrict__ col, S *__restrict__ v, size_t plane)
{
    const long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    if (t >= (long long)nsl * 32) return;
    const int sl = (int)(t >> 5), lane = (int)(t & 31);
    const int r = order[sl * (32 / K) + lane / K], k = lane % K;
    const int b = r >= 0 ? rp[r] : 0, len = r >= 0 ? rp[r + 1] - b : 0;
    const int g0 = sptr[sl], g1 = sptr[sl + 1];
    for (int g = g0; g < g1; g++) {
        const int j = (g - g0) * K + k;
        const size_t idx = (size_t)g * 32 + lane;
        const bool in = j < len;
        col[idx] = in ? ci[b + j] : 0;
        store_sliced(v, idx, plane, bv + 4 * (size_t)(in ? b + j : 0), in);
    }
}

// the same for an operator in pair form
template <class S>
__global__ void k_slice_fill_pair(int nsl, int K, const int *__restrict__ rp, const int *__restrict__ ci,
                                  const v2<S> *__restrict__ pv, const S *__restrict__ alpha,
                                  const int *__restrict__ order, const int *__restrict__ sptr, int *__restrict__ col,
                                  v2<S> *__restrict__ v, S *__restrict__ al)
{
    const long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    if (t >= (long long)nsl * 32) return;
    const int sl = (int)(t >> 5), lane = (int)(t & 31);
    const int r = order[sl * (32 / K) + lane / K], k = lane % K;
    const int b = r >= 0 ? rp[r] : 0, len = r >= 0 ? rp[r + 1] - b : 0;
    const int g0 = sptr[sl], g1 = sptr[sl + 1];
    for (int g = g0; g < g1; g++) {
        const int j = (g - g0) * K + k;
        const size_t idx = (size_t)g * 32 + lane;
        const bool in = j < len;
        col[idx] = in ? ci[b + j] : 0;
        v[idx] = in ? pv[b + j] : V2<S>::mk((S)0, (S)0);
        al[idx] = in ? alpha[b + j] : (S)0;
    }
}

// first slice of every block: the lower bound of b * groups / blocks in sptr
__global__ void k_slice_blocks(int nsl, long long groups, int blocks, const int *__restrict__ sptr,
                               int *__restrict__ bsl)
{
    const int w = blockIdx.x * blockDim.x + threadIdx.x;
    if (w > blocks) return;
    if (w == blocks) {
        bsl[w] = nsl;
        return;
    }
    const long long g = groups * w / blocks;
    int lo = 0, hi = nsl;
    while (lo < hi) {
        const int m = (lo + hi) >> 1;
        if (sptr[m] < g) lo = m + 1;
        else hi = m;
    }
    bsl[w] = lo;
}

// ------------------------------------------------------------------ fused epilogues
// Vectors the FP64 finest-level stencil gathers are kept in the (v + u, u)
// form (SU): two operations per node pair instead of three.
template <class S, bool SU> __device__ __forceinline__ v2<S> to_su(S v, S u)
{
    return V2<S>::mk(SU ? v + u : v, u);
}

// pre-smoothing, degree 2 from zero, d0 = D^{-1} f / theta precomputed:
// x1 = d0, r1 = f - A d0, d1 = c1 d0 + c2 D^{-1} r1, u = x1 + d1
template <class S> struct EpiPre {
    const v2<S> *__restrict__ f;
    const v2<S> *__restrict__ invd;
    const v2<S> *__restrict__ d0;
    v2<S> *__restrict__ u;
    S c1, c2;
    __device__ __forceinline__ void operator()(int p, S y0, S y1) const {
        const v2<S> fp = f[p], id = invd[p], dp = d0[p];
        const S r0 = fp.x - y0, r1 = fp.y - y1;
        u[p] = V2<S>::mk(dp.x + (c1 * dp.x + c2 * id.x * r0), dp.y + (c1 * dp.y + c2 * id.y * r1));
    }
};

// restriction output f_c = R r together with d0_c = D_c^{-1} f_c / theta_c
template <class S> struct EpiStoreD0 {
    v2<S> *__restrict__ f;
    v2<S> *__restrict__ d0;
    const v2<S> *__restrict__ invd;
    S it;
    __device__ __forceinline__ void operator()(int p, S y0, S y1) const {
        f[p] = V2<S>::mk(y0, y1);
        const v2<S> id = invd[p];
        d0[p] = V2<S>::mk(y0 * id.x * it, y1 * id.y * it);
    }
};

template <class S> struct EpiResid {  // r = f - A u
    const v2<S> *__restrict__ f;
    v2<S> *__restrict__ r;
    __device__ __forceinline__ void operator()(int p, S y0, S y1) const {
        const v2<S> fp = f[p];
        r[p] = V2<S>::mk(fp.x - y0, fp.y - y1);
    }
};

template <class S> struct EpiAdd {  // u += P e_c
    v2<S> *__restrict__ u;
    __device__ __forceinline__ void operator()(int p, S y0, S y1) const {
        const v2<S> a = u[p];
        u[p] = V2<S>::mk(a.x + y0, a.y + y1);
    }
};

// the same for the finest P in pair form; u in (v + u, u) form in FP64
template <class S, bool SU> struct EpiAddPair {
    v2<S> *__restrict__ u;
    const v2<S> *__restrict__ kappa;
    __device__ __forceinline__ void operator()(int p, S y0, S y1) const {
        const v2<S> a = u[p], k = kappa[p];
        const S e1 = k.y * y1;
        u[p] = V2<S>::mk(SU ? a.x + fma(k.x, y0, e1) : a.x + k.x * y0, a.y + e1);
    }
};

// post-smoothing, first half: r0 = f - A u, d0 = D^{-1} r0 / theta, w = u + d0
template <class S> struct EpiPost1 {
    const v2<S> *__restrict__ f;
    const v2<S> *__restrict__ invd;
    const v2<S> *__restrict__ u;
    v2<S> *__restrict__ r;
    v2<S> *__restrict__ d;
    v2<S> *__restrict__ w;
    S it;
    __device__ __forceinline__ void operator()(int p, S y0, S y1) const {
        const v2<S> fp = f[p], id = invd[p], up = u[p];
        const S r0 = fp.x - y0, r1 = fp.y - y1;
        const S d0 = r0 * id.x * it, d1 = r1 * id.y * it;
        r[p] = V2<S>::mk(r0, r1);
        d[p] = V2<S>::mk(d0, d1);
        w[p] = V2<S>::mk(up.x + d0, up.y + d1);
    }
};

// post-smoothing, second half: r1 = r0 - A d0, d1 = c1 d0 + c2 D^{-1} r1, u = w + d1
// (OSU: u in (v + u, u) form, which the finest prolongation in pair form gathers)
template <class S, bool OSU = false> struct EpiPost2 {
    const v2<S> *__restrict__ r;
    const v2<S> *__restrict__ d;
    const v2<S> *__restrict__ invd;
    const v2<S> *__restrict__ w;
    v2<S> *__restrict__ u;
    S c1, c2;
    __device__ __forceinline__ void operator()(int p, S y0, S y1) const {
        const v2<S> rp_ = r[p], dp = d[p], id = invd[p], wp = w[p];
        const S r0 = rp_.x - y0, r1 = rp_.y - y1;
        u[p] = to_su<S, OSU>(wp.x + (c1 * dp.x + c2 * id.x * r0), wp.y + (c1 * dp.y + c2 * id.y * r1));
    }
};

// ------------------------------------------------------------------ per-level views
// Value and vector pointers of one level in precision S (index arrays are shared).
template <class S> struct LV {
    const S *Av, *Pv, *Rv;
    const v2<S> *invd;
    v2<S> *f, *u, *r, *d, *w;
};

template <class S> static LV<S> view(amg_hierarchy *h, int l);

template <class S> static const v2<S> *kappa_of(const Level &L);
template <> const double2 *kappa_of<double>(const Level &L) { return (const double2 *)L.kappa.p; }
template <> const float2 *kappa_of<float>(const Level &L) { return (const float2 *)L.kappa32.p; }

template <> LV<double> view<double>(amg_hierarchy *h, int l)
{
    Level &L = h->lev[l];
    LV<double> v;
    v.Av = L.A.v.p;
    v.Pv = L.P.v.p;
    v.Rv = L.R.v.p;
    v.invd = (const double2 *)L.invdiag.p;
    v.f = (double2 *)L.f.p;
    v.u = (double2 *)L.u.p;
    v.r = (double2 *)L.r.p;
    v.d = (double2 *)L.d.p;
    v.w = (double2 *)L.w.p;
    return v;
}
template <> LV<float> view<float>(amg_hierarchy *h, int l)
{
    Level &L = h->lev[l];
    LV<float> v;
    v.Av = L.A32.p;
    v.Pv = L.P32.p;
    v.Rv = L.R32.p;
    v.invd = (const float2 *)L.invdiag32.p;
    v.f = (float2 *)L.f32.p;
    v.u = (float2 *)L.u32.p;
    v.r = (float2 *)L.r32.p;
    v.d = (float2 *)L.d32.p;
    v.w = (float2 *)L.w32.p;
    return v;
}

template <class S> static const S *sliced_vals(const SlicedOp &o);
template <> const double *sliced_vals<double>(const SlicedOp &o) { return o.v.p; }
template <> const float *sliced_vals<float>(const SlicedOp &o) { return o.v32.p; }
template <class S> static const S *sliced_alpha(const SlicedOp &o);
template <> const double *sliced_alpha<double>(const SlicedOp &o) { return o.alpha.p; }
template <> const float *sliced_alpha<float>(const SlicedOp &o) { return o.alpha32.p; }

template <class M, class G, class E>
static int launch_sliced(const SlicedOp &o, int K, M mat, G g, E e, cudaStream_t s)
{
    if (o.K != K || !mat.v) return BD_ESTATE;
    switch (K) {
    case 1: k_bsell<1><<<o.blocks, kSlicedTPB, 0, s>>>(o.sptr.p, o.bsl.p, o.order.p, o.col.p, mat, g, e); break;
    case 2: k_bsell<2><<<o.blocks, kSlicedTPB, 0, s>>>(o.sptr.p, o.bsl.p, o.order.p, o.col.p, mat, g, e); break;
    case 4: k_bsell<4><<<o.blocks, kSlicedTPB, 0, s>>>(o.sptr.p, o.bsl.p, o.order.p, o.col.p, mat, g, e); break;
    default: k_bsell<8><<<o.blocks, kSlicedTPB, 0, s>>>(o.sptr.p, o.bsl.p, o.order.p, o.col.p, mat, g, e); break;
    }
    ::bd::note_launch();
    BD_LAUNCH_CHECK();
    return BD_OK;
}

static bool sliced_k_ok(int K) { return K == 1 || K == 2 || K == 4 || K == 8; }

// Build M's sliced form with K lanes per row in the V-cycle's precision (the
// sorted row order is kept across rebuilds of the same operator, and buffers
// large enough already are reused).  Stream-ordered on s.
template <class T> static int ensure(DBuf<T> &b, size_t n)
{
    return b.p && b.n >= n ? BD_OK : b.alloc(n);
}

static int build_sliced(const BSR &M, const PairOp *pr, int K, bool fp32, SlicedOp &o, cudaStream_t s)
{
    if (M.nbr <= 0 || M.nb <= 0 || !sliced_k_ok(K)) return BD_EINVAL;
    const int rows = M.nbr, H = 32 / K;
    o.K = 0;
    if (o.rows != rows || !o.order.p) {
        const size_t padded = ((size_t)rows + 31) / 32 * 32;
        BD_TRY(o.order.alloc(padded));
        BD_CUDA(cudaMemsetAsync(o.order.p, 0xff, sizeof(int) * padded, s));  // -1 past the last row
        k_slice_order<<<(rows + kSliceWindow - 1) / kSliceWindow, 256, 0, s>>>(rows, M.rp.p, o.order.p);
        ::bd::note_launch();
        BD_LAUNCH_CHECK();
        o.rows = rows;
    }
    o.nsl = (rows + H - 1) / H;
    BD_TRY(ensure(o.cnt, (size_t)o.nsl));
    BD_TRY(ensure(o.sptr, (size_t)o.nsl + 1));
    k_slice_groups<<<(o.nsl + 255) / 256, 256, 0, s>>>(o.nsl, K, M.rp.p, o.order.p, o.cnt.p);
    ::bd::note_launch();
    BD_LAUNCH_CHECK();
    BD_TRY(exclusive_scan(o.cnt.p, o.sptr.p, o.nsl, &o.groups, s));
    const size_t ent = (size_t)o.groups * 32;
    BD_TRY(ensure(o.col, ent));
    const long long fill_threads = (long long)o.nsl * 32;
    const int fill_grid = (int)((fill_threads + 255) / 256);
    if (fp32) o.v.release();
    else o.v32.release();
    if (pr) {
        if (fp32) {
            BD_TRY(ensure(o.v32, 2 * ent));
            BD_TRY(ensure(o.alpha32, ent));
            k_slice_fill_pair<float><<<fill_grid, 256, 0, s>>>(o.nsl, K, M.rp.p, pr->ci.p, (const float2 *)pr->v32.p,
                                                               pr->alpha32.p, o.order.p, o.sptr.p, o.col.p,
                                                               (float2 *)o.v32.p, o.alpha32.p);
        } else {
            BD_TRY(ensure(o.v, 2 * ent));
            BD_TRY(ensure(o.alpha, ent));
            k_slice_fill_pair<double><<<fill_grid, 256, 0, s>>>(o.nsl, K, M.rp.p, pr->ci.p, (const double2 *)pr->v.p,
                                                                pr->alpha.p, o.order.p, o.sptr.p, o.col.p,
                                                                (double2 *)o.v.p, o.alpha.p);
        }
    } else if (fp32) {
        BD_TRY(ensure(o.v32, 4 * ent));
        k_slice_fill<float><<<fill_grid, 256, 0, s>>>(o.nsl, K, M.rp.p, M.ci.p, M.v.p, o.order.p, o.sptr.p,
                                                     o.col.p, o.v32.p, ent);
    } else {
        BD_TRY(ensure(o.v, 4 * ent));
        k_slice_fill<double><<<fill_grid, 256, 0, s>>>(o.nsl, K, M.rp.p, M.ci.p, M.v.p, o.order.p, o.sptr.p,
                                                      o.col.p, o.v.p, ent);
    }
    ::bd::note_launch();
    BD_LAUNCH_CHECK();
    // one resident wave, a slice per warp at least
    const long long cap = (long long)kSM * (fp32 ? SlicedMinB<float>::v : SlicedMinB<double>::v);
    o.blocks = (int)std::min<long long>(cap, ((long long)o.nsl + kSlicedTPB / 32 - 1) / (kSlicedTPB / 32));
    BD_TRY(ensure(o.bsl, (size_t)o.blocks + 1));
    k_slice_blocks<<<o.blocks / 256 + 1, 256, 0, s>>>(o.nsl, o.groups, o.blocks, o.sptr.p, o.bsl.p);
    ::bd::note_launch();
    BD_LAUNCH_CHECK();
    o.K = K;
    return BD_OK;
}

static void drop_sliced(SlicedOp &o)
{
    o.K = 0;
    o.cnt.release();
    o.col.release();
    o.v.release();
    o.v32.release();
    o.alpha.release();
    o.alpha32.release();
    o.sptr.release();
    o.bsl.release();
}

static const BSR &op_of(const Level &L, int op) { return op == 0 ? L.A : (op == 1 ? L.R : L.P); }
static const PairOp *pair_of(const Level &L, int op)
{
    return op > 0 && L.pair[op - 1].valid ? &L.pair[op - 1] : nullptr;
}
// sliced form of operator op with K lanes per row
static int build_op(Level &L, int op, int K, bool fp32, cudaStream_t s)
{
    return build_sliced(op_of(L, op), pair_of(L, op), K, fp32, L.sl[op], s);
}

// Operator op (0: A, 1: R, 2: P) of level L in the form its lanes entry names.
template <class S, class G, class E>
static int apply_op(const Level &L, int op, const S *csr_vals, G g, E e, cudaStream_t s)
{
    const int T = L.lanes[op];
    const SlicedOp &o = L.sl[op];
    if (T < 0) return launch_sliced(o, -T, MatSliced<S>{sliced_vals<S>(o), (size_t)o.groups * 32}, g, e, s);
    return launch_bsr<S>(op_of(L, op), csr_vals, T, g, e, s);
}

// The finest R or P in pair form; the caller applies kappa.
template <class S, class G, class E>
static int apply_pair(const Level &L, int op, G g, E e, cudaStream_t s)
{
    const int T = L.lanes[op];
    const SlicedOp &o = L.sl[op];
    if (T < 0) return launch_sliced(o, -T, MatPair<S>{(const v2<S> *)sliced_vals<S>(o), sliced_alpha<S>(o)}, g, e, s);
    const BSR &M = op_of(L, op);
    return launch_bsr_rows(M.nbr, M.rp.p, pair_of(L, op)->ci.p, mat_pair<S>(*pair_of(L, op)), T, g, e, s);
}

// Pair form of P (rows: fine nodes, own entry: the node's aggregate) or of its
// transpose R (rows: aggregates, own entries: the members).  L lanes per row: own
// entries keep their order at the front, the others theirs behind.
template <int L, bool IS_R>
__global__ void k_pair_fill(int rows, const int *__restrict__ rp, const int *__restrict__ ci,
                            const double *__restrict__ bv, const int *__restrict__ agg,
                            const double *__restrict__ kappa, int *__restrict__ oci, double2 *__restrict__ ov,
                            double *__restrict__ oal, float2 *__restrict__ ov32, float *__restrict__ oal32)
{
    const int lane = threadIdx.x & 31, l = lane & (L - 1);
    const unsigned group = (L == 32 ? 0xffffffffu : ((1u << (L & 31)) - 1u) << (lane & ~(L - 1)));
    const unsigned before = group & ((1u << lane) - 1u);
    const int row = (int)(grid_index(blockIdx.x, blockDim.x, threadIdx.x) / L);
    const bool act = row < rows;
    const int b = act ? rp[row] : 0, e = act ? rp[row + 1] : 0;
    int len = e - b, nown = 0;
    for (int o = 16; o; o >>= 1) len = max(len, __shfl_xor_sync(0xffffffffu, len, o));  // of the warp's rows
    for (int i = l; i < ((len + L - 1) / L) * L; i += L) {
        const int t = b + i;
        const bool own = t < e && (IS_R ? agg[ci[t]] == row : ci[t] == agg[row]);
        nown += __popc(__ballot_sync(0xffffffffu, own) & group);
    }
    int po = b, pn = b + nown;  // next own and next other position
    for (int i = l; i < ((len + L - 1) / L) * L; i += L) {
        const int t = b + i;
        const bool in = t < e;
        const int q = in ? ci[t] : 0;
        const bool own = in && (IS_R ? agg[q] == row : q == agg[row]);
        const unsigned mo = __ballot_sync(0xffffffffu, own), mn = __ballot_sync(0xffffffffu, in && !own);
        if (in) {
            const int pos = own ? po + __popc(mo & before) : pn + __popc(mn & before);
            const int node = IS_R ? q : row;
            const double kv = kappa[2 * node], ku = kappa[2 * node + 1];
            const double *a = bv + 4 * (size_t)t;
            // P's block [a00 a01; a10 a11]; R holds its transpose
            const double a01 = IS_R ? a[2] : a[1];
            const double ki = a01 / kv, ke = a[3] / ku - ki, al = own ? (a[0] - a01) / kv : 0.0;
            oci[pos] = own ? (q | ~kColMask) : q;
            if (ov) {
                ov[pos] = make_double2(ki, ke);
                oal[pos] = al;
            } else {
                ov32[pos] = make_float2((float)ki, (float)ke);
                oal32[pos] = (float)al;
            }
        }
        po += __popc(mo & group);
        pn += __popc(mn & group);
    }
}

__global__ void k_kappa(long long n, const double *__restrict__ invd, double omega, double *__restrict__ k64,
                        float *__restrict__ k32)
{
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n;
         i += (long long)gridDim.x * blockDim.x) {
        const double k = -omega * invd[i];
        k64[i] = k;
        if (k32) k32[i] = (float)k;
    }
}

static int build_pairs(Level &L, bool fp32, cudaStream_t s)
{
    const long long n = 2LL * L.N;
    BD_TRY(L.kappa.alloc((size_t)n));
    if (fp32) BD_TRY(L.kappa32.alloc((size_t)n));
    k_kappa<<<grid_for(n, 256), 256, 0, s>>>(n, L.invdiag.p, fine_omega(L), L.kappa.p, L.kappa32.p);
    ::bd::note_launch();
    for (int op = 1; op <= 2; op++) {
        const BSR &M = op_of(L, op);
        PairOp &o = L.pair[op - 1];
        BD_TRY(o.ci.alloc((size_t)M.nb));
        if (fp32) {
            BD_TRY(o.v32.alloc(2 * (size_t)M.nb));
            BD_TRY(o.alpha32.alloc((size_t)M.nb));
        } else {
            BD_TRY(o.v.alloc(2 * (size_t)M.nb));
            BD_TRY(o.alpha.alloc((size_t)M.nb));
        }
        if (op == 1)
            k_pair_fill<32, true><<<(int)((32LL * M.nbr + 255) / 256), 256, 0, s>>>(
                M.nbr, M.rp.p, M.ci.p, M.v.p, L.agg.p, L.kappa.p, o.ci.p, (double2 *)o.v.p, o.alpha.p,
                (float2 *)o.v32.p, o.alpha32.p);
        else
            k_pair_fill<8, false><<<(int)((8LL * M.nbr + 255) / 256), 256, 0, s>>>(
                M.nbr, M.rp.p, M.ci.p, M.v.p, L.agg.p, L.kappa.p, o.ci.p, (double2 *)o.v.p, o.alpha.p,
                (float2 *)o.v32.p, o.alpha32.p);
        ::bd::note_launch();
        o.valid = true;
    }
    BD_LAUNCH_CHECK();
    return BD_OK;
}

// The sliced form (FP64 only: in FP32 block-CSR with more lanes was as fast
// or faster on every level) where it beat block-CSR inside the V-cycle (us per
// V-cycle, forms.time_forms): many short, ragged rows (the prolongators of levels
// of 65536 rows and more: sorted rows leave few idle lanes, one lane per row needs
// no reduction), rows of 64 to 400 blocks on 24576 rows and more (8 lanes; the
// 128x128x32 slab's second level, 32001 rows: 145 -> 137, on the 13197 rows of
// 96x96x24 block-CSR wins, 78 against 93) and, on levels of 65536 rows and more,
// rows in between and long ones (4 lanes; 256x256x64, 249682 rows: 840 -> 743).
// Restrictions from 96 blocks a row from 8192 rows on.  Longer rows still and
// everything else: the block-CSR rule.  Between those slabs (80x80x20, 112x112x28,
// 144x144x36, 160x160x40, 192x192x48, 224x224x56, A1's 7885 to 171480 rows) the rule's
// A1 is the fastest form to within 1 %, but for 6 % at 7885 rows (8 lanes) and 8 % at
// 63151 (sliced 4); R0 and P0 to within 4 % but for R0 at 63151 rows (8 lanes 60.3,
// 4 lanes 66.7) and P0 at 137781 (1 lane 15.0, sliced 17.7); R1 of 9114 and 14710 rows
// takes 41.8 and 57.7 sliced where 16 and 8 lanes take 31.2 and 46.3.
//
// The finest R and P in pair form have their own crossovers.  R: few lanes
// where rows fill the GPU (T rows >= 200 K), else up to 16 (31542 rows: 8 lanes
// 35.8, sliced 8 38.9; 13197 rows: 16 lanes 23.2, 8 24.8; 249682 rows: 4 lanes
// 199, 8 211).  P: one lane per row on a million rows and more (256x256x64: FP64
// sliced 254, one lane 240; FP32 two lanes 127, one 107); the rule above below.
constexpr int kSlicedMinRows = 8192;
static int lanes_rule(const BSR &A, bool fp32, bool sliced_ok, const PairOp *pr = nullptr)
{
    const double avg = A.nbr > 0 ? (double)A.nb / A.nbr : 1.0;
    if (avg >= kLongRow) return lanes_for(A, fp32);
    if (pr && !fp32 && avg >= 48.0 && A.nbr >= 4096) {
        int T = 4;
        while (T < 16 && (long long)A.nbr * T < 200000) T <<= 1;
        return T;
    }
    if (pr && avg < 48.0 && A.nbr >= 1 << 20) return 1;
    if (sliced_ok && !fp32 && A.nbr >= kSlicedMinRows) {
        if (A.nbr >= 65536 && avg <= 24.0) return -1;
        if (avg < 400.0 && (A.nbr == A.nbc ? avg >= 64.0 && A.nbr >= 24576 && A.nbr < 65536 : avg >= 96.0)) return -8;
        if (A.nbr >= 65536) return -4;  // middle-length rows of a big level
    }
    return lanes_for(A, fp32);
}

// ------------------------------------------------------------------ finest level, layered stencil
int fine_raw_copy(FineStencil &F, const bd_system *sys, cudaStream_t s)
{
    F.NX = sys->mesh.nx + 1;
    F.NY = sys->mesh.ny + 1;
    F.NZ = sys->mesh.nz + 1;
    F.sym = sys->sym;
    BD_TRY(F.raw.alloc((size_t)9 * F.NZ * kFineRaw));
    BD_CUDA(cudaMemcpyAsync(F.raw.p, sys->raw.p, F.raw.bytes(), cudaMemcpyDeviceToDevice, s));
    return BD_OK;
}

int build_fine_stencil(amg_hierarchy *h, const bd_system *sys, cudaStream_t s)
{
    BD_TRY(fine_raw_copy(h->fine, sys, s));
    h->fine.valid = true;
    return BD_OK;
}

// Packed row from a raw one; a pair's coefficient is taken from its member
// that exists on this row type.
template <bool SYM>
__global__ void k_fine_pack(int rows, const double *__restrict__ raw, double c2, double it, double omega,
                            double *__restrict__ tab, float *__restrict__ tab32)
{
    using Row = FineRow<SYM>;
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= rows) return;
    const double *o = raw + (size_t)t * kFineRaw;
    const int ti = t % 3, tj = (t % 9) / 3;
    auto put = [&](int k, double x, double y) {
        const size_t e = (size_t)t * Row::LEN + k;
        if (tab) ((double2 *)tab)[e] = make_double2(x, y);
        if (tab32) ((float2 *)tab32)[e] = make_float2((float)x, (float)y);
    };
    for (int z = 0; z < (SYM ? 2 : 3); z++) {
        const int b = 9 * (z == 0 ? 1 : (z == 1 ? 2 : 0));  // dz = 0, +1, -1
        for (int k = 0; k < Row::NP; k++) {
            const int q = SYM ? fine_pair_pos(k, ti, tj) : k;
            put(z * Row::G + k, o[2 * (b + q)], o[2 * (b + q) + 1]);
        }
        put(z * Row::G + Row::NP, z == 0 ? o[54] : 0.0, 0.0);
    }
    // the inverse diagonal, as k_invdiag forms it from the assembled blocks
    const bool exists = o[55] > 0.0;
    const double dv = exists ? 1.0 / (o[54] + o[26]) : 0.0, du = exists ? 1.0 / (o[26] + o[27]) : 0.0;
    put(Row::IDC2, c2 * dv, c2 * du);
    put(Row::IDT, dv * it, du * it);
    put(Row::KAPPA, -omega * dv, -omega * du);
    put(Row::KAPPA + 1, 0.0, 0.0);
}

int fine_pack(const FineStencil &F, bool sym, double c2, double inv_theta, double omega, double *tab, float *tab32,
              cudaStream_t s)
{
    const int rows = 9 * F.NZ, grid = (rows + 63) / 64;
    if (sym) k_fine_pack<true><<<grid, 64, 0, s>>>(rows, F.raw.p, c2, inv_theta, omega, tab, tab32);
    else k_fine_pack<false><<<grid, 64, 0, s>>>(rows, F.raw.p, c2, inv_theta, omega, tab, tab32);
    ::bd::note_launch();
    BD_LAUNCH_CHECK();
    return BD_OK;
}

// One finest-level launch: make(SYM) gives the epilogue for the table's form.
template <class S, bool SU, class F>
static int fine_apply(const amg_hierarchy *h, const v2<S> *x, F make, cudaStream_t s)
{
    const FineGrid g = fine_grid<S>(h->fine, h->lev[0].ch_c1);
    const long long units = (long long)g.ncb * g.NZ;
    if (h->fine.sym)
        k_fine<S, true, SU><<<fine_blocks<S, true>(units), kFineTPB, 0, s>>>(g, x, make(std::true_type{}));
    else
        k_fine<S, false, SU><<<fine_blocks<S, false>(units), kFineTPB, 0, s>>>(g, x, make(std::false_type{}));
    ::bd::note_launch();
    BD_LAUNCH_CHECK();
    return BD_OK;
}

// ------------------------------------------------------------------ live kernel timing
int prof_begin(amg_hierarchy *h, cudaStream_t s, int label, bool fine)
{
    if (!h->prof || (!fine && h->prof < 2)) return -1;
    if (h->ev_used * 2 + 2 > (int)h->ev.size()) {
        if (h->ev.size() >= 8192) prof_collect(h);  // bounded pool: drain (synchronises)
        while (h->ev_used * 2 + 2 > (int)h->ev.size()) {
            cudaEvent_t e;
            if (cudaEventCreate(&e) != cudaSuccess) return -1;
            h->ev.push_back(e);
            if (h->ev.size() % 2 == 0) {
                h->ev_bytes.push_back(0.0);
                h->ev_flops.push_back(0.0);
                h->ev_ops.push_back(0.0);
                h->ev_label.push_back(-1);
            }
        }
    }
    int slot = h->ev_used++;
    h->ev_bytes[slot] = 0.0;
    h->ev_flops[slot] = 0.0;
    h->ev_ops[slot] = 0.0;
    h->ev_label[slot] = label;
    cudaEventRecord(h->ev[2 * slot], s);
    return slot;
}

// bytes/flops > 0 mark a finest-operator application (amg_kernel_profile sums)
void prof_end(amg_hierarchy *h, int slot, double bytes, double flops, cudaStream_t s, double ops)
{
    if (slot < 0) return;
    cudaEventRecord(h->ev[2 * slot + 1], s);
    h->ev_bytes[slot] = bytes;
    h->ev_flops[slot] = flops;
    h->ev_ops[slot] = ops;
}

void prof_collect(amg_hierarchy *h)
{
    for (int i = 0; i < h->ev_used; i++) {
        cudaEventSynchronize(h->ev[2 * i + 1]);
        float ms = 0.0f;
        if (cudaEventElapsedTime(&ms, h->ev[2 * i], h->ev[2 * i + 1]) != cudaSuccess) continue;
        if (h->ev_bytes[i] > 0.0) {
            h->prof_sum.launches++;
            h->prof_sum.total_ms += ms;
            h->prof_sum.bytes += h->ev_bytes[i];
            h->prof_sum.flops += h->ev_flops[i];
            h->prof_sum.fp64_ops += h->ev_ops[i];
        }
        const int lab = h->ev_label[i];
        if (h->prof >= 2 && lab >= 0 && lab < 256) {
            h->trace_ms[lab] += ms;
            h->trace_n[lab]++;
        }
    }
    h->ev_used = 0;
}

// Algorithmic bytes of one finest-level operator application in precision S:
// the operator once (the stencil's table; block CSR: four values and a column
// per block, row offsets) and `vec` per-node vector streams of two S each.
template <class S>
static double fine_bytes(const amg_hierarchy *h, const Level &L, int vec)
{
    const double sz = (double)sizeof(S);
    double mat = h->fine.valid ? 2 * sz * fine_row_len(h->fine.sym) * 9.0 * h->fine.NZ
                               : (4 * sz + 4.0) * (double)L.A.nb + 4.0 * (L.N + 1);
    return mat + 2 * sz * vec * (double)L.N;
}
// FP64 pipe operations per node of the stencil (a fused multiply-add, an add
// and a multiply count one each): two operators of 4 adds and 15 FMA in the
// symmetric form, 27 FMA in the general one, and the row tail (c M v + a, a + b
// and v = (v + u) - u).
static double fine_node_ops(const amg_hierarchy *h) { return (h->fine.sym ? 38.0 : 54.0) + 3.0; }
// Flops one finest-level launch executes (an FMA counts 2); the epilogue's few
// per node are not counted.
static double fine_flops(const amg_hierarchy *h, const Level &L)
{
    if (h->fine.valid) return (h->fine.sym ? 68.0 : 108.0) * L.N;
    return 8.0 * (double)L.A.nb;
}
// FP64 pipe operations of one finest-level launch of the FP64 V-cycle or of the
// PCG's A p: the stencil's per node and the fused step as its epilogue issues
// it: pre-smoother 7, residual 2, first post-smoothing half 4, second half 11
// (16 with the PCG's z statistics), A p with p.Ap 2.  The FP32 V-cycle's
// launches issue none.  Block-CSR finest levels: 4 FMA per 2x2 block,
// epilogues not counted.
enum FineRole { FR_PRE, FR_RESID, FR_POST1, FR_POST2, FR_POST2Z, FR_AP };
template <class S>
static double fine_ops(const amg_hierarchy *h, const Level &L, int role)
{
    if (!h->fine.valid) return sizeof(S) == 8 || role == FR_AP ? 4.0 * (double)L.A.nb : 0.0;
    if (sizeof(S) == 4 && role != FR_AP) return 0.0;
    static const double epi[] = {7.0, 2.0, 4.0, 11.0, 16.0, 2.0};
    return (fine_node_ops(h) + epi[role]) * (double)L.N;
}

// ------------------------------------------------------------------ coarsest level
// x = C r in FP64 whatever the storage precision, C the inverse of the
// rank-one-fixed coarsest operator with the projection orthogonal to its null
// vector folded in (k_coarse_project): one dense mat-vec, a warp per row, the rows
// spread evenly over the SMs.  Larger FP32 right-hand sides are widened once per
// block in shared memory (a conversion costs the FP64 pipe what a multiply-add
// does).  The separate projection made every block reduce z.r first: 62
// unknowns 12.1 us in one block, 1942 unknowns 21.5 us; event-timed inside the
// solve 14.8 -> 6.3 and 22.1 -> 16.1 (FP32 24.3 -> 18.1), bound by the latency of
// streaming 30 MB with 13 warps per SM (two blocks' worth of loads in flight need
// the 64 registers the launch bound leaves).
template <class S, bool STAGE>
__global__ void __launch_bounds__(1024, 1) k_coarse_solve(int n, const double *__restrict__ C, const S *__restrict__ r,
                                                       S *__restrict__ x)
{
    extern __shared__ double2 rs[];
    if constexpr (STAGE) {
        for (int j = threadIdx.x; j < n / 2; j += blockDim.x) {
            const v2<S> v = ((const v2<S> *)r)[j];
            rs[j] = make_double2(widen(v.x), widen(v.y));
        }
        __syncthreads();
    }
    const int lane = threadIdx.x & 31, i = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    if (i >= n) return;
    const double *row = C + (size_t)i * n;
    double s0 = 0.0, s1 = 0.0;
    if (n & 1) {
        for (int j = lane; j < n; j += 32) s0 = fma(row[j], widen(r[j]), s0);
    } else {  // even rows start on 16 bytes
#pragma unroll 8
        for (int j = lane; j < n / 2; j += 32) {
            const double2 c = ((const double2 *)row)[j];
            double2 v;
            if constexpr (STAGE) {
                v = rs[j];
            } else {
                const v2<S> t = ((const v2<S> *)r)[j];
                v = make_double2(widen(t.x), widen(t.y));
            }
            s0 = fma(c.x, v.x, s0);
            s1 = fma(c.y, v.y, s1);
        }
    }
    s0 += s1;
    for (int o = 16; o; o >>= 1) s0 += __shfl_xor_sync(0xffffffffu, s0, o);
    if (lane == 0) x[i] = (S)s0;
}

template <class S> static int launch_coarse(int n, const double *C, const S *r, S *x, cudaStream_t s)
{
    const int w = std::min(32, (n + kSM - 1) / kSM), grid = (n + w - 1) / w;  // rows (warps) per block
    if (sizeof(S) == 4 && w > 2 && !(n & 1))
        k_coarse_solve<S, true><<<grid, 32 * w, sizeof(double) * (size_t)n, s>>>(n, C, r, x);
    else
        k_coarse_solve<S, false><<<grid, 32 * w, 0, s>>>(n, C, r, x);
    ::bd::note_launch();
    BD_LAUNCH_CHECK();
    return BD_OK;
}
int coarse_solve(int n, const double *C, const double *r, double *x, cudaStream_t s) { return launch_coarse(n, C, r, x, s); }
int coarse_solve(int n, const double *C, const float *r, float *x, cudaStream_t s) { return launch_coarse(n, C, r, x, s); }

template <class S>
__global__ void k_copy2(int N, const v2<S> *__restrict__ a, v2<S> *__restrict__ b)
{
    for (int i = share_lo(N) + threadIdx.x, e = share_hi(N); i < e; i += blockDim.x) b[i] = a[i];
}

template <class S, bool SU = false>
__global__ void k_scale_d0(int N, const v2<S> *__restrict__ f, const v2<S> *__restrict__ invd, S it,
                           v2<S> *__restrict__ d0)
{
    for (int i = share_lo(N) + threadIdx.x, e = share_hi(N); i < e; i += blockDim.x) {
        const v2<S> a = f[i], b = invd[i];
        d0[i] = to_su<S, SU>(a.x * b.x * it, a.y * b.y * it);
    }
}

// FP64 residual in, FP32 right-hand side and d0 of the finest level out
__global__ void k_in32(int N, const double2 *__restrict__ r, const float2 *__restrict__ invd, float it,
                       float2 *__restrict__ f, float2 *__restrict__ d0)
{
    for (int i = share_lo(N) + threadIdx.x, e = share_hi(N); i < e; i += blockDim.x) {
        const double2 a = r[i];
        const float2 b = invd[i];
        const float f0 = narrow(a.x), f1 = narrow(a.y);
        f[i] = make_float2(f0, f1);
        d0[i] = make_float2(f0 * b.x * it, f1 * b.y * it);
    }
}

__global__ void k_out64(int N, const float2 *__restrict__ u, double2 *__restrict__ z)
{
    for (int i = share_lo(N) + threadIdx.x, e = share_hi(N); i < e; i += blockDim.x) {
        const float2 a = u[i];
        z[i] = make_double2(widen(a.x), widen(a.y));
    }
}

__global__ void k_to_f32(long long n, const double *__restrict__ a, float *__restrict__ b)
{
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n;
         i += (long long)gridDim.x * blockDim.x)
        b[i] = (float)a[i];
}

// The PCG's z statistics computed by the V-cycle's last finest-level kernel
// (defined with the PCG reductions below).
struct ZOut;
static int launch_fine_z(amg_hierarchy *h, const LV<double> &lv, const double2 *u, const ZOut &zo, cudaStream_t s);
// the z statistics of the FP32 V-cycle's output
static int launch_z_from32(amg_hierarchy *h, const float2 *u, const ZOut &zo, cudaStream_t s);

// One V-cycle in precision S; f0/u0 are the finest level's right-hand side and
// output (d0 of the finest level must already be in lev[0]'s d vector).  On a
// stencil finest level in FP64 its gathered vectors (d0, the iterate u until the
// last smoothing step, the post-smoother's d) are kept in (v + u, u) form; the
// output u0 is in (v, u) form either way.  zo (PCG only): the last
// post-smoothing step on a stencil finest level writes the FP64 result to
// zo->z and sums the z statistics (*zdone set); u0 then holds the iterate
// before that step.
template <class S>
static int vcycle_impl(amg_hierarchy *h, const v2<S> *f0, v2<S> *u0, cudaStream_t s, const ZOut *zo = nullptr,
                       bool *zdone = nullptr)
{
    constexpr bool SU = std::is_same<S, double>::value;
    const int nl = h->nlev;
    const bool deg2 = h->opts.cheb_degree == 2;
    // level whose smoothed correction the finest P in pair form gathers: kept in
    // (v + u, u) form in FP64 (an addition per coarse node instead of per entry)
    auto OSU = [&](int l) { return SU && l == 1 && h->fine.valid && deg2 && nl > 2; };
    auto down = [&](int l) -> int {
        Level &L = h->lev[l];
        const LV<S> lv = view<S>(h, l);
        const bool fine = l == 0 && h->fine.valid;
        const v2<S> *f = l == 0 ? f0 : lv.f;
        v2<S> *u = l == 0 ? u0 : lv.u;
        v2<S> *d0 = lv.d;
        if (deg2) {
            int sl = prof_begin(h, s, 16 * l + R_PRE, l == 0);
            if (fine)
                BD_TRY((fine_apply<S, SU>(h, d0, [&](auto sym) { return FinePre<S, sym.value, SU>{f, u}; }, s)));
            else
                BD_TRY(apply_op<S>(L, 0, lv.Av, GatherVec<S>{d0},
                                   EpiPre<S>{f, lv.invd, d0, u, (S)L.ch_c1, (S)L.ch_c2}, s));
            prof_end(h, sl, l == 0 ? fine_bytes<S>(h, L, fine ? 3 : 4) : 0.0, fine_flops(h, L), s,
                     fine_ops<S>(h, L, FR_PRE));
        } else {
            int sl = prof_begin(h, s, 16 * l + R_PRE, false);
            k_copy2<S><<<grid_for(L.N, 256), 256, 0, s>>>(L.N, d0, u); ::bd::note_launch();
            BD_LAUNCH_CHECK();
            prof_end(h, sl, 0.0, 0.0, s);
        }
        int sr = prof_begin(h, s, 16 * l + R_RESID, l == 0);
        if (fine)
            BD_TRY((fine_apply<S, SU>(h, u, [&](auto sym) { return FineResid<S, sym.value, SU>{f, lv.r}; }, s)));
        else
            BD_TRY(apply_op<S>(L, 0, lv.Av, GatherVec<S>{u}, EpiResid<S>{f, lv.r}, s));
        prof_end(h, sr, l == 0 ? fine_bytes<S>(h, L, 3) : 0.0, fine_flops(h, L), s, fine_ops<S>(h, L, FR_RESID));
        const Level &C = h->lev[l + 1];
        const LV<S> cv = view<S>(h, l + 1);
        int sx = prof_begin(h, s, 16 * l + R_RESTRICT, false);
        const EpiStoreD0<S> rest{cv.f, cv.d, cv.invd, (S)C.ch_inv_theta};
        if (fine) BD_TRY((apply_pair<S>(L, 1, GatherVec<S, SU>{lv.r}, rest, s)));
        else BD_TRY(apply_op<S>(L, 1, lv.Rv, GatherVec<S>{lv.r}, rest, s));
        prof_end(h, sx, 0.0, 0.0, s);
        return BD_OK;
    };
    auto up = [&](int l) -> int {
        Level &L = h->lev[l];
        const LV<S> lv = view<S>(h, l);
        const bool fine = l == 0 && h->fine.valid;
        const v2<S> *f = l == 0 ? f0 : lv.f;
        v2<S> *u = l == 0 ? u0 : lv.u;
        const LV<S> cv = view<S>(h, l + 1);
        int sp = prof_begin(h, s, 16 * l + R_PROLONG, false);
        if (fine) {
            const EpiAddPair<S, SU> add{u, kappa_of<S>(L)};
            if (OSU(1)) BD_TRY((apply_pair<S>(L, 2, GatherVec<S, SU>{cv.u}, add, s)));
            else BD_TRY((apply_pair<S>(L, 2, GatherVec<S>{cv.u}, add, s)));
        } else BD_TRY(apply_op<S>(L, 2, lv.Pv, GatherVec<S>{cv.u}, EpiAdd<S>{u}, s));
        prof_end(h, sp, 0.0, 0.0, s);
        int s1 = prof_begin(h, s, 16 * l + R_POST1, l == 0);
        if (fine)
            BD_TRY((fine_apply<S, SU>(h, u, [&](auto sym) {
                return FinePost1<S, sym.value, SU>{f, lv.r, lv.d, deg2 ? nullptr : lv.w};
            }, s)));
        else
            BD_TRY(apply_op<S>(L, 0, lv.Av, GatherVec<S>{u},
                               EpiPost1<S>{f, lv.invd, u, lv.r, lv.d, lv.w, (S)L.ch_inv_theta}, s));
        prof_end(h, s1, l == 0 ? fine_bytes<S>(h, L, fine ? 4 : 6) : 0.0, fine_flops(h, L), s,
                 fine_ops<S>(h, L, FR_POST1));
        if (deg2) {
            int s2 = prof_begin(h, s, 16 * l + R_POST2, l == 0);
            double bytes = l == 0 ? fine_bytes<S>(h, L, fine ? 4 : 5) : 0.0;
            // FP64: the post-smoother's last kernel carries the PCG's z statistics
            // (FP32: a pass of their own over u, vcycle_run)
            const bool fuse_z = fine && zo && sizeof(S) == 8;
            if (fuse_z) {
                if constexpr (SU) BD_TRY(launch_fine_z(h, lv, u, *zo, s));
                if (zdone) *zdone = true;
                bytes += 16.0 * L.N;  // u is not stored; z is, and the PCG's r is read
            } else if (fine) {
                BD_TRY((fine_apply<S, SU>(h, lv.d, [&](auto sym) {
                    return FinePost2<S, sym.value, SU>{lv.r, u, u};
                }, s)));
            } else if (OSU(l)) {
                BD_TRY(apply_op<S>(L, 0, lv.Av, GatherVec<S>{lv.d},
                                   EpiPost2<S, true>{lv.r, lv.d, lv.invd, lv.w, u, (S)L.ch_c1, (S)L.ch_c2}, s));
            } else {
                BD_TRY(apply_op<S>(L, 0, lv.Av, GatherVec<S>{lv.d},
                                   EpiPost2<S>{lv.r, lv.d, lv.invd, lv.w, u, (S)L.ch_c1, (S)L.ch_c2}, s));
            }
            prof_end(h, s2, bytes, fine_flops(h, L), s, fine_ops<S>(h, L, fuse_z ? FR_POST2Z : FR_POST2));
        } else {
            int s2 = prof_begin(h, s, 16 * l + R_POST2, false);
            k_copy2<S><<<grid_for(L.N, 256), 256, 0, s>>>(L.N, lv.w, u); ::bd::note_launch();
            BD_LAUNCH_CHECK();
            prof_end(h, s2, 0.0, 0.0, s);
        }
        return BD_OK;
    };
    for (int l = 0; l < nl - 1; l++) BD_TRY(down(l));
    {
        const LV<S> cv = view<S>(h, nl - 1);
        const S *f = (const S *)(nl == 1 ? f0 : cv.f);
        S *u = (S *)(nl == 1 ? u0 : cv.u);
        int sc = prof_begin(h, s, R_COARSE, false);
        BD_TRY(coarse_solve(h->nc, h->cinv.p, f, u, s));
        prof_end(h, sc, 0.0, 0.0, s);
    }
    for (int l = nl - 2; l >= 0; l--) BD_TRY(up(l));
    return BD_OK;
}

// z = B r with FP64 vectors at the boundary, in the hierarchy's precision.
// d0_ready: the producer of r already wrote the finest level's input (D0Out);
// zo, zdone (PCG): the z statistics are taken as well; an FP32 V-cycle then
// leaves its output in the finest level's u (the PCG widens it where it reads it)
// and z_dev unwritten.
static int vcycle_run(amg_hierarchy *h, const double *r_dev, double *z_dev, cudaStream_t s, bool d0_ready,
                      const ZOut *zo, bool *zdone)
{
    Level &L0 = h->lev[0];
    if (zdone) *zdone = false;
    if (h->prec32) {
        const LV<float> v0 = view<float>(h, 0);
        if (!d0_ready) {
            int si = prof_begin(h, s, R_VIN, false);
            k_in32<<<grid_for(L0.N, 256), 256, 0, s>>>(L0.N, (const double2 *)r_dev, v0.invd,
                                                       (float)L0.ch_inv_theta, v0.f, v0.d); ::bd::note_launch();
            BD_LAUNCH_CHECK();
            prof_end(h, si, 0.0, 0.0, s);
        }
        BD_TRY((vcycle_impl<float>(h, v0.f, v0.u, s)));
        if (zo) {
            int sz = prof_begin(h, s, R_ZSTATS, false);
            BD_TRY(launch_z_from32(h, v0.u, *zo, s));
            prof_end(h, sz, 0.0, 0.0, s);
            if (zdone) *zdone = true;
        } else {
            int so = prof_begin(h, s, R_VOUT, false);
            k_out64<<<grid_for(L0.N, 256), 256, 0, s>>>(L0.N, v0.u, (double2 *)z_dev); ::bd::note_launch();
            BD_LAUNCH_CHECK();
            prof_end(h, so, 0.0, 0.0, s);
        }
        return BD_OK;
    }
    // FP64 stencil: the finest level's gathered vectors in (v + u, u) form
    const LV<double> v0 = view<double>(h, 0);
    const bool su = h->fine.valid;
    if (h->nlev > 1 && !d0_ready) {
        int si = prof_begin(h, s, R_VIN, false);
        if (su)
            k_scale_d0<double, true><<<grid_for(L0.N, 256), 256, 0, s>>>(L0.N, (const double2 *)r_dev, v0.invd,
                                                                         L0.ch_inv_theta, v0.d);
        else
            k_scale_d0<double, false><<<grid_for(L0.N, 256), 256, 0, s>>>(L0.N, (const double2 *)r_dev, v0.invd,
                                                                          L0.ch_inv_theta, v0.d);
        ::bd::note_launch();
        BD_LAUNCH_CHECK();
        prof_end(h, si, 0.0, 0.0, s);
    }
    return vcycle_impl<double>(h, (const double2 *)r_dev, (double2 *)z_dev, s, zo, zdone);
}

int vcycle_device(amg_hierarchy *h, const double *r_dev, double *z_dev, cudaStream_t s)
{
    return vcycle_run(h, r_dev, z_dev, s, false, nullptr, nullptr);
}

__global__ void k_f_stats(int N, const double2 *__restrict__ f, Fin fin)
{
    double a = 0.0, b = 0.0;
    share_stream(N, [&](int i) { return f[i]; }, [&](int, const double2 &v) {
        a += v.y;
        b = fma(v.x, v.x, fma(v.y, v.y, b));
    });
    block_finish<2>(a, b, 0.0, 0.0, fin);
}

__global__ void k_project_f(int N, const double2 *__restrict__ f, double2 *__restrict__ fp, Fin fin)
{
    const double m = fin.scal[S_MEANF];
    double a = 0.0;
    share_stream(N, [&](int i) { return f[i]; }, [&](int i, double2 v) {
        v.y -= m;
        fp[i] = v;
        a = fma(v.x, v.x, fma(v.y, v.y, a));
    });
    block_finish<1>(a, 0.0, 0.0, 0.0, fin);
}

__global__ void k_zero2(int N, double2 *x)
{
    for (int i = share_lo(N) + threadIdx.x, e = share_hi(N); i < e; i += blockDim.x)
        x[i] = make_double2(0.0, 0.0);
}

// x = 0 when (mode 0) the solve is cold, or (mode 1) the right-hand side is zero
__global__ void k_zero_if(int N, double2 *__restrict__ x, const double *__restrict__ scal, int mode)
{
    const bool z = mode == 0 ? scal[S_WARM] == 0.0 : scal[S_NF2] == 0.0;
    if (!z) return;
    for (int i = share_lo(N) + threadIdx.x, e = share_hi(N); i < e; i += blockDim.x)
        x[i] = make_double2(0.0, 0.0);
}

// The next V-cycle's finest-level input, written by the kernel that forms the
// PCG residual r, so that the V-cycle needs no pass of its own over r.  FP64:
// d0 = D^{-1} r / theta, in (v + u, u) form for a stencil finest level
// (mode 1) or in (v, u) form (mode 2); FP32 V-cycle (mode 3): f = (float) r
// and d0 = D^{-1} f / theta in FP32.  The same arithmetic as k_scale_d0 and
// k_in32.
struct D0Out {
    int mode = 0;  // 0: nothing to write
    double2 *d64 = nullptr;
    const double2 *invd64 = nullptr;
    double it = 0.0;
    float2 *f32 = nullptr, *d32 = nullptr;
    const float2 *invd32 = nullptr;
    float it32 = 0.0f;
    // D^{-1} of a row (FP64 or FP32 by the mode)
    struct Pre {
        double2 b64;
        float2 b32;
    };
    __device__ __forceinline__ Pre load(int p) const
    {
        Pre q{};
        if (mode == 1 || mode == 2) q.b64 = invd64[p];
        else if (mode == 3) q.b32 = invd32[p];
        return q;
    }
    __device__ __forceinline__ void operator()(int p, double r0, double r1, const Pre &q) const
    {
        if (mode == 1 || mode == 2) {
            const double v = r0 * q.b64.x * it, u = r1 * q.b64.y * it;
            d64[p] = mode == 1 ? make_double2(v + u, u) : make_double2(v, u);
        } else if (mode == 3) {
            const float f0 = narrow(r0), f1 = narrow(r1);
            f32[p] = make_float2(f0, f1);
            d32[p] = make_float2(f0 * q.b32.x * it32, f1 * q.b32.y * it32);
        }
    }
    __device__ __forceinline__ void operator()(int p, double r0, double r1) const { (*this)(p, r0, r1, load(p)); }
};

// FP64 finest-level operator with a reduction epilogue (block CSR form, T lanes).
// MODE 0: out = A x, partial x.(A x).  MODE 1: out = f - A x (if out), partials
// ||f - A x||^2 and sum of x_u.  x is in (v, u) form.
template <int T, int MODE>
__global__ void __launch_bounds__(256) k_bsr_reduce(int N, const int *__restrict__ rp,
                                                     const int *__restrict__ ci,
                                                     const double *__restrict__ v,
                                                     const double2 *__restrict__ x,
                                                     const double2 *__restrict__ f,
                                                     double2 *__restrict__ out, Fin fin, D0Out d0)
{
    const int lane = threadIdx.x & (T - 1);
    const int groups = (gridDim.x * blockDim.x) / T;
    const int warp_first = ((blockIdx.x * blockDim.x + threadIdx.x) & ~31) / T;
    const int g_in_warp = (threadIdx.x & 31) / T;
    double acc = 0.0, xs = 0.0;
    for (int pw = warp_first; pw < N; pw += groups) {
        const int p = pw + g_in_warp;
        const bool act = p < N;
        double y0 = 0.0, y1 = 0.0;
        const int e = act ? rp[p + 1] : 0;
        for (int t = act ? rp[p] + lane : 0; t < e; t += T) {
            const int q = ci[t];
            const BlkS<double> a = load_blk(v, (size_t)t);
            const double2 xq = x[q];
            y0 = fma(a.a00, xq.x, fma(a.a01, xq.y, y0));
            y1 = fma(a.a10, xq.x, fma(a.a11, xq.y, y1));
        }
        group_sum2<T>(y0, y1);
        if (act && lane == 0) {
            const double2 xp = x[p];
            if (MODE == 0) {
                out[p] = make_double2(y0, y1);
                acc += xp.x * y0 + xp.y * y1;
            } else {
                const double2 fp = f[p];
                const double r0 = fp.x - y0, r1 = fp.y - y1;
                if (out) out[p] = make_double2(r0, r1);
                d0(p, r0, r1);
                acc += r0 * r0 + r1 * r1;
                xs += xp.y;
            }
        }
    }
    block_finish<MODE == 0 ? 1 : 2, 256>(acc, xs, 0.0, 0.0, fin);
}

// The same with the stencil: SU in MODE 0 (the search direction is stored as
// (v + u, u)), plain in MODE 1.
template <int MODE> struct FineReduce {
    const double2 *__restrict__ f;
    double2 *__restrict__ out;
    D0Out d0;
    double acc, xs;
    __device__ __forceinline__ double2 load(int p, bool ok) const
    {
        return MODE == 0 ? make_double2(0.0, 0.0) : fine_ld<double>(f, p, ok);
    }
    __device__ __forceinline__ void operator()(int p, const double2 *, double2 fp, double2 c, double, double y0, double y1)
    {
        if (MODE == 0) {
            out[p] = make_double2(y0, y1);
            acc = fma(c.x - c.y, y0, fma(c.y, y1, acc));
        } else {
            const double r0 = fp.x - y0, r1 = fp.y - y1;
            if (out) out[p] = make_double2(r0, r1);
            d0(p, r0, r1);
            acc += r0 * r0 + r1 * r1;
            xs += c.y;
        }
    }
};

template <int MODE, bool SYM>
__global__ void __launch_bounds__(kFineTPB, FineMinB<double, SYM>::v)
    k_fine_reduce(FineGrid g, const double2 *__restrict__ x, FineReduce<MODE> e, Fin fin)
{
    fine_block<double, SYM, MODE == 0>(g, x, e);
    block_finish<MODE == 0 ? 1 : 2, kFineTPB>(e.acc, e.xs, 0.0, 0.0, fin);
}

template <int MODE, bool SYM>
static void launch_fine_reduce(const amg_hierarchy *h, const double2 *x, const double2 *f, double2 *out,
                               const Fin &fin, cudaStream_t s, const D0Out &d0)
{
    const FineGrid g = fine_grid<double>(h->fine, h->lev[0].ch_c1);
    k_fine_reduce<MODE, SYM><<<fine_blocks<double, SYM>((long long)g.ncb * g.NZ), kFineTPB, 0, s>>>(
        g, x, FineReduce<MODE>{f, out, d0, 0.0, 0.0}, fin);
    ::bd::note_launch();
}

// MODE 0 applies A to the search direction (in (v+u, u) form when the finest
// level is a stencil); MODE 1 forms f - A x for an iterate in (v, u) form.
template <int MODE>
static void fine_reduce(const amg_hierarchy *h, const double2 *x, const double2 *f, double2 *out,
                        const Fin &fin, cudaStream_t s, const D0Out &d0 = D0Out{})
{
    const Level &L0 = h->lev[0];
    if (h->fine.valid) {
        if (h->fine.sym) launch_fine_reduce<MODE, true>(h, x, f, out, fin, s, d0);
        else launch_fine_reduce<MODE, false>(h, x, f, out, fin, s, d0);
        return;
    }
    const BSR &A = L0.A;
    switch (std::min(lanes_for(A, false), 32)) {
    case 1: k_bsr_reduce<1, MODE><<<kRedBlocks, 256, 0, s>>>(A.nbr, A.rp.p, A.ci.p, A.v.p, x, f, out, fin, d0); ::bd::note_launch(); break;
    case 2: k_bsr_reduce<2, MODE><<<kRedBlocks, 256, 0, s>>>(A.nbr, A.rp.p, A.ci.p, A.v.p, x, f, out, fin, d0); ::bd::note_launch(); break;
    case 4: k_bsr_reduce<4, MODE><<<kRedBlocks, 256, 0, s>>>(A.nbr, A.rp.p, A.ci.p, A.v.p, x, f, out, fin, d0); ::bd::note_launch(); break;
    case 8: k_bsr_reduce<8, MODE><<<kRedBlocks, 256, 0, s>>>(A.nbr, A.rp.p, A.ci.p, A.v.p, x, f, out, fin, d0); ::bd::note_launch(); break;
    case 16: k_bsr_reduce<16, MODE><<<kRedBlocks, 256, 0, s>>>(A.nbr, A.rp.p, A.ci.p, A.v.p, x, f, out, fin, d0); ::bd::note_launch(); break;
    default: k_bsr_reduce<32, MODE><<<kRedBlocks, 256, 0, s>>>(A.nbr, A.rp.p, A.ci.p, A.v.p, x, f, out, fin, d0); ::bd::note_launch(); break;
    }
}

// sums of z_u and r_u, and r.z (FP64 V-cycle)
__global__ void k_z_stats(int N, const double2 *__restrict__ z, const double2 *__restrict__ r, Fin fin)
{
    double a = 0.0, b = 0.0, c = 0.0;
    struct In {
        double2 z, r;
    };
    share_stream(N, [&](int i) { return In{z[i], r[i]}; }, [&](int, const In &q) {
        a += q.z.y;
        b += q.r.y;
        c = fma(q.r.x, q.z.x, fma(q.r.y, q.z.y, c));
    });
    block_finish<3>(a, b, c, 0.0, fin);
}

// The V-cycle's last finest-level kernel with the z statistics fused in: the
// post-smoothed iterate is the preconditioned residual z, stored in FP64, and
// the sums k_z_stats forms (z_u, r_u, r.z, r.z_old) are taken in FP64 in the
// same pass (stage 3).
struct ZOut {
    double2 *z;
    const double2 *r;
    const float2 *uold;  // FP32 V-cycle: its previous output
    Fin fin;
};

template <bool SYM> struct FineZ {
    FinePost2<double, SYM, true> post;
    double2 *z;  // may be the iterate's own storage
    const double2 *__restrict__ r;
    double a, b, c;
    struct Pre {
        typename FinePost2<double, SYM, true>::Pre q;
        double2 r;
    };
    __device__ __forceinline__ Pre load(int p, bool ok) const { return {post.load(p, ok), fine_ld<double>(r, p, ok)}; }
    __device__ __forceinline__ void operator()(int p, const double2 *t, const Pre &q, double2 x, double c1, double y0, double y1)
    {
        const double2 u = post.value(t, q.q, x, c1, y0, y1);
        z[p] = u;
        a += u.y;
        b += q.r.y;
        c = fma(q.r.x, u.x, fma(q.r.y, u.y, c));
    }
};

template <bool SYM>
__global__ void __launch_bounds__(kFineTPB, FineMinB<double, SYM>::v)
    k_fine_z(FineGrid g, const double2 *__restrict__ x, FineZ<SYM> e, Fin fin)
{
    fine_block<double, SYM, true>(g, x, e);
    block_finish<3, kFineTPB>(e.a, e.b, e.c, 0.0, fin);
}

static int launch_fine_z(amg_hierarchy *h, const LV<double> &lv, const double2 *u, const ZOut &zo, cudaStream_t s)
{
    const FineGrid g = fine_grid<double>(h->fine, h->lev[0].ch_c1);
    auto launch = [&](auto sym) {
        constexpr bool SYM = decltype(sym)::value;
        k_fine_z<SYM><<<fine_blocks<double, SYM>((long long)g.ncb * g.NZ), kFineTPB, 0, s>>>(
            g, lv.d, FineZ<SYM>{{lv.r, u, nullptr}, zo.z, zo.r, 0.0, 0.0, 0.0}, zo.fin);
    };
    if (h->fine.sym) launch(std::true_type{});
    else launch(std::false_type{});
    ::bd::note_launch();
    BD_LAUNCH_CHECK();
    return BD_OK;
}

// Statistics (z_u, r_u, r.z, r.z_old) of z = (double) u, the FP32 V-cycle's
// output, in FP64 (stage 3).  z and the previous projected z are not stored:
// both are the FP32 outputs, widened exactly, less their mean (S_MEANZ still holds
// the previous one here), so the PCG reads 32 bytes per node instead of moving
// 56 here and 48 instead of 80 in the direction's update.  Bound by the FP64
// operations, seven a node once the conversions are integer work (256x256x64:
// 93 + 55 -> 69 + 41 us, 128x128x32: 24.3 + 10.4 -> 20.2 + 10.2).
__global__ void __launch_bounds__(kVecThreads, 4)
    k_z_from32(int N, const float2 *__restrict__ u, ZOut zo)
{
    const double mo = zo.fin.scal[S_MEANZ];
    double a = 0.0, b = 0.0, c = 0.0, d = 0.0;
    struct In {
        float2 v, w;
        double2 r;
    };
    share_stream(N, [&](int i) { return In{u[i], zo.uold[i], zo.r[i]}; }, [&](int, const In &q) {
        const double zx = widen(q.v.x), zy = widen(q.v.y);
        a += zy;
        b += q.r.y;
        c = fma(q.r.x, zx, fma(q.r.y, zy, c));
        d = fma(q.r.x, widen(q.w.x), fma(q.r.y, widen(q.w.y) - mo, d));
    });
    block_finish<4>(a, b, c, d, zo.fin);
}

static int launch_z_from32(amg_hierarchy *h, const float2 *u, const ZOut &zo, cudaStream_t s)
{
    k_z_from32<<<kVecBlocks, kVecThreads, 0, s>>>(h->lev[0].N, u, zo);
    ::bd::note_launch();
    BD_LAUNCH_CHECK();
    return BD_OK;
}

// p = z - mean(z_u) e_u (first iteration) or that + beta p, stored in (v+u, u)
// form when SU; z as the V-cycle left it (FP64, or its FP32 output, which is
// kept for the next flexible beta).
template <bool SU, class Z>
__global__ void __launch_bounds__(kVecThreads, 4)
    k_p_update(int N, const Z *__restrict__ z, double2 *__restrict__ p, Z *__restrict__ zold,
                           const double *__restrict__ scal, int first)
{
    const double mz = scal[S_MEANZ], beta = scal[S_BETA];
    if (first < 0) first = scal[S_IT] == 0.0;
    struct In {
        Z z;
        double2 p;
    };
    share_stream(N, [&](int i) { return In{z[i], p[i]}; }, [&](int i, const In &q) {
        if (zold) zold[i] = q.z;
        const double zx = widen(q.z.x), zy = widen(q.z.y) - mz;
        const double2 zs = make_double2(SU ? zx + zy : zx, zy);
        p[i] = first ? zs : make_double2(zs.x + beta * q.p.x, zs.y + beta * q.p.y);
    });
}

template <bool SU>
__global__ void __launch_bounds__(kVecThreads, 4)
    k_xr_update(int N, double2 *__restrict__ x, double2 *__restrict__ r,
                            const double2 *__restrict__ p, const double2 *__restrict__ q, Fin fin, D0Out d0)
{
    const double alpha = fin.scal[S_ALPHA];
    double acc = 0.0;
    struct In {
        double2 x, r, p, q;
        D0Out::Pre b;
    };
    share_stream(N, [&](int i) { return In{x[i], r[i], p[i], q[i], d0.load(i)}; }, [&](int i, const In &in) {
        double2 xi = in.x, ri = in.r;
        const double2 pi = in.p, qi = in.q;
        const double pv = SU ? pi.x - pi.y : pi.x;
        xi.x += alpha * pv;
        xi.y += alpha * pi.y;
        ri.x -= alpha * qi.x;
        ri.y -= alpha * qi.y;
        x[i] = xi;
        r[i] = ri;
        d0(i, ri.x, ri.y, in.b);
        acc = fma(ri.x, ri.x, fma(ri.y, ri.y, acc));
    });
    block_finish<1>(acc, 0.0, 0.0, 0.0, fin);
}

__global__ void k_project_x(int N, double2 *__restrict__ x, const double *__restrict__ scal)
{
    const double m = scal[S_MEANX];
    for (int i = share_lo(N) + threadIdx.x, e = share_hi(N); i < e; i += blockDim.x) x[i].y -= m;
}

static void p_update(amg_hierarchy *h, int N, double2 *p, double *scal, int first, cudaStream_t s)
{
    auto run = [&](auto su) {
        constexpr bool SU = decltype(su)::value;
        if (h->prec32)
            k_p_update<SU><<<kVecBlocks, kVecThreads, 0, s>>>(N, (const float2 *)h->lev[0].u32.p, p, (float2 *)h->uold.p,
                                                             scal, first);
        else
            k_p_update<SU><<<kVecBlocks, kVecThreads, 0, s>>>(N, (const double2 *)h->z.p, p, (double2 *)nullptr, scal,
                                                             first);
    };
    if (h->fine.valid) run(std::true_type{});
    else run(std::false_type{});
    note_launch();
}

static void xr_update(const amg_hierarchy *h, int N, double2 *x, double2 *r, const double2 *p,
                      const double2 *q, const Fin &fin, cudaStream_t s, const D0Out &d0)
{
    if (h->fine.valid) k_xr_update<true><<<kVecBlocks, kVecThreads, 0, s>>>(N, x, r, p, q, fin, d0);
    else k_xr_update<false><<<kVecBlocks, kVecThreads, 0, s>>>(N, x, r, p, q, fin, d0);
    note_launch();
}

// What the producer of the PCG residual writes for the next V-cycle (see
// D0Out); mode 0 where the V-cycle has no smoothing level and is FP64.
static D0Out d0_out(amg_hierarchy *h)
{
    D0Out d;
    Level &L0 = h->lev[0];
    if (h->prec32) {
        d.mode = 3;
        d.f32 = (float2 *)L0.f32.p;
        d.d32 = (float2 *)L0.d32.p;
        d.invd32 = (const float2 *)L0.invdiag32.p;
        d.it32 = (float)L0.ch_inv_theta;
    } else if (h->nlev > 1) {
        d.mode = h->fine.valid ? 1 : 2;
        d.d64 = (double2 *)L0.d.p;
        d.invd64 = (const double2 *)L0.invdiag.p;
        d.it = L0.ch_inv_theta;
    }
    return d;
}

// ------------------------------------------------------------------ lane autotuning
// Candidates: block-CSR with powers of two from (average blocks per row)/16
// lanes per row to 4x the average, 64/128/256 meaning a thread block per row
// (rows of 32 blocks and more only), and, where the operator may take it, the
// sliced form with 1, 2, 4 and 8 lanes per row (FP64, operators of 8192 rows
// and more).  Each runs once untimed, then three times back to back, and the
// median counts (the V-cycle applies a level's operator several times in a
// row: smoother, residual).  Single launches do not rank every operator as the
// V-cycle does: on the 128x128x32 slab they put the sliced form first for the
// middle level's A, which inside the V-cycle is 5 % slower than block-CSR with
// 4 lanes, warm or after an L2 flush; the row-length rule holds the choices
// measured inside the V-cycle.  The launches of all block-CSR candidates are
// queued with their events and read after one synchronisation; each sliced
// candidate is built, timed and synchronised in turn (the next one reuses its
// buffers).
constexpr int kLaneCands = 13, kLaneReps = 3;
constexpr long long kTuneMinBlocks = 20000;  // smaller operators keep the rule

struct TuneEvents {
    cudaEvent_t e[kLaneCands][kLaneReps][2] = {};
    int create()
    {
        for (auto &c : e)
            for (auto &r : c)
                for (cudaEvent_t &v : r) BD_CUDA(cudaEventCreate(&v));
        return BD_OK;
    }
    ~TuneEvents()
    {
        for (auto &c : e)
            for (auto &r : c)
                for (cudaEvent_t v : r)
                    if (v) cudaEventDestroy(v);
    }
};

// block-CSR candidates of M, at most kLaneCands - 4
static int csr_candidates(const BSR &M, int *cand)
{
    const double avg = M.nbr > 0 ? (double)M.nb / M.nbr : 1.0;
    int Tlo = 1, Thi = 256, nc = 0;
    while (Tlo * 16 < avg && Tlo < 32) Tlo <<= 1;
    while (Thi > 1 && Thi > 4.0 * avg) Thi >>= 1;
    if (avg < 32.0) Thi = std::min(Thi, 32);
    Thi = std::max(Thi, Tlo);
    for (int T = Tlo; T <= Thi && nc < kLaneCands - 4; T <<= 1) cand[nc++] = T;
    return nc;
}

// candidate c, once untimed and then kLaneReps times between events
template <class F> static int time_candidate(F run, cudaEvent_t (*ev)[2], cudaStream_t s)
{
    BD_TRY(run());
    for (int k = 0; k < kLaneReps; k++) {
        BD_CUDA(cudaEventRecord(ev[k][0], s));
        BD_TRY(run());
        BD_CUDA(cudaEventRecord(ev[k][1], s));
    }
    return BD_OK;
}

// the fastest median wins unless the rule's choice (when among the
// candidates) is within 3 % of it: near-ties then resolve the same way
// on every run
static int pick_candidate(const int *cand, int nc, int rule, const TuneEvents &ev, int *pick)
{
    float best = 0.0f, t_rule = -1.0f;
    int bestT = rule;
    for (int c = 0; c < nc; c++) {
        float t[kLaneReps];
        for (int k = 0; k < kLaneReps; k++) BD_CUDA(cudaEventElapsedTime(&t[k], ev.e[c][k][0], ev.e[c][k][1]));
        const float med = std::max(std::min(t[0], t[1]), std::min(std::max(t[0], t[1]), t[2]));
        if (cand[c] == rule) t_rule = med;
        if (c == 0 || med < best) {
            best = med;
            bestT = cand[c];
        }
    }
    *pick = (t_rule >= 0.0f && t_rule <= 1.03f * best) ? rule : bestT;
    return BD_OK;
}

int tune_csr_lanes(const BSR &M, const std::function<int(int)> &run, cudaStream_t s, int *lanes)
{
    if (M.nb < kTuneMinBlocks) return BD_OK;
    int cand[kLaneCands];
    const int nc = csr_candidates(M, cand);
    TuneEvents ev;
    BD_TRY(ev.create());
    for (int c = 0; c < nc; c++) BD_TRY(time_candidate([&] { return run(cand[c]); }, ev.e[c], s));
    BD_CUDA(cudaStreamSynchronize(s));
    return pick_candidate(cand, nc, *lanes, ev, lanes);
}

template <class S>
static int tune_operator(Level &L, int op, bool sliced_ok, const v2<S> *x, const v2<S> *f, v2<S> *out,
                         const S *vals, TuneEvents &ev, cudaStream_t s)
{
    const BSR &M = op == 0 ? L.A : (op == 1 ? L.R : L.P);
    const bool fp32 = sizeof(S) == 4;
    const EpiResid<S> epi{f, out};
    int cand[kLaneCands], nc = csr_candidates(M, cand);
    const int ncsr = nc;
    if (sliced_ok && !fp32 && M.nbr >= kSlicedMinRows)
        for (int K = 1; K <= 8; K <<= 1) cand[nc++] = -K;
    const int rule = L.lanes[op];
    auto run = [&]() {
        return pair_of(L, op) ? apply_pair<S>(L, op, GatherVec<S, sizeof(S) == 8>{x}, epi, s)
                              : apply_op<S>(L, op, vals, GatherVec<S>{x}, epi, s);
    };
    for (int c = 0; c < nc; c++) {
        if (cand[c] < 0) BD_TRY(build_op(L, op, -cand[c], fp32, s));
        L.lanes[op] = cand[c];
        BD_TRY(time_candidate(run, ev.e[c], s));
        if (cand[c] < 0 || c + 1 == ncsr) BD_CUDA(cudaStreamSynchronize(s));
    }
    BD_CUDA(cudaStreamSynchronize(s));
    int pick = rule;
    BD_TRY(pick_candidate(cand, nc, rule, ev, &pick));
    L.lanes[op] = pick;
    if (pick > 0) drop_sliced(L.sl[op]);
    else if (L.sl[op].K != -pick) BD_TRY(build_op(L, op, -pick, fp32, s));
    return BD_OK;
}

// Time the candidate forms of every block operator the V-cycle applies (A
// below the finest level, or on it where it is not a stencil; R and P) on
// this GPU and keep the fastest.  The workspace vectors serve as operands;
// their contents do not matter.  The form changes the order of a row's sum,
// so the choice is fixed per hierarchy: every solve with it is reproducible.
template <class S>
static int autotune_lanes(amg_hierarchy *h, cudaStream_t s)
{
    TuneEvents ev;
    BD_TRY(ev.create());
    for (int l = 0; l < h->nlev - 1; l++) {
        Level &L = h->lev[l];
        const LV<S> lv = view<S>(h, l), cv = view<S>(h, l + 1);
        for (int op = 0; op < 3; op++) {
            if (op == 0 && l == 0 && h->fine.valid) continue;
            const BSR &M = op == 0 ? L.A : (op == 1 ? L.R : L.P);
            if (M.nb < kTuneMinBlocks) continue;
            const S *vals = op == 0 ? lv.Av : (op == 1 ? lv.Rv : lv.Pv);
            const v2<S> *x = op == 0 ? lv.u : (op == 1 ? lv.r : cv.u);
            const v2<S> *f = op == 1 ? cv.f : lv.f;
            v2<S> *out = op == 0 ? lv.r : (op == 1 ? cv.r : lv.w);
            BD_TRY(tune_operator<S>(L, op, op > 0 || l > 0, x, f, out, vals, ev, s));
        }
    }
    return BD_OK;
}

// ------------------------------------------------------------------ workspace
// vectors of n entries each as parts of one allocation (256-byte aligned)
template <class T> static int carve(DBuf<char> &work, size_t n, std::initializer_list<DBuf<T> *> parts)
{
    const size_t step = (n * sizeof(T) + 255) / 256 * 256;
    BD_TRY(work.alloc(step * parts.size()));
    size_t k = 0;
    for (DBuf<T> *d : parts) d->view((T *)(work.p + step * k++), n);
    return BD_OK;
}

int prepare_solve(amg_hierarchy *h, cudaStream_t s)
{
    const bool p32 = h->prec32;
    for (int l = 0; l < h->nlev; l++) {
        Level &L = h->lev[l];
        size_t n = 2 * (size_t)L.N;
        if (p32) {
            BD_TRY(carve(L.work, n, {&L.f32, &L.u32, &L.r32, &L.d32, &L.w32}));
            BD_TRY(L.invdiag32.alloc(n));
            const bool a32 = l > 0 || !h->fine.valid;  // the stencil has its own FP32 table
            if (a32) BD_TRY(L.A32.alloc(4 * (size_t)L.A.nb));
            k_to_f32<<<grid_for(n, 256), 256, 0, s>>>((long long)n, L.invdiag.p, L.invdiag32.p); ::bd::note_launch();
            if (a32) {
                k_to_f32<<<grid_for(4 * L.A.nb, 256), 256, 0, s>>>(4 * L.A.nb, L.A.v.p, L.A32.p); ::bd::note_launch();
            }
            if (l < h->nlev - 1 && a32) {  // the finest level has them in pair form
                BD_TRY(L.P32.alloc(4 * (size_t)L.P.nb));
                BD_TRY(L.R32.alloc(4 * (size_t)L.R.nb));
                k_to_f32<<<grid_for(4 * L.P.nb, 256), 256, 0, s>>>(4 * L.P.nb, L.P.v.p, L.P32.p); ::bd::note_launch();
                k_to_f32<<<grid_for(4 * L.R.nb, 256), 256, 0, s>>>(4 * L.R.nb, L.R.v.p, L.R32.p); ::bd::note_launch();
            }
            BD_LAUNCH_CHECK();
        } else {
            BD_TRY(carve(L.work, n, {&L.f, &L.u, &L.r, &L.d, &L.w}));
        }
        if (l < h->nlev - 1) {
            double lo = h->opts.eig_lo * L.lam, hi = h->opts.eig_hi * L.lam;
            double theta = 0.5 * (hi + lo), delta = 0.5 * (hi - lo);
            double sigma = theta / delta, rho0 = 1.0 / sigma;
            double rho1 = 1.0 / (2.0 * sigma - rho0);
            L.ch_inv_theta = 1.0 / theta;
            L.ch_c1 = rho1 * rho0;
            L.ch_c2 = 2.0 * rho1 / delta;
        }
    }
    if (h->fine.valid) {
        FineStencil &F = h->fine;
        const Level &L0 = h->lev[0];
        const size_t len = 2 * (size_t)fine_row_len(F.sym) * 9 * F.NZ;
        BD_TRY(F.tab.alloc(len));
        if (p32) BD_TRY(F.tab32.alloc(len));
        BD_TRY(fine_pack(F, F.sym, L0.ch_c2, L0.ch_inv_theta, fine_omega(L0), F.tab.p, F.tab32.p, s));
    }
    if (h->fine.valid && h->nlev > 1) BD_TRY(build_pairs(h->lev[0], p32, s));
    size_t n0 = 2 * (size_t)h->lev[0].N;
    BD_TRY(carve(h->work, n0, {&h->x, &h->r, &h->z, &h->p, &h->q, &h->fp, &h->fin}));
    if (p32) {
        BD_TRY(h->uold.alloc(n0));
        BD_CUDA(cudaMemsetAsync(h->uold.p, 0, h->uold.bytes(), s));
    }
    BD_TRY(h->partial.alloc(kPart * (size_t)kRedBlocks));
    BD_TRY(h->counter.alloc(1));
    BD_CUDA(cudaMemsetAsync(h->counter.p, 0, sizeof(unsigned int), s));
    BD_TRY(h->scal.alloc(S_NSLOTS));
    if (!h->host_scal) BD_CUDA(cudaMallocHost((void **)&h->host_scal, sizeof(double) * S_NSLOTS));
    if (!h->host_init) BD_CUDA(cudaMallocHost((void **)&h->host_init, sizeof(double) * S_NSLOTS));
    // lanes per block row of the V-cycle's block-CSR operators
    // (the sliced form for A only below the finest level: the PCG's fused
    // A p and residual reductions on a block-CSR finest level use
    // block-CSR; nothing on the coarsest level, which is solved densely)
    for (int l = 0; l < h->nlev; l++) {
        Level &L = h->lev[l];
        const bool last = l == h->nlev - 1;
        L.lanes[0] = lanes_rule(L.A, p32, l > 0 && !last);
        L.lanes[1] = last ? 0 : lanes_rule(L.R, p32, true, pair_of(L, 1));
        L.lanes[2] = last ? 0 : lanes_rule(L.P, p32, true, pair_of(L, 2));
        for (int op = 0; op < 3; op++) {
            if (L.lanes[op] < 0)
                BD_TRY(build_op(L, op, -L.lanes[op], p32, s));
            else drop_sliced(L.sl[op]);
        }
    }
    if (h->opts.autotune) BD_TRY(p32 ? autotune_lanes<float>(h, s) : autotune_lanes<double>(h, s));
    BD_CUDA(cudaStreamSynchronize(s));
    return BD_OK;
}

static int read_scal(amg_hierarchy *h, cudaStream_t s)
{
    BD_CUDA(cudaMemcpyAsync(h->host_scal, h->scal.p, sizeof(double) * S_NSLOTS, cudaMemcpyDeviceToHost, s));
    BD_CUDA(cudaStreamSynchronize(s));
    return BD_OK;
}

static Fin make_fin(amg_hierarchy *h, int stage, int first, cudaGraphConditionalHandle cond = 0)
{
    Fin f;
    f.scal = h->scal.p;
    f.partial = h->partial.p;
    f.counter = h->counter.p;
    f.stage = stage;
    f.N = h->lev[0].N;
    f.first = first;
    f.flex = h->prec32 ? 1 : 0;
    f.cond = cond;
    return f;
}

// Projected PCG on device vectors (f_dev, x_dev: 2N doubles each), host-driven
// loop: one residual read-back per iteration.  With an FP32 V-cycle the
// preconditioner is not exactly symmetric, so beta takes the flexible
// (Polak-Ribiere) form.
static int pcg_solve_loop(amg_hierarchy *h, const double *f_dev, double *x_dev, int warm,
                          const solve_options *o, cudaStream_t s, solve_info *info)
{
    Level &L0 = h->lev[0];
    const int N = L0.N;
    double2 *x = (double2 *)x_dev, *r = (double2 *)h->r.p, *z = (double2 *)h->z.p;
    double2 *p = (double2 *)h->p.p, *q = (double2 *)h->q.p, *fp = (double2 *)h->fp.p;
    double *scal = h->scal.p;
    cudaEvent_t e0 = nullptr, e1 = nullptr;
    BD_CUDA(cudaEventCreate(&e0));
    BD_CUDA(cudaEventCreate(&e1));
    BD_CUDA(cudaEventRecord(e0, s));
    BD_CUDA(cudaMemsetAsync(scal, 0, sizeof(double) * S_NSLOTS, s));
    k_f_stats<<<kVecBlocks, kVecThreads, 0, s>>>(N, (const double2 *)f_dev, make_fin(h, 0, 0)); ::bd::note_launch();
    k_project_f<<<kVecBlocks, kVecThreads, 0, s>>>(N, (const double2 *)f_dev, fp, make_fin(h, 1, 0)); ::bd::note_launch();
    if (!warm) {
        k_zero2<<<kVecBlocks, kVecThreads, 0, s>>>(N, x); ::bd::note_launch();
    }
    const D0Out d0 = d0_out(h);
    fine_reduce<1>(h, x, fp, r, make_fin(h, 2, 0), s, d0);
    BD_LAUNCH_CHECK();
    BD_TRY(read_scal(h, s));
    double ff = h->host_scal[S_FF], sumfu = h->host_scal[S_SUMFU];
    double nf = sqrt(h->host_scal[S_NF2]);
    double rr = sqrt(h->host_scal[S_RR]);
    int status = BD_OK, it = 0;
    if (o->strict && ff > 0.0) {
        double null_part = fabs(sumfu) / sqrt((double)N);
        if (null_part > 1e-8 * sqrt(ff)) status = BD_EINCONSISTENT;
    }
    if (status == BD_OK && nf == 0.0) {
        k_zero2<<<kVecBlocks, kVecThreads, 0, s>>>(N, x); ::bd::note_launch();
        BD_LAUNCH_CHECK();
        rr = 0.0;
    } else if (status == BD_OK && !(rr <= o->rtol * nf)) {
        status = BD_ENOTCONV;
        while (it < o->max_it) {
            const ZOut zo{z, r, (const float2 *)h->uold.p, make_fin(h, 3, it == 0)};
            bool zd = false;
            BD_TRY(vcycle_run(h, (const double *)r, (double *)z, s, true, &zo, &zd));
            if (!zd) {
                int sz = prof_begin(h, s, R_ZSTATS, false);
                k_z_stats<<<kVecBlocks, kVecThreads, 0, s>>>(N, z, r, zo.fin); ::bd::note_launch();
                prof_end(h, sz, 0.0, 0.0, s);
            }
            int su = prof_begin(h, s, R_PUPDATE, false);
            p_update(h, N, p, scal, it == 0, s);
            prof_end(h, su, 0.0, 0.0, s);
            // the FP64 PCG operator counts among the finest-operator launches
            // when the V-cycle is FP64 too (one kernel family per profile)
            int sq = prof_begin(h, s, R_AP, !h->prec32);
            fine_reduce<0>(h, p, nullptr, q, make_fin(h, 4, 0), s);
            prof_end(h, sq, h->prec32 ? 0.0 : fine_bytes<double>(h, L0, 2), fine_flops(h, L0), s,
                     fine_ops<double>(h, L0, FR_AP));
            int sx = prof_begin(h, s, R_XRUPDATE, false);
            xr_update(h, N, x, r, p, q, make_fin(h, 2, 0), s, d0);
            prof_end(h, sx, 0.0, 0.0, s);
            BD_LAUNCH_CHECK();
            BD_TRY(read_scal(h, s));
            it++;
            if (h->host_scal[S_BREAK] != 0.0) {
                status = BD_EBREAKDOWN;
                break;
            }
            rr = sqrt(h->host_scal[S_RR]);
            if (!std::isfinite(rr)) {
                status = BD_EBREAKDOWN;
                break;
            }
            if (rr <= o->rtol * nf) {
                status = BD_OK;
                break;
            }
        }
    }
    // true residual and projection of x
    fine_reduce<1>(h, x, fp, nullptr, make_fin(h, 5, 0), s);
    k_project_x<<<kVecBlocks, kVecThreads, 0, s>>>(N, x, scal); ::bd::note_launch();
    BD_LAUNCH_CHECK();
    BD_CUDA(cudaEventRecord(e1, s));
    BD_TRY(read_scal(h, s));
    prof_collect(h);
    float ms = 0.0f;
    cudaEventElapsedTime(&ms, e0, e1);
    cudaEventDestroy(e0);
    cudaEventDestroy(e1);
    if (info) {
        info->status = status;
        info->iters = it;
        info->rel_res = nf > 0.0 ? rr / nf : 0.0;
        info->true_rel_res = nf > 0.0 ? sqrt(h->host_scal[S_TRR]) / nf : 0.0;
        info->solve_ms = ms;
    }
    return status;
}

// ------------------------------------------------------------------ graph form
// The whole solve as one CUDA graph: the pre-loop kernels, a WHILE node whose
// body is one PCG iteration (V-cycle included), the post-loop kernels.  The
// body's last reduction decides convergence, breakdown or max_it on the device
// and sets the node's condition, so a solve costs one graph launch and one
// host synchronisation.  The loop is bounded by max_it.  The graph works on the
// hierarchy's own buffers (right-hand side in `fin`, iterate in `x`).
void drop_capture(cudaStream_t s)
{
    cudaStreamCaptureStatus cs;
    if (cudaStreamIsCapturing(s, &cs) == cudaSuccess && cs != cudaStreamCaptureStatusNone) {
        cudaGraph_t g = nullptr;
        cudaStreamEndCapture(s, &g);
        if (g) cudaGraphDestroy(g);
    }
    cudaGetLastError();
}

int while_handle(cudaStream_t s, WhileNode *w)
{
    cudaStreamCaptureStatus cs;
    cudaGraph_t g = nullptr;
    const cudaGraphNode_t *deps = nullptr;
    size_t nd = 0;
    BD_CUDA(cudaStreamGetCaptureInfo(s, &cs, nullptr, &g, &deps, nullptr, &nd));
    BD_CUDA(cudaGraphConditionalHandleCreate(&w->cond, g, 0, 0));
    return BD_OK;
}

int while_begin(cudaStream_t s, cudaStream_t s2, WhileNode *w)
{
    cudaStreamCaptureStatus cs;
    cudaGraph_t g = nullptr;
    const cudaGraphNode_t *deps = nullptr;
    size_t nd = 0;
    BD_CUDA(cudaStreamGetCaptureInfo(s, &cs, nullptr, &g, &deps, nullptr, &nd));
    cudaGraphNodeParams np = {};
    np.type = cudaGraphNodeTypeConditional;
    np.conditional.handle = w->cond;
    np.conditional.type = cudaGraphCondTypeWhile;
    np.conditional.size = 1;
    BD_CUDA(cudaGraphAddNode(&w->node, g, deps, nullptr, nd, &np));
    BD_CUDA(cudaStreamBeginCaptureToGraph(s2, np.conditional.phGraph_out[0], nullptr, nullptr, 0,
                                          cudaStreamCaptureModeThreadLocal));
    return BD_OK;
}

int while_end(cudaStream_t s, cudaStream_t s2, WhileNode *w)
{
    cudaGraph_t body = nullptr;
    BD_CUDA(cudaStreamEndCapture(s2, &body));
    BD_CUDA(cudaStreamUpdateCaptureDependencies(s, &w->node, nullptr, 1, cudaStreamSetCaptureDependencies));
    return BD_OK;
}

// Capture one whole solve of h into the graph being captured on stream s:
// pre-loop kernels, a WHILE node whose body (captured on s2) is one PCG
// iteration and whose condition the device sets, post-loop kernels.  Operates
// on h's own buffers (f in h->fin, x in h->x, scalars in h->scal).
static int capture_solve(amg_hierarchy *h, cudaStream_t s, cudaStream_t s2)
{
    Level &L0 = h->lev[0];
    const int N = L0.N;
    double2 *x = (double2 *)h->x.p, *r = (double2 *)h->r.p, *z = (double2 *)h->z.p;
    double2 *p = (double2 *)h->p.p, *q = (double2 *)h->q.p, *fp = (double2 *)h->fp.p;
    const double2 *fin = (const double2 *)h->fin.p;
    double *scal = h->scal.p;
    // kernel-node counts per section (the launch counter counts executions, so
    // the increments made while capturing are taken back below)
    const long long c0 = launch_count();
    k_f_stats<<<kVecBlocks, kVecThreads, 0, s>>>(N, fin, make_fin(h, 0, 0)); ::bd::note_launch();
    k_project_f<<<kVecBlocks, kVecThreads, 0, s>>>(N, fin, fp, make_fin(h, 1, 0)); ::bd::note_launch();
    k_zero_if<<<kVecBlocks, kVecThreads, 0, s>>>(N, x, scal, 0); ::bd::note_launch();
    BD_LAUNCH_CHECK();
    WhileNode w;
    BD_TRY(while_handle(s, &w));
    const D0Out d0 = d0_out(h);
    fine_reduce<1>(h, x, fp, r, make_fin(h, 6, 0, w.cond), s, d0);
    BD_LAUNCH_CHECK();
    BD_TRY(while_begin(s, s2, &w));
    const long long c1 = launch_count();
    const ZOut zo{z, r, (const float2 *)h->uold.p, make_fin(h, 3, -1)};
    bool zd = false;
    BD_TRY(vcycle_run(h, (const double *)r, (double *)z, s2, true, &zo, &zd));
    if (!zd) {
        k_z_stats<<<kVecBlocks, kVecThreads, 0, s2>>>(N, z, r, zo.fin); ::bd::note_launch();
    }
    p_update(h, N, p, scal, -1, s2);
    fine_reduce<0>(h, p, nullptr, q, make_fin(h, 4, 0), s2);
    xr_update(h, N, x, r, p, q, make_fin(h, 7, 0, w.cond), s2, d0);
    BD_LAUNCH_CHECK();
    const long long c2 = launch_count();
    BD_TRY(while_end(s, s2, &w));
    k_zero_if<<<kVecBlocks, kVecThreads, 0, s>>>(N, x, scal, 1); ::bd::note_launch();
    fine_reduce<1>(h, x, fp, nullptr, make_fin(h, 5, 0), s);
    k_project_x<<<kVecBlocks, kVecThreads, 0, s>>>(N, x, scal); ::bd::note_launch();
    BD_LAUNCH_CHECK();
    const long long c3 = launch_count();
    h->graph_pre = c1 - c0;
    h->graph_body = c2 - c1;
    h->graph_post = c3 - c2;
    note_launches(-(c3 - c0));
    return BD_OK;
}

static int capture_graph(amg_hierarchy *h)
{
    BD_CUDA(cudaStreamBeginCapture(h->cap_stream, cudaStreamCaptureModeThreadLocal));
    BD_TRY(capture_solve(h, h->cap_stream, h->cap_stream2));
    BD_CUDA(cudaStreamEndCapture(h->cap_stream, &h->graph));
    BD_CUDA(cudaGraphInstantiate(&h->graph_exec, h->graph, 0));
    return BD_OK;
}

static int build_graph(amg_hierarchy *h)
{
    if (!h->cap_stream) BD_CUDA(cudaStreamCreateWithFlags(&h->cap_stream, cudaStreamNonBlocking));
    if (!h->cap_stream2) BD_CUDA(cudaStreamCreateWithFlags(&h->cap_stream2, cudaStreamNonBlocking));
    int st = capture_graph(h);
    if (st != BD_OK) {
        drop_capture(h->cap_stream2);
        drop_capture(h->cap_stream);
        if (h->graph_exec) cudaGraphExecDestroy(h->graph_exec);
        if (h->graph) cudaGraphDestroy(h->graph);
        h->graph_exec = nullptr;
        h->graph = nullptr;
    }
    return st;
}

// Enqueue one graph-form solve on `s` (inputs copied in, the graph, the
// iterate copied out, the device scalars copied to the pinned host block);
// pcg_graph_finish waits for it.  Only one solve per hierarchy may be in flight.
static int report_from_scal(amg_hierarchy *h, const double *sc, float ms, solve_info *info);

static int pcg_graph_launch(amg_hierarchy *h, const double *f_dev, double *x_dev, int warm,
                            const solve_options *o, cudaStream_t s)
{
    const size_t bytes = sizeof(double) * 2 * (size_t)h->lev[0].N;
    if (!h->ev_solve[0]) {
        BD_CUDA(cudaEventCreate(&h->ev_solve[0]));
        BD_CUDA(cudaEventCreate(&h->ev_solve[1]));
    }
    BD_CUDA(cudaEventRecord(h->ev_solve[0], s));
    if (f_dev != h->fin.p) BD_CUDA(cudaMemcpyAsync(h->fin.p, f_dev, bytes, cudaMemcpyDeviceToDevice, s));
    if (warm && x_dev != h->x.p) BD_CUDA(cudaMemcpyAsync(h->x.p, x_dev, bytes, cudaMemcpyDeviceToDevice, s));
    for (int i = 0; i < S_NSLOTS; i++) h->host_init[i] = 0.0;
    h->host_init[S_RTOL] = o->rtol;
    h->host_init[S_MAXIT] = (double)o->max_it;
    h->host_init[S_WARM] = warm ? 1.0 : 0.0;
    BD_CUDA(cudaMemcpyAsync(h->scal.p, h->host_init, sizeof(double) * S_NSLOTS, cudaMemcpyHostToDevice, s));
    BD_CUDA(cudaGraphLaunch(h->graph_exec, s));
    if (x_dev != h->x.p) BD_CUDA(cudaMemcpyAsync(x_dev, h->x.p, bytes, cudaMemcpyDeviceToDevice, s));
    BD_CUDA(cudaEventRecord(h->ev_solve[1], s));
    BD_CUDA(cudaMemcpyAsync(h->host_scal, h->scal.p, sizeof(double) * S_NSLOTS, cudaMemcpyDeviceToHost, s));
    return BD_OK;
}

static int pcg_graph_finish(amg_hierarchy *h, cudaStream_t s, solve_info *info)
{
    BD_CUDA(cudaStreamSynchronize(s));
    float ms = 0.0f;
    cudaEventElapsedTime(&ms, h->ev_solve[0], h->ev_solve[1]);
    return report_from_scal(h, h->host_scal, ms, info);
}

static int pcg_solve_graph(amg_hierarchy *h, const double *f_dev, double *x_dev, int warm,
                           const solve_options *o, cudaStream_t s, solve_info *info)
{
    BD_TRY(pcg_graph_launch(h, f_dev, x_dev, warm, o, s));
    return pcg_graph_finish(h, s, info);
}

bool solve_graph_off()
{
    static const bool off = [] {
        const char *e = getenv("BD_SOLVE_GRAPH");
        return e && e[0] == '0';
    }();
    return off;
}

static bool graph_form(amg_hierarchy *h, const solve_options *o)
{
    if (h->prof || o->strict || h->graph_failed || solve_graph_off()) return false;
    if (!h->graph_exec && build_graph(h) != BD_OK) h->graph_failed = true;
    return h->graph_exec != nullptr;
}

// Split form for callers that overlap several hierarchies' solves: begin
// enqueues the solve (graph form) or runs it to completion (host-driven loop),
// end waits and reports.
int pcg_solve_begin(amg_hierarchy *h, const double *f_dev, double *x_dev, int warm,
                    const solve_options *o, cudaStream_t s, solve_info *info, bool *pending)
{
    if (graph_form(h, o)) {
        *pending = true;
        return pcg_graph_launch(h, f_dev, x_dev, warm, o, s);
    }
    *pending = false;
    return pcg_solve_loop(h, f_dev, x_dev, warm, o, s, info);
}

int pcg_solve_end(amg_hierarchy *h, cudaStream_t s, solve_info *info) { return pcg_graph_finish(h, s, info); }

// The graph form unless live kernel timing is on (its CUDA events bracket
// single launches), strict mode is requested (checked on the host before the
// loop), the graph could not be built, or BD_SOLVE_GRAPH=0 is set.
int pcg_solve_device(amg_hierarchy *h, const double *f_dev, double *x_dev, int warm,
                     const solve_options *o, cudaStream_t s, solve_info *info)
{
    if (graph_form(h, o)) return pcg_solve_graph(h, f_dev, x_dev, warm, o, s, info);
    return pcg_solve_loop(h, f_dev, x_dev, warm, o, s, info);
}

// Report of one solve from its scalar block (graph form): status, iterations,
// residuals; counts its kernel executions.
static int report_from_scal(amg_hierarchy *h, const double *sc, float ms, solve_info *info)
{
    note_launches(h->graph_pre + h->graph_post + (long long)sc[S_IT] * h->graph_body);
    return info_from_scal(sc, ms, info);
}

int info_from_scal(const double *sc, float ms, solve_info *info)
{
    const double nf = sqrt(sc[S_NF2]);
    const int status = (int)sc[S_STATUS];
    if (info) {
        info->status = status;
        info->iters = (int)sc[S_IT];
        info->rel_res = nf > 0.0 ? sqrt(sc[S_RR]) / nf : 0.0;
        info->true_rel_res = nf > 0.0 ? sqrt(sc[S_TRR]) / nf : 0.0;
        info->solve_ms = ms;
    }
    return status;
}

// ------------------------------------------------------------------ batched solves
// Many independent solves as one CUDA graph: branch k copies f_k and x_k into
// hierarchy k's buffers, runs its whole solve (capture_solve) and copies x and
// the scalar block back; the branches have no edges between them, so one
// launch runs all of them concurrently on the GPU.
struct BatchGraph {
    std::vector<amg_hierarchy *> h;
    std::vector<const double *> f;
    std::vector<double *> x;
    std::vector<cudaStream_t> st;
    std::vector<cudaEvent_t> join;
    cudaStream_t origin = nullptr, body = nullptr;
    cudaEvent_t fork = nullptr, ev[2] = {nullptr, nullptr};
    cudaGraph_t graph = nullptr;
    cudaGraphExec_t exec = nullptr;
    DBuf<double> init_dev;          // count x S_NSLOTS initial scalar blocks
    double *host_init = nullptr;    // pinned, count x S_NSLOTS
    double *host_scal = nullptr;    // pinned, count x S_NSLOTS (results)

    void drop_graph()
    {
        if (exec) cudaGraphExecDestroy(exec);
        if (graph) cudaGraphDestroy(graph);
        exec = nullptr;
        graph = nullptr;
    }
    ~BatchGraph()
    {
        drop_graph();
        for (cudaStream_t q : st) cudaStreamDestroy(q);
        for (cudaEvent_t e : join) cudaEventDestroy(e);
        if (origin) cudaStreamDestroy(origin);
        if (body) cudaStreamDestroy(body);
        if (fork) cudaEventDestroy(fork);
        if (ev[0]) cudaEventDestroy(ev[0]);
        if (ev[1]) cudaEventDestroy(ev[1]);
        if (host_init) cudaFreeHost(host_init);
        if (host_scal) cudaFreeHost(host_scal);
    }
};

static int batch_capture(BatchGraph &b)
{
    const int count = (int)b.h.size();
    BD_CUDA(cudaStreamBeginCapture(b.origin, cudaStreamCaptureModeThreadLocal));
    BD_CUDA(cudaEventRecord(b.fork, b.origin));
    for (int k = 0; k < count; k++) {
        amg_hierarchy *h = b.h[k];
        cudaStream_t s = b.st[k];
        const size_t bytes = sizeof(double) * 2 * (size_t)h->lev[0].N;
        BD_CUDA(cudaStreamWaitEvent(s, b.fork, 0));
        BD_CUDA(cudaMemcpyAsync(h->scal.p, b.init_dev.p + (size_t)k * S_NSLOTS, sizeof(double) * S_NSLOTS,
                                cudaMemcpyDeviceToDevice, s));
        BD_CUDA(cudaMemcpyAsync(h->fin.p, b.f[k], bytes, cudaMemcpyDeviceToDevice, s));
        BD_CUDA(cudaMemcpyAsync(h->x.p, b.x[k], bytes, cudaMemcpyDeviceToDevice, s));
        BD_TRY(capture_solve(h, s, b.body));
        BD_CUDA(cudaMemcpyAsync(b.x[k], h->x.p, bytes, cudaMemcpyDeviceToDevice, s));
        BD_CUDA(cudaMemcpyAsync(b.host_scal + (size_t)k * S_NSLOTS, h->scal.p, sizeof(double) * S_NSLOTS,
                                cudaMemcpyDeviceToHost, s));
        BD_CUDA(cudaEventRecord(b.join[k], s));
        BD_CUDA(cudaStreamWaitEvent(b.origin, b.join[k], 0));
    }
    BD_CUDA(cudaStreamEndCapture(b.origin, &b.graph));
    BD_CUDA(cudaGraphInstantiate(&b.exec, b.graph, 0));
    return BD_OK;
}

}  // namespace bd

using namespace bd;

struct amg_batch {
    bd::BatchGraph g;
};

extern "C" int amg_batch_create(amg_hierarchy *const *h, int count, amg_batch **out)
{
    if (!out) return BD_EINVAL;
    *out = nullptr;
    if (!h || count < 1) return BD_EINVAL;
    for (int k = 0; k < count; k++) {
        if (!h[k]) return BD_EINVAL;
        for (int j = 0; j < k; j++)
            if (h[j] == h[k]) return BD_EINVAL;  // one hierarchy's buffers serve one branch
    }
    amg_batch *b = new (std::nothrow) amg_batch();
    if (!b) return BD_ENOMEM;
    BatchGraph &g = b->g;
    g.h.assign(h, h + count);
    int st = BD_OK;
    auto ok = [&](cudaError_t e) {
        if (e != cudaSuccess && st == BD_OK) st = BD_ECUDA;
    };
    ok(cudaStreamCreateWithFlags(&g.origin, cudaStreamNonBlocking));
    ok(cudaStreamCreateWithFlags(&g.body, cudaStreamNonBlocking));
    ok(cudaEventCreateWithFlags(&g.fork, cudaEventDisableTiming));
    ok(cudaEventCreate(&g.ev[0]));
    ok(cudaEventCreate(&g.ev[1]));
    g.st.assign(count, nullptr);
    g.join.assign(count, nullptr);
    for (int k = 0; k < count && st == BD_OK; k++) {
        ok(cudaStreamCreateWithFlags(&g.st[k], cudaStreamNonBlocking));
        ok(cudaEventCreateWithFlags(&g.join[k], cudaEventDisableTiming));
    }
    const size_t nsc = (size_t)count * S_NSLOTS;
    if (st == BD_OK) st = g.init_dev.alloc(nsc);
    if (st == BD_OK) ok(cudaMallocHost((void **)&g.host_init, sizeof(double) * nsc));
    if (st == BD_OK) ok(cudaMallocHost((void **)&g.host_scal, sizeof(double) * nsc));
    if (st != BD_OK) {
        delete b;
        return st;
    }
    for (amg_hierarchy *hk : g.h) hk->batch_refs++;
    *out = b;
    return BD_OK;
}

extern "C" int amg_batch_solve(amg_batch *b, const double *const *f, double *const *x, const solve_options *opts,
                               void *stream, solve_info *info)
{
    if (!b || !f || !x) return BD_EINVAL;
    BatchGraph &g = b->g;
    const int count = (int)g.h.size();
    solve_options o;
    solve_options_default(&o);
    if (opts) o = *opts;
    if (!(o.rtol > 0.0) || o.max_it < 0 || o.strict) return BD_EINVAL;
    for (int k = 0; k < count; k++)
        if (!f[k] || !x[k]) return BD_EINVAL;
    // the graph is tied to the vectors it copies from and to
    bool same = g.exec != nullptr;
    for (int k = 0; k < count && same; k++) same = g.f[k] == f[k] && g.x[k] == x[k];
    if (!same) {
        g.drop_graph();
        g.f.assign(f, f + count);
        g.x.assign(x, x + count);
        const int st = batch_capture(g);
        if (st != BD_OK) {
            drop_capture(g.body);
            for (cudaStream_t q : g.st) drop_capture(q);
            drop_capture(g.origin);
            g.drop_graph();
            return st;
        }
    }
    cudaStream_t s = (cudaStream_t)stream;
    for (int k = 0; k < count; k++) {
        double *hi = g.host_init + (size_t)k * S_NSLOTS;
        for (int i = 0; i < S_NSLOTS; i++) hi[i] = 0.0;
        hi[S_RTOL] = o.rtol;
        hi[S_MAXIT] = (double)o.max_it;
        hi[S_WARM] = o.warm_start ? 1.0 : 0.0;
    }
    BD_CUDA(cudaMemcpyAsync(g.init_dev.p, g.host_init, sizeof(double) * count * S_NSLOTS,
                            cudaMemcpyHostToDevice, s));
    BD_CUDA(cudaEventRecord(g.ev[0], s));
    BD_CUDA(cudaGraphLaunch(g.exec, s));
    BD_CUDA(cudaEventRecord(g.ev[1], s));
    BD_CUDA(cudaStreamSynchronize(s));
    float ms = 0.0f;
    cudaEventElapsedTime(&ms, g.ev[0], g.ev[1]);
    int worst = BD_OK;
    for (int k = 0; k < count; k++) {
        const int stk = report_from_scal(g.h[k], g.host_scal + (size_t)k * S_NSLOTS, ms, info ? info + k : nullptr);
        if (stk != BD_OK && worst == BD_OK) worst = stk;
    }
    return worst;
}

extern "C" void amg_batch_destroy(amg_batch *b)
{
    if (!b) return;
    for (amg_hierarchy *hk : b->g.h) hk->batch_refs--;
    delete b;
}

extern "C" int amg_set_level_lanes(amg_hierarchy *h, int level, const int lanes[3], void *stream)
{
    if (!h || !lanes || level < 0 || level >= h->nlev) return BD_EINVAL;
    if (h->batch_refs > 0) return BD_ESTATE;
    Level &L = h->lev[level];
    const bool last = level == h->nlev - 1;
    for (int op = 0; op < 3; op++) {
        const int T = lanes[op];
        if (T == 0) continue;
        const bool applied = !last && !(op == 0 && level == 0 && h->fine.valid);
        const bool csr_ok = T > 0 && T <= 256 && (T & (T - 1)) == 0;
        const bool sliced_ok = T < 0 && sliced_k_ok(-T) && !(op == 0 && level == 0);
        if (!applied || !(csr_ok || sliced_ok)) return BD_EINVAL;
    }
    cudaStream_t s = (cudaStream_t)stream;
    BD_CUDA(cudaStreamSynchronize(s));
    // The captured whole-solve graph holds the old launches and buffers: drop
    // it before any buffer changes, so that no error return below leaves a
    // graph that reads freed or rebuilt memory (the next solve captures anew).
    if (h->graph_exec) cudaGraphExecDestroy(h->graph_exec);
    if (h->graph) cudaGraphDestroy(h->graph);
    h->graph_exec = nullptr;
    h->graph = nullptr;
    h->graph_failed = false;
    for (int op = 0; op < 3; op++) {
        const int T = lanes[op];
        if (T == 0) continue;
        const BSR &M = op == 0 ? L.A : (op == 1 ? L.R : L.P);
        if (T < 0) {
            const int rc = build_op(L, op, -T, h->prec32, s);
            if (rc != BD_OK) {
                // a half-built sliced form is unusable: fall back to the
                // block-CSR form the rule gives, which needs no extra buffers
                drop_sliced(L.sl[op]);
                L.lanes[op] = lanes_for(M, h->prec32);
                return rc;
            }
        } else {
            drop_sliced(L.sl[op]);
        }
        L.lanes[op] = T;
        scalar_set_lanes(h, level, op, T);
    }
    return BD_OK;
}

extern "C" int amg_vcycle(amg_hierarchy *h, const double *r, double *z, int on_device, void *stream)
{
    if (!h || !r || !z) return BD_EINVAL;
    cudaStream_t s = (cudaStream_t)stream;
    size_t bytes = sizeof(double) * 2 * (size_t)h->lev[0].N;
    if (on_device) {
        BD_TRY(vcycle_device(h, r, z, s));
        BD_CUDA(cudaStreamSynchronize(s));
        prof_collect(h);
        return BD_OK;
    }
    BD_TRY(copy_in(h->r.p, r, bytes, 0, s));
    BD_TRY(vcycle_device(h, h->r.p, h->z.p, s));
    BD_TRY(copy_out(z, h->z.p, bytes, 0, s));
    BD_CUDA(cudaStreamSynchronize(s));
    prof_collect(h);
    return BD_OK;
}

extern "C" int amg_profile_enable(amg_hierarchy *h, int enable)
{
    if (!h || enable < 0 || enable > 2) return BD_EINVAL;
    prof_collect(h);
    if (enable && !h->prof) {  // fresh sums when switched on
        h->prof_sum = amg_kernel_profile{};
        for (int i = 0; i < 256; i++) {
            h->trace_ms[i] = 0.0;
            h->trace_n[i] = 0;
        }
    }
    h->prof = enable;
    return BD_OK;
}

extern "C" int amg_profile_breakdown(const amg_hierarchy *h, double *ms, long long *count)
{
    if (!h || !ms || !count) return BD_EINVAL;
    for (int i = 0; i < 256; i++) {
        ms[i] = h->trace_ms[i];
        count[i] = h->trace_n[i];
    }
    return BD_OK;
}

extern "C" int amg_profile_read(const amg_hierarchy *h, amg_kernel_profile *out)
{
    if (!h || !out) return BD_EINVAL;
    *out = h->prof_sum;
    out->precision = h->prec32 ? 1 : 0;
    return BD_OK;
}

extern "C" int amg_solve(amg_hierarchy *h, const double *f, double *x, int on_device,
                         const solve_options *opts, void *stream, solve_info *info)
{
    if (!h || !f || !x) return BD_EINVAL;
    solve_options o;
    solve_options_default(&o);
    if (opts) o = *opts;
    if (!(o.rtol > 0.0) || o.max_it < 0) return BD_EINVAL;
    cudaStream_t s = (cudaStream_t)stream;
    size_t bytes = sizeof(double) * 2 * (size_t)h->lev[0].N;
    if (on_device) return pcg_solve_device(h, f, x, o.warm_start, &o, s, info);
    // host arrays: f and x are staged in device buffers
    DBuf<double> fdev;
    BD_TRY(fdev.alloc(2 * (size_t)h->lev[0].N));
    BD_TRY(copy_in(fdev.p, f, bytes, 0, s));
    if (o.warm_start) BD_TRY(copy_in(h->x.p, x, bytes, 0, s));
    int st = pcg_solve_device(h, fdev.p, h->x.p, o.warm_start, &o, s, info);
    BD_TRY(copy_out(x, h->x.p, bytes, 0, s));
    BD_CUDA(cudaStreamSynchronize(s));
    return st;
}
