// amg_stack.cu -- the stacked batch (many hierarchies solved together).
//
// Level l of a stack holds level l of every member hierarchy that has one,
// the members' operators placed block-diagonally and their vectors end to
// end, so each step of the V-cycle (Algorithm 2: Chebyshev pre-smoothing,
// residual, restriction, coarsest solve, prolongation, post-smoothing) is one
// kernel launch over all members instead of one launch per member.  Within a
// level the members that smooth there come first (rows [0, Ns)), the members
// whose coarsest level it is follow; their dense solves run together in one
// launch (a warp per row).  The projected PCG of Section 2.2
// keeps its scalars per member (null-space means, alpha, beta, residual norm,
// the stopping test): every reduction runs over chunks of at most kStChunk
// nodes that never span two members, and the last block to finish adds each
// member's chunk sums in chunk order, so the result does not depend on
// scheduling.  One CUDA graph per batch solve: the iteration body under a
// WHILE node whose condition the last reduction of an iteration sets on the
// device (some member still iterating); members that have converged, broken
// down or reached max_it keep their iterate.
#include <algorithm>
#include <cmath>
#include <new>
#include <type_traits>
#include <vector>

#include "amg_bsr.cuh"
#include "amg_internal.cuh"
#include "fine_stencil.cuh"

namespace bd {
namespace {

constexpr int kStChunk = 1024;   // nodes per reduction chunk
constexpr int kStThreads = 256;  // threads of the reduction and vector kernels

// per-member device scalars
enum {
    T_MEANF = 0, T_NF2, T_RR, T_RZ, T_PQ, T_ALPHA, T_BETA, T_MEANZ, T_BREAK, T_IT, T_STATUS,
    T_ACTIVE, T_TRR, T_MEANX, T_RTOL, T_MAXIT, T_WARM, T_NSLOTS
};

// node -> member, and each member's Chebyshev coefficients on one level:
// coef[4k] = 1/theta, coef[4k+1] = c1, coef[4k+2] = c2
struct StCoef {
    const int *__restrict__ mem;
    const double *__restrict__ coef;
    __device__ __forceinline__ const double *at(int p) const { return coef + 4 * mem[p]; }
};

// Epilogues of the stacked V-cycle: the single-hierarchy Chebyshev steps
// (Saad, Alg. 12.1 on D^{-1}A, degree 2) with the coefficients of the row's
// member.
template <class S> struct StPre {  // from zero: u = d0 + (c1 d0 + c2 D^{-1} (f - A d0))
    const v2<S> *__restrict__ f;
    const v2<S> *__restrict__ invd;
    const v2<S> *__restrict__ d0;
    v2<S> *__restrict__ u;
    StCoef c;
    __device__ __forceinline__ void operator()(int p, S y0, S y1) const
    {
        const double *k = c.at(p);
        const S c1 = narrow_to<S>(k[1]), c2 = narrow_to<S>(k[2]);
        const v2<S> fp = f[p], id = invd[p], dp = d0[p];
        const S r0 = fp.x - y0, r1 = fp.y - y1;
        u[p] = V2<S>::mk(dp.x + (c1 * dp.x + c2 * id.x * r0), dp.y + (c1 * dp.y + c2 * id.y * r1));
    }
};
template <class S> struct StResid {  // r = f - A u
    const v2<S> *__restrict__ f;
    v2<S> *__restrict__ r;
    __device__ __forceinline__ void operator()(int p, S y0, S y1) const
    {
        const v2<S> fp = f[p];
        r[p] = V2<S>::mk(fp.x - y0, fp.y - y1);
    }
};
template <class S> struct StStoreD0 {  // f_c = R r and d0_c = D_c^{-1} f_c / theta_c
    v2<S> *__restrict__ f;
    v2<S> *__restrict__ d0;
    const v2<S> *__restrict__ invd;
    StCoef c;
    __device__ __forceinline__ void operator()(int p, S y0, S y1) const
    {
        const S it = narrow_to<S>(c.at(p)[0]);
        const v2<S> id = invd[p];
        f[p] = V2<S>::mk(y0, y1);
        d0[p] = V2<S>::mk(y0 * id.x * it, y1 * id.y * it);
    }
};
template <class S> struct StAdd {  // u += P e_c
    v2<S> *__restrict__ u;
    __device__ __forceinline__ void operator()(int p, S y0, S y1) const
    {
        const v2<S> a = u[p];
        u[p] = V2<S>::mk(a.x + y0, a.y + y1);
    }
};
template <class S> struct StPost1 {  // r = f - A u, d = D^{-1} r / theta, w = u + d
    const v2<S> *__restrict__ f;
    const v2<S> *__restrict__ invd;
    const v2<S> *__restrict__ u;
    v2<S> *__restrict__ r;
    v2<S> *__restrict__ d;
    v2<S> *__restrict__ w;
    StCoef c;
    __device__ __forceinline__ void operator()(int p, S y0, S y1) const
    {
        const S it = narrow_to<S>(c.at(p)[0]);
        const v2<S> fp = f[p], id = invd[p], up = u[p];
        const S r0 = fp.x - y0, r1 = fp.y - y1;
        const S d0 = r0 * id.x * it, d1 = r1 * id.y * it;
        r[p] = V2<S>::mk(r0, r1);
        d[p] = V2<S>::mk(d0, d1);
        w[p] = V2<S>::mk(up.x + d0, up.y + d1);
    }
};
template <class S> struct StPost2 {  // u = w + (c1 d + c2 D^{-1} (r - A d))
    const v2<S> *__restrict__ r;
    const v2<S> *__restrict__ d;
    const v2<S> *__restrict__ invd;
    const v2<S> *__restrict__ w;
    v2<S> *__restrict__ u;
    StCoef c;
    __device__ __forceinline__ void operator()(int p, S y0, S y1) const
    {
        const double *k = c.at(p);
        const S c1 = narrow_to<S>(k[1]), c2 = narrow_to<S>(k[2]);
        const v2<S> rp_ = r[p], dp = d[p], id = invd[p], wp = w[p];
        const S r0 = rp_.x - y0, r1 = rp_.y - y1;
        u[p] = V2<S>::mk(wp.x + (c1 * dp.x + c2 * id.x * r0), wp.y + (c1 * dp.y + c2 * id.y * r1));
    }
};
struct StStore {  // q = A p (FP64, PCG)
    double2 *__restrict__ q;
    __device__ __forceinline__ void operator()(int p, double y0, double y1) const { q[p] = make_double2(y0, y1); }
};

// u += P e_c on a stencil finest level, P in pair form (PairOp): kappa scales
// the row; u in (v + u, u) form in FP64
template <class S, bool SU> struct StAddPair {
    v2<S> *__restrict__ u;
    const v2<S> *__restrict__ kappa;
    __device__ __forceinline__ void operator()(int p, S y0, S y1) const
    {
        const v2<S> a = u[p], k = kappa[p];
        const S e1 = k.y * y1;
        u[p] = V2<S>::mk(SU ? a.x + fma(k.x, y0, e1) : a.x + k.x * y0, a.y + e1);
    }
};

// ------------------------------------------------------------------ assembly of the stack
__global__ void k_st_shift(long long n, const int *__restrict__ src, int *__restrict__ dst, int add)
{
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x)
        dst[i] = src[i] + add;
}
__global__ void k_st_fill(long long n, int *__restrict__ dst, int v)
{
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x)
        dst[i] = v;
}

__global__ void k_st_f32(long long n, const double *__restrict__ src, float *__restrict__ dst)
{
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x)
        dst[i] = (float)src[i];
}

// ------------------------------------------------------------------ coarsest levels
struct StCoarseJob {
    const double *C;     // n x n projected inverse of the member's coarsest operator
    int n;               // unknowns
    int level;           // stack level holding the member's coarsest level
    long long off;       // first unknown of the member on that level
};
template <class S> struct StLevelPtrs {
    S *f[kMaxLevels];
    S *u[kMaxLevels];
};

// x = C r in FP64 for every member at once (blockIdx.y: the member), a warp per
// row, as the single-hierarchy coarsest solve.
template <class S>
__global__ void __launch_bounds__(128) k_st_coarse(const StCoarseJob *__restrict__ jobs, StLevelPtrs<S> lp)
{
    const StCoarseJob J = jobs[blockIdx.y];
    const int lane = threadIdx.x & 31, i = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    if (i >= J.n) return;
    const v2<S> *r = (const v2<S> *)(lp.f[J.level] + J.off);
    const double2 *row = (const double2 *)(J.C + (size_t)i * J.n);
    double s0 = 0.0, s1 = 0.0;
#pragma unroll 4
    for (int j = lane; j < J.n / 2; j += 32) {
        const double2 c = row[j];
        const v2<S> v = r[j];
        s0 = fma(c.x, widen(v.x), s0);
        s1 = fma(c.y, widen(v.y), s1);
    }
    s0 += s1;
    for (int o = 16; o; o >>= 1) s0 += __shfl_xor_sync(0xffffffffu, s0, o);
    if (lane == 0) lp.u[J.level][J.off + i] = (S)s0;
}

// ------------------------------------------------------------------ PCG reductions
// Context of the per-member reductions on the finest level.
struct StRed {
    double *scal;                  // count x T_NSLOTS
    double *part;                  // chunks x 4
    unsigned int *counter;
    const int *cmem, *cbeg, *cend; // member and node range of each chunk
    const int *mc0, *mc1;          // chunk range of each member
    const int *nn;                 // finest-level nodes of each member
    int count, flex;
    cudaGraphConditionalHandle cond;
};

// Vectors of the finest level (FP64 PCG vectors in (v, u) pairs; the V-cycle's
// input f0, d0 and output u0 in its precision S).
template <class S> struct StPcg {
    const double2 *fin;
    double2 *fp, *x, *r, *p, *q;
    v2<S> *f0, *d0;
    v2<S> *uold;                   // FP32 V-cycle: its previous output (flexible beta)
    const v2<S> *u0, *invd0;
    StCoef c0;
    const int *mem;                // finest-level node -> member
    int psu;                       // p stored as (v + u, u) (stencil finest level)
    int dsu;                       // FP64 V-cycle: d0 stored as (v + u, u)
};

enum { R_FSTATS = 0, R_PROJF, R_INIT, R_ZSTATS, R_PQ, R_XR, R_TRUE };

// V-cycle input from the residual: f0 = r (FP32 copy; the FP64 V-cycle reads
// r itself) and d0 = D^{-1} r / theta.
template <class S>
__device__ __forceinline__ void st_vin(const StPcg<S> &v, int i, double2 ri)
{
    const double it = v.c0.at(i)[0];
    const S rv = narrow_to<S>(ri.x), ru = narrow_to<S>(ri.y), itS = narrow_to<S>(it);
    if (sizeof(S) == 4) v.f0[i] = V2<S>::mk(rv, ru);
    const v2<S> id = v.invd0[i];
    const S dv = rv * id.x * itS, du = ru * id.y * itS;
    v.d0[i] = V2<S>::mk(v.dsu ? dv + du : dv, du);
}

// Per-member totals -> scalars (last block, one thread per member).  Returns
// whether the member keeps iterating (stages that open or close an iteration).
__device__ bool st_finish(int MODE, const StRed &R, int k, double a, double b, double c, double d)
{
    double *sc = R.scal + (size_t)k * T_NSLOTS;
    const double N = (double)R.nn[k];
    switch (MODE) {
    case R_FSTATS:
        sc[T_MEANF] = a / N;
        return false;
    case R_PROJF:
        sc[T_NF2] = a;
        return false;
    case R_INIT: {
        sc[T_RR] = a;
        const double nf = sqrt(sc[T_NF2]);
        const bool go = nf > 0.0 && !(sqrt(a) <= sc[T_RTOL] * nf) && sc[T_MAXIT] > 0.0;
        sc[T_IT] = 0.0;
        sc[T_BREAK] = 0.0;
        sc[T_STATUS] = go ? (double)BD_ENOTCONV : (double)BD_OK;
        sc[T_ACTIVE] = go ? 1.0 : 0.0;
        return go;
    }
    case R_ZSTATS: {
        if (sc[T_ACTIVE] == 0.0) return false;
        const double mz = a / N, rz = c - mz * b;  // r . (z projected)
        const double num = R.flex ? rz - d : rz;   // flexible (Polak-Ribiere) or standard beta
        sc[T_MEANZ] = mz;
        sc[T_BETA] = sc[T_IT] == 0.0 ? 0.0 : num / sc[T_RZ];
        sc[T_RZ] = rz;
        return false;
    }
    case R_PQ: {
        if (sc[T_ACTIVE] == 0.0) return false;
        sc[T_PQ] = a;
        if (!(a > 0.0) || !isfinite(a) || !isfinite(sc[T_RZ])) sc[T_BREAK] = 1.0;
        sc[T_ALPHA] = sc[T_RZ] / a;
        return false;
    }
    case R_XR: {
        if (sc[T_ACTIVE] == 0.0) return false;
        sc[T_RR] = a;
        const double it = sc[T_IT] + 1.0;
        sc[T_IT] = it;
        const double nf = sqrt(sc[T_NF2]), rr = sqrt(a);
        bool go = true;
        if (sc[T_BREAK] != 0.0 || !isfinite(rr)) {
            sc[T_STATUS] = (double)BD_EBREAKDOWN;
            go = false;
        } else if (rr <= sc[T_RTOL] * nf) {
            sc[T_STATUS] = (double)BD_OK;
            go = false;
        } else if (it >= sc[T_MAXIT]) {
            go = false;  // status stays BD_ENOTCONV
        }
        sc[T_ACTIVE] = go ? 1.0 : 0.0;
        return go;
    }
    case R_TRUE:
        sc[T_TRR] = a;
        sc[T_MEANX] = b / N;
        return false;
    }
    return false;
}

// One block per chunk: the chunk's sums (in a fixed order: every thread's
// nodes ascending, then warp k adds column k of the block's values) go to
// part[chunk]; the last block to arrive adds each member's chunks in chunk
// order and applies the stage.  Element-wise work of the stage rides along.
template <int MODE, class S>
__global__ void __launch_bounds__(kStThreads) k_st_red(StRed R, StPcg<S> v)
{
    constexpr int NV = (MODE == R_ZSTATS) ? 4 : ((MODE == R_TRUE) ? 2 : 1);
    __shared__ double buf[NV][kStThreads];
    __shared__ double tot[4];
    __shared__ bool last;
    const int c = blockIdx.x;
    const int m = R.cmem[c];
    const double *sc = R.scal + (size_t)m * T_NSLOTS;
    double acc[4] = {0.0, 0.0, 0.0, 0.0};
    const int b = R.cbeg[c], e = R.cend[c];
    if (MODE == R_FSTATS) {
        for (int i = b + threadIdx.x; i < e; i += blockDim.x) acc[0] += v.fin[i].y;
    } else if (MODE == R_PROJF) {
        const double mf = sc[T_MEANF];
        const bool warm = sc[T_WARM] != 0.0;
        for (int i = b + threadIdx.x; i < e; i += blockDim.x) {
            double2 f = v.fin[i];
            f.y -= mf;
            v.fp[i] = f;
            if (!warm) v.x[i] = make_double2(0.0, 0.0);
            acc[0] += f.x * f.x + f.y * f.y;
        }
    } else if (MODE == R_INIT) {  // q = A x already formed
        for (int i = b + threadIdx.x; i < e; i += blockDim.x) {
            const double2 f = v.fp[i], q = v.q[i];
            const double2 ri = make_double2(f.x - q.x, f.y - q.y);
            v.r[i] = ri;
            st_vin<S>(v, i, ri);
            acc[0] += ri.x * ri.x + ri.y * ri.y;
        }
    } else if (MODE == R_ZSTATS) {
        if (sc[T_ACTIVE] != 0.0) {
            const double mzo = sc[T_MEANZ];
            for (int i = b + threadIdx.x; i < e; i += blockDim.x) {
                const v2<S> u = v.u0[i];
                const double2 zi = make_double2(widen(u.x), widen(u.y)), ri = v.r[i];
                acc[0] += zi.y;
                acc[1] += ri.y;
                acc[2] = fma(ri.x, zi.x, fma(ri.y, zi.y, acc[2]));
                if (R.flex) {
                    // the previous z: its FP32 values less their mean (still in T_MEANZ)
                    const v2<S> o = v.uold[i];
                    acc[3] = fma(ri.x, widen(o.x), fma(ri.y, widen(o.y) - mzo, acc[3]));
                }
            }
        }
    } else if (MODE == R_PQ) {  // q = A p already formed
        if (sc[T_ACTIVE] != 0.0)
            for (int i = b + threadIdx.x; i < e; i += blockDim.x) {
                const double2 p = v.p[i], q = v.q[i];
                const double pv = v.psu ? p.x - p.y : p.x;
                acc[0] = fma(pv, q.x, fma(p.y, q.y, acc[0]));
            }
    } else if (MODE == R_XR) {
        if (sc[T_ACTIVE] != 0.0) {
            const double al = sc[T_ALPHA];
            for (int i = b + threadIdx.x; i < e; i += blockDim.x) {
                const double2 p = v.p[i], q = v.q[i];
                double2 xi = v.x[i], ri = v.r[i];
                xi.x += al * (v.psu ? p.x - p.y : p.x);
                xi.y += al * p.y;
                ri.x -= al * q.x;
                ri.y -= al * q.y;
                v.x[i] = xi;
                v.r[i] = ri;
                st_vin<S>(v, i, ri);
                acc[0] = fma(ri.x, ri.x, fma(ri.y, ri.y, acc[0]));
            }
        }
    } else if (MODE == R_TRUE) {  // q = A x of the final iterate
        for (int i = b + threadIdx.x; i < e; i += blockDim.x) {
            const double2 f = v.fp[i], q = v.q[i], xi = v.x[i];
            const double t0 = f.x - q.x, t1 = f.y - q.y;
            acc[0] += t0 * t0 + t1 * t1;
            acc[1] += xi.y;
        }
    }
    // block sums in a fixed order
#pragma unroll
    for (int k = 0; k < NV; k++) buf[k][threadIdx.x] = acc[k];
    __syncthreads();
    {
        const int w = threadIdx.x >> 5, l = threadIdx.x & 31;
        if (w < NV) {
            double t = buf[w][l];
            for (int i = l + 32; i < kStThreads; i += 32) t += buf[w][i];
            for (int o = 16; o; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
            if (l == 0) tot[w] = t;
        }
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        double *o = R.part + 4 * (size_t)c;
#pragma unroll
        for (int k = 0; k < NV; k++) o[k] = tot[k];
        __threadfence();
        const unsigned int ticket = atomicAdd(R.counter, 1u);
        last = ticket == gridDim.x - 1;
    }
    __syncthreads();
    if (!last) return;
    __threadfence();
    bool go = false;
    for (int k = threadIdx.x; k < R.count; k += blockDim.x) {
        double s[4] = {0.0, 0.0, 0.0, 0.0};
        for (int cc = R.mc0[k]; cc < R.mc1[k]; cc++) {
            const double *q = R.part + 4 * (size_t)cc;
#pragma unroll
            for (int j = 0; j < NV; j++) s[j] += __ldcg(q + j);
        }
        go |= st_finish(MODE, R, k, s[0], s[1], s[2], s[3]);
    }
    go = __syncthreads_or(go);
    if (threadIdx.x == 0) {
        if (MODE == R_INIT || MODE == R_XR) cudaGraphSetConditional(R.cond, go ? 1u : 0u);
        *R.counter = 0u;
    }
}

// p = z - mean(z_u) e_u (first iteration) or that + beta p, stored in (v + u, u)
// form when psu; z is the V-cycle's output, kept in FP32 for the next flexible
// beta.  Members no longer iterating keep p.
template <class S>
__global__ void k_st_p(int N, StPcg<S> v, const double *__restrict__ scal)
{
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < N; i += gridDim.x * blockDim.x) {
        const int m = v.mem[i];
        if (m < 0) continue;  // padding after a member's last node
        const double *sc = scal + (size_t)m * T_NSLOTS;
        if (sc[T_ACTIVE] == 0.0) continue;
        const v2<S> u = v.u0[i];
        if (v.uold) v.uold[i] = u;
        const double zx = widen(u.x), zy = widen(u.y) - sc[T_MEANZ];
        const double2 zs = make_double2(v.psu ? zx + zy : zx, zy);
        if (sc[T_IT] == 0.0) {
            v.p[i] = zs;
        } else {
            const double beta = sc[T_BETA];
            const double2 pi = v.p[i];
            v.p[i] = make_double2(zs.x + beta * pi.x, zs.y + beta * pi.y);
        }
    }
}

// x <- x - mean(x_u) e_u (mean-zero u_e), or zero for a zero right-hand side.
__global__ void k_st_project_x(int N, double2 *__restrict__ x, const int *__restrict__ mem,
                               const double *__restrict__ scal)
{
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < N; i += gridDim.x * blockDim.x) {
        if (mem[i] < 0) continue;  // padding
        const double *sc = scal + (size_t)mem[i] * T_NSLOTS;
        double2 xi = x[i];
        if (!(sc[T_NF2] > 0.0)) xi = make_double2(0.0, 0.0);
        else xi.y -= sc[T_MEANX];
        x[i] = xi;
    }
}

}  // namespace

// ------------------------------------------------------------------ stack levels
struct StLevel {
    int N = 0;                 // nodes of the members present on this level
    int Ns = 0;                // nodes of the members that smooth here: rows [0, Ns)
    int rowsA = 0;             // rows of the stacked A (N on the finest level, Ns below)
    BSR A, R, P;               // FP64 values (A of the finest level always: the PCG's A p)
    DBuf<float> A32, R32, P32; // FP32 V-cycle values
    // a stencil finest level: R and P in pair form (their A32, P32 stay empty)
    PairOp pair[2];
    DBuf<double> kappa;
    DBuf<float> kappa32;
    int lanes[3] = {0, 0, 0};
    DBuf<int> mem;             // member of each node
    DBuf<double> coef;         // 3 per member
    DBuf<double> f, u, r, d, w, invd;          // FP64 V-cycle (f unused on the finest level)
    DBuf<float> f32, u32, r32, d32, w32, invd32;
    // finest level only, when every member's is a stencil: the members' packed
    // tables and, per V-cycle precision, their grids in stack order (the first
    // nsmooth smooth; the PCG applies all of them in FP64)
    bool fine = false, sym = false;
    int nsmooth = 0;
    long long units = 0, units_smooth = 0;
    DBuf<double> tab;
    DBuf<float> tab32;
    DBuf<FineGrid> grid, grid32;
    // FP64 V-cycle on the stencil finest level: its gathered vectors in
    // (v + u, u) form
    bool su = false;
};

}  // namespace bd

using namespace bd;

struct amg_stack {
    int count = 0;
    bool p32 = false;
    int L = 0;                                // stack levels
    std::vector<amg_hierarchy *> h;
    StLevel lev[kMaxLevels];
    std::vector<int> nlev;                    // levels of each member
    std::vector<long long> off0;              // first node of each member on the finest level
    std::vector<int> n0;                      // finest-level nodes of each member
    DBuf<StCoarseJob> jobs;
    int max_nc = 0;
    // PCG on the finest level
    DBuf<double> fin, x, r, p, q, fp;
    DBuf<float> uold;
    DBuf<int> cmem, cbeg, cend, mc0, mc1, nn;
    int nchunks = 0;
    DBuf<double> part, scal;
    DBuf<unsigned int> counter;
    double *host_init = nullptr, *host_scal = nullptr;
    // graph of one batch solve
    std::vector<const double *> gf;
    std::vector<double *> gx;
    cudaGraph_t graph = nullptr;
    cudaGraphExec_t exec = nullptr;
    cudaStream_t cap = nullptr, cap2 = nullptr;
    cudaEvent_t ev[2] = {nullptr, nullptr};
    long long n_pre = 0, n_body = 0, n_post = 0;

    void drop_graph()
    {
        if (exec) cudaGraphExecDestroy(exec);
        if (graph) cudaGraphDestroy(graph);
        exec = nullptr;
        graph = nullptr;
    }
    ~amg_stack()
    {
        drop_graph();
        if (cap) cudaStreamDestroy(cap);
        if (cap2) cudaStreamDestroy(cap2);
        if (ev[0]) cudaEventDestroy(ev[0]);
        if (ev[1]) cudaEventDestroy(ev[1]);
        if (host_init) cudaFreeHost(host_init);
        if (host_scal) cudaFreeHost(host_scal);
        for (amg_hierarchy *hk : h) hk->batch_refs--;
    }
};

namespace bd {
namespace {

// One member's block rows [0, nbr) of M appended to the stacked operator at
// row `row0` / block `blk0`, its columns shifted by `col0`: full blocks (FP64
// and/or FP32 values), or M's pair form into OP.
int st_append(const BSR &M, int nbr, const float *v32, const PairOp *pr, BSR &O, DBuf<float> *O32, PairOp *OP, int row0,
              long long blk0, int col0, bool fp64, cudaStream_t s)
{
    if (nbr <= 0) return BD_OK;
    int nb = 0;
    BD_CUDA(cudaMemcpyAsync(&nb, M.rp.p + nbr, sizeof(int), cudaMemcpyDeviceToHost, s));
    BD_CUDA(cudaStreamSynchronize(s));
    k_st_shift<<<grid_for(nbr, 256), 256, 0, s>>>(nbr, M.rp.p, O.rp.p + row0, (int)blk0); ::bd::note_launch();
    auto copy = [&](auto *dst, const auto *src, int per) {
        return cudaMemcpyAsync(dst + per * blk0, src, sizeof(*dst) * per * (size_t)nb, cudaMemcpyDeviceToDevice, s);
    };
    if (nb > 0) {
        // (an own entry's column keeps its sign bit: q + col0 < 2^31)
        k_st_shift<<<grid_for(nb, 256), 256, 0, s>>>(nb, pr ? pr->ci.p : M.ci.p, (pr ? OP->ci.p : O.ci.p) + blk0, col0);
        ::bd::note_launch();
        if (pr && O32) {
            BD_CUDA(copy(OP->v32.p, pr->v32.p, 2));
            BD_CUDA(copy(OP->alpha32.p, pr->alpha32.p, 1));
        } else if (pr) {
            BD_CUDA(copy(OP->v.p, pr->v.p, 2));
            BD_CUDA(copy(OP->alpha.p, pr->alpha.p, 1));
        } else {
            if (fp64) BD_CUDA(copy(O.v.p, M.v.p, 4));
            if (O32 && v32) {
                BD_CUDA(copy(O32->p, v32, 4));
            } else if (O32) {  // a stencil finest level keeps no FP32 blocks (stacked with a block-CSR one)
                k_st_f32<<<grid_for(4LL * nb, 256), 256, 0, s>>>(4LL * nb, M.v.p, O32->p + 4 * blk0);
                ::bd::note_launch();
            }
        }
    }
    BD_LAUNCH_CHECK();
    return BD_OK;
}

// Stacked operator over `rows` (member list with each member's block rows,
// first node on the row level and first node on the column level).
struct StPart {
    const BSR *M;
    const float *v32;
    const PairOp *pr;  // pair form to stack instead of the blocks (all parts, or none)
    int nbr;
    long long row0;
    long long col0;
};
// rows: the stacked operator's rows, the parts' rows at their row0 (ascending)
// and empty rows in between (the finest level's padding to multiples of 32)
int st_build(const std::vector<StPart> &parts, long long rows, int ncols, bool fp64, bool fp32, BSR &O,
             DBuf<float> &O32, PairOp *OP, cudaStream_t s)
{
    long long blocks = 0;
    for (const StPart &pt : parts) blocks += pt.nbr > 0 ? pt.M->nb : 0;  // full operators: nbr == M->nbr
    if (rows > 2147483647LL || blocks > 2147483647LL) return BD_ERANGE;
    O.nbr = (int)rows;
    O.nbc = ncols;
    O.nb = blocks;
    const size_t nb = (size_t)std::max<long long>(blocks, 1);
    const bool pairs = OP && !parts.empty() && parts[0].pr;
    BD_TRY(O.rp.alloc((size_t)rows + 1));
    if (pairs) {
        BD_TRY(OP->ci.alloc(nb));
        if (fp32) {
            BD_TRY(OP->v32.alloc(2 * nb));
            BD_TRY(OP->alpha32.alloc(nb));
        } else {
            BD_TRY(OP->v.alloc(2 * nb));
            BD_TRY(OP->alpha.alloc(nb));
        }
        OP->valid = true;
    } else {
        BD_TRY(O.ci.alloc(nb));
        if (fp64) BD_TRY(O.v.alloc(4 * nb));
        if (fp32) BD_TRY(O32.alloc(4 * nb));
    }
    long long blk = 0, next = 0;
    for (const StPart &pt : parts) {
        if (pt.nbr <= 0) continue;
        if (pt.row0 > next) {  // empty rows before this part
            k_st_fill<<<grid_for(pt.row0 - next, 256), 256, 0, s>>>(pt.row0 - next, O.rp.p + next, (int)blk);
            ::bd::note_launch();
        }
        BD_TRY(st_append(*pt.M, pt.nbr, pt.v32, pairs ? pt.pr : nullptr, O, fp32 ? &O32 : nullptr, OP, (int)pt.row0, blk,
                         (int)pt.col0, fp64, s));
        blk += pt.M->nb;
        next = pt.row0 + pt.nbr;
    }
    k_st_fill<<<grid_for(rows + 1 - next, 256), 256, 0, s>>>(rows + 1 - next, O.rp.p + next, (int)blocks);
    ::bd::note_launch();
    BD_LAUNCH_CHECK();
    return BD_OK;
}

// The members' stencils as one launch: tables packed in one form (symmetric
// only if every member's is) and each member's first node and work unit.
int st_fine_build(amg_stack *b, const std::vector<int> &order, const std::vector<long long> &off, cudaStream_t s)
{
    StLevel &S = b->lev[0];
    S.sym = true;
    size_t rows = 0;
    for (int k : order) {
        S.sym = S.sym && b->h[k]->fine.sym;
        rows += 9 * (size_t)b->h[k]->fine.NZ;
    }
    const size_t len = 2 * (size_t)fine_row_len(S.sym);
    BD_TRY(S.tab.alloc(rows * len));
    if (b->p32) BD_TRY(S.tab32.alloc(rows * len));
    std::vector<FineGrid> g64, g32;
    size_t at = 0;
    long long units = 0;
    for (int k : order) {
        const FineStencil &F = b->h[k]->fine;
        const Level &L0 = b->h[k]->lev[0];
        double *t64 = S.tab.p + at * len;
        float *t32 = b->p32 ? S.tab32.p + at * len : nullptr;
        BD_TRY(fine_pack(F, S.sym, L0.ch_c2, L0.ch_inv_theta, fine_omega(L0), t64, t32, s));
        FineGrid g = fine_grid<double>(F, L0.ch_c1);
        g.off = (int)off[k];
        g.unit0 = (int)units;
        g.tab = t64;
        g64.push_back(g);
        g.tab = t32;
        g32.push_back(g);
        units += (long long)g.ncb * g.NZ;
        if (units > 2147483647LL) return BD_ERANGE;
        at += 9 * (size_t)F.NZ;
        if (b->nlev[k] > 1) {
            S.nsmooth++;
            S.units_smooth = units;
        }
    }
    S.units = units;
    BD_TRY(S.grid.alloc(g64.size()));
    BD_TRY(S.grid32.alloc(g32.size()));
    BD_CUDA(cudaMemcpyAsync(S.grid.p, g64.data(), sizeof(FineGrid) * g64.size(), cudaMemcpyHostToDevice, s));
    BD_CUDA(cudaMemcpyAsync(S.grid32.p, g32.data(), sizeof(FineGrid) * g32.size(), cudaMemcpyHostToDevice, s));
    BD_CUDA(cudaStreamSynchronize(s));  // the lists live on the host stack
    return BD_OK;
}

template <class T> int st_vec(DBuf<T> &b, long long n, cudaStream_t s)
{
    BD_TRY(b.alloc((size_t)std::max<long long>(n, 1)));
    BD_CUDA(cudaMemsetAsync(b.p, 0, b.bytes(), s));
    return BD_OK;
}

int st_create(amg_stack *b, cudaStream_t s)
{
    const int count = b->count;
    b->nlev.resize(count);
    int L = 0;
    for (int k = 0; k < count; k++) {
        b->nlev[k] = b->h[k]->nlev;
        L = std::max(L, b->nlev[k]);
    }
    b->L = L;
    bool fine0 = true;
    for (int k = 0; k < count; k++) fine0 = fine0 && b->h[k]->fine.valid;
    b->lev[0].fine = fine0;
    // member order and node offsets per level: smoothing members, then the
    // members whose coarsest level it is; on a stencil finest level every
    // member starts on a multiple of 32 nodes
    std::vector<std::vector<int>> order(L);
    std::vector<std::vector<long long>> off(L, std::vector<long long>(count, -1));
    for (int l = 0; l < L; l++) {
        long long o = 0;
        int ns = 0;
        for (int pass = 0; pass < 2; pass++)
            for (int k = 0; k < count; k++) {
                const int last = b->nlev[k] - 1;
                if ((pass == 0 && last > l) || (pass == 1 && last == l)) {
                    order[l].push_back(k);
                    off[l][k] = o;
                    const long long nk = b->h[k]->lev[l].N;
                    o += (l == 0 && fine0) ? (nk + 31) / 32 * 32 : nk;
                    if (pass == 0) ns = (int)o;
                }
            }
        if (o > 1073741823LL) return BD_ERANGE;
        b->lev[l].N = (int)o;
        b->lev[l].Ns = ns;
    }
    const bool p32 = b->p32;
    for (int l = 0; l < L; l++) {
        StLevel &S = b->lev[l];
        // A: every member on the finest level (the PCG applies it), the smoothing ones below
        std::vector<StPart> pa, pr, pp;
        for (int k : order[l]) {
            const Level &Lk = b->h[k]->lev[l];
            const bool smooth = b->nlev[k] - 1 > l;
            if ((l == 0 && !fine0) || (l > 0 && smooth))
                pa.push_back({&Lk.A, p32 ? Lk.A32.p : nullptr, nullptr, Lk.A.nbr, off[l][k], off[l][k]});
            const bool pairs = l == 0 && fine0;
            if (smooth)
                pp.push_back({&Lk.P, p32 ? Lk.P32.p : nullptr, pairs ? &Lk.pair[1] : nullptr, Lk.P.nbr, off[l][k],
                              off[l + 1][k]});
        }
        if (l + 1 < L)
            for (int k : order[l + 1]) {
                const Level &Lk = b->h[k]->lev[l];
                pr.push_back({&Lk.R, p32 ? Lk.R32.p : nullptr, l == 0 && fine0 ? &Lk.pair[0] : nullptr, Lk.R.nbr,
                              off[l + 1][k], off[l][k]});
            }
        BD_TRY(st_build(pa, l == 0 ? S.N : S.Ns, S.N, l == 0 || !p32, p32, S.A, S.A32, nullptr, s));
        S.rowsA = S.A.nbr;
        if (!pp.empty()) {
            BD_TRY(st_build(pp, S.Ns, b->lev[l + 1].N, !p32, p32, S.P, S.P32, &S.pair[1], s));
            BD_TRY(st_build(pr, b->lev[l + 1].N, S.N, !p32, p32, S.R, S.R32, &S.pair[0], s));
        }
        if (l == 0 && fine0) BD_TRY(st_fine_build(b, order[0], off[0], s));
        // node -> member (-1 on padding), Chebyshev coefficients, inverse diagonals
        BD_TRY(S.mem.alloc((size_t)std::max(S.N, 1)));
        BD_CUDA(cudaMemsetAsync(S.mem.p, 0xff, S.mem.bytes(), s));
        std::vector<double> coef(4 * (size_t)count, 0.0);
        for (int k : order[l]) {
            const Level &Lk = b->h[k]->lev[l];
            k_st_fill<<<grid_for(Lk.N, 256), 256, 0, s>>>(Lk.N, S.mem.p + off[l][k], k); ::bd::note_launch();
            coef[4 * k] = Lk.ch_inv_theta;
            coef[4 * k + 1] = Lk.ch_c1;
            coef[4 * k + 2] = Lk.ch_c2;
        }
        BD_TRY(S.coef.alloc(coef.size()));
        BD_CUDA(cudaMemcpyAsync(S.coef.p, coef.data(), sizeof(double) * coef.size(), cudaMemcpyHostToDevice, s));
        BD_CUDA(cudaStreamSynchronize(s));  // coef lives on the host stack
        const long long n2 = 2LL * S.N;
        if (l == 0 && fine0) {
            if (p32) BD_TRY(st_vec(S.kappa32, n2, s));
            else BD_TRY(st_vec(S.kappa, n2, s));
            for (int k : order[l]) {
                const Level &Lk = b->h[k]->lev[0];
                if (b->nlev[k] <= 1) continue;
                if (p32)
                    BD_CUDA(cudaMemcpyAsync(S.kappa32.p + 2 * off[l][k], Lk.kappa32.p, sizeof(float) * 2 * Lk.N,
                                            cudaMemcpyDeviceToDevice, s));
                else
                    BD_CUDA(cudaMemcpyAsync(S.kappa.p + 2 * off[l][k], Lk.kappa.p, sizeof(double) * 2 * Lk.N,
                                            cudaMemcpyDeviceToDevice, s));
            }
        }
        if (p32) {
            BD_TRY(st_vec(S.invd32, n2, s));
            for (int k : order[l])
                BD_CUDA(cudaMemcpyAsync(S.invd32.p + 2 * off[l][k], b->h[k]->lev[l].invdiag32.p,
                                        sizeof(float) * 2 * b->h[k]->lev[l].N, cudaMemcpyDeviceToDevice, s));
            BD_TRY(st_vec(S.f32, n2, s));
            BD_TRY(st_vec(S.u32, n2, s));
            BD_TRY(st_vec(S.r32, n2, s));
            BD_TRY(st_vec(S.d32, n2, s));
            BD_TRY(st_vec(S.w32, n2, s));
        } else {
            BD_TRY(st_vec(S.invd, n2, s));
            for (int k : order[l])
                BD_CUDA(cudaMemcpyAsync(S.invd.p + 2 * off[l][k], b->h[k]->lev[l].invdiag.p,
                                        sizeof(double) * 2 * b->h[k]->lev[l].N, cudaMemcpyDeviceToDevice, s));
            // FP64 on a stencil: its gathered vectors in (v + u, u) form
            S.su = l == 0 && fine0;
            if (l > 0) BD_TRY(st_vec(S.f, n2, s));
            BD_TRY(st_vec(S.u, n2, s));
            BD_TRY(st_vec(S.r, n2, s));
            BD_TRY(st_vec(S.d, n2, s));
            BD_TRY(st_vec(S.w, n2, s));
        }
        S.lanes[0] = lanes_for(S.A, p32);
        if (!pp.empty()) {
            S.lanes[1] = lanes_for(S.R, p32);
            S.lanes[2] = lanes_for(S.P, p32);
        }
    }
    // coarsest-level jobs
    std::vector<StCoarseJob> jobs(count);
    for (int k = 0; k < count; k++) {
        const amg_hierarchy *hk = b->h[k];
        const int c = b->nlev[k] - 1;
        jobs[k] = {hk->cinv.p, hk->nc, c, 2 * off[c][k]};
        b->max_nc = std::max(b->max_nc, hk->nc);
    }
    BD_TRY(b->jobs.alloc(count));
    BD_CUDA(cudaMemcpyAsync(b->jobs.p, jobs.data(), sizeof(StCoarseJob) * count, cudaMemcpyHostToDevice, s));
    // PCG vectors and reduction chunks of the finest level
    const long long n2 = 2LL * b->lev[0].N;
    BD_TRY(st_vec(b->fin, n2, s));
    BD_TRY(st_vec(b->x, n2, s));
    BD_TRY(st_vec(b->r, n2, s));
    BD_TRY(st_vec(b->p, n2, s));
    BD_TRY(st_vec(b->q, n2, s));
    BD_TRY(st_vec(b->fp, n2, s));
    if (p32) BD_TRY(st_vec(b->uold, n2, s));
    b->off0.assign(count, 0);
    b->n0.assign(count, 0);
    std::vector<int> cm, cb, ce, m0(count, 0), m1(count, 0), nn(count, 0);
    for (int k : order[0]) {
        const int N = b->h[k]->lev[0].N;
        b->off0[k] = off[0][k];
        b->n0[k] = N;
        nn[k] = N;
        m0[k] = (int)cm.size();
        for (int a = 0; a < N; a += kStChunk) {
            cm.push_back(k);
            cb.push_back((int)(off[0][k] + a));
            ce.push_back((int)(off[0][k] + std::min(N, a + kStChunk)));
        }
        m1[k] = (int)cm.size();
    }
    b->nchunks = (int)cm.size();
    BD_TRY(b->cmem.alloc(cm.size()));
    BD_TRY(b->cbeg.alloc(cb.size()));
    BD_TRY(b->cend.alloc(ce.size()));
    BD_TRY(b->mc0.alloc(count));
    BD_TRY(b->mc1.alloc(count));
    BD_TRY(b->nn.alloc(count));
    BD_CUDA(cudaMemcpyAsync(b->cmem.p, cm.data(), sizeof(int) * cm.size(), cudaMemcpyHostToDevice, s));
    BD_CUDA(cudaMemcpyAsync(b->cbeg.p, cb.data(), sizeof(int) * cb.size(), cudaMemcpyHostToDevice, s));
    BD_CUDA(cudaMemcpyAsync(b->cend.p, ce.data(), sizeof(int) * ce.size(), cudaMemcpyHostToDevice, s));
    BD_CUDA(cudaMemcpyAsync(b->mc0.p, m0.data(), sizeof(int) * count, cudaMemcpyHostToDevice, s));
    BD_CUDA(cudaMemcpyAsync(b->mc1.p, m1.data(), sizeof(int) * count, cudaMemcpyHostToDevice, s));
    BD_CUDA(cudaMemcpyAsync(b->nn.p, nn.data(), sizeof(int) * count, cudaMemcpyHostToDevice, s));
    BD_TRY(b->part.alloc(4 * (size_t)std::max(b->nchunks, 1)));
    BD_TRY(b->scal.alloc((size_t)count * T_NSLOTS));
    BD_TRY(b->counter.alloc(1));
    BD_CUDA(cudaMemsetAsync(b->counter.p, 0, sizeof(unsigned int), s));
    BD_CUDA(cudaMallocHost((void **)&b->host_init, sizeof(double) * count * T_NSLOTS));
    BD_CUDA(cudaMallocHost((void **)&b->host_scal, sizeof(double) * count * T_NSLOTS));
    BD_CUDA(cudaStreamCreateWithFlags(&b->cap, cudaStreamNonBlocking));
    BD_CUDA(cudaStreamCreateWithFlags(&b->cap2, cudaStreamNonBlocking));
    BD_CUDA(cudaEventCreate(&b->ev[0]));
    BD_CUDA(cudaEventCreate(&b->ev[1]));
    BD_CUDA(cudaStreamSynchronize(s));
    return BD_OK;
}

// ------------------------------------------------------------------ stacked V-cycle
template <class S> struct StView {
    const S *Av, *Rv, *Pv;
    v2<S> *f, *u, *r, *d, *w;
    const v2<S> *invd;
};
template <class S> StView<S> st_view(amg_stack *b, int l);
template <> StView<double> st_view<double>(amg_stack *b, int l)
{
    StLevel &S = b->lev[l];
    return {S.A.v.p, S.R.v.p, S.P.v.p, (double2 *)(l == 0 ? b->r.p : S.f.p), (double2 *)S.u.p,
            (double2 *)S.r.p, (double2 *)S.d.p, (double2 *)S.w.p, (const double2 *)S.invd.p};
}
template <> StView<float> st_view<float>(amg_stack *b, int l)
{
    StLevel &S = b->lev[l];
    return {S.A32.p, S.R32.p, S.P32.p, (float2 *)S.f32.p, (float2 *)S.u32.p, (float2 *)S.r32.p,
            (float2 *)S.d32.p, (float2 *)S.w32.p, (const float2 *)S.invd32.p};
}

template <class S> const v2<S> *st_kappa(const StLevel &Lv);
template <> const double2 *st_kappa<double>(const StLevel &Lv) { return (const double2 *)Lv.kappa.p; }
template <> const float2 *st_kappa<float>(const StLevel &Lv) { return (const float2 *)Lv.kappa32.p; }
template <class S> const FineGrid *st_grids(const StLevel &Lv);
template <> const FineGrid *st_grids<double>(const StLevel &Lv) { return Lv.grid.p; }
template <> const FineGrid *st_grids<float>(const StLevel &Lv) { return Lv.grid32.p; }

// The stencil finest level of every member (all) or of those that smooth;
// make(SYM) gives the epilogue for the tables' form.
template <class S, bool SU, class F>
int st_fine(const StLevel &Lv, bool all, const v2<S> *x, F make, cudaStream_t s)
{
    const int count = all ? (int)Lv.grid.n : Lv.nsmooth;
    if (count <= 0) return BD_OK;
    const long long units = all ? Lv.units : Lv.units_smooth;
    if (Lv.sym)
        k_fine_many<S, true, SU><<<fine_blocks<S, true>(units), kFineTPB, 0, s>>>(st_grids<S>(Lv), count, x,
                                                                                  make(std::true_type{}));
    else
        k_fine_many<S, false, SU><<<fine_blocks<S, false>(units), kFineTPB, 0, s>>>(st_grids<S>(Lv), count, x,
                                                                                    make(std::false_type{}));
    ::bd::note_launch();
    BD_LAUNCH_CHECK();
    return BD_OK;
}

// Block-CSR operator of stack level l on rows [0, rows).
template <class S, class E>
int st_apply(const StLevel &Lv, int rows, const S *vals, const v2<S> *x, E e, cudaStream_t s)
{
    return launch_bsr_rows(rows, Lv.A.rp.p, Lv.A.ci.p, MatFull<S>{vals}, Lv.lanes[0], GatherVec<S>{x}, e, s);
}

template <class S>
int st_vcycle(amg_stack *b, cudaStream_t s)
{
    constexpr bool SU = std::is_same<S, double>::value;
    const int L = b->L;
    for (int l = 0; l + 1 < L; l++) {
        StLevel &Lv = b->lev[l];
        if (Lv.Ns <= 0) continue;
        const StView<S> v = st_view<S>(b, l), cv = st_view<S>(b, l + 1);
        const StCoef c{Lv.mem.p, Lv.coef.p}, cc{b->lev[l + 1].mem.p, b->lev[l + 1].coef.p};
        if (l == 0 && Lv.fine) {
            BD_TRY((st_fine<S, SU>(Lv, false, v.d, [&](auto sym) { return FinePre<S, sym.value, SU>{v.f, v.u}; }, s)));
            BD_TRY((st_fine<S, SU>(Lv, false, v.u, [&](auto sym) { return FineResid<S, sym.value, SU>{v.f, v.r}; }, s)));
        } else {
            BD_TRY(st_apply<S>(Lv, Lv.Ns, v.Av, v.d, StPre<S>{v.f, v.invd, v.d, v.u, c}, s));
            BD_TRY(st_apply<S>(Lv, Lv.Ns, v.Av, v.u, StResid<S>{v.f, v.r}, s));
        }
        const StStoreD0<S> rest{cv.f, cv.d, cv.invd, cc};
        if (Lv.pair[0].valid)
            BD_TRY((launch_bsr_rows(Lv.R.nbr, Lv.R.rp.p, Lv.pair[0].ci.p, mat_pair<S>(Lv.pair[0]), Lv.lanes[1],
                                    GatherVec<S, SU>{v.r}, rest, s)));
        else
            BD_TRY(launch_bsr<S>(Lv.R, v.Rv, Lv.lanes[1], GatherVec<S>{v.r}, rest, s));
    }
    StLevelPtrs<S> lp{};
    for (int l = 0; l < L; l++) {
        const StView<S> v = st_view<S>(b, l);
        lp.f[l] = (S *)v.f;
        lp.u[l] = (S *)v.u;
    }
    const dim3 grid((std::max(b->max_nc, 1) + 3) / 4, b->count);
    k_st_coarse<S><<<grid, 128, 0, s>>>(b->jobs.p, lp); ::bd::note_launch();
    BD_LAUNCH_CHECK();
    for (int l = L - 2; l >= 0; l--) {
        StLevel &Lv = b->lev[l];
        if (Lv.Ns <= 0) continue;
        const StView<S> v = st_view<S>(b, l), cv = st_view<S>(b, l + 1);
        const StCoef c{Lv.mem.p, Lv.coef.p};
        if (l == 0 && Lv.fine) {
            BD_TRY((launch_bsr_rows(Lv.P.nbr, Lv.P.rp.p, Lv.pair[1].ci.p, mat_pair<S>(Lv.pair[1]), Lv.lanes[2],
                                    GatherVec<S>{cv.u}, StAddPair<S, SU>{v.u, st_kappa<S>(Lv)}, s)));
            BD_TRY((st_fine<S, SU>(Lv, false, v.u, [&](auto sym) {
                return FinePost1<S, sym.value, SU>{v.f, v.r, v.d, nullptr};
            }, s)));
            BD_TRY((st_fine<S, SU>(Lv, false, v.d, [&](auto sym) {
                return FinePost2<S, sym.value, SU>{v.r, v.u, v.u};
            }, s)));
            continue;
        }
        BD_TRY(launch_bsr<S>(Lv.P, v.Pv, Lv.lanes[2], GatherVec<S>{cv.u}, StAdd<S>{v.u}, s));
        BD_TRY(st_apply<S>(Lv, Lv.Ns, v.Av, v.u, StPost1<S>{v.f, v.invd, v.u, v.r, v.d, v.w, c}, s));
        BD_TRY(st_apply<S>(Lv, Lv.Ns, v.Av, v.d, StPost2<S>{v.r, v.d, v.invd, v.w, v.u, c}, s));
    }
    return BD_OK;
}

// ------------------------------------------------------------------ stacked PCG graph
template <class S>
StPcg<S> st_pcg(amg_stack *b)
{
    const StView<S> v0 = st_view<S>(b, 0);
    StPcg<S> v;
    v.fin = (const double2 *)b->fin.p;
    v.fp = (double2 *)b->fp.p;
    v.x = (double2 *)b->x.p;
    v.r = (double2 *)b->r.p;
    v.p = (double2 *)b->p.p;
    v.q = (double2 *)b->q.p;
    v.uold = b->p32 ? (v2<S> *)b->uold.p : nullptr;
    v.f0 = v0.f;
    v.d0 = v0.d;
    v.u0 = v0.u;
    v.invd0 = v0.invd;
    v.c0 = StCoef{b->lev[0].mem.p, b->lev[0].coef.p};
    v.mem = b->lev[0].mem.p;
    v.psu = b->lev[0].fine ? 1 : 0;
    v.dsu = b->lev[0].su ? 1 : 0;
    return v;
}

StRed st_red(amg_stack *b, cudaGraphConditionalHandle cond)
{
    return {b->scal.p, b->part.p, b->counter.p, b->cmem.p, b->cbeg.p, b->cend.p, b->mc0.p, b->mc1.p, b->nn.p,
            b->count, b->p32 ? 1 : 0, cond};
}

// q = A x on the finest level; su: x is stored in (v + u, u) form (the PCG's p
// on a stencil level)
int st_apply_a(amg_stack *b, const double2 *x, double2 *q, cudaStream_t s, bool su = false)
{
    StLevel &S = b->lev[0];
    if (S.fine) {
        auto store = [&](auto) { return FineStore<double>{q}; };
        return su ? st_fine<double, true>(S, true, x, store, s) : st_fine<double, false>(S, true, x, store, s);
    }
    return launch_bsr_rows(S.N, S.A.rp.p, S.A.ci.p, MatFull<double>{S.A.v.p}, lanes_for(S.A, false),
                           GatherVec<double>{x}, StStore{q}, s);
}

template <class S>
int st_capture(amg_stack *b)
{
    cudaStream_t s = b->cap, s2 = b->cap2;
    const int count = b->count, N0 = b->lev[0].N;
    const StPcg<S> v = st_pcg<S>(b);
    const int nch = b->nchunks;
    const int vg = grid_for(N0, kStThreads);
    BD_CUDA(cudaStreamBeginCapture(s, cudaStreamCaptureModeThreadLocal));
    const long long c0 = launch_count();
    BD_CUDA(cudaMemcpyAsync(b->scal.p, b->host_init, sizeof(double) * count * T_NSLOTS, cudaMemcpyHostToDevice, s));
    for (int k = 0; k < count; k++) {
        const size_t bytes = sizeof(double) * 2 * (size_t)b->n0[k];
        BD_CUDA(cudaMemcpyAsync(b->fin.p + 2 * b->off0[k], b->gf[k], bytes, cudaMemcpyDeviceToDevice, s));
        BD_CUDA(cudaMemcpyAsync(b->x.p + 2 * b->off0[k], b->gx[k], bytes, cudaMemcpyDeviceToDevice, s));
    }
    k_st_red<R_FSTATS, S><<<nch, kStThreads, 0, s>>>(st_red(b, 0), v); ::bd::note_launch();
    k_st_red<R_PROJF, S><<<nch, kStThreads, 0, s>>>(st_red(b, 0), v); ::bd::note_launch();
    BD_TRY(st_apply_a(b, v.x, v.q, s));
    BD_LAUNCH_CHECK();
    cudaStreamCaptureStatus cs;
    cudaGraph_t g = nullptr;
    const cudaGraphNode_t *deps = nullptr;
    size_t nd = 0;
    BD_CUDA(cudaStreamGetCaptureInfo(s, &cs, nullptr, &g, &deps, nullptr, &nd));
    cudaGraphConditionalHandle cond;
    BD_CUDA(cudaGraphConditionalHandleCreate(&cond, g, 0, 0));
    k_st_red<R_INIT, S><<<nch, kStThreads, 0, s>>>(st_red(b, cond), v); ::bd::note_launch();
    BD_LAUNCH_CHECK();
    BD_CUDA(cudaStreamGetCaptureInfo(s, &cs, nullptr, &g, &deps, nullptr, &nd));
    cudaGraphNodeParams np = {};
    np.type = cudaGraphNodeTypeConditional;
    np.conditional.handle = cond;
    np.conditional.type = cudaGraphCondTypeWhile;
    np.conditional.size = 1;
    cudaGraphNode_t wnode;
    BD_CUDA(cudaGraphAddNode(&wnode, g, deps, nullptr, nd, &np));
    cudaGraph_t body = np.conditional.phGraph_out[0];
    const long long c1 = launch_count();
    BD_CUDA(cudaStreamBeginCaptureToGraph(s2, body, nullptr, nullptr, 0, cudaStreamCaptureModeThreadLocal));
    BD_TRY(st_vcycle<S>(b, s2));
    k_st_red<R_ZSTATS, S><<<nch, kStThreads, 0, s2>>>(st_red(b, 0), v); ::bd::note_launch();
    k_st_p<S><<<vg, kStThreads, 0, s2>>>(N0, v, b->scal.p); ::bd::note_launch();
    BD_TRY(st_apply_a(b, v.p, v.q, s2, v.psu != 0));
    k_st_red<R_PQ, S><<<nch, kStThreads, 0, s2>>>(st_red(b, 0), v); ::bd::note_launch();
    k_st_red<R_XR, S><<<nch, kStThreads, 0, s2>>>(st_red(b, cond), v); ::bd::note_launch();
    BD_LAUNCH_CHECK();
    cudaGraph_t body_out = nullptr;
    BD_CUDA(cudaStreamEndCapture(s2, &body_out));
    const long long c2 = launch_count();
    BD_CUDA(cudaStreamUpdateCaptureDependencies(s, &wnode, nullptr, 1, cudaStreamSetCaptureDependencies));
    BD_TRY(st_apply_a(b, v.x, v.q, s));
    k_st_red<R_TRUE, S><<<nch, kStThreads, 0, s>>>(st_red(b, 0), v); ::bd::note_launch();
    k_st_project_x<<<vg, kStThreads, 0, s>>>(N0, v.x, b->lev[0].mem.p, b->scal.p); ::bd::note_launch();
    BD_LAUNCH_CHECK();
    for (int k = 0; k < count; k++) {
        const size_t bytes = sizeof(double) * 2 * (size_t)b->n0[k];
        BD_CUDA(cudaMemcpyAsync(b->gx[k], b->x.p + 2 * b->off0[k], bytes, cudaMemcpyDeviceToDevice, s));
    }
    BD_CUDA(cudaMemcpyAsync(b->host_scal, b->scal.p, sizeof(double) * count * T_NSLOTS, cudaMemcpyDeviceToHost, s));
    const long long c3 = launch_count();
    BD_CUDA(cudaStreamEndCapture(s, &b->graph));
    BD_CUDA(cudaGraphInstantiate(&b->exec, b->graph, 0));
    b->n_pre = c1 - c0;
    b->n_body = c2 - c1;
    b->n_post = c3 - c2;
    note_launches(-(c3 - c0));
    return BD_OK;
}

void end_capture(cudaStream_t s)
{
    cudaStreamCaptureStatus cs;
    if (cudaStreamIsCapturing(s, &cs) == cudaSuccess && cs != cudaStreamCaptureStatusNone) {
        cudaGraph_t g = nullptr;
        cudaStreamEndCapture(s, &g);
        if (g) cudaGraphDestroy(g);
    }
    cudaGetLastError();
}

}  // namespace
}  // namespace bd

// ------------------------------------------------------------------ public
extern "C" int amg_stack_create(amg_hierarchy *const *h, int count, void *stream, amg_stack **out)
{
    if (!out) return BD_EINVAL;
    *out = nullptr;
    if (!h || count < 1) return BD_EINVAL;
    for (int k = 0; k < count; k++) {
        if (!h[k] || h[k]->nlev < 1) return BD_EINVAL;
        if (h[k]->prec32 != h[0]->prec32) return BD_EINVAL;     // one V-cycle precision per stack
        if (h[k]->opts.cheb_degree != 2) return BD_EINVAL;     // Appendix A's degree-2 smoother only
    }
    amg_stack *b = new (std::nothrow) amg_stack();
    if (!b) return BD_ENOMEM;
    b->count = count;
    b->p32 = h[0]->prec32;
    b->h.assign(h, h + count);
    for (amg_hierarchy *hk : b->h) hk->batch_refs++;  // their forms may not change while stacked
    const int st = bd::st_create(b, (cudaStream_t)stream);
    if (st != BD_OK) {
        delete b;
        return st;
    }
    *out = b;
    return BD_OK;
}

extern "C" int amg_stack_solve(amg_stack *b, const double *const *f, double *const *x, const solve_options *opts,
                               void *stream, solve_info *info)
{
    if (!b || !f || !x) return BD_EINVAL;
    const int count = b->count;
    solve_options o;
    solve_options_default(&o);
    if (opts) o = *opts;
    if (!(o.rtol > 0.0) || o.max_it < 0 || o.strict) return BD_EINVAL;
    for (int k = 0; k < count; k++)
        if (!f[k] || !x[k]) return BD_EINVAL;
    bool same = b->exec != nullptr;
    for (int k = 0; k < count && same; k++) same = b->gf[k] == f[k] && b->gx[k] == x[k];
    if (!same) {
        b->drop_graph();
        b->gf.assign(f, f + count);
        b->gx.assign(x, x + count);
        const int st = b->p32 ? bd::st_capture<float>(b) : bd::st_capture<double>(b);
        if (st != BD_OK) {
            bd::end_capture(b->cap2);
            bd::end_capture(b->cap);
            b->drop_graph();
            return st;
        }
    }
    for (int k = 0; k < count; k++) {
        double *hi = b->host_init + (size_t)k * bd::T_NSLOTS;
        for (int i = 0; i < bd::T_NSLOTS; i++) hi[i] = 0.0;
        hi[bd::T_RTOL] = o.rtol;
        hi[bd::T_MAXIT] = (double)o.max_it;
        hi[bd::T_WARM] = o.warm_start ? 1.0 : 0.0;
    }
    cudaStream_t s = (cudaStream_t)stream;
    BD_CUDA(cudaEventRecord(b->ev[0], s));
    BD_CUDA(cudaGraphLaunch(b->exec, s));
    BD_CUDA(cudaEventRecord(b->ev[1], s));
    BD_CUDA(cudaStreamSynchronize(s));
    float ms = 0.0f;
    cudaEventElapsedTime(&ms, b->ev[0], b->ev[1]);
    int worst = BD_OK;
    double loops = 0.0;
    for (int k = 0; k < count; k++) {
        const double *sc = b->host_scal + (size_t)k * bd::T_NSLOTS;
        loops = std::max(loops, sc[bd::T_IT]);
        const double nf = std::sqrt(sc[bd::T_NF2]);
        const int stk = (int)sc[bd::T_STATUS];
        if (info) {
            info[k].status = stk;
            info[k].iters = (int)sc[bd::T_IT];
            info[k].rel_res = nf > 0.0 ? std::sqrt(sc[bd::T_RR]) / nf : 0.0;
            info[k].true_rel_res = nf > 0.0 ? std::sqrt(sc[bd::T_TRR]) / nf : 0.0;
            info[k].solve_ms = ms;
            info[k].total_iters = (long long)sc[bd::T_IT];
        }
        if (stk != BD_OK && worst == BD_OK) worst = stk;
    }
    bd::note_launches(b->n_pre + b->n_post + (long long)loops * b->n_body);
    return worst;
}

extern "C" int amg_stack_info(const amg_stack *b, int *levels, long long *launches_per_iteration)
{
    if (!b) return BD_EINVAL;
    if (levels) *levels = b->L;
    if (launches_per_iteration) *launches_per_iteration = b->n_body;
    return BD_OK;
}

extern "C" void amg_stack_destroy(amg_stack *b) { delete b; }
