// amg_scalar.cu -- the elliptic solve of the decoupled scheme (Section 2.2,
// Eq. 6) on its one field.
//
// bd_elliptic_setup builds the block hierarchy of [I, 0; 0, Ai + Ae]: every
// level's operators are block diagonal and the scheme's right-hand side and
// iterate have a zero v field, which the V-cycle and the PCG preserve.  Here the
// same solve runs on the u_e field alone: the finest level as a scalar layered
// stencil, the coarse operators with the (u, u) entry of each block (12 instead
// of 36 bytes, one FP64 multiply-add instead of four), the coarsest inverse's
// (u, u) part, scalar vectors.  128x128x32, per PCG iteration: 1087 -> 343 us.
// The PCG's recurrences, stopping test and graph are those of the block solve
// (amg_solve.cu).
#include <algorithm>
#include <cmath>
#include <cstdlib>
#include <new>
#include <type_traits>

#include "amg_bsr.cuh"
#include "fine_scalar.cuh"
#include "pcg_reduce.cuh"
#include "scalar.cuh"

namespace bd {

// ------------------------------------------------------------------ tables
template <bool SYM>
__global__ void k_sc_pack(int rows, const double *__restrict__ raw, double a, double b, double m, double c2, double it,
                          double *__restrict__ tab, float *__restrict__ tab32)
{
    using Row = ScRow<SYM>;
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= rows) return;
    const double *o = raw + (size_t)t * kFineRaw;
    const int ti = t % 3, tj = (t % 9) / 3;
    auto put = [&](int k, double x) {
        tab[(size_t)t * Row::LEN + k] = x;
        if (tab32) tab32[(size_t)t * Row::LEN + k] = (float)x;
    };
    for (int k = 0; k < Row::LEN; k++) put(k, 0.0);
    for (int z = 0; z < (SYM ? 2 : 3); z++) {
        const int base = 9 * (z == 0 ? 1 : (z == 1 ? 2 : 0));  // dz = 0, +1, -1
        for (int k = 0; k < Row::NP; k++) {
            const int q = base + (SYM ? fine_pair_pos(k, ti, tj) : k);
            const double v = a * o[2 * q] + b * o[2 * q + 1];
            put(z * Row::G + k, q == 13 ? v + m * o[54] : v);
        }
    }
    const double du = o[55] > 0.0 ? 1.0 / (o[26] + o[27]) : 0.0;  // of Ai + Ae
    put(Row::IDC2, c2 * du);
    put(Row::IDT, du * it);
}

int sc_pack(const FineStencil &F, double a, double b, double m, double c1, double c2, double inv_theta, bool fp32,
            ScOp &op, cudaStream_t s)
{
    op.sym = F.sym;
    op.g.NX = F.NX;
    op.g.NXY = F.NX * F.NY;
    op.g.NZ = F.NZ;
    op.g.ncb = (op.g.NXY + kFineTPB - 1) / kFineTPB;
    op.g.c1 = c1;
    const int rows = 9 * F.NZ, grid = (rows + 63) / 64;
    const size_t len = (size_t)rows * (F.sym ? ScRow<true>::LEN : ScRow<false>::LEN);
    BD_TRY(op.tab.alloc(len));
    if (fp32) BD_TRY(op.tab32.alloc(len));
    if (F.sym) k_sc_pack<true><<<grid, 64, 0, s>>>(rows, F.raw.p, a, b, m, c2, inv_theta, op.tab.p, op.tab32.p);
    else k_sc_pack<false><<<grid, 64, 0, s>>>(rows, F.raw.p, a, b, m, c2, inv_theta, op.tab.p, op.tab32.p);
    ::bd::note_launch();
    BD_LAUNCH_CHECK();
    return BD_OK;
}

namespace {

// (u, u) entries of a block operator; of an interleaved vector its u_e field;
// of the coarsest inverse its (u, u) part
__global__ void k_uu(long long nb, const double *__restrict__ v, double *__restrict__ a, float *__restrict__ a32)
{
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < nb; i += (long long)gridDim.x * blockDim.x) {
        if (a) a[i] = v[4 * i + 3];
        else a32[i] = (float)v[4 * i + 3];
    }
}
__global__ void k_u_field(int n, const double *__restrict__ v, double *__restrict__ a, float *__restrict__ a32)
{
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
        if (a) a[i] = v[2 * (size_t)i + 1];
        if (a32) a32[i] = (float)v[2 * (size_t)i + 1];
    }
}
__global__ void k_uu_dense(int n, const double *__restrict__ c, double *__restrict__ a)
{
    for (int e = blockIdx.x * blockDim.x + threadIdx.x; e < n * n; e += gridDim.x * blockDim.x)
        a[e] = c[(size_t)(2 * (e / n) + 1) * (2 * n) + 2 * (e % n) + 1];
}

// ------------------------------------------------------------------ coarse operators
template <class S> struct MatOne {
    using Sc = S;
    static constexpr bool OWN = false;
    const S *__restrict__ v;
    struct Acc {
        S y = 0;
    };
    template <class G> __device__ __forceinline__ void step(Acc &A, size_t t, int q, const G &g) const
    {
        A.y = fma(v[t], g(q), A.y);
    }
    __device__ __forceinline__ void finish(const Acc &A, S &y0, S &y1) const
    {
        y0 = A.y;
        y1 = 0;
    }
};
template <class S> struct GatherOne {
    const S *__restrict__ x;
    __device__ __forceinline__ S operator()(int q) const { return x[q]; }
};

// Chebyshev steps (degree 2) and transfers, as the block V-cycle's epilogues.
template <class S> struct E1Pre {
    const S *__restrict__ f, *__restrict__ invd, *__restrict__ d0;
    S *__restrict__ u;
    S c1, c2;
    __device__ __forceinline__ void operator()(int p, S y, S) const
    {
        const S d = d0[p];
        u[p] = d + (c1 * d + c2 * invd[p] * (f[p] - y));
    }
};
template <class S> struct E1Resid {
    const S *__restrict__ f;
    S *__restrict__ r;
    __device__ __forceinline__ void operator()(int p, S y, S) const { r[p] = f[p] - y; }
};
template <class S> struct E1Restrict {
    S *__restrict__ f, *__restrict__ d0;
    const S *__restrict__ invd;
    S it;
    __device__ __forceinline__ void operator()(int p, S y, S) const
    {
        f[p] = y;
        d0[p] = y * invd[p] * it;
    }
};
template <class S> struct E1Add {
    S *__restrict__ u;
    __device__ __forceinline__ void operator()(int p, S y, S) const { u[p] += y; }
};
template <class S> struct E1Post1 {
    const S *__restrict__ f, *__restrict__ invd;
    S *__restrict__ r, *__restrict__ d;
    S it;
    __device__ __forceinline__ void operator()(int p, S y, S) const
    {
        const S r0 = f[p] - y;
        r[p] = r0;
        d[p] = r0 * invd[p] * it;
    }
};
template <class S> struct E1Post2 {
    const S *__restrict__ r, *__restrict__ d, *__restrict__ invd;
    S *u;
    S c1, c2;
    __device__ __forceinline__ void operator()(int p, S y, S) const
    {
        const S d0 = d[p];
        u[p] = (u[p] + d0) + (c1 * d0 + c2 * invd[p] * (r[p] - y));
    }
};

// the same on the stencil (t: c2 D^{-1}, D^{-1} / theta)
template <class S> struct S1Pre {
    const S *__restrict__ f;
    S *__restrict__ u;
    __device__ __forceinline__ S load(int p, bool ok) const { return ok ? f[p] : (S)0; }
    __device__ __forceinline__ void operator()(int p, const S *t, S fp, S c, S c1, S y)
    {
        u[p] = c + (c1 * c + t[0] * (fp - y));
    }
};
template <class S> struct S1Resid {
    const S *__restrict__ f;
    S *__restrict__ r;
    __device__ __forceinline__ S load(int p, bool ok) const { return ok ? f[p] : (S)0; }
    __device__ __forceinline__ void operator()(int p, const S *, S fp, S, S, S y) { r[p] = fp - y; }
};
template <class S> struct S1Post1 {
    const S *__restrict__ f;
    S *__restrict__ r, *__restrict__ d;
    __device__ __forceinline__ S load(int p, bool ok) const { return ok ? f[p] : (S)0; }
    __device__ __forceinline__ void operator()(int p, const S *t, S fp, S, S, S y)
    {
        const S r0 = fp - y;
        r[p] = r0;
        d[p] = r0 * t[1];
    }
};
template <class S> struct S1Post2 {
    const S *__restrict__ r;
    S *u;
    struct Pre {
        S r, u;
    };
    __device__ __forceinline__ Pre load(int p, bool ok) const { return {ok ? r[p] : (S)0, ok ? u[p] : (S)0}; }
    __device__ __forceinline__ void operator()(int p, const S *t, const Pre &q, S c, S c1, S y)
    {
        u[p] = (q.u + c) + fma(c1, c, t[0] * (q.r - y));
    }
};

// ------------------------------------------------------------------ PCG kernels
__global__ void k1_f_stats(int N, const double *__restrict__ f, Fin fin)
{
    double a = 0.0, b = 0.0;
    for (int i = share_lo(N) + threadIdx.x, e = share_hi(N); i < e; i += blockDim.x) {
        const double v = f[i];
        a += v;
        b += v * v;
    }
    block_finish<2>(a, b, 0.0, 0.0, fin);
}
// f projected (mean removed); x cleared when the solve is cold
__global__ void k1_project_f(int N, const double *__restrict__ f, double *__restrict__ fp, double *__restrict__ x, Fin fin)
{
    const double m = fin.scal[S_MEANF];
    const bool cold = fin.scal[S_WARM] == 0.0;
    double a = 0.0;
    for (int i = share_lo(N) + threadIdx.x, e = share_hi(N); i < e; i += blockDim.x) {
        const double v = f[i] - m;
        fp[i] = v;
        if (cold) x[i] = 0.0;
        a += v * v;
    }
    block_finish<1>(a, 0.0, 0.0, 0.0, fin);
}
// The next V-cycle's finest-level input from the residual.
template <class S> struct S1In {
    S *__restrict__ f;  // FP32 V-cycle: its right-hand side (FP64 reads r itself)
    S *__restrict__ d;
    const S *__restrict__ invd;
    S it;
    __device__ __forceinline__ S load(int p) const { return d ? invd[p] : (S)0; }
    __device__ __forceinline__ void operator()(int p, double r, S b) const
    {
        const S v = narrow_to<S>(r);
        if (sizeof(S) == 4) f[p] = v;
        if (d) d[p] = v * b * it;
    }
    __device__ __forceinline__ void operator()(int p, double r) const { (*this)(p, r, load(p)); }
};
// MODE 0: q = A p and p.q; 1: r = f - A x (stored if out), ||r||^2 and sum x
template <int MODE, class S> struct S1Reduce {
    const double *__restrict__ f;
    double *__restrict__ out;
    S1In<S> in;
    double acc, xs;
    __device__ __forceinline__ double load(int p, bool ok) const { return MODE && ok ? f[p] : 0.0; }
    __device__ __forceinline__ void operator()(int p, const double *, double fp, double c, double, double y)
    {
        if (MODE == 0) {
            out[p] = y;
            acc = fma(c, y, acc);
        } else {
            const double r = fp - y;
            if (out) {
                out[p] = r;
                in(p, r);
            }
            acc += r * r;
            xs += c;
        }
    }
};
template <int MODE, bool SYM, class S>
__global__ void __launch_bounds__(kFineTPB, ScMinB<double>::v)
    k1_reduce(ScGrid g, const double *__restrict__ x, S1Reduce<MODE, S> e, Fin fin)
{
    sc_block<double, SYM>(g, x, e);
    block_finish<MODE == 0 ? 1 : 2, kFineTPB>(e.acc, e.xs, 0.0, 0.0, fin);
}
// last post-smoothing step with the z statistics (FP64 V-cycle)
struct S1Z {
    S1Post2<double> post;
    double *z;
    const double *__restrict__ r;
    double a, b, c;
    struct Pre {
        S1Post2<double>::Pre q;
        double r;
    };
    __device__ __forceinline__ Pre load(int p, bool ok) const { return {post.load(p, ok), ok ? r[p] : 0.0}; }
    __device__ __forceinline__ void operator()(int p, const double *t, const Pre &q, double x, double c1, double y)
    {
        const double u = (q.q.u + x) + fma(c1, x, t[0] * (q.q.r - y));
        z[p] = u;
        a += u;
        b += q.r;
        c = fma(q.r, u, c);
    }
};
template <bool SYM>
__global__ void __launch_bounds__(kFineTPB, ScMinB<double>::v)
    k1_z(ScGrid g, const double *__restrict__ x, S1Z e, Fin fin)
{
    sc_block<double, SYM>(g, x, e);
    block_finish<3, kFineTPB>(e.a, e.b, e.c, 0.0, fin);
}
// z from the V-cycle's output u and its statistics (FP32, or a single level)
template <class S>
__global__ void k1_z_from(int N, const S *u, const double *__restrict__ r, const double *__restrict__ zold, double *z, Fin fin)
{
    double a = 0.0, b = 0.0, c = 0.0, d = 0.0;
    struct In {
        S u;
        double r, o;
    };
    share_stream(N, [&](int i) { return In{u[i], r[i], zold ? zold[i] : 0.0}; }, [&](int i, const In &q) {
        const double zi = widen(q.u);
        z[i] = zi;
        a += zi;
        b += q.r;
        c += q.r * zi;
        d += q.r * q.o;
    });
    block_finish<4>(a, b, c, d, fin);
}
__global__ void k1_p_update(int N, double *__restrict__ z, double *__restrict__ p, double *__restrict__ zold,
                            const double *__restrict__ scal)
{
    const double mz = scal[S_MEANZ], beta = scal[S_BETA];
    const bool first = scal[S_IT] == 0.0;
    struct In {
        double z, p;
    };
    share_stream(N, [&](int i) { return In{z[i], p[i]}; }, [&](int i, const In &q) {
        const double zi = q.z - mz;
        if (zold) zold[i] = zi;
        p[i] = first ? zi : zi + beta * q.p;
    });
}
template <class S>
__global__ void k1_xr_update(int N, double *__restrict__ x, double *__restrict__ r, const double *__restrict__ p,
                             const double *__restrict__ q, S1In<S> in, Fin fin)
{
    const double alpha = fin.scal[S_ALPHA];
    double acc = 0.0;
    struct In {
        double x, r, p, q;
        S b;
    };
    share_stream(N, [&](int i) { return In{x[i], r[i], p[i], q[i], in.load(i)}; }, [&](int i, const In &v) {
        const double ri = v.r - alpha * v.q;
        x[i] = v.x + alpha * v.p;
        r[i] = ri;
        in(i, ri, v.b);
        acc += ri * ri;
    });
    block_finish<1>(acc, 0.0, 0.0, 0.0, fin);
}
// x to mean zero, or zero for a zero right-hand side
__global__ void k1_project_x(int N, double *__restrict__ x, const double *__restrict__ scal)
{
    const double m = scal[S_MEANX];
    const bool zero = scal[S_NF2] == 0.0;
    for (int i = share_lo(N) + threadIdx.x, e = share_hi(N); i < e; i += blockDim.x) x[i] = zero ? 0.0 : x[i] - m;
}

template <class S> struct Buf;
template <> struct Buf<double> {
    template <class D> static double *p(D &d) { return d.p64.p; }
};
template <> struct Buf<float> {
    template <class D> static float *p(D &d) { return d.p32.p; }
};
// a scalar vector or value array in the V-cycle's precision
struct Arr {
    DBuf<double> p64;
    DBuf<float> p32;
    int alloc(size_t n, bool fp32) { return fp32 ? p32.alloc(n) : p64.alloc(n); }
};

struct ScLevel {
    Arr A, P, R, invd, f, u, r, d;
    int lanes[3] = {1, 1, 1};
    // the forms setup chose, here and for the block operators (amg_set_level_lanes)
    int chosen[3] = {1, 1, 1}, block[3] = {0, 0, 0};
};

}  // namespace

struct ScalarEll {
    ScOp op;
    FineStencil F;
    ScLevel lev[kMaxLevels];
    DBuf<double> cinv;
    DBuf<double> fin, fp, x, r, z, p, q, zold, partial, scal;
    DBuf<unsigned int> counter;
    cudaGraph_t graph = nullptr;
    cudaGraphExec_t exec = nullptr;
    cudaStream_t cap = nullptr, cap2 = nullptr;
    cudaEvent_t ev[2] = {nullptr, nullptr};
    double *host = nullptr;  // pinned: initial scalars, then results
    bool failed = false;
    long long pre = 0, body = 0, post = 0;
    void drop_graph()
    {
        if (exec) cudaGraphExecDestroy(exec);
        if (graph) cudaGraphDestroy(graph);
        exec = nullptr;
        graph = nullptr;
        failed = false;
    }
    ~ScalarEll()
    {
        drop_graph();
        if (cap) cudaStreamDestroy(cap);
        if (cap2) cudaStreamDestroy(cap2);
        if (ev[0]) cudaEventDestroy(ev[0]);
        if (ev[1]) cudaEventDestroy(ev[1]);
        if (host) cudaFreeHost(host);
    }
};

namespace {

template <class S, class E>
int csr(const BSR &M, Arr &v, int T, const S *x, E e, cudaStream_t s)
{
    return launch_bsr_rows(M.nbr, M.rp.p, M.ci.p, MatOne<S>{Buf<S>::p(v)}, T, GatherOne<S>{x}, e, s);
}

// Time the lanes of every coarse operator (amg_options.autotune).  The workspace
// vectors serve as operands; their contents do not matter.
template <class S> int tune(amg_hierarchy *h, ScalarEll &E, cudaStream_t s)
{
    auto P = [&](Arr &a) { return Buf<S>::p(a); };
    for (int l = 0; l < h->nlev - 1; l++) {
        Level &L = h->lev[l];
        ScLevel &C = E.lev[l], &D = E.lev[l + 1];
        if (l > 0)
            BD_TRY(tune_csr_lanes(L.A, [&](int T) {
                return csr<S>(L.A, C.A, T, (const S *)P(C.u), E1Resid<S>{P(C.f), P(C.r)}, s);
            }, s, &C.lanes[0]));
        BD_TRY(tune_csr_lanes(L.R, [&](int T) {
            return csr<S>(L.R, C.R, T, (const S *)P(C.r), E1Resid<S>{P(D.f), P(D.r)}, s);
        }, s, &C.lanes[1]));
        BD_TRY(tune_csr_lanes(L.P, [&](int T) {
            return csr<S>(L.P, C.P, T, (const S *)P(D.u), E1Resid<S>{P(C.f), P(C.d)}, s);
        }, s, &C.lanes[2]));
    }
    return BD_OK;
}

}  // namespace

int scalar_build(amg_hierarchy *h, const bd_system *sys, cudaStream_t s)
{
    h->scalar.reset();
    if (h->opts.cheb_degree != 2) return BD_OK;  // the block solve serves degree 1
    auto up = std::make_shared<ScalarEll>();
    ScalarEll &E = *up;
    const bool p32 = h->prec32;
    const int nl = h->nlev;
    Level &L0 = h->lev[0];
    BD_TRY(fine_raw_copy(E.F, sys, s));
    BD_TRY(sc_pack(E.F, 1.0, 1.0, 0.0, L0.ch_c1, L0.ch_c2, L0.ch_inv_theta, p32, E.op, s));
    for (int l = 0; l < nl; l++) {
        Level &L = h->lev[l];
        ScLevel &C = E.lev[l];
        auto uu = [&](const BSR &M, Arr &a) {
            BD_TRY(a.alloc((size_t)M.nb, p32));
            k_uu<<<grid_for(M.nb, 256), 256, 0, s>>>(M.nb, M.v.p, a.p64.p, a.p32.p); ::bd::note_launch();
            return BD_OK;
        };
        for (Arr *a : {&C.invd, &C.f, &C.u, &C.r, &C.d}) BD_TRY(a->alloc((size_t)L.N, p32));
        k_u_field<<<grid_for(L.N, 256), 256, 0, s>>>(L.N, L.invdiag.p, C.invd.p64.p, C.invd.p32.p); ::bd::note_launch();
        if (l == nl - 1) break;
        if (l > 0) BD_TRY(uu(L.A, C.A));
        BD_TRY(uu(L.P, C.P));
        BD_TRY(uu(L.R, C.R));
        // one value per entry: rows are bound by latency and bytes, as FP32 blocks.
        // Every power of two timed for every operator inside the elliptic iteration
        // (48x48x12 to 160x160x40, both precisions): the rule's choice is the fastest to
        // within 3 us of 95 to 340 an iteration, but for A2 at 128x128x32 in FP64 (2956
        // rows of 241: 128 threads, 64 take 11 of 343 less) and R0, P0 and A1 at
        // 160x160x40 (6, 11 and 9 of 550 with half the lanes).
        C.lanes[0] = lanes_for(L.A, true);
        C.lanes[1] = lanes_for(L.R, true);
        C.lanes[2] = lanes_for(L.P, true);
    }
    if (h->opts.autotune) BD_TRY(p32 ? tune<float>(h, E, s) : tune<double>(h, E, s));
    for (int l = 0; l < nl - 1; l++)
        for (int op = 0; op < 3; op++) {
            E.lev[l].chosen[op] = E.lev[l].lanes[op];
            E.lev[l].block[op] = h->lev[l].lanes[op];
        }
    const int n = h->nc / 2;
    BD_TRY(E.cinv.alloc((size_t)n * n));
    k_uu_dense<<<grid_for((long long)n * n, 256), 256, 0, s>>>(n, h->cinv.p, E.cinv.p); ::bd::note_launch();
    BD_LAUNCH_CHECK();
    const size_t N = (size_t)L0.N;
    for (DBuf<double> *v : {&E.fin, &E.fp, &E.x, &E.r, &E.z, &E.p, &E.q}) BD_TRY(v->alloc(N));
    if (p32) {
        BD_TRY(E.zold.alloc(N));
        BD_CUDA(cudaMemsetAsync(E.zold.p, 0, E.zold.bytes(), s));
    }
    BD_TRY(E.partial.alloc(kPart * (size_t)kRedBlocks));
    BD_TRY(E.scal.alloc(S_NSLOTS));
    BD_TRY(E.counter.alloc(1));
    BD_CUDA(cudaMemsetAsync(E.counter.p, 0, sizeof(unsigned int), s));
    BD_CUDA(cudaMallocHost((void **)&E.host, 2 * sizeof(double) * S_NSLOTS));
    BD_CUDA(cudaStreamCreateWithFlags(&E.cap, cudaStreamNonBlocking));
    BD_CUDA(cudaStreamCreateWithFlags(&E.cap2, cudaStreamNonBlocking));
    BD_CUDA(cudaEventCreate(&E.ev[0]));
    BD_CUDA(cudaEventCreate(&E.ev[1]));
    BD_CUDA(cudaStreamSynchronize(s));
    h->scalar = up;
    return BD_OK;
}

void scalar_set_lanes(amg_hierarchy *h, int level, int op, int T)
{
    if (!h->scalar) return;
    h->scalar->drop_graph();
    ScLevel &C = h->scalar->lev[level];
    C.lanes[op] = T == C.block[op] ? C.chosen[op] : std::abs(T);
}

namespace {

// One V-cycle on the u_e field; the finest level's input is in lev[0].d and f0.
// FP64: the last step writes z and its statistics (zf) unless there is one level.
template <class S>
int vcycle1(amg_hierarchy *h, const S *f0, const Fin &zf, cudaStream_t s)
{
    ScalarEll &E = *h->scalar;
    const int nl = h->nlev, N0 = h->lev[0].N;
    auto P = [&](Arr &a) { return Buf<S>::p(a); };
    for (int l = 0; l < nl - 1; l++) {
        Level &L = h->lev[l];
        ScLevel &C = E.lev[l], &D = E.lev[l + 1];
        const S *f = l == 0 ? f0 : P(C.f);
        if (l == 0) {
            BD_TRY(sc_apply(E.op, (const S *)P(C.d), [&] { return S1Pre<S>{f, P(C.u)}; }, s));
            BD_TRY(sc_apply(E.op, (const S *)P(C.u), [&] { return S1Resid<S>{f, P(C.r)}; }, s));
        } else {
            BD_TRY(csr<S>(L.A, C.A, C.lanes[0], P(C.d), E1Pre<S>{f, P(C.invd), P(C.d), P(C.u), (S)L.ch_c1, (S)L.ch_c2}, s));
            BD_TRY(csr<S>(L.A, C.A, C.lanes[0], P(C.u), E1Resid<S>{f, P(C.r)}, s));
        }
        BD_TRY(csr<S>(L.R, C.R, C.lanes[1], P(C.r),
                      E1Restrict<S>{P(D.f), P(D.d), P(D.invd), (S)h->lev[l + 1].ch_inv_theta}, s));
    }
    ScLevel &K = E.lev[nl - 1];
    BD_TRY(coarse_solve(h->nc / 2, E.cinv.p, nl == 1 ? f0 : (const S *)P(K.f), P(K.u), s));
    for (int l = nl - 2; l >= 0; l--) {
        Level &L = h->lev[l];
        ScLevel &C = E.lev[l], &D = E.lev[l + 1];
        const S *f = l == 0 ? f0 : P(C.f);
        BD_TRY(csr<S>(L.P, C.P, C.lanes[2], P(D.u), E1Add<S>{P(C.u)}, s));
        if (l > 0) {
            BD_TRY(csr<S>(L.A, C.A, C.lanes[0], P(C.u),
                          E1Post1<S>{f, P(C.invd), P(C.r), P(C.d), (S)L.ch_inv_theta}, s));
            BD_TRY(csr<S>(L.A, C.A, C.lanes[0], P(C.d),
                          E1Post2<S>{P(C.r), P(C.d), P(C.invd), P(C.u), (S)L.ch_c1, (S)L.ch_c2}, s));
            continue;
        }
        BD_TRY(sc_apply(E.op, (const S *)P(C.u), [&] { return S1Post1<S>{f, P(C.r), P(C.d)}; }, s));
        if constexpr (std::is_same<S, double>::value) {
            const S1Z e{{P(C.r), P(C.u)}, E.z.p, E.r.p, 0.0, 0.0, 0.0};
            if (E.op.sym) k1_z<true><<<E.op.blocks<S>(), kFineTPB, 0, s>>>(E.op.grid<S>(), P(C.d), e, zf);
            else k1_z<false><<<E.op.blocks<S>(), kFineTPB, 0, s>>>(E.op.grid<S>(), P(C.d), e, zf);
            ::bd::note_launch();
            BD_LAUNCH_CHECK();
            return BD_OK;
        } else {
            BD_TRY(sc_apply(E.op, (const S *)P(C.d), [&] { return S1Post2<S>{P(C.r), P(C.u)}; }, s));
        }
    }
    k1_z_from<S><<<kVecBlocks, kVecThreads, 0, s>>>(N0, P(E.lev[0].u), E.r.p, h->prec32 ? E.zold.p : nullptr, E.z.p, zf);
    ::bd::note_launch();
    BD_LAUNCH_CHECK();
    return BD_OK;
}

template <int MODE, class S>
int reduce1(ScalarEll &E, const double *x, const S1Reduce<MODE, S> &e, const Fin &fin, cudaStream_t s)
{
    if (E.op.sym) k1_reduce<MODE, true, S><<<E.op.blocks<double>(), kFineTPB, 0, s>>>(E.op.grid<double>(), x, e, fin);
    else k1_reduce<MODE, false, S><<<E.op.blocks<double>(), kFineTPB, 0, s>>>(E.op.grid<double>(), x, e, fin);
    ::bd::note_launch();
    BD_LAUNCH_CHECK();
    return BD_OK;
}

template <class S> int capture(amg_hierarchy *h)
{
    ScalarEll &E = *h->scalar;
    const int N = h->lev[0].N;
    cudaStream_t s = E.cap, s2 = E.cap2;
    ScLevel &C0 = E.lev[0];
    auto fin = [&](int stage, cudaGraphConditionalHandle cond = 0) {
        return Fin{E.scal.p, E.partial.p, E.counter.p, stage, N, -1, h->prec32 ? 1 : 0, cond};
    };
    const S1In<S> in{Buf<S>::p(C0.f), h->nlev > 1 ? Buf<S>::p(C0.d) : nullptr, Buf<S>::p(C0.invd),
                     (S)h->lev[0].ch_inv_theta};
    BD_CUDA(cudaStreamBeginCapture(s, cudaStreamCaptureModeThreadLocal));
    const long long c0 = launch_count();
    k1_f_stats<<<kVecBlocks, kVecThreads, 0, s>>>(N, E.fin.p, fin(0)); ::bd::note_launch();
    k1_project_f<<<kVecBlocks, kVecThreads, 0, s>>>(N, E.fin.p, E.fp.p, E.x.p, fin(1)); ::bd::note_launch();
    BD_LAUNCH_CHECK();
    WhileNode w;
    BD_TRY(while_handle(s, &w));
    BD_TRY((reduce1<1, S>(E, E.x.p, S1Reduce<1, S>{E.fp.p, E.r.p, in, 0.0, 0.0}, fin(6, w.cond), s)));
    BD_TRY(while_begin(s, s2, &w));
    const long long c1 = launch_count();
    const S *f0;
    if constexpr (std::is_same<S, double>::value) f0 = E.r.p;
    else f0 = C0.f.p32.p;
    BD_TRY(vcycle1<S>(h, f0, fin(3), s2));
    k1_p_update<<<kVecBlocks, kVecThreads, 0, s2>>>(N, E.z.p, E.p.p, h->prec32 ? E.zold.p : nullptr, E.scal.p);
    ::bd::note_launch();
    BD_TRY((reduce1<0, S>(E, E.p.p, S1Reduce<0, S>{nullptr, E.q.p, in, 0.0, 0.0}, fin(4), s2)));
    k1_xr_update<S><<<kVecBlocks, kVecThreads, 0, s2>>>(N, E.x.p, E.r.p, E.p.p, E.q.p, in, fin(7, w.cond));
    ::bd::note_launch();
    BD_LAUNCH_CHECK();
    const long long c2 = launch_count();
    BD_TRY(while_end(s, s2, &w));
    BD_TRY((reduce1<1, S>(E, E.x.p, S1Reduce<1, S>{E.fp.p, nullptr, in, 0.0, 0.0}, fin(5), s)));
    k1_project_x<<<kVecBlocks, kVecThreads, 0, s>>>(N, E.x.p, E.scal.p); ::bd::note_launch();
    BD_LAUNCH_CHECK();
    const long long c3 = launch_count();
    BD_CUDA(cudaStreamEndCapture(s, &E.graph));
    BD_CUDA(cudaGraphInstantiate(&E.exec, E.graph, 0));
    E.pre = c1 - c0;
    E.body = c2 - c1;
    E.post = c3 - c2;
    note_launches(-(c3 - c0));
    return BD_OK;
}

}  // namespace

bool scalar_ready(amg_hierarchy *h, const solve_options *o)
{
    if (!h->scalar || h->prof || o->strict || solve_graph_off()) return false;
    ScalarEll &E = *h->scalar;
    if (!E.exec && !E.failed) {
        const int st = h->prec32 ? capture<float>(h) : capture<double>(h);
        if (st != BD_OK) {
            drop_capture(E.cap2);
            drop_capture(E.cap);
            E.drop_graph();
            E.failed = true;
        }
    }
    return E.exec != nullptr;
}

int scalar_solve(amg_hierarchy *h, const double *f, double *x, const solve_options *o, cudaStream_t s, solve_info *info)
{
    ScalarEll &E = *h->scalar;
    const size_t bytes = sizeof(double) * (size_t)h->lev[0].N;
    double *in = E.host, *out = E.host + S_NSLOTS;
    for (int i = 0; i < S_NSLOTS; i++) in[i] = 0.0;
    in[S_RTOL] = o->rtol;
    in[S_MAXIT] = (double)o->max_it;
    in[S_WARM] = 1.0;
    BD_CUDA(cudaEventRecord(E.ev[0], s));
    BD_CUDA(cudaMemcpyAsync(E.fin.p, f, bytes, cudaMemcpyDeviceToDevice, s));
    BD_CUDA(cudaMemcpyAsync(E.x.p, x, bytes, cudaMemcpyDeviceToDevice, s));
    BD_CUDA(cudaMemcpyAsync(E.scal.p, in, sizeof(double) * S_NSLOTS, cudaMemcpyHostToDevice, s));
    BD_CUDA(cudaGraphLaunch(E.exec, s));
    BD_CUDA(cudaMemcpyAsync(x, E.x.p, bytes, cudaMemcpyDeviceToDevice, s));
    BD_CUDA(cudaEventRecord(E.ev[1], s));
    BD_CUDA(cudaMemcpyAsync(out, E.scal.p, sizeof(double) * S_NSLOTS, cudaMemcpyDeviceToHost, s));
    BD_CUDA(cudaStreamSynchronize(s));
    float ms = 0.0f;
    cudaEventElapsedTime(&ms, E.ev[0], E.ev[1]);
    note_launches(E.pre + E.post + (long long)out[S_IT] * E.body);
    return info_from_scal(out, ms, info);
}

}  // namespace bd
