// bd_decoupled.cu -- the paper's own time-stepping scheme (Section 2.2,
// Eqs. 4-7 as printed): per step the gating update (Eq. 4), the elliptic
// system (Ai + Ae) u_e^n = -Ai v^n (Eq. 6) by AMG-PCG, then the parabolic
// system (c M + Ai) v^{n+1} = c M v^n - Ai u_e^n + M (I_app - chi I_ion)
// (Eq. 7, ionic sign as in the coupled step) by CG, Jacobi-preconditioned or
// unpreconditioned (the paper's GPU runs leave it unpreconditioned).
//
// The elliptic hierarchy is the block hierarchy of [I, 0; 0, Ai + Ae]
// (bd_elliptic_setup), solved on its one field (amg_scalar.cu).  Ai and c M + Ai
// are scalar layered stencils (fine_scalar.cuh).  The parabolic CG runs as one
// CUDA graph: three kernels per iteration under a WHILE node whose condition the
// last reduction sets; the host synchronises once per solve, where a host-driven
// loop read 1216 partial sums back twice per iteration (128x128x32, 24
// iterations: 3.9 -> 1.25 ms).  Reductions sum in a fixed order, so it is
// reproducible run to run.
#include <cmath>
#include <new>

#include "amg_internal.cuh"
#include "fine_scalar.cuh"
#include "pcg_reduce.cuh"
#include "scalar.cuh"

namespace bd {
namespace {

// elliptic right-hand side -Ai v
struct DEllRhs {
    double *__restrict__ f;
    __device__ __forceinline__ int load(int, bool) const { return 0; }
    __device__ __forceinline__ void operator()(int p, const double *, int, double, double, double y) { f[p] = -y; }
};

// gating update (Eq. 4) and parabolic right-hand side (Eq. 7); y = Ai u_e
struct DParRhs {
    const double *__restrict__ M, *__restrict__ stim, *__restrict__ v;
    double *__restrict__ w, *__restrict__ b;
    double chi, cm, dt;
    bd_rm_params rm;
    int stim_on;
    struct Pre {
        double M, stim, v, w;
    };
    __device__ __forceinline__ Pre load(int p, bool ok) const
    {
        return ok ? Pre{M[p], stim_on ? stim[p] : 0.0, v[p], w[p]} : Pre{0.0, 0.0, 0.0, 0.0};
    }
    __device__ __forceinline__ void operator()(int p, const double *, const Pre &q, double, double, double y)
    {
        const double c = (chi * cm) / dt;
        const double wn = (q.w + dt * rm.eta2 * q.v / rm.vp) / (1.0 + dt * rm.eta2 * rm.eta3);
        const double iion = rm.G * q.v * (1.0 - q.v / rm.vth) * (1.0 - q.v / rm.vp) + rm.eta1 * q.v * wn;
        b[p] = c * q.M * q.v - y + q.M * (q.stim - chi * iion);
        w[p] = wn;
    }
};

// r = b - A v; partials r.r, r.D^{-1}r, b.b
struct DResid {
    const double *__restrict__ b, *__restrict__ dinv;
    double *__restrict__ r;
    double rr, rz, bb;
    struct Pre {
        double b, d;
    };
    __device__ __forceinline__ Pre load(int p, bool ok) const { return ok ? Pre{b[p], dinv[p]} : Pre{0.0, 0.0}; }
    __device__ __forceinline__ void operator()(int p, const double *, const Pre &q, double, double, double y)
    {
        const double rv = q.b - y;
        r[p] = rv;
        rr += rv * rv;
        rz += rv * (q.d * rv);
        bb += q.b * q.b;
    }
};
template <bool SYM>
__global__ void __launch_bounds__(kFineTPB, ScMinB<double>::v)
    k_par_resid(ScGrid g, const double *__restrict__ v, DResid e, Fin fin)
{
    sc_block<double, SYM>(g, v, e);
    block_finish<3, kFineTPB>(e.rr, e.rz, e.bb, 0.0, fin);
}

// q = A p; partial p.q
struct DApply {
    double *__restrict__ q;
    double pq;
    __device__ __forceinline__ int load(int, bool) const { return 0; }
    __device__ __forceinline__ void operator()(int p, const double *, int, double c, double, double y)
    {
        q[p] = y;
        pq = fma(c, y, pq);
    }
};
template <bool SYM>
__global__ void __launch_bounds__(kFineTPB, ScMinB<double>::v)
    k_par_apply(ScGrid g, const double *__restrict__ p, DApply e, Fin fin)
{
    sc_block<double, SYM>(g, p, e);
    block_finish<1, kFineTPB>(e.pq, 0.0, 0.0, 0.0, fin);
}

// p = D^{-1} r, + beta p after the first iteration
__global__ void k_par_direction(int N, const double *__restrict__ dinv, const double *__restrict__ r,
                                double *__restrict__ p, const double *__restrict__ scal)
{
    const double beta = scal[S_BETA];
    const bool first = scal[S_IT] == 0.0;
    struct In {
        double d, r, p;
    };
    share_stream(N, [&](int i) { return In{dinv[i], r[i], p[i]}; }, [&](int i, const In &q) {
        const double z = q.d * q.r;
        p[i] = first ? z : fma(beta, q.p, z);
    });
}

// v += alpha p, r -= alpha q; partials r.r, r.D^{-1}r
__global__ void k_par_update(int N, const double *__restrict__ p, const double *__restrict__ q,
                             const double *__restrict__ dinv, double *__restrict__ v, double *__restrict__ r, Fin fin)
{
    const double alpha = fin.scal[S_ALPHA];
    struct In {
        double p, q, d, v, r;
    };
    double rr = 0.0, rz = 0.0;
    if (fin.scal[S_BREAK] == 0.0)
        share_stream(N, [&](int i) { return In{p[i], q[i], dinv[i], v[i], r[i]}; }, [&](int i, const In &k) {
            v[i] = fma(alpha, k.p, k.v);
            const double rv = fma(-alpha, k.q, k.r);
            r[i] = rv;
            rr += rv * rv;
            rz += rv * (k.d * rv);
        });
    block_finish<2>(rr, rz, 0.0, 0.0, fin);
}

// v = 0 for a zero right-hand side
__global__ void k_par_zero(int N, double *__restrict__ v, const double *__restrict__ scal)
{
    if (scal[S_NF2] != 0.0) return;
    for (int i = share_lo(N) + threadIdx.x, e = share_hi(N); i < e; i += blockDim.x) v[i] = 0.0;
}

// inverse diagonal of c M + Ai (ones when unpreconditioned)
__global__ void k_par_dinv(int N, const int *__restrict__ rp, const int *__restrict__ ci,
                           const double *__restrict__ Ki, const double *__restrict__ M, double c, int jacobi,
                           double *__restrict__ dinv)
{
    for (int p = blockIdx.x * blockDim.x + threadIdx.x; p < N; p += gridDim.x * blockDim.x) {
        double d = c * M[p];
        for (int t = rp[p]; t < rp[p + 1]; t++)
            if (ci[t] == p) d = d + Ki[t];
        dinv[p] = jacobi ? 1.0 / d : 1.0;
    }
}

// (0, u) pairs of the block solve
__global__ void k_split(int N, const double2 *__restrict__ xe, double *__restrict__ ue)
{
    for (int p = blockIdx.x * blockDim.x + threadIdx.x; p < N; p += gridDim.x * blockDim.x) ue[p] = xe[p].y;
}
__global__ void k_join(int N, const double *__restrict__ ue, double2 *__restrict__ xe)
{
    for (int p = blockIdx.x * blockDim.x + threadIdx.x; p < N; p += gridDim.x * blockDim.x)
        xe[p] = make_double2(0.0, ue[p]);
}

}  // namespace
}  // namespace bd

struct bd_dsim {
    const bd_system *sys = nullptr;
    amg_hierarchy *h = nullptr;
    bd_rm_params rm{};
    int N = 0, jacobi = 1;
    long long step = 0;
    double stim_ms = 0.0;
    bd::FineStencil raw;
    bd::ScOp ki, par;              // Ai; c M + Ai
    bd::DBuf<double> v, w, stim, ue;  // N each
    bd::DBuf<double> f;            // elliptic right-hand side
    bd::DBuf<double> xe, fe;       // block solve only: (0, u_e) pairs
    bd::DBuf<double> b, r, p, q, dinv, partial, scal;
    bd::DBuf<unsigned int> counter;
    double *host = nullptr;        // pinned: initial scalars, then results
    cudaEvent_t ev[2] = {nullptr, nullptr};
    cudaGraph_t graph = nullptr;
    cudaGraphExec_t exec = nullptr;
    cudaStream_t cap = nullptr, cap2 = nullptr;
    bool graph_failed = false;
    ~bd_dsim()
    {
        if (exec) cudaGraphExecDestroy(exec);
        if (graph) cudaGraphDestroy(graph);
        if (cap) cudaStreamDestroy(cap);
        if (cap2) cudaStreamDestroy(cap2);
        if (host) cudaFreeHost(host);
        if (ev[0]) cudaEventDestroy(ev[0]);
        if (ev[1]) cudaEventDestroy(ev[1]);
    }
};

using namespace bd;

namespace {

constexpr int kParBody = 3;  // kernels of an iteration

Fin par_fin(bd_dsim *S, int stage, cudaGraphConditionalHandle cond = 0)
{
    return Fin{S->scal.p, S->partial.p, S->counter.p, stage, S->N, -1, 0, cond};
}

int par_resid(bd_dsim *S, const Fin &fin, cudaStream_t s)
{
    const DResid e{S->b.p, S->dinv.p, S->r.p, 0.0, 0.0, 0.0};
    const int grid = S->par.blocks<double>();
    if (S->par.sym) k_par_resid<true><<<grid, kFineTPB, 0, s>>>(S->par.grid<double>(), S->v.p, e, fin);
    else k_par_resid<false><<<grid, kFineTPB, 0, s>>>(S->par.grid<double>(), S->v.p, e, fin);
    note_launch();
    BD_LAUNCH_CHECK();
    return BD_OK;
}

int par_body(bd_dsim *S, cudaGraphConditionalHandle cond, cudaStream_t s)
{
    const int N = S->N, grid = S->par.blocks<double>();
    k_par_direction<<<kVecBlocks, kVecThreads, 0, s>>>(N, S->dinv.p, S->r.p, S->p.p, S->scal.p); note_launch();
    const DApply e{S->q.p, 0.0};
    if (S->par.sym) k_par_apply<true><<<grid, kFineTPB, 0, s>>>(S->par.grid<double>(), S->p.p, e, par_fin(S, 10));
    else k_par_apply<false><<<grid, kFineTPB, 0, s>>>(S->par.grid<double>(), S->p.p, e, par_fin(S, 10));
    note_launch();
    k_par_update<<<kVecBlocks, kVecThreads, 0, s>>>(N, S->p.p, S->q.p, S->dinv.p, S->v.p, S->r.p, par_fin(S, 8, cond));
    note_launch();
    BD_LAUNCH_CHECK();
    return BD_OK;
}

int par_post(bd_dsim *S, cudaStream_t s)
{
    k_par_zero<<<kVecBlocks, kVecThreads, 0, s>>>(S->N, S->v.p, S->scal.p); note_launch();
    return par_resid(S, par_fin(S, 11), s);
}

int par_capture(bd_dsim *S)
{
    if (!S->cap) BD_CUDA(cudaStreamCreateWithFlags(&S->cap, cudaStreamNonBlocking));
    if (!S->cap2) BD_CUDA(cudaStreamCreateWithFlags(&S->cap2, cudaStreamNonBlocking));
    const long long c0 = launch_count();
    BD_CUDA(cudaStreamBeginCapture(S->cap, cudaStreamCaptureModeThreadLocal));
    WhileNode w;
    BD_TRY(while_handle(S->cap, &w));
    BD_TRY(par_resid(S, par_fin(S, 9, w.cond), S->cap));
    BD_TRY(while_begin(S->cap, S->cap2, &w));
    BD_TRY(par_body(S, w.cond, S->cap2));
    BD_TRY(while_end(S->cap, S->cap2, &w));
    BD_TRY(par_post(S, S->cap));
    BD_CUDA(cudaStreamEndCapture(S->cap, &S->graph));
    BD_CUDA(cudaGraphInstantiate(&S->exec, S->graph, 0));
    note_launches(-(launch_count() - c0));
    return BD_OK;
}

// (c M + Ai) v = b by (Jacobi-)CG from the current v; iterations, the recurrence
// and true residuals and the device time into info
int parabolic_cg(bd_dsim *S, const solve_options *o, cudaStream_t s, solve_info *info)
{
    double *in = S->host, *out = S->host + S_NSLOTS;
    for (int i = 0; i < S_NSLOTS; i++) in[i] = 0.0;
    in[S_RTOL] = o->rtol;
    in[S_MAXIT] = (double)o->max_it;
    BD_CUDA(cudaEventRecord(S->ev[0], s));
    BD_CUDA(cudaMemcpyAsync(S->scal.p, in, sizeof(double) * S_NSLOTS, cudaMemcpyHostToDevice, s));
    if (!S->exec && !S->graph_failed && !solve_graph_off() && par_capture(S) != BD_OK) {
        drop_capture(S->cap2);
        drop_capture(S->cap);
        if (S->graph) cudaGraphDestroy(S->graph);
        S->graph = nullptr;
        S->exec = nullptr;
        S->graph_failed = true;
    }
    auto fetch = [&]() {
        BD_CUDA(cudaMemcpyAsync(out, S->scal.p, sizeof(double) * S_NSLOTS, cudaMemcpyDeviceToHost, s));
        BD_CUDA(cudaStreamSynchronize(s));
        return BD_OK;
    };
    if (S->exec) {
        BD_CUDA(cudaGraphLaunch(S->exec, s));
    } else {
        BD_TRY(par_resid(S, par_fin(S, 9), s));
        for (;;) {
            BD_TRY(fetch());
            if (out[S_WARM] == 0.0) break;
            BD_TRY(par_body(S, 0, s));
        }
        BD_TRY(par_post(S, s));
    }
    BD_CUDA(cudaEventRecord(S->ev[1], s));
    BD_TRY(fetch());
    if (S->exec) note_launches(3 + (long long)out[S_IT] * kParBody);
    float ms = 0.0f;
    cudaEventElapsedTime(&ms, S->ev[0], S->ev[1]);
    return info_from_scal(out, ms, info);
}

// (Ai + Ae) u_e = f from the current u_e
int elliptic_solve(bd_dsim *S, const solve_options *o, cudaStream_t s, solve_info *info)
{
    if (scalar_ready(S->h, o)) return scalar_solve(S->h, S->f.p, S->ue.p, o, s, info);
    const size_t n = 2 * (size_t)S->N;
    if (!S->xe.p) {
        BD_TRY(S->xe.alloc(n));
        BD_TRY(S->fe.alloc(n));
    }
    const int grid = grid_for(S->N, 256);
    k_join<<<grid, 256, 0, s>>>(S->N, S->f.p, (double2 *)S->fe.p); note_launch();
    k_join<<<grid, 256, 0, s>>>(S->N, S->ue.p, (double2 *)S->xe.p); note_launch();
    BD_LAUNCH_CHECK();
    const int st = pcg_solve_device(S->h, S->fe.p, S->xe.p, 1, o, s, info);
    k_split<<<grid, 256, 0, s>>>(S->N, (const double2 *)S->xe.p, S->ue.p); note_launch();
    BD_LAUNCH_CHECK();
    return st;
}

}  // namespace

extern "C" int bd_dsim_create(const bd_system *sys, amg_hierarchy *h_elliptic, const bd_rm_params *rm,
                              const double *stim, int stim_on_device, double stim_ms, int jacobi, void *stream,
                              bd_dsim **out)
{
    if (!sys || !h_elliptic || !out) return BD_EINVAL;
    *out = nullptr;
    if (h_elliptic->lev[0].N != sys->N || h_elliptic->fine.valid) return BD_EINVAL;
    cudaStream_t s = (cudaStream_t)stream;
    bd_dsim *S = new (std::nothrow) bd_dsim();
    if (!S) return BD_ENOMEM;
    S->sys = sys;
    S->h = h_elliptic;
    if (rm) S->rm = *rm;
    else bd_rm_params_default(&S->rm);
    S->N = sys->N;
    S->jacobi = jacobi ? 1 : 0;
    S->stim_ms = stim ? stim_ms : 0.0;
    const size_t N = (size_t)sys->N;
    int st = BD_OK;
    for (DBuf<double> *d : {&S->v, &S->w, &S->stim, &S->ue, &S->f, &S->b, &S->r, &S->p, &S->q, &S->dinv})
        if (st == BD_OK) st = d->alloc(N);
    if (st || (st = S->partial.alloc(kPart * (size_t)kRedBlocks)) || (st = S->scal.alloc(S_NSLOTS)) ||
        (st = S->counter.alloc(1))) {
        delete S;
        return st;
    }
    if (cudaMallocHost((void **)&S->host, 2 * sizeof(double) * S_NSLOTS) != cudaSuccess ||
        cudaEventCreate(&S->ev[0]) != cudaSuccess || cudaEventCreate(&S->ev[1]) != cudaSuccess) {
        delete S;
        return BD_ECUDA;
    }
    const bd_params &P = sys->params;
    if (cudaMemsetAsync(S->v.p, 0, S->v.bytes(), s) || cudaMemsetAsync(S->w.p, 0, S->w.bytes(), s) ||
        cudaMemsetAsync(S->stim.p, 0, S->stim.bytes(), s) || cudaMemsetAsync(S->ue.p, 0, S->ue.bytes(), s) ||
        cudaMemsetAsync(S->counter.p, 0, S->counter.bytes(), s)) {
        delete S;
        return BD_ECUDA;
    }
    if ((st = fine_raw_copy(S->raw, sys, s)) ||
        (st = sc_pack(S->raw, 1.0, 0.0, 0.0, 0.0, 0.0, 0.0, false, S->ki, s)) ||
        (st = sc_pack(S->raw, 1.0, 0.0, 1.0, 0.0, 0.0, 0.0, false, S->par, s))) {
        delete S;
        return st;
    }
    k_par_dinv<<<grid_for(sys->N, 256), 256, 0, s>>>(sys->N, sys->A.rp.p, sys->A.ci.p, sys->Ki.p, sys->M.p,
                                                     (P.chi * P.cm) / P.dt, S->jacobi, S->dinv.p); note_launch();
    if (cudaGetLastError() != cudaSuccess) {
        delete S;
        return BD_ECUDA;
    }
    if (stim && (st = copy_in(S->stim.p, stim, N * sizeof(double), stim_on_device, s))) {
        delete S;
        return st;
    }
    if (cudaStreamSynchronize(s) != cudaSuccess) {
        delete S;
        return BD_ECUDA;
    }
    *out = S;
    return BD_OK;
}

extern "C" int bd_dsim_set_state(bd_dsim *S, const double *v, const double *ue, const double *w, int on_device,
                                 void *stream)
{
    if (!S) return BD_EINVAL;
    cudaStream_t s = (cudaStream_t)stream;
    const size_t bytes = sizeof(double) * (size_t)S->N;
    if (v) BD_TRY(copy_in(S->v.p, v, bytes, on_device, s));
    if (w) BD_TRY(copy_in(S->w.p, w, bytes, on_device, s));
    if (ue) BD_TRY(copy_in(S->ue.p, ue, bytes, on_device, s));
    BD_CUDA(cudaStreamSynchronize(s));
    return BD_OK;
}

extern "C" int bd_dsim_get_state(const bd_dsim *S, double *v, double *ue, double *w, int on_device, void *stream)
{
    if (!S) return BD_EINVAL;
    cudaStream_t s = (cudaStream_t)stream;
    const size_t bytes = sizeof(double) * (size_t)S->N;
    if (v) BD_TRY(copy_out(v, S->v.p, bytes, on_device, s));
    if (w) BD_TRY(copy_out(w, S->w.p, bytes, on_device, s));
    if (ue) BD_TRY(copy_out(ue, S->ue.p, bytes, on_device, s));
    BD_CUDA(cudaStreamSynchronize(s));
    return BD_OK;
}

extern "C" int bd_dsim_step(bd_dsim *S, int nsteps, const solve_options *opts, void *stream,
                            solve_info *elliptic, solve_info *parabolic)
{
    if (!S || nsteps < 0) return BD_EINVAL;
    solve_options o;
    solve_options_default(&o);
    if (opts) o = *opts;
    if (!(o.rtol > 0.0) || o.max_it < 0) return BD_EINVAL;
    cudaStream_t s = (cudaStream_t)stream;
    const bd_system *sys = S->sys;
    const bd_params &P = sys->params;
    solve_info ie{}, ip{};
    long long te = 0, tp = 0;
    int st = BD_OK;
    for (int k = 0; k < nsteps && st == BD_OK; k++) {
        const double t = (double)S->step * P.dt;
        // Eq. 6: (Ai + Ae) u_e^n = -Ai v^n, warm from the previous u_e
        BD_TRY(sc_apply(S->ki, (const double *)S->v.p, [&] { return DEllRhs{S->f.p}; }, s));
        st = elliptic_solve(S, &o, s, &ie);
        te += ie.iters;
        if (st != BD_OK) break;
        // Eqs. 4 and 7, then the parabolic solve warm from v^n
        BD_TRY(sc_apply(S->ki, (const double *)S->ue.p, [&] {
            return DParRhs{sys->M.p, S->stim.p, S->v.p, S->w.p, S->b.p, P.chi, P.cm, P.dt, S->rm, t < S->stim_ms};
        }, s));
        st = parabolic_cg(S, &o, s, &ip);
        tp += ip.iters;
        S->step++;
    }
    ie.total_iters = te;
    ip.total_iters = tp;
    if (elliptic) *elliptic = ie;
    if (parabolic) *parabolic = ip;
    return st;
}

extern "C" void bd_dsim_destroy(bd_dsim *S) { delete S; }
