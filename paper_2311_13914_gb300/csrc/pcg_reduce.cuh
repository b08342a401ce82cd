// pcg_reduce.cuh -- deterministic reductions of the PCG kernels with the
// recurrence's scalar stage applied by the last block: shared by the block
// system's solve (amg_solve.cu) and the decoupled scheme's scalar ones
// (amg_scalar.cu).
#pragma once

#include "amg_internal.cuh"

namespace bd {

// ------------------------------------------------------------------ vector kernels' shares
// Block b's share [share_lo(n), share_hi(n)) of n rows or nodes: the grid
// splits the 32-row slices in equal contiguous parts, so with one resident
// wave of blocks every SM gets the same work (a grid-stride loop leaves the
// SMs whose blocks drew one row fewer per thread idle for part of the launch).
static __device__ __forceinline__ int share_lo(int n)
{
    return (int)((((long long)n + 31) >> 5) * blockIdx.x / gridDim.x) * 32;
}
static __device__ __forceinline__ int share_hi(int n)
{
    return min(n, (int)((((long long)n + 31) >> 5) * (blockIdx.x + 1) / gridDim.x) * 32);
}

// body(i, ld(i)) for the block's share of n, the next entry's values loaded before
// the present ones are used.  The warps of a block start together, and without
// that all wait for their loads, then all queue for the FP64 pipe, one after the
// other (256x256x64 nodes, x and r: 91 -> 88 us; 96x96x24, an iteration with the
// FP32 V-cycle: 181.5 -> 179.2).
template <class L, class B> static __device__ __forceinline__ void share_stream(int n, const L &ld, B &&body)
{
    const int e = share_hi(n);
    int i = share_lo(n) + threadIdx.x;
    if (i >= e) return;
    auto cur = ld(i);
    for (;;) {
        const int k = i + blockDim.x;
        const bool more = k < e;
        const auto nxt = ld(more ? k : i);
        body(i, cur);
        if (!more) return;
        cur = nxt;
        i = k;
    }
}

// ------------------------------------------------------------------ PCG reductions
// scal[] slots of the device scalars
enum {
    S_SUMFU = 0, S_FF, S_NF2, S_RR, S_RZ, S_PQ, S_ALPHA, S_BETA, S_MEANZ,
    S_BREAK, S_MEANF, S_TRR, S_MEANX,
    // device-side loop control of the graph form
    S_RTOL, S_MAXIT, S_WARM, S_IT, S_STATUS,
    S_NSLOTS
};
constexpr int kPart = 4;  // partial sums per block
// Grid of the PCG vector kernels: one resident wave of fewer, larger blocks
// than kRedBlocks, so the last block's reduction of the partials is shorter.
constexpr int kVecBlocks = 608, kVecThreads = 256;
constexpr int kMaxBlockThreads = 256;  // largest block of a reduction kernel

// What the last block of a reduction kernel does with the totals.
// first < 0: "first iteration" is read from the device iteration counter
// (graph form).  Stages 6 and 7 are the graph form's loop control: 6 opens
// the loop after the initial residual, 7 closes an iteration; both set the
// WHILE node's condition.
struct Fin {
    double *scal;
    double *partial;
    unsigned int *counter;
    int stage, N, first, flex;
    cudaGraphConditionalHandle cond;
};

static __device__ void finish_stage(const Fin &f, double a, double b, double c, double d)
{
    double *scal = f.scal;
    const int N = f.N;
    const int first = f.first < 0 ? (scal[S_IT] == 0.0) : f.first;
    switch (f.stage) {
    case 0:  // f statistics: sum f_u, ||f||^2
        scal[S_SUMFU] = a;
        scal[S_FF] = b;
        scal[S_MEANF] = a / N;
        break;
    case 1:  // ||fp||^2
        scal[S_NF2] = a;
        break;
    case 2:  // ||r||^2
        scal[S_RR] = a;
        break;
    case 3: {  // z statistics: sum z_u, sum r_u, r.z, r.z_old
        double mz = a / N;
        double rz = c - mz * b;  // r . (z projected)
        scal[S_MEANZ] = mz;
        // standard CG: beta = rz_new / rz_old; flexible (Polak-Ribiere):
        // beta = (r.z_new - r.z_old) / rz_old with z_old the previous projected z
        double num = f.flex ? rz - d : rz;
        scal[S_BETA] = first ? 0.0 : num / scal[S_RZ];
        scal[S_RZ] = rz;
        break;
    }
    case 4:  // p.q
        scal[S_PQ] = a;
        if (!(a > 0.0) || !isfinite(a) || !isfinite(scal[S_RZ])) scal[S_BREAK] = 1.0;
        scal[S_ALPHA] = scal[S_RZ] / a;
        break;
    case 5:  // true residual and mean of x_u
        scal[S_TRR] = a;
        scal[S_MEANX] = b / N;
        break;
    case 6: {  // initial ||r||^2; open the loop unless already converged
        scal[S_RR] = a;
        const double nf = sqrt(scal[S_NF2]);
        const bool go = nf > 0.0 && !(sqrt(a) <= scal[S_RTOL] * nf) && scal[S_MAXIT] > 0.0;
        scal[S_IT] = 0.0;
        scal[S_STATUS] = go ? (double)BD_ENOTCONV : (double)BD_OK;
        cudaGraphSetConditional(f.cond, go ? 1u : 0u);
        break;
    }
    case 7: {  // ||r||^2 after the update; close or continue the loop
        scal[S_RR] = a;
        const double it = scal[S_IT] + 1.0;
        scal[S_IT] = it;
        const double nf = sqrt(scal[S_NF2]), rr = sqrt(a);
        bool go = true;
        if (scal[S_BREAK] != 0.0 || !isfinite(rr)) {
            scal[S_STATUS] = (double)BD_EBREAKDOWN;
            go = false;
        } else if (rr <= scal[S_RTOL] * nf) {
            scal[S_STATUS] = (double)BD_OK;
            go = false;
        } else if (it >= scal[S_MAXIT]) {
            go = false;  // status stays BD_ENOTCONV
        }
        cudaGraphSetConditional(f.cond, go ? 1u : 0u);
        break;
    }
    // the decoupled scheme's parabolic CG (no null space; its loop also runs
    // host-driven, without a condition: S_WARM then tells the host to go on)
    case 9: {  // initial ||r||^2, r.z, ||b||^2
        scal[S_RR] = a;
        scal[S_RZ] = b;
        scal[S_NF2] = c;
        const double nf = sqrt(c);
        const bool done = nf == 0.0 || sqrt(a) <= scal[S_RTOL] * nf;
        if (nf == 0.0) scal[S_RR] = 0.0;
        scal[S_IT] = 0.0;
        scal[S_STATUS] = done ? (double)BD_OK : (double)BD_ENOTCONV;
        const bool go = !done && scal[S_MAXIT] > 0.0;
        scal[S_WARM] = go ? 1.0 : 0.0;
        if (f.cond) cudaGraphSetConditional(f.cond, go ? 1u : 0u);
        break;
    }
    case 10:  // p.q
        scal[S_PQ] = a;
        if (!(a > 0.0) || !isfinite(a)) scal[S_BREAK] = 1.0;
        scal[S_ALPHA] = scal[S_RZ] / a;
        break;
    case 8: {  // ||r||^2 and r.z after the update (none after a breakdown)
        bool go = false;
        if (scal[S_BREAK] != 0.0) {
            scal[S_STATUS] = (double)BD_EBREAKDOWN;
        } else {
            scal[S_RR] = a;
            const double it = scal[S_IT] + 1.0;
            scal[S_IT] = it;
            if (sqrt(a) <= scal[S_RTOL] * sqrt(scal[S_NF2])) scal[S_STATUS] = (double)BD_OK;
            else go = it < scal[S_MAXIT];
            scal[S_BETA] = b / scal[S_RZ];
            scal[S_RZ] = b;
        }
        scal[S_WARM] = go ? 1.0 : 0.0;
        if (f.cond) cudaGraphSetConditional(f.cond, go ? 1u : 0u);
        break;
    }
    case 11:  // true residual
        scal[S_TRR] = a;
        break;
    }
}

// Block sums of the first NV of a thread's values, in a fixed order: every
// thread stores its values, then warp k adds column k (the entries of lanes
// l, l + 32, ... in index order) and folds its 32 lane sums by shuffles into
// tot[k].  That is 12 FP64 warp additions per value and block for 256 threads
// (36 for 1024), where a shuffle tree in every warp costs 45 for 256.
template <int NV, int BT>
static __device__ __forceinline__ void block_sum(const double (&v)[4], double (*buf)[BT], double *tot)
{
#pragma unroll
    for (int k = 0; k < NV; k++) buf[k][threadIdx.x] = v[k];
    __syncthreads();
    const int w = threadIdx.x >> 5, l = threadIdx.x & 31;
    if (w < NV) {
        double t = buf[w][l];
        for (int i = l + 32; i < (int)blockDim.x; i += 32) t += buf[w][i];
        for (int o = 16; o; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
        if (l == 0) tot[w] = t;
    }
    __syncthreads();
}

// Block sums -> partial[blockIdx]; the last block to arrive reduces all
// partials in a fixed order (independent of which block is last, so the
// result is reproducible) and applies the stage.  No waiting: blocks that are
// not last simply exit.  NV of (a, b, c, d) are live; the stage sees zeros for
// the rest.  Needs blockDim.x <= BT and a multiple of 32 (the shared buffer
// holds BT values per sum: kernels of 256 threads keep the rest of shared
// memory for L1).
template <int NV, int BT = kMaxBlockThreads>
static __device__ void block_finish(double a, double b, double c, double d, const Fin &f)
{
    __shared__ double buf[NV][BT];
    __shared__ double tot[4];
    __shared__ bool last;
    double v[4] = {a, b, c, d};
    block_sum<NV, BT>(v, buf, tot);
    if (threadIdx.x == 0) {
        double *o = f.partial + kPart * blockIdx.x;
#pragma unroll
        for (int k = 0; k < NV; k++) o[k] = tot[k];
        __threadfence();
        const unsigned int ticket = atomicAdd(f.counter, 1u);
        last = ticket == gridDim.x - 1;
    }
    __syncthreads();
    if (!last) return;
    __threadfence();
#pragma unroll
    for (int k = 0; k < 4; k++) v[k] = 0.0;
    // L2 loads (the partials were published by the other blocks' fences and
    // tickets), not volatile ones, so that the unrolled loads of several
    // partials are in flight together: the last block's serial tail
#pragma unroll 4
    for (int i = threadIdx.x; i < (int)gridDim.x; i += blockDim.x) {
        const double *q = f.partial + kPart * i;
#pragma unroll
        for (int k = 0; k < NV; k++) v[k] += __ldcg(q + k);
    }
    block_sum<NV, BT>(v, buf, tot);
    if (threadIdx.x == 0) {
        finish_stage(f, tot[0], NV > 1 ? tot[1] : 0.0, NV > 2 ? tot[2] : 0.0, NV > 3 ? tot[3] : 0.0);
        *f.counter = 0u;
    }
}

}  // namespace bd
