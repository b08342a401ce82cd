// fine_scalar.cuh -- one scalar operator of an assembled slab (a combination of
// Ki, Ke and the lumped mass) as a layered stencil: the decoupled scheme's
// elliptic and parabolic operators and the products with Ai in their
// right-hand sides.  The walk, the row types and the symmetric form are those of
// the block operator (fine_stencil.cuh) with one value per node: 4 adds and 15
// multiply-adds, where block CSR took four multiply-adds and 36 bytes per block
// (elliptic, 27 blocks a row) or 12 bytes per node pair (Ai in CSR).
#pragma once

#include "fine_stencil.cuh"

namespace bd {

// Packed row: dz = 0 group (NP coefficients), dz = +1 group, in the general form
// dz = -1, each padded to whole 16-byte words; c2 D^{-1}; D^{-1} / theta.
template <bool SYM> struct ScRow {
    static constexpr int NP = SYM ? 5 : 9;
    static constexpr int G = SYM ? 8 : 12;
    static constexpr int UP = G, DN = 2 * G;
    static constexpr int IDC2 = (SYM ? 2 : 3) * G, IDT = IDC2 + 1;
    static constexpr int LEN = IDC2 + 4;
};

struct ScGrid {
    int NX = 0, NXY = 0, NZ = 0, ncb = 0;
    double c1 = 0.0;
    const void *tab = nullptr;
};

template <int NP> __device__ __forceinline__ void sc_group(const double *__restrict__ t, double (&c)[NP])
{
    const double2 *q = (const double2 *)t;
#pragma unroll
    for (int k = 0; k < NP; k += 2) {
        const double2 v = q[k / 2];
        c[k] = v.x;
        if (k + 1 < NP) c[k + 1] = v.y;
    }
}
template <int NP> __device__ __forceinline__ void sc_group(const float *__restrict__ t, float (&c)[NP])
{
    const float4 *q = (const float4 *)t;
#pragma unroll
    for (int k = 0; k < NP; k += 4) {
        const float4 v = q[k / 4];
        c[k] = v.x;
        if (k + 1 < NP) c[k + 1] = v.y;
        if (k + 2 < NP) c[k + 2] = v.z;
        if (k + 3 < NP) c[k + 3] = v.w;
    }
}
template <class S, int NP> __device__ __forceinline__ S sc_mac(const S (&c)[NP], const S (&s)[NP], S a)
{
#pragma unroll
    for (int k = 0; k < NP; k++) a = fma(c[k], s[k], a);
    return a;
}

// Outputs of planes [z0, z1) of column `col` (fine_march with one value).
template <class S, bool SYM, class E>
__device__ __forceinline__ void sc_march(const ScGrid &g, const S *__restrict__ x, int col, int z0, int z1, E &epi)
{
    using Row = ScRow<SYM>;
    constexpr int NP = Row::NP, pl = 9 * Row::LEN;
    const bool act = col < g.NXY;
    const int i = col % g.NX, j = col / g.NX, NY = g.NXY / g.NX;
    const bool l = act && i > 0, r = act && i < g.NX - 1, d = act && j > 0, u = act && j < NY - 1;
    const int type = 3 * (j == 0 ? 0 : (j == NY - 1 ? 2 : 1)) + (i == 0 ? 0 : (i == g.NX - 1 ? 2 : 1));
    const S *__restrict__ tab = (const S *)g.tab + (act ? type : 0) * Row::LEN;
    const S c1 = (S)g.c1;
    S n[9], s[NP];
    auto ld = [&](int q, bool ok) -> S { return ok ? x[q] : (S)0; };
    auto load = [&](int k) {
        const bool ok = k < g.NZ;
        const int q = k * g.NXY + col;
        n[0] = ld(q - g.NX - 1, ok && d && l);
        n[1] = ld(q - g.NX, ok && d);
        n[2] = ld(q - g.NX + 1, ok && d && r);
        n[3] = ld(q - 1, ok && l);
        n[4] = ld(q, ok && act);
        n[5] = ld(q + 1, ok && r);
        n[6] = ld(q + g.NX - 1, ok && u && l);
        n[7] = ld(q + g.NX, ok && u);
        n[8] = ld(q + g.NX + 1, ok && u && r);
    };
    auto sums = [&]() {
        if constexpr (SYM) {
            s[0] = n[4];
            s[1] = n[3] + n[5];
            s[2] = n[1] + n[7];
            s[3] = n[0] + n[8];
            s[4] = n[2] + n[6];
        } else {
#pragma unroll
            for (int m = 0; m < 9; m++) s[m] = n[m];
        }
    };
    S a = 0, up[NP];
    if (z0 > 0) {
        load(z0 - 1);
        sc_group(tab + (SYM ? (z0 - 1) * pl + Row::UP : z0 * pl + Row::DN), up);
        sums();
        load(z0);
        a = sc_mac(up, s, a);
    } else {
        load(z0);
    }
    const S *t = tab + z0 * pl;
    int p = z0 * g.NXY + col;
    auto own = [&](S ao) {
        S c[NP];
        sc_group(t, c);
        ao = sc_mac(c, s, ao);
        sc_group(t + Row::UP, up);
        return ao;
    };
    auto below = [&]() {
        if constexpr (SYM) {
            return sc_mac(up, s, (S)0);
        } else {
            S c[NP];
            sc_group(t + pl + Row::DN, c);
            return sc_mac(c, s, (S)0);
        }
    };
    S cen = n[4];
    sums();
    load(z0 + 1);
    a = own(a);
    for (int k = z0 + 1; k < z1; k++) {
        const auto pre = epi.load(p, act);
        const S cm = cen, *tm = t;
        const S an = below();
        cen = n[4];
        sums();
        load(k + 1);
        a = sc_mac(up, s, a);
        if (act) epi(p, tm + Row::IDC2, pre, cm, c1, a);
        t += pl;
        p += g.NXY;
        a = own(an);
    }
    const auto pre = epi.load(p, act);
    if (z1 < g.NZ) {
        sums();
        a = sc_mac(up, s, a);
    }
    if (act) epi(p, t + Row::IDC2, pre, cen, c1, a);
}

template <class S, bool SYM, class E>
__device__ __forceinline__ void sc_block(const ScGrid &g, const S *__restrict__ x, E &epi)
{
    const long long U = (long long)g.ncb * g.NZ;
    const int u1 = (int)(U * (blockIdx.x + 1) / gridDim.x);
    for (int un = (int)(U * blockIdx.x / gridDim.x); un < u1;) {
        const int cb = un / g.NZ, z0 = un - cb * g.NZ;
        const int z1 = min(g.NZ, z0 + (u1 - un));
        sc_march<S, SYM>(g, x, cb * kFineTPB + threadIdx.x, z0, z1, epi);
        un += z1 - z0;
    }
}

// Four blocks per SM: half the FP64 work of the block operator per plane.
template <class S> struct ScMinB { static constexpr int v = sizeof(S) == 8 ? 4 : 8; };

template <class S, bool SYM, class E>
__global__ void __launch_bounds__(kFineTPB, ScMinB<S>::v) k_sc(ScGrid g, const S *__restrict__ x, E epi)
{
    sc_block<S, SYM>(g, x, epi);
}

// One scalar operator: its table and grid.
struct ScOp {
    bool sym = false;
    ScGrid g;
    DBuf<double> tab;
    DBuf<float> tab32;
    template <class S> ScGrid grid() const
    {
        ScGrid q = g;
        q.tab = sizeof(S) == 8 ? (const void *)tab.p : (const void *)tab32.p;
        return q;
    }
    template <class S> int blocks() const
    {
        const long long units = (long long)g.ncb * g.NZ;
        // as fine_blocks: short walks only where the slab fills the GPU
        const int w = sizeof(S) == 8 && units < 20LL * kSM ? 2 : ScMinB<S>::v;
        return (int)std::max<long long>(1, std::min<long long>(units, (long long)kSM * w));
    }
};

// make(SYM) gives the epilogue
template <class S, class F> static int sc_apply(const ScOp &A, const S *x, F make, cudaStream_t s)
{
    if (A.sym) k_sc<S, true><<<A.blocks<S>(), kFineTPB, 0, s>>>(A.grid<S>(), x, make());
    else k_sc<S, false><<<A.blocks<S>(), kFineTPB, 0, s>>>(A.grid<S>(), x, make());
    ::bd::note_launch();
    BD_LAUNCH_CHECK();
    return BD_OK;
}

// The table of a Ki + b Ke + m (c M) from the raw rows, with the Chebyshev
// scalings of the inverse diagonal of Ai + Ae.
int sc_pack(const FineStencil &F, double a, double b, double m, double c1, double c2, double inv_theta, bool fp32,
            ScOp &op, cudaStream_t s);

}  // namespace bd
