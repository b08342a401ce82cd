// fine_stencil.cuh -- the finest level of an assembled slab as a layered
// stencil: operator application with fused Chebyshev epilogues, shared by the
// V-cycle and PCG of one hierarchy (amg_solve.cu) and of a stack of them
// (amg_stack.cu).
//
// The fibre field of the Bidomain slab depends on z alone (Section 2.1's
// tensor on uniform Q1 hexahedra), so a row of Ki and Ke depends on the node's
// plane and on whether it lies on an x or y face: nine row types per plane.
// The operator is a table of (nz + 1) x 9 rows instead of 20 (FP64) or 9
// (FP32) bytes per node pair, and so is everything else that follows from a
// row's diagonal (D^{-1} scaled for each Chebyshev step).  A launch streams
// its vectors only, and they stay in L2 at 128x128x32 nodes.
//
// Work split: a thread owns a column (i, j) and walks along z.  Every plane is
// loaded once (nine values) and used for three outputs.  Where the fibres lie
// in the plane (no z component, the usual field), a row is symmetric under
// (dx, dy) -> (-dx, -dy), so the four pairs of opposite neighbours are added
// first: 4 adds and 15 multiply-adds per node and operator instead of 27.
// That is what bounds the FP64 kernels (two FP64 operations per clock and SM);
// the general form (27 coefficients) serves every other field.  Against the
// operator stored in sliced ELL (20 and 9 bytes per node pair), event-timed per
// launch: 128x128x32 FP64 67.6 -> 51 us (residual), FP32 33 -> 10.4;
// 256x256x64 FP64 A p 462 -> 343, FP32 219 -> 37.5.  The general form: 65.8, 13.8,
// 458 and 65.4 (54 multiply-adds a node, as many as the sliced ELL's).
#pragma once

#include "amg_bsr.cuh"

namespace bd {

// One row of the packed table, in pairs of S, in groups that load as whole
// 16-byte words: (Ki, Ke) of the in-plane positions for dz = 0 and (c M, 0);
// the same for dz = +1 and a pad; in the general form for dz = -1 too (in the
// symmetric form a plane's dz = +1 coefficients are those of the plane above
// for dz = -1, and each group is loaded once for both); c2 D^{-1}; D^{-1} /
// theta; kappa = -omega D^{-1} (PairOp); a pad.  In-plane positions: symmetric form 0 centre, 1 x pair, 2 y pair, 3
// the (-1,-1), (1,1) pair, 4 the (1,-1), (-1,1) pair; general form 3 (dy + 1) +
// dx + 1.
template <bool SYM> struct FineRow {
    static constexpr int NP = SYM ? 5 : 9;
    static constexpr int G = NP + 1;          // pairs of a group
    static constexpr int CM = NP;
    static constexpr int UP = G;
    static constexpr int DN = 2 * G;          // general form only
    static constexpr int IDC2 = (SYM ? 2 : 3) * G;
    static constexpr int IDT = IDC2 + 1;
    static constexpr int KAPPA = IDC2 + 2;
    static constexpr int LEN = IDC2 + 4;
};

// One slab of a launch: extents in nodes, first node and first work unit.  A
// unit is one plane of one block of columns.
struct FineGrid {
    int NX = 0, NXY = 0, NZ = 0, ncb = 0;
    int off = 0;
    int unit0 = 0;
    double c1 = 0.0;  // Chebyshev coefficient of the degree-2 step
    const void *tab = nullptr;
};

// Resident blocks per SM.  FP64: the pipe issues two operations per clock and
// SM, so a plane of one warp keeps its scheduler's share busy for about 3000
// clocks, and two blocks (two warps per scheduler) hide every load; more of them
// only shorten the walks and add halo planes (128x128x32, residual: 4 blocks
// 61.6 us, 3 53.0, 2 51.0).  FP32: latency and L1 wavefronts; 6 blocks of 80
// registers beat 8 of 64 (256x256x64, residual: 48 -> 37.5 us).  General form, pre-smoother
// at 128x128x32 and 256x256x64: FP64 1 block 83.3 and 655 us, 2 68.3 and 472, 3 70.5
// and 482; FP32 4 blocks 15.2 and 93, 5 14.6 and 75 (36 bytes of a thread's registers
// spilled), 6 15.2 and 84.
constexpr int kFineTPB = 128;
template <class S, bool SYM> struct FineMinB { static constexpr int v = sizeof(S) == 8 ? 2 : (SYM ? 6 : 5); };

template <class S> __device__ __forceinline__ v2<S> fine_ld(const v2<S> *__restrict__ x, int q, bool ok)
{
    return ok ? x[q] : V2<S>::mk((S)0, (S)0);
}

// (v + u, u) of a loaded pair; the vector may be stored that way (SU)
template <class S, bool SU> __device__ __forceinline__ v2<S> fine_su(v2<S> a)
{
    return SU ? a : V2<S>::mk(a.x + a.y, a.y);
}

// A group of a table row.
template <int G> __device__ __forceinline__ void fine_group(const double2 *__restrict__ t, double2 (&c)[G])
{
#pragma unroll
    for (int k = 0; k < G; k++) c[k] = t[k];
}
template <int G> __device__ __forceinline__ void fine_group(const float2 *__restrict__ t, float2 (&c)[G])
{
    const float4 *q = (const float4 *)t;
#pragma unroll
    for (int k = 0; k < G / 2; k++) {
        const float4 v = q[k];
        c[2 * k] = make_float2(v.x, v.y);
        c[2 * k + 1] = make_float2(v.z, v.w);
    }
}

// (a, b) += (Ki part, Ke part) of a group applied to a plane's sums
template <class S, int NP>
__device__ __forceinline__ void fine_mac(const v2<S> (&c)[NP + 1], const v2<S> (&s)[NP], S &a, S &b)
{
#pragma unroll
    for (int k = 0; k < NP; k++) {
        a = fma(c[k].x, s[k].x, a);
        b = fma(c[k].y, s[k].y, b);
    }
}

// Outputs of planes [z0, z1) of column `col`.  Every output adds its terms in
// the order plane below, own plane, plane above, so the result does not depend
// on how the planes are split.  The next plane's nine values are loaded before
// a plane's arithmetic, which hides their latency behind it even with one or
// two warps per scheduler.
template <class S, bool SYM, bool SU, class E>
__device__ __forceinline__ void fine_march(const FineGrid &g, const v2<S> *__restrict__ x, int col, int z0, int z1,
                                           E &epi)
{
    using Row = FineRow<SYM>;
    constexpr int NP = Row::NP;
    const bool act = col < g.NXY;
    const int i = col % g.NX, j = col / g.NX, NY = g.NXY / g.NX;
    const bool l = act && i > 0, r = act && i < g.NX - 1, d = act && j > 0, u = act && j < NY - 1;
    const int type = 3 * (j == 0 ? 0 : (j == NY - 1 ? 2 : 1)) + (i == 0 ? 0 : (i == g.NX - 1 ? 2 : 1));
    constexpr int pl = 9 * Row::LEN;
    const v2<S> *__restrict__ tab = (const v2<S> *)g.tab + (act ? type : 0) * Row::LEN;
    const v2<S> *__restrict__ xb = x + g.off;
    const S c1 = (S)g.c1;
    v2<S> n[9], s[NP];
    auto load = [&](int k) {
        const bool ok = k < g.NZ;
        const int q = k * g.NXY + col;
        n[0] = fine_ld<S>(xb, q - g.NX - 1, ok && d && l);
        n[1] = fine_ld<S>(xb, q - g.NX, ok && d);
        n[2] = fine_ld<S>(xb, q - g.NX + 1, ok && d && r);
        n[3] = fine_ld<S>(xb, q - 1, ok && l);
        n[4] = fine_ld<S>(xb, q, ok && act);
        n[5] = fine_ld<S>(xb, q + 1, ok && r);
        n[6] = fine_ld<S>(xb, q + g.NX - 1, ok && u && l);
        n[7] = fine_ld<S>(xb, q + g.NX, ok && u);
        n[8] = fine_ld<S>(xb, q + g.NX + 1, ok && u && r);
    };
    auto sums = [&]() {
        if constexpr (SYM) {
            s[0] = fine_su<S, SU>(n[4]);
            s[1] = fine_su<S, SU>(V2<S>::mk(n[3].x + n[5].x, n[3].y + n[5].y));
            s[2] = fine_su<S, SU>(V2<S>::mk(n[1].x + n[7].x, n[1].y + n[7].y));
            s[3] = fine_su<S, SU>(V2<S>::mk(n[0].x + n[8].x, n[0].y + n[8].y));
            s[4] = fine_su<S, SU>(V2<S>::mk(n[2].x + n[6].x, n[2].y + n[6].y));
        } else {
#pragma unroll
            for (int m = 0; m < 9; m++) s[m] = fine_su<S, SU>(n[m]);
        }
    };
    S a = 0, b = 0, cv = 0;  // the output of the plane at hand and its c M v
    v2<S> up[NP + 1], cen = V2<S>::mk((S)0, (S)0);
    if (z0 > 0) {  // the plane below output z0
        load(z0 - 1);
        fine_group(tab + (SYM ? (z0 - 1) * pl + Row::UP : z0 * pl + Row::DN), up);
        sums();
        load(z0);
        fine_mac<S, NP>(up, s, a, b);
    } else {
        load(z0);
    }
    const v2<S> *t = tab + z0 * pl;  // the row of plane k
    int p = g.off + z0 * g.NXY + col;
    auto own = [&](S &ao, S &bo) {   // own-plane terms of output k
        v2<S> c[NP + 1];
        fine_group(t, c);
        cv = c[NP].x * (SU ? cen.x - cen.y : cen.x);
        fine_mac<S, NP>(c, s, ao, bo);
        fine_group(t + Row::UP, up);
    };
    auto below = [&](S &an, S &bn) {  // plane k's terms of output k + 1
        an = bn = 0;
        if constexpr (SYM) {
            fine_mac<S, NP>(up, s, an, bn);
        } else {
            v2<S> c[NP + 1];
            fine_group(t + pl + Row::DN, c);
            fine_mac<S, NP>(c, s, an, bn);
        }
    };
    {
        cen = n[4];
        sums();
        load(z0 + 1);
        own(a, b);
    }
    for (int k = z0 + 1; k < z1; k++) {  // output k - 1 is completed by plane k
        const auto pre = epi.load(p, act);
        const v2<S> cm = cen, *tm = t;
        const S cvm = cv;
        S an, bn;
        below(an, bn);
        cen = n[4];
        sums();
        load(k + 1);
        fine_mac<S, NP>(up, s, a, b);
        if (act) epi(p, tm, pre, cm, c1, cvm + a, a + b);
        a = an;
        b = bn;
        t += pl;
        p += g.NXY;
        own(a, b);
    }
    const auto pre = epi.load(p, act);
    if (z1 < g.NZ) {
        sums();
        fine_mac<S, NP>(up, s, a, b);
    }
    if (act) epi(p, t, pre, cen, c1, cv + a, a + b);
}

// A block's share of the units: planes of column blocks, in order, so that all
// blocks get the same number of planes to within one.
template <class S, bool SYM, bool SU, class E>
__device__ __forceinline__ void fine_share(const FineGrid &g, int u0, int u1, const v2<S> *__restrict__ x, E &epi)
{
    for (int un = u0; un < u1;) {
        const int cb = un / g.NZ, z0 = un - cb * g.NZ;
        const int z1 = min(g.NZ, z0 + (u1 - un));
        fine_march<S, SYM, SU>(g, x, cb * kFineTPB + threadIdx.x, z0, z1, epi);
        un += z1 - z0;
    }
}

template <class S, bool SYM, bool SU, class E>
__device__ __forceinline__ void fine_block(const FineGrid &g, const v2<S> *__restrict__ x, E &epi)
{
    const long long U = (long long)g.ncb * g.NZ;
    fine_share<S, SYM, SU>(g, (int)(U * blockIdx.x / gridDim.x), (int)(U * (blockIdx.x + 1) / gridDim.x), x, epi);
}

// ------------------------------------------------------------------ epilogues
// The Chebyshev steps (Saad, Alg. 12.1 on D^{-1} A, degree 2) with the row's
// constants from the table.  `c` is the gathered vector's own entry as stored.
// In the (v + u, u) form u_s = v + u of a result needs the sum of its parts.
template <class S, bool SYM> struct FineConst {
    using Row = FineRow<SYM>;
    static __device__ __forceinline__ v2<S> idc2(const v2<S> *t) { return t[Row::IDC2]; }
    static __device__ __forceinline__ v2<S> idt(const v2<S> *t) { return t[Row::IDT]; }
    static __device__ __forceinline__ v2<S> kappa(const v2<S> *t) { return t[Row::KAPPA]; }
};

// pre-smoothing from zero: u = d0 + (c1 d0 + c2 D^{-1} (f - A d0)), d0 gathered
template <class S, bool SYM, bool SU> struct FinePre {
    const v2<S> *__restrict__ f;
    v2<S> *__restrict__ u;
    __device__ __forceinline__ v2<S> load(int p, bool ok) const { return fine_ld<S>(f, p, ok); }
    __device__ __forceinline__ void operator()(int p, const v2<S> *t, v2<S> fp, v2<S> c, S c1, S y0, S y1)
    {
        const v2<S> k = FineConst<S, SYM>::idc2(t);
        const S m0 = k.x * (fp.x - y0), m1 = k.y * (fp.y - y1);
        if (SU) u[p] = V2<S>::mk(fma(1 + c1, c.x, m0 + m1), fma(1 + c1, c.y, m1));
        else u[p] = V2<S>::mk(c.x + (c1 * c.x + m0), c.y + (c1 * c.y + m1));
    }
};

// what the restriction gathers: kappa (f - A u), kappa R's row scaling (PairOp);
// in (v + u, u) form in FP64, plain in FP32 (whose additions are free)
template <class S, bool SYM, bool SU> struct FineResid {
    const v2<S> *__restrict__ f;
    v2<S> *__restrict__ r;
    __device__ __forceinline__ v2<S> load(int p, bool ok) const { return fine_ld<S>(f, p, ok); }
    __device__ __forceinline__ void operator()(int p, const v2<S> *t, v2<S> fp, v2<S>, S, S y0, S y1)
    {
        const v2<S> k = FineConst<S, SYM>::kappa(t);
        const S t1 = k.y * (fp.y - y1), r0 = fp.x - y0;
        r[p] = V2<S>::mk(SU ? fma(k.x, r0, t1) : k.x * r0, t1);
    }
};

// post-smoothing, first half: r = f - A u, d = D^{-1} r / theta.  The iterate
// w = u + d is formed again by the second half (one add) instead of stored,
// except for degree 1, whose result it is (w given).
template <class S, bool SYM, bool SU> struct FinePost1 {
    const v2<S> *__restrict__ f;
    v2<S> *__restrict__ r;
    v2<S> *__restrict__ d;
    v2<S> *__restrict__ w;
    __device__ __forceinline__ v2<S> load(int p, bool ok) const { return fine_ld<S>(f, p, ok); }
    __device__ __forceinline__ void operator()(int p, const v2<S> *t, v2<S> fp, v2<S> c, S, S y0, S y1)
    {
        const v2<S> k = FineConst<S, SYM>::idt(t);
        const S r0 = fp.x - y0, r1 = fp.y - y1;
        const S d1 = r1 * k.y, d0 = SU ? r0 * k.x + d1 : r0 * k.x;
        r[p] = V2<S>::mk(r0, r1);
        d[p] = V2<S>::mk(d0, d1);
        if (w) {
            const S ws = c.x + d0, wu = c.y + d1;
            w[p] = V2<S>::mk(SU ? ws - wu : ws, wu);
        }
    }
};

// post-smoothing, second half: u = (u + d) + (c1 d + c2 D^{-1} (r - A d)), d
// gathered; the result in plain (v, u) form
template <class S, bool SYM, bool SU> struct FinePost2 {
    const v2<S> *__restrict__ r;
    const v2<S> *uin;  // stored as the gathered vectors are; may be u itself
    v2<S> *u;
    struct Pre {
        v2<S> r, u;
    };
    __device__ __forceinline__ Pre load(int p, bool ok) const { return {fine_ld<S>(r, p, ok), fine_ld<S>(uin, p, ok)}; }
    __device__ __forceinline__ v2<S> value(const v2<S> *t, const Pre &q, v2<S> c, S c1, S y0, S y1) const
    {
        const v2<S> k = FineConst<S, SYM>::idc2(t);
        const S m0 = k.x * (q.r.x - y0), m1 = k.y * (q.r.y - y1);
        const S uu = (q.u.y + c.y) + fma(c1, c.y, m1);
        const S us = (q.u.x + c.x) + fma(c1, c.x, SU ? m0 + m1 : m0);
        return V2<S>::mk(SU ? us - uu : us, uu);
    }
    __device__ __forceinline__ void operator()(int p, const v2<S> *t, const Pre &q, v2<S> c, S c1, S y0, S y1)
    {
        u[p] = value(t, q, c, c1, y0, y1);
    }
};

template <class S> struct FineStore {  // q = A x
    v2<S> *__restrict__ q;
    __device__ __forceinline__ int load(int, bool) const { return 0; }
    __device__ __forceinline__ void operator()(int p, const v2<S> *, int, v2<S>, S, S y0, S y1)
    {
        q[p] = V2<S>::mk(y0, y1);
    }
};

// ------------------------------------------------------------------ launches
template <class S, bool SYM, bool SU, class E>
__global__ void __launch_bounds__(kFineTPB, FineMinB<S, SYM>::v) k_fine(FineGrid g, const v2<S> *__restrict__ x, E epi)
{
    fine_block<S, SYM, SU>(g, x, epi);
}

// Several slabs in one launch (their units end to end).
template <class S, bool SYM, bool SU, class E>
__global__ void __launch_bounds__(kFineTPB, FineMinB<S, SYM>::v)
    k_fine_many(const FineGrid *__restrict__ gs, int count, const v2<S> *__restrict__ x, E epi)
{
    const FineGrid e = gs[count - 1];
    const long long U = e.unit0 + (long long)e.ncb * e.NZ;
    int u0 = (int)(U * blockIdx.x / gridDim.x);
    const int u1 = (int)(U * (blockIdx.x + 1) / gridDim.x);
    int lo = 0, hi = count - 1;  // the last slab whose units start at or before u0
    while (lo < hi) {
        const int m = (lo + hi + 1) >> 1;
        if (gs[m].unit0 <= u0) lo = m;
        else hi = m - 1;
    }
    for (; u0 < u1; lo++) {
        const FineGrid g = gs[lo];
        const int end = min(u1 - g.unit0, g.ncb * g.NZ);
        fine_share<S, SYM, SU>(g, u0 - g.unit0, end, x, epi);
        u0 = g.unit0 + end;
    }
}

// Blocks of a launch over `units`: one resident wave of equal shares.  FP64
// slabs of few planes take one block per SM, since every walk starts with the
// plane below it (77x53x19: 17.8 -> 17.0 us).
template <class S, bool SYM> static int fine_blocks(long long units)
{
    const int w = sizeof(S) == 8 && units < 10LL * kSM ? 1 : FineMinB<S, SYM>::v;
    return (int)std::max<long long>(1, std::min<long long>(units, (long long)kSM * w));
}

template <class S> static const void *fine_tab(const FineStencil &F);
template <> const void *fine_tab<double>(const FineStencil &F) { return F.tab.p; }
template <> const void *fine_tab<float>(const FineStencil &F) { return F.tab32.p; }

template <class S> static FineGrid fine_grid(const FineStencil &F, double c1)
{
    FineGrid g;
    g.NX = F.NX;
    g.NXY = F.NX * F.NY;
    g.NZ = F.NZ;
    g.ncb = (g.NXY + kFineTPB - 1) / kFineTPB;
    g.c1 = c1;
    g.tab = fine_tab<S>(F);
    return g;
}

// In-plane stencil position (3 (dy + 1) + dx + 1) a symmetric pair's coefficient is
// read from: its member that exists on row type (ti, tj).
__device__ __forceinline__ int fine_pair_pos(int k, int ti, int tj)
{
    if (k == 0) return 4;
    if (k == 1) return ti == 2 ? 3 : 5;
    if (k == 2) return tj == 2 ? 1 : 7;
    if (k == 3) return (ti == 2 || tj == 2) ? 0 : 8;
    return (ti == 2 || tj == 0) ? 6 : 2;
}

// Table of one slab from its raw rows and the level's Chebyshev constants, in
// the symmetric or the general form.
int fine_pack(const FineStencil &F, bool sym, double c2, double inv_theta, double omega, double *tab, float *tab32,
              cudaStream_t s);
// the prolongator smoother's omega on a level (0 on a hierarchy's only level)
inline double fine_omega(const Level &L) { return L.lam > 0.0 ? 4.0 / (3.0 * L.lam) : 0.0; }
constexpr int fine_row_len(bool sym) { return sym ? FineRow<true>::LEN : FineRow<false>::LEN; }

}  // namespace bd
