"""Workloads of the Bidomain SA-AMG-PCG library, called as a user's program calls them.

listed() names them, draw() gives more of the same ranges, prepare() makes what a program
has in hand before the call (inputs on the GPU, hierarchies, stacks), run() is one pass
through the public entry points and returns its whole outputs, work() the arithmetic and
traffic a pass cannot do without, exact() the same outputs from plain torch in FP64.

Kinds and their ranges (elements of the slab, all of them the repository's own meshes or
sizes between them):
  dot      reproducible inner product of device vectors, 1e3 .. 1e7 entries
  vcycle   one V-cycle as a preconditioner, 16x16x8 .. 192x192x48, FP64 or FP32 V-cycle
  solve    one cold AMG-PCG solve to rtol 1e-8, 16x16x8 .. 256x256x64, FP64 or FP32 V-cycle
  step     a simulation from rest: several time steps and the state read back, 16x16x8 ..
           192x192x48, FP64 or FP32 V-cycle
  fresh    a new slab: assembly, hierarchy setup and its first solve, 16x16x8 .. 128x128x32
  csr      a solve of a caller's own matrix (tissue with a conductivity of its own in every
           element), 12x12x6 .. 64x64x16
  stack    many uneven slabs solved together, 8 .. 64 of them, FP64 or FP32 V-cycle
  dsim     time steps of the decoupled scheme, 16x16x8 .. 128x128x32, Jacobi-CG or plain CG
  serve    the continuous-batching server on several simulations, 2 .. 8 requests
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2311_13914_gb300 import binding as B
from paper_2311_13914_gb300 import workloads as W

RTOL = 1e-8


def listed():
    return [
        # the reproducible inner product a caller uses on vectors of the 128x128x32 slab:
        # the shortest call of the library, launch- and latency-bound
        dict(name="dot_paper", kind="dot", n=1098306),
        # the V-cycle alone as the preconditioner of a caller's own Krylov loop
        dict(name="vcycle_f64", kind="vcycle", nx=96, ny=96, nz=24, hz=2, precision=0),
        # the small slab's single solve: short kernels on a level of 8125 nodes
        dict(name="solve_small_f64", kind="solve", nx=24, ny=24, nz=12, hz=1, precision=0, limit=100),
        # odd extents and ragged tails, a mid-size slab's single solve
        dict(name="solve_odd_f64", kind="solve", nx=77, ny=53, nz=19, hz=1, precision=0, limit=100),
        # precision form at the largest size: 8.6 M unknowns, FP32 V-cycle in FP64 CG
        dict(name="solve_large_f32", kind="solve", nx=256, ny=256, nz=64, hz=2, precision=1, limit=2000),
        # the headline simulation: 128x128x32 from rest under the corner stimulus, FP64
        dict(name="step_paper_f64", kind="step", nx=128, ny=128, nz=32, hz=2, precision=0, limit=2000, steps=5),
        # the same simulation with the FP32 V-cycle
        dict(name="step_paper_f32", kind="step", nx=128, ny=128, nz=32, hz=2, precision=1, limit=2000, steps=5),
        # a slab that is seen for the first time: assembly, setup and one solve
        dict(name="fresh_paper_f64", kind="fresh", nx=128, ny=128, nz=32, hz=2, precision=0, limit=2000),
        # a caller's matrix with element-wise conductivities (no slab structure to use)
        dict(name="csr_f64", kind="csr", nx=48, ny=48, nz=12, hz=1),
        # 64 uneven slabs in one launch per step, FP32 V-cycle
        dict(name="stack64_f32", kind="stack", count=64, meshes=2, precision=1),
        # the decoupled scheme: elliptic AMG-PCG and parabolic Jacobi-CG per step
        dict(name="dsim_paper", kind="dsim", nx=128, ny=128, nz=32, hz=2, jacobi=True, steps=2),
        # six simulations through the server: admission, setup, overlapped steps, results
        dict(name="serve6_f32", kind="serve", count=6, meshes=3, precision=1),
    ]


def _size(rng, lo, hi, cap):
    """Element counts, each spread over the logarithm of its range, at most `cap` nodes;
    elements once or twice as high as wide."""
    while True:
        n = [int(round(math.exp(rng.uniform(math.log(a), math.log(b))))) for a, b in zip(lo, hi)]
        if (n[0] + 1) * (n[1] + 1) * (n[2] + 1) <= cap:
            return dict(nx=n[0], ny=n[1], nz=n[2], hz=rng.choice([1, 2]))


def draw(rng):
    kind = rng.choice(["dot", "vcycle", "solve", "solve", "step", "step", "fresh", "csr", "stack", "dsim", "serve"])
    prec = rng.randrange(2)
    if kind == "dot":
        return dict(kind=kind, n=int(round(math.exp(rng.uniform(math.log(1e3), math.log(1e7))))))
    if kind == "vcycle":
        return dict(kind=kind, precision=prec, **_size(rng, (16, 16, 8), (192, 192, 48), 1_900_000))
    if kind == "solve":
        return dict(kind=kind, precision=prec, limit=rng.choice([100, 2000]),
                    **_size(rng, (16, 16, 8), (256, 256, 64), 4_293_185 if prec else 2_000_000))
    if kind == "step":
        return dict(kind=kind, precision=prec, limit=rng.choice([100, 2000]), steps=rng.randint(1, 5),
                    **_size(rng, (16, 16, 8), (192, 192, 48), 1_000_000))
    if kind == "fresh":
        return dict(kind=kind, precision=prec, limit=rng.choice([100, 2000]),
                    **_size(rng, (16, 16, 8), (128, 128, 32), 549_153))
    if kind == "csr":
        return dict(kind=kind, **_size(rng, (12, 12, 6), (64, 64, 16), 71_825))
    if kind == "stack":
        return dict(kind=kind, count=rng.randint(8, 64), meshes=rng.randrange(1000), precision=prec)
    if kind == "dsim":
        return dict(kind=kind, jacobi=rng.random() < 0.7, steps=rng.randint(1, 2),
                    **_size(rng, (16, 16, 8), (128, 128, 32), 549_153))
    return dict(kind="serve", count=rng.randint(2, 8), meshes=rng.randrange(1000), precision=prec)


# ------------------------------------------------------------------ inputs
def _mesh(case):
    """A slab 1 cm wide of elements as high as they are wide, or twice that: with hz = 2
    the 1 x 1 x 0.5 cm slabs of 96x96x24 to 256x256x64 elements, with 1 that of 24x24x12."""
    h = 1.0 / case["nx"]
    return dict(nx=case["nx"], ny=case["ny"], nz=case["nz"], lx=1.0, ly=case["ny"] * h, lz=case["hz"] * case["nz"] * h)


def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed) % (1 << 62))


def _fibres(mesh, seed):
    rng = np.random.Generator(np.random.PCG64(int(seed)))
    return W.fibre_table(mesh, 120.0, float(rng.uniform(-30.0, 30.0)))


def _rhs(n, seed):
    """N(0, 1) entries, consistent with the null vector (0, 1)."""
    f = torch.randn(n, generator=_gen(seed), device="cuda", dtype=torch.float64)
    f[1::2] -= f[1::2].mean()
    return f


def _stimulus(mesh, seed):
    """The corner stimulus with an amplitude of its own for every seed."""
    rng = np.random.Generator(np.random.PCG64(int(seed) + 17))
    return W.stimulus(mesh, amplitude=8.0e4 * float(rng.uniform(0.75, 1.25)))


def _front(mesh, seed):
    """A state in mid-propagation: a smooth depolarisation front at a seeded radius and
    the recovery variable behind it."""
    rng = np.random.Generator(np.random.PCG64(int(seed) + 29))
    r0 = float(rng.uniform(0.3, 0.6))
    ax = [torch.linspace(0, mesh[k], mesh[n] + 1, device="cuda", dtype=torch.float64)
          for k, n in (("lz", "nz"), ("ly", "ny"), ("lx", "nx"))]
    z, y, x = torch.meshgrid(*ax, indexing="ij")
    d = torch.sqrt(x * x + y * y + z * z) - r0
    v = 100.0 / (1.0 + torch.exp(d / 0.05))
    w = 0.3 / (1.0 + torch.exp((d + 0.2) / 0.1))
    return v.reshape(-1).contiguous(), w.reshape(-1).contiguous()


def _slabs(case, seed):
    """The batched workload's meshes; fibres and conductivities of the seed's."""
    rng = np.random.Generator(np.random.PCG64(int(seed) + 5))
    out = []
    for m, p, _ in W.batch_slabs(case["count"], seed=case["meshes"]):
        fib = W.fibre_table(m, float(rng.uniform(60.0, 150.0)), float(rng.uniform(-30.0, 30.0)))
        for key, f in zip(("sil", "sit", "sel", "set"), rng.uniform(0.8, 1.2, 4)):
            p[key] = W.DEFAULT_PARAMS[key] * float(f)
        out.append((m, p, fib))
    return out


def _requests(case, seed):
    """Server requests: nx = ny = 4k, nz = k, a few time steps each."""
    size = np.random.Generator(np.random.PCG64(case["meshes"]))
    rng = np.random.Generator(np.random.PCG64(int(seed) + 5))
    out = []
    for i in range(case["count"]):
        k, steps = int(size.integers(8, 17)), int(size.integers(4, 9))
        m = W.mesh(4 * k, 4 * k, k)
        fib = W.fibre_table(m, 120.0, float(rng.uniform(-30.0, 30.0)))
        out.append((m, fib, _stimulus(m, int(seed) + i), steps))
    return out


def _opts(case):
    return B.amg_options_default(precision=case.get("precision", 0), coarse_eq_limit=case.get("limit", 100))


def prepare(case, seed):
    kind = case["kind"]
    if kind == "dot":
        g = _gen(seed)
        x = torch.randn(case["n"], generator=g, device="cuda", dtype=torch.float64)
        y = torch.randn(case["n"], generator=g, device="cuda", dtype=torch.float64)
        return dict(case=case, x=x, y=y, out=torch.zeros(1, dtype=torch.float64, device="cuda"))
    if kind == "stack":
        slabs = _slabs(case, seed)
        sys_, hs, ns = [], [], []
        for m, p, fib in slabs:
            s = B.bd_assemble(m, p, fib)
            sys_.append(s)
            hs.append(B.amg_setup(s, _opts(case)))
            ns.append(2 * W.n_nodes(m))
        f = torch.cat([_rhs(n, seed + k) for k, n in enumerate(ns)])
        x = torch.zeros_like(f)
        at = np.concatenate([[0], np.cumsum(ns)])
        cut = lambda t: [t[int(a):int(b)] for a, b in zip(at[:-1], at[1:])]  # noqa: E731
        return dict(case=case, sys=sys_, h=hs, stack=B.amg_stack_create(hs), f=cut(f), x=cut(x), xall=x,
                    opts=B.solve_options_default(rtol=RTOL))
    if kind == "serve":
        return dict(case=case, reqs=_requests(case, seed))
    m = _mesh(case)
    n = 2 * W.n_nodes(m)
    fib = _fibres(m, seed)
    st = dict(case=case, mesh=m, n=n, opts=B.solve_options_default(rtol=RTOL))
    if kind == "fresh":
        return dict(st, fib=torch.tensor(fib.reshape(-1), device="cuda"), f=_rhs(n, seed))
    if kind == "csr":
        h = B.amg_setup_from_csr(n, *_csr(m, fib, _element_scale(m, seed)))
        return dict(st, h=h, f=_rhs(n, seed), x=torch.zeros(n, dtype=torch.float64, device="cuda"))
    s = B.bd_assemble(m, W.DEFAULT_PARAMS, fib)
    if kind == "dsim":
        v, w = _front(m, seed)
        return dict(st, sys=s, h=B.bd_elliptic_setup(s, _opts(case)), v=v, w=w,
                    stim=torch.tensor(_stimulus(m, seed), device="cuda"))
    h = B.amg_setup(s, _opts(case))
    st.update(sys=s, h=h)
    if kind == "step":
        N = n // 2
        st.update(stim=torch.tensor(_stimulus(m, seed), device="cuda"),
                  out=tuple(torch.zeros(N, dtype=torch.float64, pin_memory=True) for _ in range(3)))
        return st
    return dict(st, f=_rhs(n, seed), x=torch.zeros(n, dtype=torch.float64, device="cuda"))


# ------------------------------------------------------------------ one pass
def run(st):
    case, kind = st["case"], st["case"]["kind"]
    if kind == "dot":
        return B.bd_dot_exact_noalloc(st["x"], st["y"], st["out"])
    if kind == "vcycle":
        return B.amg_vcycle(st["h"], st["f"], st["x"])
    if kind in ("solve", "csr"):
        x, info = B.amg_solve(st["h"], st["f"], st["x"], st["opts"])
        return dict(x=x, iters=info["iters"])
    if kind == "step":
        sim = B.bd_sim_create(st["sys"], st["h"], stim=st["stim"], stim_ms=1.0)
        info = B.bd_step(sim, case["steps"], st["opts"])
        v, ue, w = B.bd_sim_get_state(sim, st["n"] // 2, out=st["out"])
        return dict(v=v, ue=ue, w=w, iters=info["total_iters"])
    if kind == "fresh":
        s = B.bd_assemble(st["mesh"], W.DEFAULT_PARAMS, st["fib"])
        h = B.amg_setup(s, _opts(case))
        x, info = B.amg_solve(h, st["f"], torch.zeros_like(st["f"]), st["opts"])
        lv = [B.amg_level_info(h, l) for l in range(B.amg_num_levels(h))]
        return dict(x=x, iters=info["iters"], lam=np.array([l["lam"] for l in lv]),
                    sizes=np.array([[l["n"], l["nnz"], l["n_agg"], l["p_nnz"]] for l in lv]))
    if kind == "stack":
        infos = B.amg_stack_solve(st["stack"], st["f"], st["x"], st["opts"])
        return dict(x=st["xall"], iters=np.array([i["iters"] for i in infos]))
    if kind == "dsim":
        sim = B.bd_dsim_create(st["sys"], st["h"], stim=st["stim"], stim_ms=1.0, jacobi=case["jacobi"])
        B.bd_dsim_set_state(sim, v=st["v"], w=st["w"])
        ell, par = B.bd_dsim_step(sim, case["steps"], st["opts"])
        v, ue, w = B.bd_dsim_get_state(sim, st["n"] // 2)
        return dict(v=v, ue=ue, w=w, iters=np.array([ell["total_iters"], par["total_iters"]]))
    srv = B.bd_server_create(B.bd_server_options_default(precision=case["precision"]))
    ids = [B.bd_server_submit(srv, m, W.DEFAULT_PARAMS, fib, stim, 1.0, steps) for m, fib, stim, steps in st["reqs"]]
    B.bd_server_drain(srv)
    return [B.bd_server_result(srv, i) for i in ids]


# ------------------------------------------------------------------ what a pass cannot do without
def _solve_work(N, iters):
    """PCG with a degree-2 smoothed V-cycle: five products with the 27-point pair of
    operators per iteration (two multiply-adds per node pair) and a quarter more on the
    coarse levels; the right-hand side read and the solution written once."""
    return dict(bytes=32.0 * N, flops=iters * 5 * 1.25 * 108.0 * N)


def work(case):
    kind = case["kind"]
    if kind == "dot":
        return dict(bytes=16.0 * case["n"] + 8, flops=2.0 * case["n"])
    if kind == "stack":
        N = sum(W.n_nodes(m) for m, _, _ in _slabs(case, 0))
        return _solve_work(N, 12)
    if kind == "serve":
        N = sum(W.n_nodes(m) * s for m, _, _, s in _requests(case, 0))
        return _solve_work(N, 11)
    N = (case["nx"] + 1) * (case["ny"] + 1) * (case["nz"] + 1)
    if kind == "vcycle":
        return dict(bytes=32.0 * N, flops=4 * 1.25 * 108.0 * N)
    if kind == "step":
        one = _solve_work(N, 17)
        return dict(bytes=case["steps"] * one["bytes"] + 24.0 * N, flops=case["steps"] * one["flops"])
    if kind == "dsim":  # one field each: an elliptic solve and a 24-iteration parabolic one
        fl = 16 * 5 * 1.25 * 54.0 * N + 24 * 54.0 * N
        return dict(bytes=case["steps"] * 32.0 * N + 24.0 * N, flops=case["steps"] * fl)
    w = _solve_work(N, 25 if N > 2_000_000 else 14)
    if kind == "fresh":  # the Galerkin products: A P and R (A P), 2x2 blocks
        w["flops"] += 2 * 27 * 7 * 16.0 * N
    return w


# ------------------------------------------------------------------ the same in plain torch, FP64
def _element_matrices(mesh, p, fib):
    """(nz, 2, 8, 8) stiffness of every element layer, 2x2x2 Gauss points."""
    h = np.array([mesh["lx"] / mesh["nx"], mesh["ly"] / mesh["ny"], mesh["lz"] / mesh["nz"]])
    g = (1.0 + np.array([-1.0, 1.0]) / math.sqrt(3.0)) / 2.0
    K = np.zeros((mesh["nz"], 2, 8, 8))
    for gx in range(2):
        for gy in range(2):
            for gz in range(2):
                xi = (g[gx], g[gy], g[gz])
                G = np.zeros((8, 3))
                for a in range(8):
                    bit = [(a >> d) & 1 for d in range(3)]
                    sh = [xi[d] if bit[d] else 1.0 - xi[d] for d in range(3)]
                    for d in range(3):
                        G[a, d] = (1.0 if bit[d] else -1.0) / h[d] * sh[(d + 1) % 3] * sh[(d + 2) % 3]
                al = fib[:, gz, :]
                for m, (sl, s_t) in enumerate(((p["sil"], p["sit"]), (p["sel"], p["set"]))):
                    D = s_t * np.eye(3) + (sl - s_t) * al[:, :, None] * al[:, None, :]
                    K[:, m] += h.prod() / 8.0 * np.einsum("ad,zde,be->zab", G, D, G)
    return K


def _element_scale(mesh, seed):
    g = _gen(seed + 3)
    return torch.exp(torch.rand((mesh["nz"], mesh["ny"], mesh["nx"]), generator=g, device="cuda",
                                dtype=torch.float64) * 2.0 - 1.0)


def _stencils(mesh, p, fib, scale=None):
    """Ki and Ke as (27, nz+1, ny+1, nx+1) coefficient arrays, and c M."""
    nx, ny, nz = mesh["nx"], mesh["ny"], mesh["nz"]
    Kel = torch.tensor(_element_matrices(mesh, p, fib), device="cuda")
    K = torch.zeros((2, 27, nz + 1, ny + 1, nx + 1), dtype=torch.float64, device="cuda")
    M = torch.zeros((nz + 1, ny + 1, nx + 1), dtype=torch.float64, device="cuda")
    vol = mesh["lx"] / nx * (mesh["ly"] / ny) * (mesh["lz"] / nz) / 8.0
    at = lambda a: (slice(a >> 2 & 1, nz + (a >> 2 & 1)), slice(a >> 1 & 1, ny + (a >> 1 & 1)),  # noqa: E731
                    slice(a & 1, nx + (a & 1)))
    for a in range(8):
        M[at(a)] += vol
        for b in range(8):
            d = [(b >> k & 1) - (a >> k & 1) for k in range(3)]
            o = 9 * (d[2] + 1) + 3 * (d[1] + 1) + d[0] + 1
            for m in range(2):
                k = Kel[:, m, a, b].view(-1, 1, 1)
                K[(m, o) + at(a)] += k if scale is None else k * scale
    return K[0], K[1], M * (p["chi"] * p["cm"] / p["dt"])


def _csr(mesh, fib, scale):
    """The block operator of element-wise scaled conductivities as a caller's scalar CSR."""
    Ki, Ke, cM = _stencils(mesh, W.DEFAULT_PARAMS, fib, scale)
    nz, ny, nx = (mesh[k] + 1 for k in ("nz", "ny", "nx"))
    N = nz * ny * nx
    Z, Y, X = torch.meshgrid(*(torch.arange(k, device="cuda") for k in (nz, ny, nx)), indexing="ij")
    o = torch.arange(27, device="cuda").view(27, 1, 1, 1)
    z, y, x = Z + torch.div(o, 9, rounding_mode="floor") - 1, Y + torch.div(o, 3, rounding_mode="floor") % 3 - 1, X + o % 3 - 1
    ok = ((z >= 0) & (z < nz) & (y >= 0) & (y < ny) & (x >= 0) & (x < nx)).view(27, N).t()
    q = (x + nx * (y + ny * z)).view(27, N).t()[ok]
    ki, ke = (t.reshape(27, N).t()[ok] for t in (Ki, Ke))
    cnt = ok.sum(1)
    row = torch.repeat_interleave(torch.arange(N, device="cuda"), cnt)
    vv = ki + torch.where(row == q, cM.reshape(-1)[row], torch.zeros_like(ki))
    start = torch.cumsum(cnt, 0) - cnt
    k = torch.arange(q.numel(), device="cuda") - start[row]
    val = torch.empty(4 * q.numel(), dtype=torch.float64, device="cuda")
    col = torch.empty(4 * q.numel(), dtype=torch.int32, device="cuda")
    for r, pair in enumerate(((vv, ki), (ki, ki + ke))):
        pos = 4 * start[row] + 2 * cnt[row] * r + 2 * k
        for c, t in enumerate(pair):
            val[pos + c] = t
            col[pos + c] = (2 * q + c).to(torch.int32)
    rp = torch.zeros(2 * N + 1, dtype=torch.int32, device="cuda")
    rp[1:] = torch.cumsum(torch.repeat_interleave(2 * cnt, 2), 0).to(torch.int32)
    return rp, col, val


def _apply(K, x):
    """27-point operator on a (nz+1, ny+1, nx+1) field."""
    p = torch.nn.functional.pad(x[None], (1, 1, 1, 1, 1, 1))[0]
    nz, ny, nx = x.shape
    y = torch.zeros_like(x)
    for o in range(27):
        a, b, c = o // 9, o // 3 % 3, o % 3
        y.addcmul_(K[o], p[a:a + nz, b:b + ny, c:c + nx])
    return y


def _cg(op, dinv, f, x, project, tol=1e-13, most=6000):
    """Jacobi-CG on (k, nz, ny, nx) fields to `tol`; `project` removes a null space."""
    f = project(f)
    r = f - op(x)
    nf = float(f.norm())
    if nf == 0.0:
        return torch.zeros_like(f)
    z = project(dinv * r)
    d, rz = z.clone(), (r * z).sum()
    for i in range(most):
        q = op(d)
        al = rz / (d * q).sum()
        x = x + al * d
        r = r - al * q
        if i % 20 == 19 and float(r.norm()) <= tol * nf:
            break
        z = project(dinv * r)
        new = (r * z).sum()
        d = z + (new / rz) * d
        rz = new
    return project(x)


class _System:
    def __init__(self, mesh, p, fib, scale=None):
        self.p, self.shape = p, tuple(mesh[k] + 1 for k in ("nz", "ny", "nx"))
        self.Ki, self.Ke, self.cM = _stencils(mesh, p, fib, scale)

    def block(self, x):
        a = _apply(self.Ki, x[0] + x[1])
        return torch.stack([self.cM * x[0] + a, a + _apply(self.Ke, x[1])])

    def solve(self, f, x=None):
        dinv = 1.0 / torch.stack([self.cM + self.Ki[13], self.Ki[13] + self.Ke[13]])
        mean0 = lambda t: torch.stack([t[0], t[1] - t[1].mean()])  # noqa: E731
        return _cg(self.block, dinv, f, torch.zeros_like(f) if x is None else x, mean0)

    def flat(self, f):
        x = self.solve(f.view(*self.shape, 2).permute(3, 0, 1, 2).contiguous())
        return x.permute(1, 2, 3, 0).reshape(-1)

    def membrane(self, v, w, stim, t):
        """(updated w, M (I_app - chi I_ion)) of the Rogers-McCulloch model."""
        p = self.p
        w = (w + p["dt"] * 0.012 * v / 100.0) / (1.0 + p["dt"] * 0.012)
        ion = 1.5 * v * (1.0 - v / 13.0) * (1.0 - v / 100.0) + 4.4 * v * w
        M = self.cM * (p["dt"] / (p["chi"] * p["cm"]))
        return w, M * ((stim if t < 1.0 else 0.0) - p["chi"] * ion)

    def coupled(self, stim, steps):
        x = torch.zeros((2,) + self.shape, dtype=torch.float64, device="cuda")
        w = torch.zeros(self.shape, dtype=torch.float64, device="cuda")
        stim = torch.as_tensor(stim, device="cuda").view(self.shape)
        for k in range(steps):
            w, g = self.membrane(x[0], w, stim, k * self.p["dt"])
            x = self.solve(torch.stack([self.cM * x[0] + g, torch.zeros_like(g)]), x)
        return [t.reshape(-1).cpu() for t in (x[0], x[1], w)]

    def decoupled(self, v, w, stim, steps):
        v, w = v.view(self.shape), w.view(self.shape)
        stim = torch.as_tensor(stim, device="cuda").view(self.shape)
        Kt = self.Ki + self.Ke
        mean0 = lambda t: t - t.mean()  # noqa: E731
        u = torch.zeros_like(v)
        for k in range(steps):
            u = _cg(lambda t: _apply(Kt, t), 1.0 / Kt[13], -_apply(self.Ki, v), u, mean0)
            w, g = self.membrane(v, w, stim, k * self.p["dt"])
            v = _cg(lambda t: self.cM * t + _apply(self.Ki, t), 1.0 / (self.cM + self.Ki[13]),
                    self.cM * v - _apply(self.Ki, u) + g, v, lambda t: t)
        return [t.reshape(-1).cpu() for t in (v, u, w)]


def exact(case, seed):
    kind = case["kind"]
    if kind == "dot":
        st = prepare(case, seed)
        prod = (st["x"] * st["y"]).cpu().numpy()  # each product rounded, then the exact sum rounded once
        return torch.tensor([math.fsum(prod)], dtype=torch.float64)
    if kind == "vcycle":
        return None  # defined by the hierarchy, which this library alone builds
    if kind == "stack":
        out = [_System(m, p, fib).flat(_rhs(2 * W.n_nodes(m), seed + k))
               for k, (m, p, fib) in enumerate(_slabs(case, seed))]
        return dict(x=torch.cat(out), iters=None)
    if kind == "serve":
        return [tuple(t.numpy() for t in _System(m, W.DEFAULT_PARAMS, fib).coupled(stim, steps))
                for m, fib, stim, steps in _requests(case, seed)]
    m = _mesh(case)
    S = _System(m, W.DEFAULT_PARAMS, _fibres(m, seed), _element_scale(m, seed) if kind == "csr" else None)
    if kind == "step":
        v, ue, w = S.coupled(_stimulus(m, seed), case["steps"])
        return dict(v=v, ue=ue, w=w, iters=None)
    if kind == "dsim":
        v, ue, w = S.decoupled(*_front(m, seed), _stimulus(m, seed), case["steps"])
        return dict(v=v.numpy(), ue=ue.numpy(), w=w.numpy(), iters=None)
    return dict(x=S.flat(_rhs(2 * W.n_nodes(m), seed)), iters=None, lam=None, sizes=None)
