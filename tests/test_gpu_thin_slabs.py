"""Slabs one element wide in x or y under fibres that leave the plane.  Such a slab has
no row type with both members of an x (or y) pair, so its in-plane symmetry says
nothing about the coupling between planes, on which the choice of the stencil's
form (68 flops a node symmetric, 108 general) rests as well.  Against the oracle, which
applies the assembled CSR operator: V-cycle 1e-10 in FP64 and 1e-4 in FP32,
solutions 1e-7, decoupled steps 1e-6 (the bounds of each path)."""
import numpy as np
import pytest

from paper_2311_13914_gb300 import workloads as W

pytestmark = pytest.mark.gpu

XZ, YZ, XYZ, XY = (0.8, 0.0, 0.6), (0.0, 0.8, 0.6), (0.6, 0.48, 0.64), (0.6, 0.8, 0.0)
OUT_OF_PLANE = [((1, 4, 3), XZ), ((1, 40, 12), XZ), ((1, 40, 12), YZ), ((4, 1, 3), YZ), ((40, 1, 12), YZ),
                ((40, 1, 12), XZ), ((1, 1, 9), XYZ), ((1, 1, 40), XZ), ((1, 1, 40), YZ), ((3, 4, 3), XZ)]
IN_PLANE = [((1, 4, 3), XY), ((1, 1, 40), XY), ((40, 1, 12), XY), ((3, 4, 3), XY)]


@pytest.fixture(scope="module")
def B():
    import torch

    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA GPU")
    from paper_2311_13914_gb300 import _build, binding

    _build.build()
    return binding


def _slab(size, fibre):
    m = W.mesh(*size)
    return m, np.tile(np.array(fibre), (m["nz"], 2, 1))


def _flops_per_node(B, h, f):
    """Flops of one finest-level launch per node: which form the stencil took."""
    B.amg_profile_enable(h, 1)
    B.amg_vcycle(h, f)
    prof = B.amg_profile_read(h)
    B.amg_profile_enable(h, 0)
    return prof["flops"] / prof["launches"] / (f.size // 2)


@pytest.mark.parametrize("size,fibre", OUT_OF_PLANE + IN_PLANE)
def test_form_and_solution(B, oracle_lib, size, fibre):
    m, fib = _slab(size, fibre)
    sysh = B.bd_assemble(m, W.DEFAULT_PARAMS, fib)
    o = oracle_lib.assemble(m, W.DEFAULT_PARAMS, fib)
    H = oracle_lib.Hierarchy(o["A"], coarse_eq_limit=30)
    f = W.rhs(o["A"].shape[0], 3)
    zo = H.vcycle(f)
    xo, _ = H.pcg(f, rtol=1e-10)
    for precision, bound in ((0, 1e-10), (1, 1e-4)):
        h = B.amg_setup(sysh, B.amg_options_default(coarse_eq_limit=30, precision=precision))
        assert B.amg_num_levels(h) > 1
        assert _flops_per_node(B, h, f) == (108 if fibre[2] else 68)
        z = B.amg_vcycle(h, f)
        assert np.linalg.norm(z - zo) <= bound * np.linalg.norm(zo)
        x, info = B.amg_solve(h, f, opts=B.solve_options_default(rtol=1e-10))
        assert info["status"] == 0 and info["true_rel_res"] <= 1.01e-10
        assert np.linalg.norm(x - xo) <= 1e-7 * np.linalg.norm(xo)


@pytest.mark.parametrize("size,fibre", [((1, 40, 12), XZ), ((40, 1, 12), YZ), ((1, 1, 40), XYZ)])
def test_decoupled_step(B, oracle_lib, size, fibre):
    m, fib = _slab(size, fibre)
    N = W.n_nodes(m)
    rng = np.random.default_rng(7)
    v, ue, w = 80.0 * rng.random(N), 0.3 * rng.standard_normal(N), 0.2 * rng.random(N)
    sysh = B.bd_assemble(m, W.DEFAULT_PARAMS, fib)
    sim = B.bd_dsim_create(sysh, B.bd_elliptic_setup(sysh, B.amg_options_default(coarse_eq_limit=30)))
    B.bd_dsim_set_state(sim, v=v, ue=ue, w=w)
    B.bd_dsim_step(sim, 2)
    o = oracle_lib.assemble(m, W.DEFAULT_PARAMS, fib)
    H = oracle_lib.Hierarchy(oracle_lib.elliptic_block(o["Ki"], o["Ke"]), coarse_eq_limit=30)
    ov, ou, ow = v.copy(), ue.copy(), w.copy()
    for _ in range(2):
        H.bd_step_decoupled(o["Ki"], o["M"], W.DEFAULT_PARAMS, np.zeros(N), ov, ou, ow, jacobi=True)
    for x, y in zip(B.bd_dsim_get_state(sim, N), (ov, ou, ow)):
        assert np.linalg.norm(x - y) <= 1e-6 * np.linalg.norm(y)


@pytest.mark.parametrize("precision", [0, 1])
def test_stack(B, oracle_lib, precision):
    """Thin out-of-plane members alone, and with a member of the symmetric form."""
    import torch

    members = [((1, 40, 12), XZ), ((40, 1, 12), YZ), ((1, 1, 9), XYZ)]
    for slabs in (members, members + [((14, 8, 9), XY)]):
        hs, fs, want = [], [], []
        for k, (size, fibre) in enumerate(slabs):
            m, fib = _slab(size, fibre)
            sysh = B.bd_assemble(m, W.DEFAULT_PARAMS, fib)
            hs.append(B.amg_setup(sysh, B.amg_options_default(coarse_eq_limit=30, precision=precision)))
            o = oracle_lib.assemble(m, W.DEFAULT_PARAMS, fib)
            f = W.rhs(o["A"].shape[0], k)
            want.append(oracle_lib.Hierarchy(o["A"], coarse_eq_limit=30).pcg(f, rtol=1e-10)[0])
            fs.append(torch.tensor(f, device="cuda"))
        xs = [torch.zeros_like(f) for f in fs]
        infos = B.amg_stack_solve(B.amg_stack_create(hs), fs, xs, B.solve_options_default(rtol=1e-10))
        for x, xo, i in zip(xs, want, infos):
            assert i["status"] == 0
            assert np.linalg.norm(x.cpu().numpy() - xo) <= 1e-7 * np.linalg.norm(xo)
