"""Finest level as a layered stencil: the symmetric form (fibres in the plane)
and the general one (fibres with a z component) against the oracle, which
applies the assembled CSR operator, at the sizes where the kernel's walks can go
wrong: slabs one element thick in each direction (no interior row type), one
column block more or less, walks that wrap over column blocks.  V-cycle 1e-10
(the solve phase's bound in FP64) and 1e-4 in FP32, solutions 1e-7; a stack mixes
both forms."""
import numpy as np
import pytest

from paper_2311_13914_gb300 import workloads as W

pytestmark = pytest.mark.gpu

MESHES = [(9, 9, 1), (1, 40, 12), (40, 1, 12), (2, 2, 60), (15, 7, 9), (14, 8, 9), (63, 31, 3), (5, 4, 300)]


@pytest.fixture(scope="module")
def B():
    import torch

    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA GPU")
    from paper_2311_13914_gb300 import _build, binding

    _build.build()
    return binding


def _fib(m, tilt):
    """Rotating fibres, lifted out of the plane by an angle that varies with z."""
    fib = W.fibre_table(m, 120.0, 5.0)
    if tilt:
        a = np.linspace(0.2, 0.7, 2 * m["nz"]).reshape(-1, 2)
        fib = fib * np.cos(a)[..., None]
        fib[..., 2] = np.sin(a)
    return fib


@pytest.mark.parametrize("tilt", [False, True])
@pytest.mark.parametrize("size", MESHES)
def test_stencil_forms_match_oracle(B, oracle_lib, size, tilt):
    m = W.mesh(*size)
    fib = _fib(m, tilt)
    sysh = B.bd_assemble(m, W.DEFAULT_PARAMS, fib)
    o = oracle_lib.assemble(m, W.DEFAULT_PARAMS, fib)
    H = oracle_lib.Hierarchy(o["A"], coarse_eq_limit=30)
    n = o["A"].shape[0]
    f = W.rhs(n, 3)
    zo = H.vcycle(f)
    xo, _ = H.pcg(f, rtol=1e-10)
    for precision, bound in ((0, 1e-10), (1, 1e-4)):
        h = B.amg_setup(sysh, B.amg_options_default(coarse_eq_limit=30, precision=precision))
        assert B.amg_num_levels(h) > 1
        z = B.amg_vcycle(h, f)
        assert np.linalg.norm(z - zo) <= bound * np.linalg.norm(zo)
        x, info = B.amg_solve(h, f, opts=B.solve_options_default(rtol=1e-10))
        assert info["status"] == 0 and info["true_rel_res"] <= 1.01e-10
        assert np.linalg.norm(x - xo) <= 1e-7 * np.linalg.norm(xo)


@pytest.mark.parametrize("precision", [0, 1])
def test_stack_of_both_forms(B, precision):
    import torch

    hs, fs, xs, ref = [], [], [], []
    for k, (size, tilt) in enumerate([((15, 7, 9), True), ((14, 8, 9), False), ((1, 1, 1), False), ((2, 2, 60), True)]):
        m = W.mesh(*size)
        sysh = B.bd_assemble(m, W.DEFAULT_PARAMS, _fib(m, tilt))
        h = B.amg_setup(sysh, B.amg_options_default(coarse_eq_limit=30, precision=precision))
        f = torch.tensor(W.rhs(2 * W.n_nodes(m), k), device="cuda")
        ref.append(B.amg_solve(h, f, torch.zeros_like(f)))
        hs.append(h)
        fs.append(f)
        xs.append(torch.zeros_like(f))
    for (xr, ir), x, i in zip(ref, xs, B.amg_stack_solve(B.amg_stack_create(hs), fs, xs)):
        assert i["status"] == 0 and abs(i["iters"] - ir["iters"]) <= 1
        assert float((x - xr).norm()) <= 1e-7 * float(xr.norm())


@pytest.mark.parametrize("precision", [0, 1])
def test_stack_of_stencil_and_csr_members(B, precision):
    """A member given as a caller's CSR has no stencil: the whole stack then runs
    on blocks, the slab's included."""
    import torch

    m = W.mesh(14, 8, 9)
    sysh = B.bd_assemble(m, W.DEFAULT_PARAMS, _fib(m, False))
    rp, ci, v, _ = B.bd_system_export(sysh)
    n = rp.size - 1
    o = B.amg_options_default(coarse_eq_limit=30, precision=precision)
    hs = [B.amg_setup(sysh, o), B.amg_setup_from_csr(n, rp, ci, v, o)]
    fs = [torch.tensor(W.rhs(n, k), device="cuda") for k in range(2)]
    ref = [B.amg_solve(h, f, torch.zeros_like(f))[0] for h, f in zip(hs, fs)]
    xs = [torch.zeros_like(f) for f in fs]
    for x, xr, i in zip(xs, ref, B.amg_stack_solve(B.amg_stack_create(hs), fs, xs)):
        assert i["status"] == 0 and float((x - xr).norm()) <= 1e-7 * float(xr.norm())
