"""The decoupled scheme's scalar solves: the elliptic solve on its one field
against the block solve of the same hierarchy (live timing selects it) and the
whole step against the oracle, over both stencil forms, thin slabs, both V-cycle
precisions, a single dense level, a coarsest level above 256 unknowns, zero
states and the iteration limit.  Solutions to 1e-6 (the scheme's parity bound)."""
import numpy as np
import pytest

from paper_2311_13914_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def B():
    import torch

    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA GPU")
    from paper_2311_13914_gb300 import _build, binding

    _build.build()
    return binding


def _case(B, size, tilt, **opts):
    m = W.mesh(*size)
    fib = W.fibre_table(m, 120.0, 5.0)
    if tilt:
        a = np.linspace(0.2, 0.7, 2 * m["nz"]).reshape(-1, 2)
        fib = fib * np.cos(a)[..., None]
        fib[..., 2] = np.sin(a)
    sysh = B.bd_assemble(m, W.DEFAULT_PARAMS, fib)
    rng = np.random.default_rng(size[0])
    N = W.n_nodes(m)
    state = (80.0 * rng.random(N), 0.3 * rng.standard_normal(N), 0.2 * rng.random(N))
    return m, fib, sysh, B.bd_elliptic_setup(sysh, B.amg_options_default(**opts)), state, N


CASES = [((15, 7, 9), False, dict(coarse_eq_limit=30)), ((15, 7, 9), True, dict(coarse_eq_limit=30)),
         ((9, 9, 1), False, {}), ((1, 40, 12), True, dict(coarse_eq_limit=30)), ((2, 2, 60), False, {}),
         ((3, 3, 3), False, dict(coarse_eq_limit=2000)), ((40, 36, 12), False, dict(coarse_eq_limit=2000))]


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("size,tilt,opts", CASES)
def test_scalar_step_matches_block_solve_and_oracle(B, oracle_lib, size, tilt, opts, precision):
    m, fib, sysh, h, (v, ue, w), N = _case(B, size, tilt, precision=precision, **opts)
    got = []
    for block in (False, True):
        sim = B.bd_dsim_create(sysh, h, jacobi=not tilt)
        B.bd_dsim_set_state(sim, v=v, ue=ue, w=w)
        B.amg_profile_enable(h, int(block))
        info = B.bd_dsim_step(sim, 2)
        B.amg_profile_enable(h, 0)
        got.append((B.bd_dsim_get_state(sim, N), info))
    (a, ia), (b, ib) = got
    assert abs(ia[0]["total_iters"] - ib[0]["total_iters"]) <= 2
    o = oracle_lib.assemble(m, W.DEFAULT_PARAMS, fib)
    H = oracle_lib.Hierarchy(oracle_lib.elliptic_block(o["Ki"], o["Ke"]), **opts)
    ov, ou, ow = v.copy(), ue.copy(), w.copy()
    for _ in range(2):
        H.bd_step_decoupled(o["Ki"], o["M"], W.DEFAULT_PARAMS, np.zeros(N), ov, ou, ow, jacobi=not tilt)
    for x, y, z in zip(a, b, (ov, ou, ow)):
        assert np.linalg.norm(x - y) <= 1e-6 * np.linalg.norm(y)
        assert np.linalg.norm(x - z) <= 1e-6 * np.linalg.norm(z)
    assert ia[0]["status"] == ia[1]["status"] == 0
    assert ia[0]["true_rel_res"] <= 1.01e-8 and ia[1]["true_rel_res"] <= 1.01e-8


def test_zero_state_and_iteration_limit(B):
    m, fib, sysh, h, (v, ue, w), N = _case(B, (15, 7, 9), False, coarse_eq_limit=30)
    sim = B.bd_dsim_create(sysh, h)
    B.bd_dsim_set_state(sim, ue=ue)  # v = 0: zero right-hand sides, u_e and v go to zero
    ie, ip = B.bd_dsim_step(sim, 1)
    assert ie["status"] == ip["status"] == 0 and ie["iters"] == ip["iters"] == 0
    assert all(not np.any(x) for x in B.bd_dsim_get_state(sim, N))
    sim = B.bd_dsim_create(sysh, h)
    B.bd_dsim_set_state(sim, v=v, w=w)
    ie, ip = B.bd_dsim_step(sim, 1, B.solve_options_default(max_it=2, rtol=1e-12), raise_on_error=False)
    assert ie["status"] == B.BD_ENOTCONV and ie["iters"] == 2  # the step stops there: v and w unchanged
    gv, _, gw = B.bd_dsim_get_state(sim, N)
    assert np.array_equal(gv, v) and np.array_equal(gw, w)
