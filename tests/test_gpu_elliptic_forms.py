"""Operator forms of an elliptic hierarchy reach the one-field operators that the
decoupled scheme applies.  The lanes per row change the order of a row's sum and so the
last bits of a step, never more than the solves' tolerance allows (1e-6, the scheme's
parity bound); the same lanes give the same bits."""
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


def _step(B, sysh, h, N):
    rng = np.random.default_rng(11)
    sim = B.bd_dsim_create(sysh, h)
    B.bd_dsim_set_state(sim, v=80.0 * rng.random(N), ue=0.3 * rng.standard_normal(N), w=0.2 * rng.random(N))
    ie, ip = B.bd_dsim_step(sim, 2)
    assert ie["status"] == ip["status"] == 0
    return np.concatenate(B.bd_dsim_get_state(sim, N))


@pytest.mark.parametrize("precision", [0, 1])
def test_set_lanes_reach_the_decoupled_step(B, precision):
    from paper_2311_13914_gb300 import forms

    m = W.mesh(24, 20, 10)
    N = W.n_nodes(m)
    sysh = B.bd_assemble(m, W.DEFAULT_PARAMS, W.fibre_table(m, 120.0, 5.0))
    h = B.bd_elliptic_setup(sysh, B.amg_options_default(precision=precision, coarse_eq_limit=30))
    levels = B.amg_num_levels(h)
    assert levels > 2
    start = [B.amg_level_lanes(h, l) for l in range(levels - 1)]

    def with_lanes(pick):
        for l in range(levels - 1):
            lanes = pick(l)
            B.amg_set_level_lanes(h, l, (lanes[0] if l else 0, lanes[1], lanes[2]))
        return _step(B, sysh, h, N)

    first = _step(B, sysh, h, N)
    some = {T: with_lanes(lambda l: (T, T, T)) for T in (2, 16, 64, -2)}
    for x in some.values():
        assert np.linalg.norm(x - first) <= 1e-6 * np.linalg.norm(first)
    assert not np.array_equal(some[2], some[16]) and not np.array_equal(some[16], some[64])
    assert np.array_equal(some[-2], some[2])
    assert np.array_equal(with_lanes(lambda l: start[l]), first)
    f = W.rhs(2 * N, 1)
    f[0::2] = 0.0
    forms.time_forms(h, f, candidates=(1, 8), reps=1, warm=1)
    assert np.array_equal(_step(B, sysh, h, N), first)


def test_tuner_reaches_the_one_field_operators(B):
    """Launches that amg_options.autotune adds to the setup: the block hierarchy of the same
    matrix tells how many of them are the block operators'.  FP32, whose candidates are
    block-CSR only, launches the same number every time."""
    m = W.mesh(48, 48, 12)
    N = W.n_nodes(m)
    sysh = B.bd_assemble(m, W.DEFAULT_PARAMS, W.fibre_table(m, 120.0, 5.0))
    opts = [B.amg_options_default(precision=1, autotune=a) for a in (0, 1)]
    plain = B.bd_elliptic_setup(sysh, opts[0])
    A = B.amg_export_level(plain, 0)["A"]

    def added(setup):
        counts = []
        for o in opts:
            before = B.bd_launch_count()
            h = setup(o)
            counts.append(B.bd_launch_count() - before)
        return counts[1] - counts[0], h

    blocks, _ = added(lambda o: B.amg_setup_from_csr(2 * N, *A, o))
    both, tuned = added(lambda o: B.bd_elliptic_setup(sysh, o))
    # the finest R and P and the second level's A have 20000 blocks and more, each at
    # least four candidates of four launches
    assert blocks > 0 and both >= blocks + 3 * 4 * 4
    x, y = _step(B, sysh, plain, N), _step(B, sysh, tuned, N)
    assert np.linalg.norm(x - y) <= 1e-6 * np.linalg.norm(x)
    assert np.array_equal(_step(B, sysh, tuned, N), y)
