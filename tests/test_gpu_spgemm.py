"""Galerkin products R (A P) of the coarse levels against scipy's, on slabs whose
levels take each way of forming them: rows hashed by part of a warp and by whole
warps, a warp per row with an accumulator per column, a thread block per row.

Both sides sum the same terms; with n terms either is within n 2^-53 of the sum of
their absolute values, so the two are within twice that."""
import numpy as np
import pytest

sp = pytest.importorskip("scipy.sparse")

pytestmark = pytest.mark.gpu

PITCH = dict(lx=1.0, ly=1.0, lz=0.5)


@pytest.mark.parametrize("n, limit, first", [((24, 24, 12), 60, 0), ((40, 33, 7), 40, 0), ((96, 96, 24), 100, 1),
                                             ((128, 128, 32), 2000, 1)])
def test_galerkin_products(n, limit, first):
    from paper_2311_13914_gb300 import binding as B, workloads as W

    m = dict(zip(("nx", "ny", "nz"), n), **PITCH)
    s = B.bd_assemble(m, W.DEFAULT_PARAMS, W.fibre_table(m, 120.0, 10.0))
    h = B.amg_setup(s, B.amg_options_default(precision=0, coarse_eq_limit=limit))
    levels = B.amg_num_levels(h)
    assert levels > first + 1
    mat = lambda t, shape: sp.csr_matrix((t[2], t[1], t[0]), shape=shape)  # noqa: E731
    fine = B.amg_export_level(h, first)
    for lv in range(first, levels - 1):
        coarse = B.amg_export_level(h, lv + 1)
        A = mat(fine["A"], (fine["n"],) * 2)
        P = mat(fine["P"], (fine["n"], coarse["n"]))
        got = mat(coarse["A"], (coarse["n"],) * 2)
        want = (P.T.tocsr() @ (A @ P)).tocsr()
        want.sort_indices()
        assert np.array_equal(got.indptr, want.indptr) and np.array_equal(got.indices, want.indices)
        size = (abs(P).T.tocsr() @ (abs(A) @ abs(P))).tocsr()
        size.sort_indices()
        terms = np.diff(P.tocsc().indptr).max() + np.diff(A.indptr).max()
        assert np.all(np.abs(got.data - want.data) <= 2 * terms * 2.0**-53 * size.data)
        fine = coarse
