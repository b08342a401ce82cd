"""The smoothed prolongator P = Pt - omega D^-1 (A Pt) of the finest level, bit for bit,
from the exported aggregates and lambda: A Pt is the product whose rows a part of a
warp hashes (rows of B of one block, 19456 rows and more).  The setup of such a slab
forms products by hashing and by dense rows."""
import numpy as np
import pytest

from paper_2311_13914_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("size", [(48, 48, 12), (39, 38, 13)])
def test_finest_prolongator_bits(size):
    from paper_2311_13914_gb300 import binding as B

    m = W.mesh(*size)
    N = W.n_nodes(m)
    assert N >= 19456
    s = B.bd_assemble(m, W.DEFAULT_PARAMS, W.fibre_table(m, 120.0, 10.0))
    before = B.bd_spgemm_path_counts()
    h = B.amg_setup(s)
    hashed, dense = (b - a for a, b in zip(before, B.bd_spgemm_path_counts()))
    assert hashed >= 3  # the squared graph, A Pt and A P of the finest level
    assert dense >= 1 or size != (48, 48, 12)
    e = B.amg_export_level(h, 0)
    rp, ci, v = e["A"]
    agg = np.asarray(e["agg"], dtype=np.int64)
    nagg = int(agg.max()) + 1
    # blocks of A: rows 2p and 2p + 1 hold the same columns
    cnt = np.diff(rp)[0::2] // 2
    row = np.repeat(np.arange(N), cnt)
    k = np.arange(row.size) - np.repeat(np.cumsum(cnt) - cnt, cnt)
    at = [rp[2 * row + r] + 2 * k for r in (0, 1)]
    col = ci[at[0]] // 2
    a = [[v[at[r] + c] for c in (0, 1)] for r in (0, 1)]
    # Pt: 1 / |aggregate|^(1/2) (B = 1 on the finest level; sums of ones are exact)
    pt = 1.0 / np.sqrt(np.bincount(agg, minlength=nagg).astype(np.float64))[agg]
    key = row * nagg + agg[col]
    cols, slot = np.unique(key, return_inverse=True)
    omega = 4.0 / (3.0 * B.amg_level_info(h, 0)["lam"])
    prow, pcol = cols // nagg, cols % nagg
    got = e["P"]
    assert np.array_equal(np.diff(got[0])[0::2] // 2, np.bincount(prow, minlength=N))
    first = np.cumsum(np.bincount(prow, minlength=N)) - np.bincount(prow, minlength=N)
    j = np.arange(cols.size) - first[prow]
    own = np.where(agg[prow] == pcol, pt[prow], 0.0)
    diag = np.zeros((2, N))
    for r in (0, 1):
        diag[r][row[row == col]] = a[r][r][row == col]
    for r in (0, 1):
        for c in (0, 1):
            ap = np.zeros(cols.size)
            np.add.at(ap, slot, a[r][c] * pt[col])  # one after the other, columns ascending
            want = (own if r == c else 0.0) - (omega / diag[r])[prow] * ap
            pos = got[0][2 * prow + r] + 2 * j + c
            assert np.array_equal(got[1][pos], 2 * pcol + c)
            assert np.array_equal(got[2][pos], want)
