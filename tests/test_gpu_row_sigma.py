"""FP64 and FP32 sigma of the row kernels (csrc/sigma_rows.cu) at the edges of their
dispatch and tiles, against the oracle's determinant-pair row-pull.

Tolerances are the sigma tolerances of the parity tests: FP64 1e-12 max|y| (sums of at
most 1e4 FP64 terms), FP32 2e-6 max|y| (x rounded to FP32 on both sides).
"""
import numpy as np
import pytest

import oracle
import synthetic

pytestmark = pytest.mark.gpu

TOL = {"fp64": 1e-12, "fp32": 2e-6}


@pytest.fixture(scope="module")
def torch():
    import torch as _t
    assert _t.cuda.is_available()
    return _t


# FP64: rows of 1 to 1716 strings (every split of a row's term list, one and several
# chunks of D, no or one electron per spin, the gather kernel below 100 long rows);
# FP32: the pair-tiled kernels from 301 strings on (even and odd row lengths, a last
# tile of one to 63 columns, every pair count per pass in use there), and the gather
# kernel beside them.
CASES = [("fp64", 6, 3, 1), ("fp64", 7, 3, 4), ("fp64", 9, 5, 4), ("fp64", 9, 0, 4),
         ("fp64", 9, 4, 0), ("fp64", 10, 5, 5), ("fp64", 11, 4, 5), ("fp64", 12, 6, 4),
         ("fp64", 12, 1, 6), ("fp64", 13, 3, 6), ("fp32", 11, 4, 4), ("fp32", 11, 6, 5),
         ("fp32", 12, 5, 7), ("fp32", 12, 3, 6), ("fp32", 13, 3, 6), ("fp32", 13, 10, 5),
         ("fp32", 14, 3, 10), ("fp32", 12, 1, 6), ("fp32", 11, 5, 2)]


@pytest.mark.parametrize("prec,n,na,nb", CASES)
def test_row_sigma(torch, prec, n, na, nb):
    from paper_2506_07430_gb300 import KPM
    I = synthetic.integrals(n, na, nb, seed=2506700 + 16 * n + na)
    sc = oracle.SlaterCondon(I.h1, I.eri, n, na, nb)
    k = KPM(I.h1, I.eri, I.dipole, n, na, nb, precision=prec)
    X = np.stack([synthetic.random_state(sc.dim, s) for s in (3, 4)])
    xt = torch.tensor(X, dtype=k.vdtype, device="cuda")
    y = k.sigma(xt).cpu().numpy().astype(np.float64)
    one = k.sigma(xt[1].contiguous()).cpu().numpy().astype(np.float64)
    again = k.sigma(xt).cpu().numpy().astype(np.float64)
    k.close()
    assert np.array_equal(y[1], one) and np.array_equal(y, again)
    rows = np.arange(sc.dim)
    if sc.dim > 20000:
        rng = np.random.default_rng(9)
        rows = np.unique(np.concatenate([rng.choice(sc.dim, 4000, replace=False),
                                         np.arange(64), np.arange(sc.dim - 64, sc.dim)]))
    for c in range(2):
        x = xt[c].cpu().numpy().astype(np.float64)
        ref = sc.sigma_rows(rows, x)
        assert np.abs(y[c][rows] - ref).max() <= TOL[prec] * np.abs(ref).max()


def test_batch_mixes_sigma_paths(torch):
    """One batch over molecules of every FP32 (gather, pair-tiled) and FP64 (row, gather)
    path: the moments are those of each molecule alone, bit for bit."""
    from paper_2506_07430_gb300 import KPM, moments_batch
    for prec, mols in (("fp32", [(6, 3, 3), (11, 5, 5), (11, 6, 4), (8, 4, 3)]),
                       ("fp64", [(8, 4, 4), (12, 1, 6), (9, 4, 5)])):
        ks, psis = [], []
        for i, (n, na, nb) in enumerate(mols):
            I = synthetic.integrals(n, na, nb, seed=2506760 + i)
            ks.append(KPM(I.h1, I.eri, I.dipole, n, na, nb, precision=prec))
            psis.append(torch.tensor(synthetic.random_state(ks[-1].dim, 60 + i), device="cuda"))
        a, b = [60.0] * len(ks), [-5.0] * len(ks)
        got = moments_batch(ks, psis, 0b101, a, b, 22)
        for i, k in enumerate(ks):
            assert np.array_equal(got[i], k.moments(psis[i], 0b101, a[i], b[i], 22)), (prec, i)
            k.close()
