"""FP64 sigma of molecules on either side of the line between the row kernel and the gather
kernel for long rows, against the oracle on sampled rows (tolerance as for every FP64 sigma:
sums of up to 1e4 terms)."""
import numpy as np
import pytest

import oracle
import synthetic

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,na,nb", [
    (14, 3, 6),     # 364 rows of 3003 strings: chunks of several entries
    (16, 3, 6),     # 560 rows of 8008: a single one
])
def test_long_rows_fp64(n, na, nb):
    import torch

    from paper_2506_07430_gb300 import KPM
    I = synthetic.integrals(n, na, nb, seed=2506860 + n)
    k = KPM(I.h1, I.eri, I.dipole, n, na, nb, precision="fp64")
    x = synthetic.random_state(k.dim, 7)
    y = k.sigma(torch.from_numpy(x).cuda()).cpu().numpy().reshape(-1)
    sc = oracle.SlaterCondon(I.h1, I.eri, n, na, nb)
    rows = np.unique(np.concatenate([
        [0, 1, k.dim // 2, k.dim - 1],
        np.random.default_rng(11).integers(0, k.dim, 400)])).astype(np.int64)
    ref = sc.sigma_rows(rows, x)
    assert np.abs(y[rows] - ref).max() <= 1e-12 * np.abs(y).max()
    k.close()
