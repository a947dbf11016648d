"""FP64 sigma of many rows of few strings each: the row kernel's staging of W is spread over
more threads than there are items, and left out where no beta string has an off-diagonal
entry.  Sampled rows against the oracle; FP64 sums of up to 1500 terms: 1e-13."""
import numpy as np
import pytest

import oracle
import synthetic

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,na,nb", [
    (18, 5, 1), (18, 5, 0), (16, 6, 1), (16, 5, 16), (14, 7, 13), (12, 6, 0), (10, 5, 1),
])
def test_short_rows_match_oracle(n, na, nb):
    import torch

    from paper_2506_07430_gb300 import KPM
    I = synthetic.integrals(n, na, nb, seed=2506970 + n)
    sc = oracle.SlaterCondon(I.h1, I.eri, n, na, nb)
    k = KPM(I.h1, I.eri, I.dipole, n, na, nb, precision="fp64")
    x = torch.randn((2, k.dim), generator=torch.Generator(device="cuda").manual_seed(4),
                    device="cuda", dtype=torch.float64)
    y = k.sigma(x).cpu().numpy()
    rows = np.unique(np.linspace(0, k.dim - 1, 400).astype(np.int64))
    for c in range(2):
        ref = sc.sigma_rows(rows, x[c].cpu().numpy())
        assert np.abs(y[c][rows] - ref).max() <= 1e-13 * np.abs(y[c]).max()
    k.close()
