"""Dipole of rows with fewer strings than the diagonal tables have entries (2^(ceil(n/2) + 1)),
which sum a string's diagonal integrals directly, and of rows just above, which look them up;
against the oracle.  FP64 sums of at most 2 * 81 + 1 terms: 1e-13 of the norm."""
import numpy as np
import pytest

import oracle
import synthetic

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,na,nb", [
    (1, 1, 0), (2, 1, 1), (3, 1, 1), (5, 2, 0), (5, 3, 5), (8, 4, 2), (8, 2, 3), (7, 3, 2),
    (9, 3, 2), (9, 2, 3), (12, 3, 2), (12, 2, 3), (16, 3, 1), (18, 2, 1), (18, 1, 2),
])
def test_dipole_short_rows(n, na, nb):
    import torch

    from paper_2506_07430_gb300 import KPM
    I = synthetic.integrals(n, na, nb, seed=2506900 + n)
    sc = oracle.SlaterCondon(I.h1, I.eri, n, na, nb)
    psi = synthetic.random_state(sc.dim, 3)
    k = KPM(I.h1, I.eri, I.dipole, n, na, nb, precision="fp64")
    for c in range(3):
        y = k.apply_dipole(c, torch.from_numpy(psi).cuda())
        k.synchronize()
        ref = sc.dipole(I.dipole[c], psi)
        assert np.linalg.norm(y.cpu().numpy() - ref) <= 1e-13 * np.linalg.norm(ref), c
    k.close()
