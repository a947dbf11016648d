"""FP64 sigma of sectors with few terms a determinant, which the gather kernel takes, and of
those just above, which the row kernel takes: against the oracle's dense H, and alone as in
one batch with a larger molecule.  FP64 sums of up to some hundred terms: 1e-13."""
import numpy as np
import pytest

import oracle
import synthetic

pytestmark = pytest.mark.gpu

# up to 34 terms | from 35; without opposite-spin entries up to 63 | from 64
MOLS = [(1, 1, 0), (2, 1, 1), (3, 2, 1), (4, 1, 1), (4, 2, 1), (5, 1, 1), (4, 2, 2), (4, 0, 2),
        (5, 0, 3), (8, 4, 0), (10, 5, 0), (3, 3, 1), (3, 1, 3), (2, 0, 0)]


def _ctx(n, na, nb):
    import torch

    from paper_2506_07430_gb300 import KPM
    I = synthetic.integrals(n, na, nb, seed=2506920 + n)
    k = KPM(I.h1, I.eri, I.dipole, n, na, nb, precision="fp64")
    return I, k, torch.from_numpy(synthetic.random_state(k.dim, 7)).cuda()


@pytest.mark.parametrize("n,na,nb", MOLS)
def test_sigma_matches_oracle(n, na, nb):
    import torch
    I, k, _ = _ctx(n, na, nb)
    H = oracle.SlaterCondon(I.h1, I.eri, n, na, nb).dense()
    x = torch.randn((3, k.dim), generator=torch.Generator(device="cuda").manual_seed(1),
                    device="cuda", dtype=torch.float64)
    y = k.sigma(x).cpu().numpy()
    ref = x.cpu().numpy() @ H
    assert np.abs(y - ref).max() <= 1e-13 * np.abs(ref).max()
    k.close()


def test_batch_equals_alone():
    from paper_2506_07430_gb300 import moments_batch
    ctx = [_ctx(*m) for m in MOLS + [(6, 3, 3)]]
    ks, psis = [c[1] for c in ctx], [c[2] for c in ctx]
    a, b = [60.0] * len(ks), [0.0] * len(ks)
    alone = [k.moments(p, 7, 60.0, 0.0, 64) for k, p in zip(ks, psis)]
    for x, y in zip(alone, moments_batch(ks, psis, 7, a, b, 64)):
        assert np.array_equal(x, y)
    for k in ks:
        k.close()
