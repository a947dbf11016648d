"""An infinity or NaN in x reaches the determinants that H connects to it and no others, on the
tiled FP32 products (which multiply by zeros) as on the FP64 row kernel."""
import numpy as np
import pytest

import oracle
import synthetic

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec,tol", [("fp32", 1e-5), ("fp64", 1e-13)])
@pytest.mark.parametrize("n,na,nb", [
    (11, 5, 5),     # 462 strings: rows in tiles of 128 with a remainder
    (15, 2, 3),     # 105 x 455
    (14, 11, 3),    # 364 x 364, fewest beta entries
])
def test_nonfinite_entries_reach_their_neighbours_only(prec, tol, n, na, nb):
    import torch

    from paper_2506_07430_gb300 import KPM
    I = synthetic.integrals(n, na, nb, seed=2506950 + n)
    H = oracle.SlaterCondon(I.h1, I.eri, n, na, nb).csr()
    k = KPM(I.h1, I.eri, I.dipole, n, na, nb, precision=prec)
    x = torch.randn((2, k.dim), generator=torch.Generator(device="cuda").manual_seed(2),
                    device="cuda", dtype=k.vdtype)
    bad = {0: float("inf"), k.dim // 3: float("nan"), k.dim - 1: float("-inf")}
    idx = torch.tensor(list(bad), device="cuda")
    x[1, idx] = 0.0
    y0 = k.sigma(x)
    x[1, idx] = torch.tensor(list(bad.values()), device="cuda", dtype=k.vdtype)
    y = k.sigma(x)
    k.synchronize()
    assert torch.equal(y[0], y0[0])
    touched = np.zeros(k.dim, bool)
    for j in bad:
        touched[H[:, [j]].nonzero()[0]] = True
    assert 0 < touched.sum() < k.dim // 2
    got = y[1].double().cpu().numpy()
    assert np.array_equal(~np.isfinite(got), touched)
    ref = y0[1].double().cpu().numpy()
    assert np.abs(got - ref)[~touched].max() <= tol * np.abs(ref).max()
    k.close()
