"""Same-spin products whose matrices differ by many orders of magnitude: with one electron of
a spin, the off-diagonal entries of its string Hamiltonian are those of h1 alone, and h1 may
be diagonal but for rounding.  FP64 is the reference; FP16 pieces hold 22 bits, BF16 pieces
of x 16."""
import numpy as np
import pytest

import synthetic

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec,tol", [("mixed", 2e-6), ("mixed_bf16", 1e-5)])
@pytest.mark.parametrize("n,na,nb", [(8, 1, 4), (8, 4, 1), (8, 1, 1)])
@pytest.mark.parametrize("off", [1e-8, 1e-35, 1e-310])
def test_tiny_off_diagonal_h1(off, n, na, nb, prec, tol):
    import torch

    from paper_2506_07430_gb300 import KPM
    I = synthetic.integrals(n, na, nb, seed=2506870)
    h1 = np.diag(np.diag(I.h1)) + off * (1.0 - np.eye(n))
    k = KPM(h1, I.eri, I.dipole, n, na, nb, precision=prec)
    ref = KPM(h1, I.eri, I.dipole, n, na, nb, precision="fp64")
    g = torch.Generator(device="cuda").manual_seed(8)
    x = torch.randn((1, k.dim), generator=g, device="cuda")
    y, z = k.sigma(x), ref.sigma(x.double())
    k.synchronize()
    ref.synchronize()
    assert torch.isfinite(y).all()
    assert ((y.double() - z).norm() / z.norm()).item() < tol
    k.close()
    ref.close()
