"""Blocks of columns on the tensor-core sigma: columns that share a set of launches give the
bits that each gives alone (counts around the three that one launch takes, column sizes
that are not multiples of the tiles, columns of very different magnitude)."""
import pytest

import synthetic

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", ["mixed", "mixed_bf16"])
@pytest.mark.parametrize("n,na,nb", [(4, 1, 2), (7, 0, 3), (9, 4, 5), (11, 6, 5)])
def test_block_columns_equal_single(prec, n, na, nb):
    import torch

    from paper_2506_07430_gb300 import KPM
    I = synthetic.integrals(n, na, nb, seed=2506820 + n)
    k = KPM(I.h1, I.eri, I.dipole, n, na, nb, precision=prec)
    g = torch.Generator(device="cuda").manual_seed(5)
    x = torch.randn((7, k.dim), generator=g, device="cuda")
    x *= torch.tensor([1.0, 1e-6, 1e5, 0.0, 3.0, 1e-20, 7.0], device="cuda")[:, None]
    one = torch.stack([k.sigma(x[c].clone()) for c in range(7)])
    for ncol in (1, 2, 3, 4, 6, 7):
        assert torch.equal(k.sigma(x[:ncol].clone()), one[:ncol]), ncol
    k.synchronize()
    k.close()
