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


@pytest.mark.parametrize("n,na,nb", [
    (12, 6, 6),     # one column: GEMM tiles of 64 columns; three: 256
    (13, 5, 5),     # one: 128; three: 256
    (12, 9, 2),     # 66 beta strings: one row tile pair of mostly padding; 64 for any count
    (10, 8, 1),     # 45 alpha strings: one column tile with a remainder
])
def test_gemm_tile_widths_same_bits(n, na, nb):
    # a tile's width leaves the order of its sums alone, so a block of three columns and its
    # columns alone agree in every bit whichever widths their grids take
    import torch

    from paper_2506_07430_gb300 import KPM
    I = synthetic.integrals(n, na, nb, seed=2506830 + n)
    k = KPM(I.h1, I.eri, I.dipole, n, na, nb, precision="mixed")
    g = torch.Generator(device="cuda").manual_seed(6)
    x = torch.randn((3, k.dim), generator=g, device="cuda")
    one = torch.stack([k.sigma(x[c].clone()) for c in range(3)])
    assert torch.equal(k.sigma(x.clone()), one)
    k.synchronize()
    k.close()
    # and with the FP64 sigma: FP16 pieces of 22 bits, FP32 sums of at most 3000 terms
    ref = KPM(I.h1, I.eri, I.dipole, n, na, nb, precision="fp64")
    y = ref.sigma(x[:1].double())
    ref.synchronize()
    assert ((one[:1].double() - y).norm() / y.norm()).item() < 2e-6
    ref.close()
