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


@pytest.mark.parametrize("prec,tol", [
    ("mixed", 2e-6),         # two FP16 pieces: 22 bits of x
    ("mixed_bf16", 1e-5),    # two BF16 pieces: 2^-17 of each entry of x at most
])
@pytest.mark.parametrize("n,na,nb", [
    (12, 2, 4),     # 66 x 495 strings: a second row of 64 x 64 tiles with two rows, odd pitch
    (11, 2, 11),    # 55 x 1: one column
    (11, 11, 2),    # 1 x 55: one row
    (16, 2, 1),     # 120 x 16
    (8, 4, 3),      # 70 x 56
])
def test_split_copies_at_tile_edges(prec, tol, n, na, nb):
    import torch

    from paper_2506_07430_gb300 import KPM
    I = synthetic.integrals(n, na, nb, seed=2506840 + n)
    k = KPM(I.h1, I.eri, I.dipole, n, na, nb, precision=prec)
    ref = KPM(I.h1, I.eri, I.dipole, n, na, nb, precision="fp64")
    g = torch.Generator(device="cuda").manual_seed(7)
    x = torch.randn((2, k.dim), generator=g, device="cuda")
    y, z = k.sigma(x), ref.sigma(x.double())
    k.synchronize()
    ref.synchronize()
    for c in range(2):
        assert ((y[c].double() - z[c]).norm() / z[c].norm()).item() < tol, c
    k.close()
    ref.close()
