"""H applied to vectors that start one element past a 16-byte boundary: rows of even length,
whose wider loads need the boundary, give the bits of the same vectors on it."""
import pytest

import synthetic

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", ["fp64", "fp32", "mixed", "mixed_bf16"])
@pytest.mark.parametrize("n,na,nb", [
    (12, 3, 5),     # 220 x 792 strings: tiled FP32 products, rows a multiple of 16 bytes
    (10, 5, 5),     # 252 x 252
    (9, 4, 2),      # 126 x 36
])
def test_sigma_of_offset_vectors(prec, n, na, nb):
    import torch

    from paper_2506_07430_gb300 import KPM
    I = synthetic.integrals(n, na, nb, seed=2506960 + n)
    k = KPM(I.h1, I.eri, I.dipole, n, na, nb, precision=prec)
    x = torch.randn((3, k.dim), generator=torch.Generator(device="cuda").manual_seed(3),
                    device="cuda", dtype=k.vdtype)
    ref = k.sigma(x)
    assert x.data_ptr() % 16 == 0
    for shift in (1, 2, 3):
        xb, yb = (torch.empty(3 * k.dim + 8, dtype=k.vdtype, device="cuda") for _ in range(2))
        xs, ys = (t[shift:shift + 3 * k.dim].view(3, k.dim) for t in (xb, yb))
        xs.copy_(x)
        assert torch.equal(k.sigma(xs, ys), ref), shift
    k.synchronize()
    k.close()
