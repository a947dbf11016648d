"""A context whose row-kernel tables do not fit in the device's free memory is made without
them: its sigma runs in the gather kernel, which needs none."""
import pytest

import synthetic

pytestmark = pytest.mark.gpu


def test_fp32_without_room_for_dense_string_hamiltonian():
    import torch

    from paper_2506_07430_gb300 import KPM
    n, na, nb = 17, 7, 3          # 19448 x 680 strings: dense F_a 1.5 GB, the rest 0.5 GB
    I = synthetic.integrals(n, na, nb, seed=2506930)
    k = KPM(I.h1, I.eri, I.dipole, n, na, nb, precision="fp32")
    x = torch.randn((1, k.dim), generator=torch.Generator(device="cuda").manual_seed(1),
                    device="cuda")
    y, z = k.sigma(x), torch.empty_like(x)
    k.synchronize()
    k.close()
    torch.cuda.empty_cache()
    hog = torch.empty(torch.cuda.mem_get_info()[0] - (1200 << 20), dtype=torch.uint8,
                      device="cuda")
    try:
        k = KPM(I.h1, I.eri, I.dipole, n, na, nb, precision="fp32")
        k.sigma(x, z)
        k.synchronize()
        k.close()
    finally:
        del hog
        torch.cuda.empty_cache()
    # FP32 sums in another order: 240 * 42 terms of either sign
    assert ((y - z).norm() / y.norm()).item() < 1e-6
