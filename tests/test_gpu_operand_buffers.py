"""The tensor-core sigma's operand buffers: as large as the widest block of columns asked for,
not larger; grown without touching what a captured graph holds."""
import numpy as np
import pytest

import synthetic

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec,pieces", [("mixed", 8), ("mixed_bf16", 12)])
def test_one_column_holds_one_column_of_splits(prec, pieces):
    import torch

    from paper_2506_07430_gb300 import KPM
    n, na, nb = 14, 5, 5                     # 2002 x 2002 determinants: 32 MB of FP16 splits
    I = synthetic.integrals(n, na, nb, seed=2506880)
    k = KPM(I.h1, I.eri, I.dipole, n, na, nb, precision=prec)       # autotuned, kernels loaded
    x = torch.ones((3, k.dim), device="cuda")
    y = torch.empty_like(x)
    assert torch.equal(x[0], x[1])
    k.close()
    free0 = torch.cuda.mem_get_info()[0]
    k = KPM(I.h1, I.eri, I.dipole, n, na, nb, precision=prec)
    free1 = torch.cuda.mem_get_info()[0]
    k.sigma(x[0], y[0])
    k.synchronize()
    one = free1 - torch.cuda.mem_get_info()[0]
    # per determinant: `pieces` bytes (rows of x padded to 2048), and 4 MB for row scales
    # and the 2 MB pages of up to eight buffers
    assert one <= pieces * 2002 * 2048 + (20 << 20), one
    k.sigma(x, y)
    k.synchronize()
    three = free1 - torch.cuda.mem_get_info()[0]
    assert three <= 3 * pieces * 2002 * 2048 + (20 << 20), three
    assert torch.equal(y[0], y[1]) and torch.equal(y[0], y[2])
    k.close()
    assert torch.cuda.mem_get_info()[0] >= free0 - (4 << 20)


@pytest.mark.parametrize("prec", ["mixed", "mixed_bf16"])
@pytest.mark.parametrize("n,na,nb", [(7, 3, 3), (9, 4, 5)])
def test_growth_leaves_captured_steps_alone(prec, n, na, nb):
    import torch

    from paper_2506_07430_gb300 import KPM
    I = synthetic.integrals(n, na, nb, seed=2506880 + n)
    res = []
    for wide in (False, True):
        k = KPM(I.h1, I.eri, I.dipole, n, na, nb, precision=prec)
        g = torch.Generator(device="cuda").manual_seed(9)
        x = torch.randn((3, k.dim), generator=g, device="cuda")
        psi = torch.from_numpy(synthetic.random_state(k.dim, 5)).cuda()
        k.recursion_begin(psi, 2, 2000.0, 0.0, 2 * 41)
        k.recursion_advance(20)                      # replayed steps of one column
        if wide:
            one = torch.stack([k.sigma(x[c].clone()) for c in range(3)])
            junk = []
            for ncol in (2, 3):                      # buffers grow
                assert torch.equal(k.sigma(x[:ncol].clone()), one[:ncol])
                junk.append(torch.full((3, 4 * k.dim), float("nan"), device="cuda"))
        k.recursion_advance(20)                      # the steps captured before
        res.append(k.recursion_moments())
        k.close()
    assert np.isfinite(res[0]).all()
    assert np.array_equal(res[0], res[1])


def test_wider_block_inside_a_capture():
    # the buffers hold one column when the capture begins: the block goes column by column
    import torch

    from paper_2506_07430_gb300 import KPM
    n, na, nb = 7, 3, 3
    I = synthetic.integrals(n, na, nb, seed=2506890)
    st = torch.cuda.Stream()
    with torch.cuda.stream(st):
        k = KPM(I.h1, I.eri, I.dipole, n, na, nb, precision="mixed", stream=st)
        g = torch.Generator(device="cuda").manual_seed(10)
        x = torch.randn((3, k.dim), generator=g, device="cuda")
        y = torch.zeros_like(x)
        one = torch.stack([k.sigma(x[c].clone()) for c in range(3)])
        st.synchronize()
        graph = torch.cuda.CUDAGraph()
        graph.capture_begin()
        k.sigma(x, y)
        graph.capture_end()
        assert torch.equal(k.sigma(x.clone()), one)          # grows
        graph.replay()
        st.synchronize()
        assert torch.equal(y, one)
        k.close()
