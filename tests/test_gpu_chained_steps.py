"""Recursion steps whose kernels start before their predecessor has ended give the bits of the
same steps with the device idle between any two: a kernel that read or wrote too early would
not.  One CTA per row, so from less than one wave (8 orbitals) to several (10, three columns).
"""
import numpy as np
import pytest

import synthetic

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,na,nb,mask", [
    (2, 1, 1, 1), (5, 0, 3, 7), (6, 3, 2, 5), (8, 4, 4, 1), (9, 4, 5, 7), (10, 5, 5, 7),
])
def test_chained_steps_same_bits(n, na, nb, mask):
    import torch

    from paper_2506_07430_gb300 import KPM, recursion_advance_batch
    I = synthetic.integrals(n, na, nb, seed=2506840 + n)
    out = []
    for way in ("idle between", "graphs", "direct", "batch"):
        k = KPM(I.h1, I.eri, I.dipole, n, na, nb, precision="fp64")
        psi = torch.from_numpy(synthetic.random_state(k.dim, 5)).cuda()
        k.graphs_enable(way == "graphs")
        k.recursion_begin(psi, mask, 200.0, 0.0, 2 * 62)
        if way == "idle between":
            for _ in range(61):
                k.recursion_advance(1)
                k.synchronize()
        elif way == "batch":
            recursion_advance_batch([k], 61)
        else:
            k.recursion_advance(61)
        out.append(k.recursion_moments())
        k.close()
    assert np.isfinite(out[0]).all()
    for o in out[1:]:
        assert np.array_equal(out[0], o)
