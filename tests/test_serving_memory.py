"""The server's account of device memory: what a request allocates on its path, no tables of
another path and no buffer uncounted; a request that fits the budget only without the
buffers that buy speed is served without them."""
import time

import numpy as np
import pytest

import synthetic

pytestmark = pytest.mark.gpu


def _psi(n, na, nb):
    from math import comb
    return synthetic.random_state(comb(n, na) * comb(n, nb), 11)


def _alone(I, n, na, nb, psi, prec, mask, nm):
    import torch

    from paper_2506_07430_gb300 import KPM
    k = KPM(I.h1, I.eri, I.dipole, n, na, nb, precision=prec)
    m = k.moments(torch.from_numpy(psi).cuda(), mask, 2000.0, 0.0, nm)
    k.close()
    return m


@pytest.mark.parametrize("n,na,nb,prec,budget_mb,bits", [
    # gather path: 191 MB of string tables; a dense F (662 MB) is never allocated
    (16, 1, 8, "fp32", 320, True),
    # pair-tiled path: 0.19 GB with the dense F (47 MB), which the budget does not hold
    (14, 7, 3, "fp32", 160, False),
    # 2002 x 2002: splits of three columns 98 MB, of one 33 MB
    (14, 5, 5, "mixed", 370, True),
])
def test_small_budget_is_enough(n, na, nb, prec, budget_mb, bits):
    from paper_2506_07430_gb300 import Server
    I = synthetic.integrals(n, na, nb, seed=2506940 + n)
    psi = _psi(n, na, nb)
    srv = Server(mem_budget_bytes=budget_mb << 20, max_slots=2, steps_per_round=8, precision=prec)
    r = srv.wait(srv.submit(I.h1, I.eri, I.dipole, n, na, nb, psi, 7, 2000.0, 0.0, 32, npoints=64))
    srv.close()
    ref = _alone(I, n, na, nb, psi, prec, 7, 32)
    if bits:
        assert np.array_equal(r["moments"], ref)
    else:   # FP32 sums in another order, 16 steps
        assert np.abs(r["moments"] - ref).max() <= 2e-6 * np.abs(ref).max()


@pytest.mark.parametrize("n,na,nb,prec", [
    (14, 7, 7, "mixed_bf16"), (14, 7, 7, "mixed"), (13, 7, 6, "fp32"), (12, 6, 6, "fp64"),
])
def test_estimate_covers_what_is_held(n, na, nb, prec):
    import torch

    from paper_2506_07430_gb300 import Server
    I = synthetic.integrals(n, na, nb, seed=2506940 + n)
    psi = _psi(n, na, nb)
    srv = Server(mem_budget_bytes=16 << 30, max_slots=1, steps_per_round=4, precision=prec)

    def submit(nm):
        return srv.submit(I.h1, I.eri, I.dipole, n, na, nb, psi, 7, 2000.0, 0.0, nm, npoints=64)

    srv.wait(submit(32))                        # kernels loaded, autotuned
    free0 = torch.cuda.mem_get_info()[0]
    i = submit(20000)
    t0 = time.time()
    while srv.stats()["resident"] == 0 and time.time() - t0 < 60:
        time.sleep(0.05)
    time.sleep(0.2)
    counted, used = srv.stats()["mem_used"], free0 - torch.cuda.mem_get_info()[0]
    assert srv.stats()["resident"] == 1
    srv.cancel(i)
    with pytest.raises(Exception):
        srv.wait(i)
    srv.close()
    assert used <= counted, (used, counted)
    assert counted <= used + (100 << 20), (used, counted)
