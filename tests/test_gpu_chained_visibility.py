"""Steps whose kernels start while their predecessor runs give the bits of the same steps
with every launch waited for on the host (CUDA_LAUNCH_BLOCKING=1, a process of its own).
Row lengths and dimensions are odd, so that neighbouring rows, columns and reduction blocks
share 32-byte sectors, and a column has several reduction blocks.
"""
import os
import subprocess
import sys

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

# norb, alpha and beta electrons, precision, mask of dipole components
CASES = [(n, na, nb, prec, mask) for n, na, nb in [(7, 3, 3), (15, 2, 3)]
         for prec in ("fp64", "fp32", "mixed", "mixed_bf16") for mask in (2, 7)]

CHILD = """
import sys
import numpy as np, torch
sys.path.insert(0, {root!r})
import synthetic
from paper_2506_07430_gb300 import KPM
out = {{}}
for i, (n, na, nb, prec, mask) in enumerate({cases!r}):
    I = synthetic.integrals(n, na, nb, seed=2506860 + n)
    k = KPM(I.h1, I.eri, I.dipole, n, na, nb, precision=prec)
    psi = torch.from_numpy(synthetic.random_state(k.dim, 5)).cuda()
    k.graphs_enable(False)
    k.recursion_begin(psi, mask, 2000.0, 0.0, 2 * 40)
    k.recursion_advance(39)
    out[str(i)] = k.recursion_moments()
    k.close()
np.savez({path!r}, **out)
"""


def test_chained_launches_equal_blocking_launches(tmp_path):
    res = []
    for blocking in ("0", "1"):
        path = str(tmp_path / f"m{blocking}.npz")
        env = dict(os.environ, CUDA_LAUNCH_BLOCKING=blocking)
        r = subprocess.run([sys.executable, "-c", CHILD.format(root=ROOT, cases=CASES, path=path)],
                           env=env, capture_output=True, text=True, timeout=300)
        assert r.returncode == 0, r.stderr[-2000:]
        res.append(np.load(path))
    for i, case in enumerate(CASES):
        a, b = res[0][str(i)], res[1][str(i)]
        assert np.isfinite(a).all(), case
        assert np.array_equal(a, b), case
