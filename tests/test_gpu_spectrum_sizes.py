"""kpm_spectrum at the sizes where the reconstruction changes what it does: moments fold
onto the nodes (N > M: images 2M - m, 2M + m, 4M - m, ...), nodes pair with their mirror
images (odd and even M, one node), fewer moments than the 32 lanes of a warp, and sums at
the rounded nodes beyond N M = 2^24.

Against the oracle's direct cosine sums.  Exact nodes: 1e-10 relative L2, as in the parity
tests.  Rounded nodes: T_n turns a node's rounding (2^-53) into n / sin(theta) times that;
N M 2^-53 bounds its relative L2 over the nodes, times 4 for both sides' own rounding.
"""
import numpy as np
import pytest

from oracle import kpm as okpm

pytestmark = pytest.mark.gpu

SIZES = [(1, 1), (5, 1), (31, 2), (32, 64), (33, 65), (64, 64), (65, 64), (127, 64), (128, 64),
         (129, 64), (257, 64), (1000, 7), (513, 514), (2049, 513), (8192, 2048), (8193, 2048),
         (70000, 241)]


@pytest.mark.parametrize("N,M", SIZES)
@pytest.mark.parametrize("kernel", ["none", "jackson"])
def test_spectrum_sizes(N, M, kernel):
    from paper_2506_07430_gb300 import spectrum
    rng = np.random.default_rng(N * 31 + M)
    mu = np.cos(np.arange(N) * 1.1) * np.exp(-np.arange(N) / 700.0) + 1e-3 * rng.standard_normal(N)
    om, it = spectrum(mu, 2.5, -1.0, M, kernel=kernel)
    om_r, it_r = okpm.spectrum(mu, 2.5, -1.0, M, kernel=kernel)
    tol = 1e-10 if N * M <= 2 ** 24 else max(1e-10, 4.0 * N * M * 2.0 ** -53)
    assert np.abs(om - om_r).max() <= 1e-13
    assert np.linalg.norm(it - it_r) <= tol * np.linalg.norm(it_r)


def test_spectrum_passes_on_a_moment_that_is_not_finite():
    """Also one whose Chebyshev polynomial vanishes at every node (n = M, 3M)."""
    from paper_2506_07430_gb300 import spectrum
    for bad in (3, 16, 48, 49):
        mu = np.ones(50)
        mu[bad] = np.nan
        assert not np.isfinite(spectrum(mu, 1.0, 0.0, 16, kernel="none")[1]).any()
