"""The 2D Fourier sums as two one-dimensional sums against the double sum of the oracle.

Tolerance: each bin is a sum of n1 + n3 rounded terms per axis; 1e-13 of the largest bin
leaves three orders of magnitude over 2^-53 sqrt(2 * 130).
"""
import numpy as np
import pytest

from oracle import heom as OH

pytestmark = pytest.mark.gpu

H = pytest.importorskip("paper_2601_20550_gb300.heom")


@pytest.fixture(scope="module", autouse=True)
def built():
    import os
    if not os.path.exists(H.LIB_PATH):
        import __graft_entry__
        __graft_entry__.build()


@pytest.mark.parametrize("n1,n3,n_t2", [(1, 1, 1), (1, 5, 2), (7, 1, 1), (2, 3, 1), (5, 129, 1), (130, 4, 2), (17, 16, 3)])
def test_fourier_sums(n1, n3, n_t2):
    rng = np.random.default_rng(n1 * 1000 + n3)
    RI, RII = (rng.standard_normal((n_t2, n1, n3)) + 1j * rng.standard_normal((n_t2, n1, n3)) for _ in range(2))
    got = H.heom_spectrum_2d(RI, RII, 4.0)
    ref, _, _ = OH.correlation_spectrum(RI, RII, 4.0)
    assert np.abs(got - ref).max() < 1e-13 * np.abs(ref).max()
