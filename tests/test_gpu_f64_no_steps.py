"""FP64 states that no step has changed come back as they are, bit for bit: zero steps, an
equilibration of no length, a steady state whose start already meets the tolerance."""
import numpy as np
import pytest

from test_gpu_f64_engine import model_of

pytestmark = pytest.mark.gpu

H = pytest.importorskip("paper_2601_20550_gb300.heom")


@pytest.mark.parametrize("levels", [(6,), (3, 3), (9,), (3, 3, 4), (4, 4, 4), (4, 5, 5)])
def test_no_steps(levels):
    h = H.heom_build_hierarchy(model_of(levels, 1))
    ground = np.zeros((1, h.n_ado, h.d, h.d), dtype=complex)
    ground[0, 0, 0, 0] = 1.0
    for tol in (0.0, 1e-9):
        assert np.array_equal(H.heom_state_download(H.heom_equilibrate(h, 0.25, 0.0, tol)), ground)
    s, its = H.heom_steady_state(h, tol=1e6)[:2]
    assert its == 0 and np.array_equal(H.heom_state_download(s), ground)
    rng = np.random.default_rng(1)
    x = rng.standard_normal(ground.shape) + 1j * rng.standard_normal(ground.shape)
    s = H.heom_state_create(h, 1, H.FP64)
    H.heom_state_upload(s, x)
    H.heom_propagate(h, s, 0.25, 0)
    assert np.array_equal(H.heom_state_download(s), x)
