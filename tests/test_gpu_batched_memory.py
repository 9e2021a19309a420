"""Device buffers of a batched FP64 response: per set a trunk, two scratch states and the
branch sets, nothing more (a call that fills the device has no room for another state).
Counted with the library's allocation injection: the fewest allocations with which the call
succeeds, for a set named twice and three times."""
import pytest

import workloads as W
from test_gpu_f64_engine import model_of

pytestmark = pytest.mark.gpu

H = pytest.importorskip("paper_2601_20550_gb300.heom")


@pytest.mark.parametrize("levels", [(3, 3), (4, 4, 4), (4, 5, 5)])
def test_buffers_per_set(levels):
    h = H.heom_build_hierarchy(model_of(levels, 1))
    eq = H.heom_equilibrate(h, 0.25, 1.0, 0.0)
    grid = W.grid(0.25, 1, 2, 2, (0.0,))

    def works(n_sets, after):
        H.heom_debug_fail_alloc(after)
        try:
            H.heom_response_2d_batched([h] * n_sets, [eq] * n_sets, grid)
            return True
        except H.HeomError as e:
            assert e.status == -2, str(e)
            return False
        finally:
            H.heom_debug_fail_alloc(-1)

    def fewest(n_sets):
        return next(k for k in range(200) if works(n_sets, k))

    # T, ta, tb, three branch sets and a placeholder for the fourth
    assert fewest(3) - fewest(2) == 7
