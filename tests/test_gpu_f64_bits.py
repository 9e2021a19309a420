"""FP64 results of a branch are its own: the same bits alone, anywhere in a batch of any
size, in any row block, and in a call with other parameter sets.  Bases and batches are
chosen so that each basis runs through every kernel that takes it: all steps in one launch
(block, cluster, grid), whole items, panels with the items' arithmetic, panels."""
import numpy as np
import pytest

import workloads as W
from test_gpu_f64_engine import model_of, propagated

pytestmark = pytest.mark.gpu

H = pytest.importorskip("paper_2601_20550_gb300.heom")


@pytest.mark.parametrize("levels,depth,batches", [
    ((6,), 6, (1, 5, 128, 500)), ((4, 4), 2, (1, 12, 300)),             # one launch: cluster, grid, block
    ((5, 5), 4, (1, 160)), ((3, 3, 3), 1, (1, 400)),                    # and whole items, several per block
    ((3, 3, 4), 1, (1, 30, 200)), ((3, 3, 5), 1, (1, 24, 200)),         # and panels of items, d = 36, 45
    ((4, 4, 3), 1, (1, 24, 200)), ((4, 3, 4), 1, (1, 24, 200)),         # d = 48
    ((4, 4, 4), 1, (1, 20, 100)), ((3, 5, 5), 1, (1, 20, 100)), ((4, 3, 6), 1, (1, 20, 100)),   # d = 64, 75, 72
    ((4, 5, 5), 1, (1, 2, 9)), ((5, 5, 6), 1, (1, 3)), ((5, 17), 1, (1, 7)),                    # panels: d = 100, 150, 85
])
def test_branches_alone_and_in_batches(levels, depth, batches):
    model = model_of(levels, depth)
    h = H.heom_build_hierarchy(model)
    rng = np.random.default_rng(sum(levels) * depth)
    one = rng.standard_normal((1, h.n_ado, h.d, h.d)) + 1j * rng.standard_normal((1, h.n_ado, h.d, h.d))
    one *= 10.0 ** rng.integers(-6, 3, size=(1, h.n_ado, 1, 1))
    ref = propagated(model, one, 2)
    assert np.isfinite(ref).all() and (ref != one).any()
    for B in batches:
        x = rng.standard_normal((B,) + one.shape[1:]) + 0j
        at = sorted({0, B // 3, B // 2, B - 1})
        x[at] = one[0]
        got = propagated(model, x, 2)
        for i in at:
            assert np.array_equal(got[i], ref[0]), (B, i)


@pytest.mark.parametrize("levels,n1,rows", [((4, 4), 12, 5), ((3, 3, 4), 9, 1), ((4, 4, 4), 9, 1), ((4, 5, 5), 5, 2)])
def test_row_blocks(levels, n1, rows):
    """Row blocks of a response against the whole one (batches of 2 rows and 2 n1 branches)."""
    h = H.heom_build_hierarchy(model_of(levels, 1))
    eq = H.heom_equilibrate(h, 0.25, 1.0, 0.0)
    grid = W.grid(0.25, 2, n1, 3, (0.0, 0.5))
    RI, RII, _ = H.heom_response_2d(h, eq, grid)
    for j in (0, n1 - rows):
        ri, rii = H.heom_response_2d_rows(h, eq, grid, j, j + rows)
        assert np.array_equal(ri, RI[:, j:j + rows]) and np.array_equal(rii, RII[:, j:j + rows])


@pytest.mark.parametrize("sets", [((3, 3), (4,), (3, 3, 3)), ((3, 3), (4, 4, 4), (4, 5, 5), (3, 4, 3)),
                                  ((4, 4, 4), (3, 3, 5), (3, 5, 5))])
def test_sets_equal_their_own_calls(sets):
    grid = W.grid(0.25, 2, 3, 3, (0.0, 0.5))
    hs = [H.heom_build_hierarchy(model_of(lv, 1)) for lv in sets]
    eqs = [H.heom_equilibrate(h, 0.25, 2.0, 0.0) for h in hs]
    RI, RII, SC = H.heom_response_2d_batched(hs, eqs, grid)
    for i, h in enumerate(hs):
        ri, rii, sc = H.heom_response_2d(h, eqs[i], grid)
        assert np.array_equal(RI[i], ri) and np.array_equal(RII[i], rii) and np.array_equal(SC[i], sc), sets[i]
