"""The FP64 engine (coupling basis, integer commutator) at the sizes where its variants
change: bases up to 48 (all steps in one launch; one block, one cluster or the whole grid
per branch), whole items in shared memory, panels of 32 columns, ragged row groups and
panels, several items per block, single-level modes.

Tolerance: 1e-12 of the largest entry after three RK4 steps, as for the other FP64 state
tests (the engine's own error is below 1e-15).
"""
import numpy as np
import pytest

import workloads as W
from oracle import heom as OH
from oracle import model as OM

pytestmark = pytest.mark.gpu

H = pytest.importorskip("paper_2601_20550_gb300.heom")


@pytest.fixture(scope="module", autouse=True)
def built():
    import os
    if not os.path.exists(H.LIB_PATH):
        import __graft_entry__
        __graft_entry__.build()


def model_of(levels, depth, K=1):
    m = W.water_model(4, depth, K_pade=K, n_prim=100)
    m["modes"] = m["modes"][:len(levels)]
    m["pairs"] = [p for p in m["pairs"] if p["s"] < len(levels) and p["t"] < len(levels)]
    for md, n in zip(m["modes"], levels):
        md["n_levels"] = n
    return m


def propagated(model, x, steps, dt=0.25):
    h = H.heom_build_hierarchy(model)
    s = H.heom_state_create(h, x.shape[0], H.FP64)
    H.heom_state_upload(s, x)
    H.heom_propagate(h, s, dt, steps)
    return H.heom_state_download(s)


@pytest.mark.parametrize("levels,depth,K,branches", [
    ((1,), 2, 1, 2), ((2,), 1, 1, 1), ((7,), 3, 1, 90), ((8,), 2, 2, 5), ((9,), 1, 1, 2),   # one mode
    ((3, 3), 2, 1, 1), ((5, 4), 3, 1, 1), ((4, 7), 2, 1, 3), ((4, 8), 1, 2, 1),            # up to d = 32
    ((5, 5), 4, 1, 160),                                                  # too much work per block for one launch
    ((3, 11), 1, 1, 2), ((3, 3, 4), 1, 1, 2), ((2, 3, 6), 1, 2, 40),      # whole items, several per block
    ((4, 4, 5), 1, 1, 1), ((3, 4, 7), 1, 1, 1), ((1, 9, 9), 1, 1, 1),     # 80, 84, 81
    ((5, 17), 1, 1, 1), ((4, 5, 5), 1, 1, 2), ((2, 8, 8), 1, 1, 1),       # panels: 85 (dense basis change), 100, 128
    ((3, 7, 8), 1, 1, 1),                                                 # 168: ragged last panel
    ((5, 7), 1, 1, 1), ((3, 4, 4), 1, 1, 1), ((3, 4, 3), 2, 1, 3), ((7, 7), 1, 1, 2),   # 33 to 48 in one launch; 49
])
def test_propagation(levels, depth, K, branches):
    model = model_of(levels, depth, K)
    prob = OM.Problem(model)
    rng = np.random.default_rng(sum(levels) + branches)
    shape = (branches, prob.nado, prob.d, prob.d)
    x = rng.standard_normal(shape) + 1j * rng.standard_normal(shape)
    x *= 10.0 ** rng.integers(-6, 3, size=(branches, prob.nado, 1, 1))     # ADOs of very different size
    got = propagated(model, x, 3)
    pick = sorted({0, branches // 2, branches - 1})
    ref = OH.propagate(prob, x[pick], 0.25, 3)
    assert np.abs(got[pick] - ref).max() < 1e-12 * np.abs(ref).max()


@pytest.mark.parametrize("levels", [(4, 4), (4, 4, 4), (4, 5, 5)])
def test_zero_and_non_finite_states(levels):
    """A zero branch stays zero; a NaN or an infinity reaches the branch that holds it (and
    its zero neighbour branches stay zero)."""
    model = model_of(levels, 1)
    d = int(np.prod(levels))
    n = OM.Problem(model).nado
    x = np.zeros((3, n, d, d), dtype=complex)
    x[1, 0, 1, 2] = np.nan
    got = propagated(model, x, 1)
    assert (got[0] == 0).all() and (got[2] == 0).all()
    assert np.isnan(got[1, 0]).any()
    x[1, 0, 1, 2] = np.inf
    assert not np.isfinite(propagated(model, x, 1)[1, 0]).all()


@pytest.mark.parametrize("scale", [1e-300, 1e-30, 1e30, 1e290])
def test_linear_in_scale(scale):
    """Scaling by powers of ten over the exponent range scales the result (down to the
    rounding of the scaling itself; 1e-300 leaves about 7 digits above the subnormals)."""
    model = model_of((4, 4, 4), 1)
    rng = np.random.default_rng(3)
    n = OM.Problem(model).nado
    x = rng.standard_normal((1, n, 64, 64)) + 1j * rng.standard_normal((1, n, 64, 64))
    a, b = propagated(model, x, 2), propagated(model, x * scale, 2)
    assert np.abs(b / scale - a).max() < (1e-6 if scale < 1e-299 else 1e-13) * np.abs(a).max()


def test_sets_of_small_and_large_bases():
    """Parameter sets on every variant in one batched call equal their own calls."""
    grid = W.grid(0.25, 2, 3, 3, (0.0, 0.5), t_eq_fs=2.0)
    for levels in (((3, 3), (4,), (3, 3, 3)), ((3, 3), (4, 4, 4), (4, 5, 5), (3, 4, 3))):
        models = [model_of(lv, 1) for lv in levels]
        hs = [H.heom_build_hierarchy(m) for m in models]
        eqs = [H.heom_equilibrate(h, 0.25, 2.0, 0.0) for h in hs]
        RI, RII, SC = H.heom_response_2d_batched(hs, eqs, grid)
        for i, m in enumerate(models):
            ri, rii, sc = H.heom_response_2d(hs[i], eqs[i], grid)
            scale = max(np.abs(ri).max(), np.abs(rii).max())
            assert np.abs(RI[i] - ri).max() <= 1e-14 * scale and np.abs(RII[i] - rii).max() <= 1e-14 * scale
            assert np.abs(SC[i] - sc).max() <= 1e-13 * np.abs(sc).max()
