"""FP32 stages and kicks in 64 x 64 register tiles: ragged tiles, and the same bits as the
32 x 32 tiles that a launch with few items takes.

Tolerance of the kicks: 2 d rounded products and additions of 2^-24, of random sign, so
4 sqrt(2 d) 2^-24 = 4e-6 of the largest at d = 130, and the two basis changes' 2^-24.
"""
import numpy as np
import pytest

import workloads as W
from oracle import heom as OH
from oracle import model as OM
from test_gpu_f64_engine import model_of

pytestmark = pytest.mark.gpu

H = pytest.importorskip("paper_2601_20550_gb300.heom")


def state(prob, branches, seed):
    rng = np.random.default_rng(seed)
    shape = (branches, prob.nado, prob.d, prob.d)
    return rng.standard_normal(shape) + 1j * rng.standard_normal(shape)


def propagated(h, x, steps=3):
    s = H.heom_state_create(h, x.shape[0], H.FP32)
    H.heom_state_upload(s, x)
    H.heom_propagate(h, s, 0.25, steps)
    return H.heom_state_download(s)


@pytest.mark.parametrize("levels,depth,branches", [
    ((5, 7), 1, 60), ((6, 6), 1, 60), ((3, 13), 2, 40), ((4, 4, 4), 2, 8), ((5, 13), 1, 20), ((4, 4, 5), 1, 12),
    ((4, 5, 5), 1, 8), ((5, 5, 5), 1, 8), ((2, 8, 8), 1, 8), ((3, 6, 8), 1, 5),
])
def test_stage_bits_do_not_depend_on_the_tiles(levels, depth, branches):
    model = model_of(levels, depth)
    prob = OM.Problem(model)
    x = state(prob, branches, sum(levels))
    h = H.heom_build_hierarchy(model, H.FP32)
    got = propagated(h, x)
    assert np.array_equal(got[-1:], propagated(h, x[-1:]))
    assert np.array_equal(got[:1], propagated(h, x[:1]))
    ref = OH.propagate(prob, x[:1], 0.25, 3)
    assert np.abs(got[:1] - ref).max() < 2e-5 * np.abs(ref).max()


@pytest.mark.parametrize("levels", [(3, 13), (5, 8), (4, 4, 4), (5, 13), (4, 4, 5), (5, 5, 5), (2, 8, 8)])
@pytest.mark.parametrize("which", [0, 1, 2])
def test_kick(levels, which):
    model = model_of(levels, 1)
    prob = OM.Problem(model)
    x = state(prob, 2, sum(levels))
    h = H.heom_build_hierarchy(model, H.FP32)
    s = H.heom_state_create(h, 2, H.FP32)
    H.heom_state_upload(s, x)
    H.heom_kick(h, s, which)
    ops = H.heom_get_operators(h)
    ref = OH.kick(x, (ops["mu"], ops["mu_plus"], ops["mu_plus"].T)[which])
    assert np.abs(H.heom_state_download(s) - ref).max() < 5e-6 * np.abs(ref).max()


def test_response_with_tiled_kicks():
    model = model_of((5, 8), 1)
    grid = W.grid(0.5, 3, 4, 4, (0.0, 1.0), t_eq_fs=5.0)
    _, _, RI, RII, _ = H.spectrum_2d(model, grid, H.FP32)
    _, RIo, RIIo, _ = OH.spectrum_2d(OM.Problem(model), grid)
    scale = max(np.abs(RIo).max(), np.abs(RIIo).max())
    assert np.abs(RI - RIo).max() < 2e-5 * scale
    assert np.abs(RII - RIIo).max() < 2e-5 * scale
