"""FP64 dipole kicks at the sizes of their two kernels (d = 40 and above: 32 x 32 tiles of
integer products), ragged tiles, extreme scales and non-finite entries.

Tolerance: 1e-13 of the largest entry, as for the kicks in test_gpu_parity; both factors
are rounded to 2^-54 of their slice's largest, a sum has at most 2 d = 200 products.  The
matrices are the library's own (at 23 levels its eigensolver and the oracle's differ by
1e-13, more than the kick is allowed).
"""
import numpy as np
import pytest

import workloads as W
from oracle import heom as OH
from oracle import model as OM
from test_gpu_f64_engine import model_of

pytestmark = pytest.mark.gpu

H = pytest.importorskip("paper_2601_20550_gb300.heom")


def kicked(model, x, which):
    """The state after the kick, and the matrix that it was kicked with."""
    h = H.heom_build_hierarchy(model)
    s = H.heom_state_create(h, x.shape[0], H.FP64)
    H.heom_state_upload(s, x)
    H.heom_kick(h, s, which)
    ops = H.heom_get_operators(h)
    return H.heom_state_download(s), (ops["mu"], ops["mu_plus"], ops["mu_plus"].T)[which]


@pytest.mark.parametrize("levels", [(23,), (4, 6), (5, 5), (4, 8), (3, 11), (3, 13), (5, 8), (3, 3, 5), (4, 4, 4), (4, 5, 5)])
@pytest.mark.parametrize("which,scale", [(0, 1.0), (1, 1e-290), (2, 1e290)])
def test_kick(levels, which, scale):
    model = model_of(levels, 1)
    prob = OM.Problem(model)
    rng = np.random.default_rng(sum(levels))
    shape = (2, prob.nado, prob.d, prob.d)
    x = rng.standard_normal(shape) + 1j * rng.standard_normal(shape)
    got, K = kicked(model, x * scale, which)
    got = got / scale
    ref = OH.kick(x, K)
    assert np.abs(got - ref).max() < 1e-13 * np.abs(ref).max()


@pytest.mark.parametrize("levels", [(5, 7), (6, 8)])
def test_kick_keeps_non_finite_entries_apart(levels):
    model = model_of(levels, 1)
    prob = OM.Problem(model)
    rng = np.random.default_rng(3)
    shape = (1, prob.nado, prob.d, prob.d)
    x = rng.standard_normal(shape) + 1j * rng.standard_normal(shape)
    y = x.copy()
    x[0, 0, 4, 33] = np.inf
    x[0, 1, 20, 2] = np.nan
    got, K = kicked(model, x, 1)
    ref = OH.kick(y, K)
    bad = np.zeros(shape, bool)
    bad[0, 0, :, 33] = bad[0, 0, 4, :] = bad[0, 1, :, 2] = bad[0, 1, 20, :] = True
    assert not np.isfinite(got[bad]).any()
    assert np.abs((got - ref)[~bad]).max() < 1e-13 * np.abs(ref).max()


@pytest.mark.parametrize("levels", [(5, 6), (5, 8)])
def test_response_with_tiled_kicks(levels):
    model = model_of(levels, 1)
    grid = W.grid(0.5, 3, 4, 4, (0.0, 1.0), t_eq_fs=5.0)
    _, _, RI, RII, SC = H.spectrum_2d(model, grid, H.FP64)
    _, RIo, RIIo, SCo = OH.spectrum_2d(OM.Problem(model), grid)
    scale = max(np.abs(RIo).max(), np.abs(RIIo).max())
    assert np.abs(RI - RIo).max() < 1e-10 * scale
    assert np.abs(RII - RIIo).max() < 1e-10 * scale
    assert np.abs(SC - SCo).max() < 1e-10 * np.abs(SCo).max()
