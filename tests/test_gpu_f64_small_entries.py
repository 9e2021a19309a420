"""Accuracy of FP64 results entry by entry.

Kicks of product-basis states: every entry of K w - w K within the rounding of its own
products, (2 d + 2) 2^-53 times the sum of their magnitudes, on states whose entries span
thirty decades as populations and coherences do.  (Relative to the largest entry, the small
ones could be lost altogether.)

Kicks inside a response, in the coupling basis: a response of no propagation is three kicks
and a trace.  Each kick of matrices of norm |mu| is good to about d 2^-53 of |mu| |w|."""
import numpy as np
import pytest

import workloads as W
from test_gpu_f64_engine import model_of

pytestmark = pytest.mark.gpu

H = pytest.importorskip("paper_2601_20550_gb300.heom")

EPS = 2.0 ** -53


def graded(rng, shape, levels):
    """Random entries times 10^(-1.5 (excitation of row + of column))."""
    N = np.indices(levels).reshape(len(levels), -1).sum(0)
    x = rng.standard_normal(shape) + 1j * rng.standard_normal(shape)
    return x * 10.0 ** (-1.5 * (N[:, None] + N[None, :]))


def matrices(h):
    ops = H.heom_get_operators(h)
    return ops["mu"], ops["mu_plus"], ops["mu_plus"].T


@pytest.mark.parametrize("levels", [(5, 7), (5, 8), (4, 4, 4), (4, 5, 5)])
@pytest.mark.parametrize("which", [0, 1, 2])
@pytest.mark.parametrize("device", [False, True])
def test_kick_of_small_entries(levels, which, device):
    h = H.heom_build_hierarchy(model_of(levels, 1))
    rng = np.random.default_rng(sum(levels) + which)
    x = graded(rng, (2, h.n_ado, h.d, h.d), levels)
    K = matrices(h)[which]
    if device:
        torch = pytest.importorskip("torch")
        xin = torch.from_numpy(x).cuda()
        out = torch.empty_like(xin)
        H.heom_kick_dev(h, xin.data_ptr(), out.data_ptr(), 2, H.FP64, which, torch.cuda.current_stream().cuda_stream)
        got = out.cpu().numpy()
    else:
        s = H.heom_state_create(h, 2, H.FP64)
        H.heom_state_upload(s, x)
        H.heom_kick(h, s, which)
        got = H.heom_state_download(s)
    xl, Kl = x.astype(np.clongdouble), K.astype(np.longdouble)
    ref = Kl @ xl - xl @ Kl
    for part in ("real", "imag"):
        size = np.abs(K) @ np.abs(getattr(x, part)) + np.abs(getattr(x, part)) @ np.abs(K)
        err = np.abs(getattr(got, part) - getattr(ref, part))
        assert (err <= (2 * h.d + 2) * EPS * size).all(), part


@pytest.mark.parametrize("levels", [(5, 7), (3, 13), (5, 8), (3, 3, 5), (4, 4, 4), (4, 5, 5)])
def test_kicks_inside_a_response(levels):
    h = H.heom_build_hierarchy(model_of(levels, 1))
    rng = np.random.default_rng(sum(levels))
    x = rng.standard_normal((1, h.n_ado, h.d, h.d)) + 1j * rng.standard_normal((1, h.n_ado, h.d, h.d))
    x = x + x.conj().transpose(0, 1, 3, 2)
    eq = H.heom_state_create(h, 1, H.FP64)
    H.heom_state_upload(eq, x)
    RI, RII, _ = H.heom_response_2d(h, eq, W.grid(0.25, 1, 1, 1, (0.0,)))
    mu, mp, mm = (m.astype(np.longdouble) for m in matrices(h))
    kick = lambda K, r: K @ r - r @ K   # noqa: E731
    r = x[0, 0].astype(np.clongdouble)
    norm = np.linalg.norm(x[0, 0]) * np.linalg.norm(np.asarray(mu, float), 2) ** 4
    for R, order in ((RI, (mm, mp, mp)), (RII, (mp, mm, mp))):
        ref = -1j * np.trace(mu @ kick(order[2], kick(order[1], kick(order[0], r))))
        assert abs(R[0, 0, 0] - complex(ref)) <= 32 * h.d * EPS * norm
