"""The gradient's kernels in the coupling eigenbasis where their tiles are ragged: one to
three modes of one to six levels, several 64 x 64 tiles of H's gradient, and a mode of
seven levels (which stays in the product basis).

Reference: the library's own forward loss, central differences with Richardson
extrapolation.  Tolerance 1e-7 of the largest entry, as in test_gpu_grad: the step is
1e-3, so the extrapolated difference is off by 1e-12 of the fifth derivative and by the
loss's rounding (1e-13) over the step.
"""
import numpy as np
import pytest

import workloads as W
from test_gpu_f64_engine import model_of

pytestmark = pytest.mark.gpu

H = pytest.importorskip("paper_2601_20550_gb300.heom")


@pytest.mark.parametrize("levels,depth,K", [
    ((6,), 3, 1), ((2, 7), 2, 1), ((5, 2), 2, 2), ((1, 6, 3), 2, 1), ((2, 3, 5), 1, 2), ((4, 5, 5), 1, 1),
])
def test_grad_against_library_fd(levels, depth, K):
    model = model_of(levels, depth, K)
    grid = W.grid(0.5, 3, 3, 4, (0.0,), t_eq_fs=10.0)
    th = H.theta_of(model)
    w = np.maximum(np.abs(th), 1.0)
    rng = np.random.default_rng(len(levels) + depth)

    def spectrum(t):
        h = H.heom_build_hierarchy(H.with_theta(model, t), H.FP64)
        e = H.heom_equilibrate(h, 0.5, 10.0, 0.0)
        return H.heom_response_2d(h, e, grid)[2]

    S_ref = spectrum(th * (1 + 0.05 * rng.uniform(-1, 1, th.size)))
    h = H.heom_build_hierarchy(model, H.FP64)
    loss, g = H.heom_response_2d_grad(h, H.heom_equilibrate(h, 0.5, 10.0, 0.0), grid, S_ref, 2)

    def central(i, step):
        e = np.zeros(th.size)
        e[i] = step
        return (np.sum((spectrum(th + e) - S_ref) ** 2) - np.sum((spectrum(th - e) - S_ref) ** 2)) / (2 * step)

    top = np.max(np.abs(g * w))
    for s in range(len(levels)):
        for i in {s, 6 + s, 9 + s} | ({3} if len(levels) > 1 else set()):
            step = 1e-3 * w[i]
            fd = (4 * central(i, step / 2) - central(i, step)) / 3
            assert abs(g[i] - fd) * w[i] < 1e-7 * top, (i, g[i], fd)
