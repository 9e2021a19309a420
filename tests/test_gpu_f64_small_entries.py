"""Accuracy of FP64 results entry by entry.

Kicks of product-basis states: every entry of K w - w K within the rounding of its own
products, (2 d + 2) 2^-53 times the sum of their magnitudes, on states whose entries span
thirty decades as populations and coherences do.  (Relative to the largest entry, the small
ones could be lost altogether.)

Kicks inside a response, in the coupling basis: a response of no propagation is three kicks
and a trace.  Each kick of matrices of norm |mu| is good to about d 2^-53 of |mu| |w|.

Propagation: each ADO to a few dozen 2^-53 of its own size and of what its neighbours bring
(norms propagated with the same steps), however much larger other ADOs are; the entries of
one ADO are not accurate beyond 2^-53 of its largest."""
import numpy as np
import pytest

import workloads as W
from test_gpu_f64_engine import model_of
from test_gpu_f64_long_modes import rhs

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


@pytest.mark.parametrize("levels,depth", [((6,), 4), ((4, 4), 2)])
def test_propagation_ado_by_ado(levels, depth):
    model = model_of(levels, depth)
    h = H.heom_build_hierarchy(model)
    ops = H.heom_get_operators(h)
    ado, bath = ops["ado"], ops["bath"].astype(np.longdouble)
    V = []
    for s, md in enumerate(model["modes"]):
        _, qk = H.heom_get_mode(h, s, levels[s])
        v = (md["V_LL"] * qk[0] + 0.5 * md["V_SL"] * qk[1]).astype(np.longdouble)
        left, right = int(np.prod(levels[:s])), int(np.prod(levels[s + 1:]))
        V.append(np.kron(np.kron(np.eye(left), v), np.eye(right)).astype(np.longdouble))
    rng = np.random.default_rng(depth)
    x = rng.standard_normal((1, h.n_ado, h.d, h.d)) + 1j * rng.standard_normal((1, h.n_ado, h.d, h.d))
    x *= (10.0 ** (-4.0 * ado.sum(1)))[None, :, None, None]
    state = H.heom_state_create(h, 1, H.FP64)
    H.heom_state_upload(state, x)
    H.heom_propagate(h, state, 0.25, 2)
    got = H.heom_state_download(state)[0]
    # sizes: |L| on the norms of the ADOs
    spread = float(np.ptp(np.linalg.eigvalsh(ops["H"])))
    L = np.diag(spread + ado @ ops["bath"][:, 1])
    index = {tuple(a): i for i, a in enumerate(ado)}
    for n, a in enumerate(ado):
        for j, b in enumerate(ops["bath"]):
            v = 2 * np.linalg.norm(np.asarray(V[int(b[0])], float), 2)
            for step, c in ((1, 1.0), (-1, a[j] * (abs(b[2]) + abs(b[3])))):
                m = list(a)
                m[j] += step
                if tuple(m) in index:
                    L[n, index[tuple(m)]] += v * c
    y, size, step = x[0].astype(np.clongdouble), np.linalg.norm(x[0], axis=(1, 2)), np.longdouble(0.25)
    for _ in range(2):
        w, z = y, size
        for q in (4, 3, 2, 1):
            w = y + step / q * rhs(w, ops["H"].astype(np.longdouble), V, ado, bath, len(levels))
            z = size + 0.25 / q * (L @ z)
        y, size = w, z
    err = np.sqrt((np.abs(got - y) ** 2).sum((1, 2)))
    assert (err <= 64 * EPS * size).all()
