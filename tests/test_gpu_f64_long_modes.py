"""FP64 propagation with modes above eight levels, whose change of basis is the dense
product: against RK4 in extended precision on the library's own matrices.

Tolerance: the two changes of basis are 2 d-term sums of FP64 products on either side,
4 (d + 2) 2^-53 of the largest entry (times sqrt(d) between largest entry and norm) at the
very worst and a few 2^-53 in practice; 5e-15 leaves room for d = 24.  Vectors of the coupling
matrix that are not those the stage's tables were made with are off by 1e-13 at these sizes."""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu

H = pytest.importorskip("paper_2601_20550_gb300.heom")


def rhs(x, Hm, V, ado, bath, modes):
    """Eq. HEOM_DB for all ADOs of one branch, extended precision."""
    index = {tuple(a): i for i, a in enumerate(ado)}
    out = np.empty_like(x)
    for n, a in enumerate(ado):
        r = -1j * (Hm @ x[n] - x[n] @ Hm) - sum(k * b[1] for k, b in zip(a, bath)) * x[n]
        for s in range(modes):
            A, B = np.zeros_like(x[n]), np.zeros_like(x[n])
            for j, b in enumerate(bath):
                if int(b[0]) != s:
                    continue
                up, dn = list(a), list(a)
                up[j] += 1
                dn[j] -= 1
                if tuple(up) in index:
                    A = A + x[index[tuple(up)]]
                if dn[j] >= 0:
                    A = A + a[j] * b[2] * x[index[tuple(dn)]]
                    B = B + a[j] * b[3] * x[index[tuple(dn)]]
            r = r - 1j * (V[s] @ A - A @ V[s]) + V[s] @ B + B @ V[s]
        out[n] = r
    return out


@pytest.mark.parametrize("levels,V_LL,V_SL", [(12, 1.0, 1.0), (16, 0.0, 0.05), (16, 0.0, 1.0), (16, 0.1, 1.0),
                                              (24, 0.1, 1.0), (24, 1.0, 0.0)])
def test_long_modes(levels, V_LL, V_SL):
    md = W.mode("morse", 3600.0, D_cm=1.0e4, n_levels=levels, n_prim=200, q_min=-5.0, q_max=20.0, V_LL=V_LL, V_SL=V_SL,
                mu1=1.0, mu2=0.0036, K_pade=1)
    h = H.heom_build_hierarchy({"modes": [md], "pairs": [], "T_K": 300.0, "depth_L": 1})
    ops = H.heom_get_operators(h)
    spread = np.ptp(np.linalg.eigvalsh(ops["H"]))
    dt = float(min(2.0 / spread, 1.0 / ops["bath"][:, 1].max()))
    rng = np.random.default_rng(levels)
    x = rng.standard_normal((1, h.n_ado, levels, levels)) + 1j * rng.standard_normal((1, h.n_ado, levels, levels))
    s = H.heom_state_create(h, 1, H.FP64)
    H.heom_state_upload(s, x)
    H.heom_propagate(h, s, dt, 2)
    got = H.heom_state_download(s)[0]
    _, qk = H.heom_get_mode(h, 0, levels)
    V = [(V_LL * qk[0] + 0.5 * V_SL * qk[1]).astype(np.longdouble)]
    Hm, ado, bath = ops["H"].astype(np.longdouble), ops["ado"], ops["bath"].astype(np.longdouble)
    y, step = x[0].astype(np.clongdouble), np.longdouble(dt)
    for _ in range(2):
        w = y
        for q in (4, 3, 2, 1):
            w = y + step / q * rhs(w, Hm, V, ado, bath, 1)
        y = w
    assert np.abs(got - y).max() <= 5e-15 * np.abs(y).max()
