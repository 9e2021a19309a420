"""The work that users of this framework have it do, as timed cases.

listed() covers the procedure of a 2D correlation spectrum end to end and stage by
stage: equilibration, t1 trunk, batched t3 scan in each arithmetic (FP64, FP32,
tensor cores), whole responses, Fourier sums, several parameter sets in one call and
the misfit gradient, from six levels of one mode (28 small matrices, launch latency)
to three modes of five or six levels each.  draw() gives more of the same ranges.

exact() restates the method in plain torch, 64 bits, on its own: mode eigenbases,
bath exponentials, hierarchy, right-hand side, classic RK4, kicks, traces, sums.
"""
import functools
import itertools
import math

import numpy as np
import torch

from paper_2601_20550_gb300 import heom as H

CM = 2.0 * math.pi * 2.99792458e-5      # 1 cm^-1 in rad/fs
KB = 0.6950348005                       # Boltzmann constant, cm^-1 / K
FP64, FP32, TC = 0, 1, 2


def listed():
    return [
        # one anharmonic mode, the smallest workload: the whole 2D spectrum of a 64 x 64 grid
        {"name": "one-mode spectrum", "kind": "response", "levels": "6", "depth": 6, "K": 1, "n1": 64, "n3": 64,
         "t2": 0, "m": 8},
        # the smallest call: one sample period (8 RK4 steps) of one branch of that model
        {"name": "one-mode steps", "kind": "propagate", "levels": "6", "depth": 6, "K": 1, "prec": FP64,
         "branches": 1, "steps": 8},
        # linear absorption of the stretch-bend pair: one branch, many steps of small matrices
        {"name": "two-mode absorption", "kind": "absorption", "levels": "44", "depth": 4, "K": 1, "n": 64, "m": 16},
        # FP64 equilibration of the five-level water model (every run's first phase)
        {"name": "five-level equilibration", "kind": "equilibrate", "levels": "555", "depth": 6, "K": 1, "steps": 4},
        # FP64 t3 scan of the four-level water model
        {"name": "four-level scan, FP64", "kind": "propagate", "levels": "444", "depth": 4, "K": 1, "prec": FP64,
         "branches": 16, "steps": 2},
        # misfit gradient over twelve parameters, four-level water model at reduced depth and grid
        {"name": "misfit gradient", "kind": "gradient", "levels": "444", "depth": 2, "K": 1, "n1": 4, "n3": 4, "m": 4,
         "ckpt": 8},
        # three parameter sets of uneven basis size in one call
        {"name": "parameter sets, FP64", "kind": "sets", "levels": "454 666 556", "depth": 1, "K": 2, "prec": FP64,
         "n1": 4, "n3": 4, "m": 4},
        # t1 trunk of the five-level model: a single FP32 branch
        {"name": "five-level trunk, FP32", "kind": "propagate", "levels": "555", "depth": 6, "K": 1, "prec": FP32,
         "branches": 1, "steps": 8},
        # six levels per mode (d = 216, beyond the tensor-core tile) in FP32
        {"name": "six-level window, FP32", "kind": "propagate", "levels": "666", "depth": 4, "K": 2, "prec": FP32,
         "branches": 2, "steps": 1},
        # mixed-precision t3 scan of the five-level model, the bulk of a spectrum's work
        {"name": "five-level scan, tensor cores", "kind": "propagate", "levels": "555", "depth": 6, "K": 1,
         "prec": TC, "branches": 32, "steps": 2},
        # a block of t1 rows of the five-level response through the host interface
        {"name": "five-level rows, tensor cores", "kind": "rows", "levels": "555", "depth": 6, "K": 1, "prec": TC,
         "j0": 0, "j1": 2, "n3": 3, "m": 8},
        # correlation spectrum from responses on the host (assembly of row blocks)
        {"name": "Fourier sums 128 x 128", "kind": "sums", "n1": 128, "n3": 128, "t2": 2},
    ]


def draw(rng):
    def log(a, b):
        return int(round(math.exp(rng.uniform(math.log(a), math.log(b)))))

    def lv(lo, hi):
        return "".join(str(rng.randint(lo, hi)) for _ in range(3))

    kind = rng.choice(["response", "small", "absorption", "equilibrate", "scan64", "gradient", "sets", "scan32",
                       "scantc", "rows", "sums"])
    if kind == "response":
        return {"kind": "response", "levels": str(rng.randint(3, 7)), "depth": rng.randint(2, 6), "K": 1,
                "n1": rng.randint(5, 64), "n3": rng.randint(5, 64), "t2": rng.randint(0, 40), "m": rng.randint(4, 8)}
    if kind == "small":
        return {"kind": "propagate", "levels": rng.choice(["4", "5", "6", "7", "33", "43"]),
                "depth": rng.randint(2, 6), "K": rng.randint(1, 2), "prec": rng.choice([FP64, FP64, FP32, TC]),
                "branches": log(1, 128), "steps": rng.randint(1, 16)}
    if kind == "absorption":
        return {"kind": "absorption", "levels": rng.choice(["33", "43", "44", "54"]), "depth": rng.randint(2, 5),
                "K": 1, "n": rng.randint(16, 64), "m": rng.randint(4, 16)}
    if kind == "equilibrate":
        return {"kind": "equilibrate", "levels": lv(3, 5), "depth": rng.randint(2, 5), "K": 1,
                "steps": rng.randint(1, 8)}
    if kind == "scan64":
        return {"kind": "propagate", "levels": lv(3, 5), "depth": rng.randint(1, 4), "K": 1, "prec": FP64,
                "branches": log(1, 10), "steps": rng.randint(1, 2)}
    if kind == "gradient":
        return {"kind": "gradient", "levels": rng.choice(["33", "44", "333", "343"]), "depth": rng.randint(1, 2),
                "K": 1, "n1": rng.randint(2, 4), "n3": rng.randint(2, 4), "m": rng.randint(2, 4),
                "ckpt": rng.randint(3, 8)}
    if kind == "sets":
        return {"kind": "sets", "levels": " ".join(lv(3, 5) for _ in range(rng.randint(2, 4))), "depth": 1,
                "K": rng.randint(1, 2), "prec": rng.choice([FP64, TC]), "n1": rng.randint(2, 5),
                "n3": rng.randint(2, 5), "m": rng.randint(2, 4)}
    if kind == "scan32":
        return {"kind": "propagate", "levels": lv(3, 6), "depth": rng.randint(2, 4), "K": 1, "prec": FP32,
                "branches": log(1, 12), "steps": rng.randint(1, 3)}
    if kind == "scantc":
        return {"kind": "propagate", "levels": lv(3, 5), "depth": rng.randint(3, 6), "K": 1, "prec": TC,
                "branches": log(2, 32), "steps": rng.randint(1, 2)}
    if kind == "rows":
        j0 = rng.randint(0, 2)
        return {"kind": "rows", "levels": lv(3, 5), "depth": rng.randint(2, 4), "K": 1,
                "prec": rng.choice([FP32, TC]), "j0": j0, "j1": j0 + rng.randint(1, 4), "n3": rng.randint(2, 5),
                "m": rng.randint(2, 8)}
    return {"kind": "sums", "n1": log(16, 128), "n3": log(16, 128), "t2": rng.randint(1, 2)}


# ---------------------------------------------------------------------------
# Models: a Morse mode, the stretch-bend pair (cubic potentials) or three Morse modes
# with cubic pair couplings drawn from the seed
# ---------------------------------------------------------------------------
def _mode(omega, n, **kw):
    md = {"potential": "morse", "omega_cm": omega, "g3_cm": 0.0, "morse_D_cm": 1.0e4, "n_levels": n, "n_prim": 100,
          "q_min": -5.0, "q_max": 20.0, "zeta_cm": 2.0 * 25.0 * omega / 100.0, "gamma_cm": 100.0, "V_LL": 0.1,
          "V_SL": 0.1, "mu1": 1.0, "mu2": 0.0036, "K_pade": 1}
    md.update(kw)
    return md


def make_model(levels, depth, K, seed=2601):
    n = [int(c) for c in levels]
    rng = np.random.default_rng(seed)
    pairs = []

    def pair(s, t, g21, g12, mu):
        pairs.append({"s": s, "t": t, "g_st_cm": 0.0, "g_s2t_cm": float(g21), "g_st2_cm": float(g12), "mu_st": mu})

    if len(n) == 1:
        modes = [_mode(3600.0, n[0], q_min=-4.0, q_max=16.0, V_SL=0.05)]
    elif len(n) == 2:
        modes = [_mode(3520.0, n[0], potential="cubic", g3_cm=-1362.9, n_prim=16, V_LL=0.0, V_SL=1.0, gamma_cm=20.0,
                       zeta_cm=27878.4, mu1=2.904, mu2=0.0093),
                 _mode(1710.0, n[1], potential="cubic", g3_cm=-218.76, n_prim=16, V_LL=0.0, V_SL=1.0, gamma_cm=80.0,
                       zeta_cm=584.82, mu1=0.7695, mu2=0.0)]
        pair(0, 1, 0.0, 128.66, 7.5e-4)
    else:
        om, D, mu = (3650.0, 3750.0, 1600.0), (1.0e4, 1.0e4, 2.0e4), (1.0, 1.0, 0.545)
        modes = [_mode(om[s], n[s], morse_D_cm=D[s], mu1=mu[s], mu2=0.0036 if s < 2 else 0.0) for s in range(3)]
        for (s, t), c in (((0, 1), 0.0), ((0, 2), 6e-4), ((1, 2), 6e-4)):
            g = rng.uniform(-50.0, 50.0, size=2)
            pair(s, t, g[0], g[1], c)
    for md in modes:
        md["K_pade"] = K
    return {"modes": modes, "pairs": pairs, "T_K": 300.0, "depth_L": depth}


def dt_of(levels):
    return 0.25 if "6" in levels[1:] or "7" in levels or len(levels) == 2 else 0.5


def ados_of(case, levels):
    D = len(levels) * (case["K"] + 1)
    L = case["depth"]
    return math.comb(L + D, D)


@functools.lru_cache(maxsize=None)
def handle(levels, depth, K, prec, seed=2601):
    """The hierarchy handle, built once per model as a user's program keeps it."""
    return H.heom_build_hierarchy(make_model(levels, depth, K, seed), prec)


def grid_of(case, dt, t2=(0.0,), n1=None):
    return {"dt_fs": dt, "steps_per_sample": case["m"], "n1": n1 or case["n1"], "n3": case["n3"],
            "t2_fs": [float(t) for t in t2]}


@functools.lru_cache(maxsize=None)
def index_set(D, L):
    return sorted((n for n in itertools.product(range(L + 1), repeat=D) if sum(n) <= L), key=lambda n: (sum(n), n))


def random_state(levels, depth, K, branches, seed, dtype=torch.complex128, equilibrium=False):
    """ADO magnitudes that fall with their level, as in a kicked equilibrium; in the product
    basis (complex128) also with the excitation of row and column."""
    n = [int(c) for c in levels]
    d = math.prod(n)
    ados = index_set(len(n) * (K + 1), depth)
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    x = torch.randn((branches, len(ados), d, d), generator=g, device="cuda", dtype=dtype)
    lev = torch.tensor([sum(a) for a in ados], device="cuda", dtype=torch.float64)
    x *= (10.0 ** -lev).to(x.real.dtype)[None, :, None, None]
    if dtype == torch.complex128:
        N = torch.tensor([sum(a) for a in itertools.product(*[range(k) for k in n])], device="cuda",
                         dtype=torch.float64)
        x *= torch.exp(-0.5 * (N[:, None] + N[None, :]))
    if equilibrium:
        x = 1e-2 * (x + x.mH)
        x[:, 0, 0, 0] += 1.0
    return x


def uploaded(h, x):
    s = H.heom_state_create(h, x.shape[0], FP64)
    H.heom_state_import_dev(s, x.data_ptr(), torch.cuda.current_stream().cuda_stream)
    torch.cuda.synchronize()
    return s


# ---------------------------------------------------------------------------
def prepare(case, seed):
    k = case["kind"]
    if k == "sums":
        rng = np.random.default_rng(seed)
        t = np.exp(-0.03 * (np.arange(case["n1"])[:, None] + np.arange(case["n3"])[None, :]))
        R = [(rng.standard_normal((case["t2"],) + t.shape) + 1j * rng.standard_normal((case["t2"],) + t.shape)) * t
             for _ in range(2)]
        return {"case": case, "RI": R[0], "RII": R[1]}
    sets = case["levels"].split()
    lv = sets[0]
    dt = min(dt_of(s) for s in sets)
    st = {"case": case, "dt": dt}
    if k == "propagate":
        st["h"] = handle(lv, case["depth"], case["K"], case["prec"])
        st["y"] = random_state(lv, case["depth"], case["K"], case["branches"], seed,
                               torch.complex128 if case["prec"] == FP64 else torch.complex64)
        st["wa"], st["wb"] = torch.empty_like(st["y"]), torch.empty_like(st["y"])
    elif k == "equilibrate":
        h = H.heom_build_hierarchy(make_model(lv, case["depth"], case["K"], seed), FP64)
        st["h"], st["out"] = h, torch.empty((1, h.n_ado, h.d, h.d), dtype=torch.complex128, device="cuda")
    elif k == "gradient":
        st["h"] = handle(lv, case["depth"], case["K"], FP64)
        st["eq"] = H.heom_equilibrate(st["h"], dt, 8 * dt)
        st["ref"] = reference_spectrum(case, seed)
    else:
        prec = case.get("prec", FP64)
        st["h"] = [handle(s, case["depth"], case["K"], prec) for s in sets]
        st["eq"] = [uploaded(h, random_state(s, case["depth"], case["K"], 1, seed + i, equilibrium=True))
                    for i, (h, s) in enumerate(zip(st["h"], sets))]
    return st


def reference_spectrum(case, seed):
    rng = np.random.default_rng(seed)
    return 10.0 * rng.standard_normal((1, case["n1"], case["n3"]))


def run(st):
    case = st["case"]
    k = case["kind"]
    if k == "sums":
        return H.heom_spectrum_2d(st["RI"], st["RII"], 4.0)
    dt = st["dt"]
    if k == "propagate":
        H.heom_propagate_dev(st["h"], st["y"].data_ptr(), st["wa"].data_ptr(), st["wb"].data_ptr(),
                             case["branches"], case["prec"], dt, case["steps"],
                             torch.cuda.current_stream().cuda_stream)
        return st["y"]
    if k == "equilibrate":
        eq = H.heom_equilibrate(st["h"], dt, case["steps"] * dt)
        H.heom_state_export_dev(eq, st["out"].data_ptr(), torch.cuda.current_stream().cuda_stream)
        torch.cuda.current_stream().synchronize()     # the state goes out of scope here
        return st["out"]
    if k == "gradient":
        return H.heom_response_2d_grad(st["h"], st["eq"], grid_of(case, dt), st["ref"], case["ckpt"])
    if k == "absorption":
        return H.heom_response_1d(st["h"][0], st["eq"][0], dt, case["m"], case["n"])
    if k == "response":
        return H.heom_response_2d(st["h"][0], st["eq"][0], grid_of(case, dt, (case["t2"] * dt,)))
    if k == "rows":
        return H.heom_response_2d_rows(st["h"][0], st["eq"][0], grid_of(case, dt, n1=case["j1"]), case["j0"],
                                       case["j1"])
    return H.heom_response_2d_batched(st["h"], st["eq"], grid_of(case, dt))


def work(case):
    """State in and out once; the products that H's structure leaves (no three-mode terms),
    the neighbour sums and one diagonal product per mode, of every ADO update."""
    if case["kind"] == "sums":
        n1, n3, t = case["n1"], case["n3"], case["t2"]
        return {"bytes": t * n1 * n3 * 40.0, "flops": t * 2.0 * 8.0 * n1 * n3 * (n1 + n3)}
    total = {"bytes": 0.0, "flops": 0.0}
    k = case["kind"]
    for lv in case["levels"].split():
        n = [int(c) for c in lv]
        d, N, M = math.prod(n), ados_of(case, lv), len(n)
        nnz = 1 + sum(a - 1 for a in n) + sum((a - 1) * (b - 1) for a, b in itertools.combinations(n, 2))
        D, L = M * (case["K"] + 1), case["depth"]
        nb = 2.0 * D * (math.comb(L - 1 + D, D) if L else 0) / N
        upd = 4.0 * d * d * (8.0 * nnz + 8.0 * nb + 16.0 * M + 8.0)
        b = 16.0 if case.get("prec", FP64) == FP64 else 8.0
        state = N * d * d * b
        if k == "propagate":
            steps, io = case["branches"] * case["steps"], 2.0 * case["branches"]
        elif k == "equilibrate":
            steps, io = case["steps"], 1.0
        elif k == "absorption":
            steps, io = (case["n"] - 1) * case["m"], 1.0
        elif k == "rows":
            B = 2 * (case["j1"] - case["j0"])
            steps, io = (case["j1"] - 1) * case["m"] + B * (case["n3"] - 1) * case["m"], 1.0
        else:
            B, m = 2 * case["n1"], case["m"]
            steps, io = (case["n1"] - 1) * m + B * ((case["n3"] - 1) * m + case.get("t2", 0)), 1.0
            if k == "gradient":
                steps = 4.0 * (steps + 8)
        total["bytes"] += io * state
        total["flops"] += steps * N * upd
    return total


# ---------------------------------------------------------------------------
# The method in plain torch, 64 bits
# ---------------------------------------------------------------------------
def mode_matrices(md):
    w, n, M = md["omega_cm"] * CM, md["n_prim"], md["n_levels"]
    if md["potential"] == "morse":
        D = md["morse_D_cm"] * CM
        x = np.linspace(md["q_min"], md["q_max"], n)
        i = np.arange(n)
        df = i[:, None] - i[None, :]
        T = np.where(df == 0, math.pi ** 2 / 3, 2.0 / np.where(df == 0, 1, df) ** 2) * (-1.0) ** df
        Hm = 0.5 * w / (x[1] - x[0]) ** 2 * T + np.diag(D * (1 - np.exp(-math.sqrt(w / (2 * D)) * x)) ** 2)
        q = [np.diag(x ** p) for p in range(5)]
    else:
        a = np.diag(np.sqrt(np.arange(1.0, n + 4)), 1)
        a = (a + a.T) / math.sqrt(2)
        q = [np.linalg.matrix_power(a, p)[:n, :n] for p in range(5)]
        Hm = w * np.diag(np.arange(n) + 0.5) + md["g3_cm"] * CM / 6 * q[3]
    E, U = np.linalg.eigh(Hm)
    U = U[:, :M].copy()
    U[:, 0] *= np.sign(U[np.argmax(np.abs(U[:, 0])), 0])
    for c in range(1, M):
        U[:, c] *= np.sign(U[:, c - 1] @ q[1] @ U[:, c])
    return E[:M], [U.T @ m @ U for m in q]


def pade(N):
    off = [1 / math.sqrt((2 * m + 1) * (2 * m + 3)) for m in range(1, 2 * N)]
    lam = np.linalg.eigvalsh(np.diag(off, 1) + np.diag(off, -1))
    xi = np.sort(2 / lam[lam > 0])
    bern = [1 / 6, -1 / 30, 1 / 42, -1 / 30]
    A = [[2 * (-1) ** m / x ** (2 * m + 2) for x in xi] for m in range(N)]
    return xi, np.linalg.solve(A, [bern[m] / math.factorial(2 * m + 2) for m in range(N)])


def jacobi_vectors(A):
    """Eigenvectors by cyclic Jacobi rotations, ascending: complex64 states are held in this basis
    and its column signs follow from the rotations."""
    A, n = A.copy(), len(A)
    Z = np.eye(n)
    for _ in range(60):
        for p in range(n - 1):
            for q in range(p + 1, n):
                if abs(A[p, q]) < 1e-300:
                    continue
                th = (A[q, q] - A[p, p]) / (2 * A[p, q])
                t = (1.0 if th >= 0 else -1.0) / (abs(th) + math.hypot(th, 1.0))
                R = np.eye(n)
                R[p, p] = R[q, q] = c = 1 / math.hypot(t, 1.0)
                R[p, q], R[q, p] = t * c, -t * c
                A, Z = R.T @ A @ R, Z @ R
        if np.linalg.norm(A - np.diag(np.diag(A))) <= 1e-15 * np.linalg.norm(A):
            break
    return Z[:, np.argsort(np.diag(A))]


def kron(ops, dims):
    out = np.ones((1, 1))
    for s, n in enumerate(dims):
        out = np.kron(out, ops.get(s, np.eye(n)))
    return out


def plain_model(model):
    """Matrices of the model as numpy arrays: H, V (per mode), mu, mu+, bath, and the basis U
    in which every V is diagonal."""
    modes, dims = model["modes"], [md["n_levels"] for md in model["modes"]]
    d = math.prod(dims)
    E, q = zip(*[mode_matrices(md) for md in modes])
    kT = KB * model["T_K"] * CM
    Hs, mu, V, U, bath = np.zeros((d, d)), np.zeros((d, d)), [], np.ones((1, 1)), []
    for s, md in enumerate(modes):
        a, b = md["V_LL"], md["V_SL"]
        lam, gam = md["zeta_cm"] * md["gamma_cm"] / (2 * md["omega_cm"]) * CM, md["gamma_cm"] * CM
        v = a * q[s][1] + b / 2 * q[s][2]
        Hs += kron({s: np.diag(E[s]) + lam * (a * a * q[s][2] + a * b * q[s][3] + b * b / 4 * q[s][4])}, dims)
        mu += kron({s: md["mu1"] * q[s][1] + md["mu2"] / 2 * q[s][2]}, dims)
        V.append(v)
        U = np.kron(U, jacobi_vectors(v))
        xi, eta = pade(md["K_pade"])
        nu = xi * kT
        den = gam ** 2 - nu ** 2
        bath.append((s, gam, 2 * lam * kT * (1 + np.sum(2 * eta * gam ** 2 / den)), -lam * gam))
        bath += [(s, nu[i], -4 * lam * gam * kT * eta[i] * nu[i] / den[i], 0.0) for i in range(len(nu))]
    for p in model["pairs"]:
        s, t = p["s"], p["t"]
        for g, i, j in ((p["g_st_cm"], 1, 1), (p["g_s2t_cm"] / 6, 2, 1), (p["g_st2_cm"] / 6, 1, 2)):
            Hs += g * CM * kron({s: q[s][i], t: q[t][j]}, dims)
        mu += p["mu_st"] * kron({s: q[s][1], t: q[t][1]}, dims)
    N = np.array([sum(x) for x in itertools.product(*[range(k) for k in dims])])
    return {"H": Hs, "V": V, "mu": mu, "mup": np.where(N[:, None] > N[None, :], mu, 0.0), "U": U, "dims": dims,
            "nu": np.array([b[1] for b in bath]), "re": np.array([b[2] for b in bath]),
            "im": np.array([b[3] for b in bath]), "of": [b[0] for b in bath]}


def on_device(pm, depth, rotate=True):
    """The model on the GPU, in the basis where every V is diagonal (rotate) or in the product basis."""
    def t(a):
        return torch.tensor(np.asarray(a), dtype=torch.float64, device="cuda")

    U = pm["U"]
    R = (lambda A: U.T @ A @ U) if rotate else (lambda A: A)
    m = {k: t(R(pm[k])) for k in ("H", "mu", "mup")}
    full = [kron({s: v}, pm["dims"]) for s, v in enumerate(pm["V"])]
    if rotate:
        m["lam"] = [t(np.diag(R(f))) for f in full]
    else:
        m["V"] = [t(f) for f in full]
    m.update({k: t(pm[k]) for k in ("nu", "re", "im")}, of=pm["of"], U=t(U))
    ados = index_set(len(pm["of"]), depth)
    at = {a: i for i, a in enumerate(ados)}
    m["n"] = t(np.array(ados, dtype=float).reshape(len(ados), -1))
    m["up"], m["down"] = [], []
    for j in range(len(pm["of"])):
        for key, step in (("up", 1), ("down", -1)):
            to = [at.get(a[:j] + (a[j] + step,) + a[j + 1:], -1) for a in ados]
            m[key].append((torch.tensor([max(x, 0) for x in to], device="cuda"), t([float(x >= 0) for x in to])))
    return m


def left(A, X):
    return torch.complex(A @ X.real, A @ X.imag)


def right(X, A):
    return torch.complex(X.real @ A, X.imag @ A)


def rhs(m, X):
    out = -1j * (left(m["H"], X) - right(X, m["H"])) - (m["n"] @ m["nu"])[None, :, None, None] * X
    for s in sorted(set(m["of"])):
        A = B = 0
        for j in (j for j, o in enumerate(m["of"]) if o == s):
            (iu, fu), (id_, fd) = m["up"][j], m["down"][j]
            Xd = X[:, id_] * (fd * m["n"][:, j])[None, :, None, None]
            A = A + X[:, iu] * fu[None, :, None, None] + m["re"][j] * Xd
            B = B + m["im"][j] * Xd
        if "lam" in m:
            la = m["lam"][s]
            out = out - 1j * (la[:, None] - la[None, :]) * A + (la[:, None] + la[None, :]) * B
        else:
            V = m["V"][s]
            out = out - 1j * (left(V, A) - right(A, V)) + left(V, B) + right(B, V)
    return out


def rk4(m, X, dt, steps):
    for _ in range(steps):
        k1 = rhs(m, X)
        k2 = rhs(m, X + 0.5 * dt * k1)
        k3 = rhs(m, X + 0.5 * dt * k2)
        X = X + dt / 6 * (k1 + 2 * k2 + 2 * k3 + rhs(m, X + dt * k3))
    return X


def kicked(X, K):
    return left(K, X) - right(X, K)


def trace(m, X):
    return (m["mu"].T * X[:, 0]).sum(dim=(-1, -2))


def responses(m, eq, g, j0=0, j1=None):
    """R_I, R_II [1][rows][n3] for one t2 (kicks mu-, mu+, mu+ and mu+, mu-, mu+)."""
    dt, k, out = g["dt_fs"], g["steps_per_sample"], []
    j1 = g["n1"] if j1 is None else j1
    mp, mm = m["mup"], m["mup"].T
    for first, second in ((mm, mp), (mp, mm)):
        trunk, rows = kicked(eq, first), []
        for j in range(j1):
            trunk = trunk if j == 0 else rk4(m, trunk, dt, k)
            if j >= j0:
                rows.append(kicked(trunk, second))
        X = rk4(m, torch.cat(rows), dt, round(g["t2_fs"][0] / dt))
        X, R = kicked(X, mp), []
        for i in range(g["n3"]):
            X = X if i == 0 else rk4(m, X, dt, k)
            R.append(-1j * trace(m, X))
        out.append(torch.stack(R, dim=1)[None])
    return out


def sums(RI, RII, dtau):
    n1, n3 = RI.shape[1:]

    def F(n, sign):
        k = torch.arange(n, device=RI.device)
        ph = 2 * math.pi / n * ((k[:, None] * k[None, :]) % n).double()
        f = torch.complex(torch.cos(ph), sign * torch.sin(ph))
        f[:, 0] *= 0.5
        return f

    return (dtau ** 2 * (F(n1, -1) @ RI @ F(n3, 1).mT + F(n1, 1) @ RII @ F(n3, 1).mT)).imag


def rotated(m, X, back=False):
    U = m["U"].T if back else m["U"]
    return right(left(U.T, X), U)


def exact(case, seed):
    k = case["kind"]
    if k == "sums":
        st = prepare(case, seed)
        return sums(torch.tensor(st["RI"], device="cuda"), torch.tensor(st["RII"], device="cuda"), 4.0)
    sets = case["levels"].split()
    dt = min(dt_of(s) for s in sets)
    model_seed = seed if k == "equilibrate" else 2601
    pms = [plain_model(make_model(s, case["depth"], case["K"], model_seed)) for s in sets]
    if k == "gradient":
        return exact_gradient(case, seed, pms[0], dt)
    ms = [on_device(pm, case["depth"]) for pm in pms]
    m = ms[0]
    if k == "propagate":
        ados, d = ados_of(case, sets[0]), len(pms[0]["H"])
        if case["branches"] * case["steps"] * ados * d ** 3 > 4e11:
            return None
        prec = case["prec"]
        x = random_state(sets[0], case["depth"], case["K"], case["branches"], seed,
                         torch.complex128 if prec == FP64 else torch.complex64).to(torch.complex128)
        for b in range(0, case["branches"], 4):      # a few branches at a time
            y = x[b:b + 4]
            y = rk4(m, rotated(m, y) if prec == FP64 else y, dt, case["steps"])
            x[b:b + 4] = rotated(m, y, back=True) if prec == FP64 else y
        return x
    if k == "equilibrate":
        d = len(pms[0]["H"])
        x = torch.zeros((1, ados_of(case, sets[0]), d, d), dtype=torch.complex128, device="cuda")
        x[0, 0, 0, 0] = 1.0
        return rotated(m, rk4(m, rotated(m, x), dt, case["steps"]), back=True)
    eqs = [rotated(m, random_state(s, case["depth"], case["K"], 1, seed + i, equilibrium=True))
           for i, (m, s) in enumerate(zip(ms, sets))]
    if k == "absorption":
        X, R = kicked(eqs[0], m["mu"]), []
        for i in range(case["n"]):
            X = X if i == 0 else rk4(m, X, dt, case["m"])
            R.append(1j * trace(m, X)[0])
        R = torch.stack(R)
        w = torch.ones(case["n"], device="cuda")
        w[0] = 0.5
        return R, (dt * case["m"] * torch.fft.ifft(w * R, norm="forward")).imag
    if k == "rows":
        return responses(m, eqs[0], grid_of(case, dt, n1=case["j1"]), case["j0"], case["j1"])
    g = grid_of(case, dt, (case.get("t2", 0) * dt,))
    got = [responses(m, eq, g) for m, eq in zip(ms, eqs)]
    got = [(a, b, sums(a, b, dt * case["m"])) for a, b in got]
    return got[0] if k == "response" else [torch.stack(x) for x in zip(*got)]


PARTS = ("H", "mu", "mup", "nu", "re", "im")


def exact_gradient(case, seed, pm, dt):
    """Loss and its gradient: reverse mode through the plain propagation, matrix derivatives by
    fourth-order differences of the plain model build."""
    m = on_device(pm, case["depth"], rotate=False)
    leaves = [m[p].requires_grad_() for p in PARTS] + [v.requires_grad_() for v in m["V"]]
    d = len(pm["H"])
    eq = torch.zeros((1, ados_of(case, case["levels"]), d, d), dtype=torch.complex128, device="cuda")
    eq[0, 0, 0, 0] = 1.0
    a, b = responses(m, rk4(m, eq, dt, 8), grid_of(case, dt))
    loss = (sums(a, b, dt * case["m"]) - torch.tensor(reference_spectrum(case, seed), device="cuda")).square().sum()
    grads = [g.cpu().numpy() for g in torch.autograd.grad(loss, leaves)]
    out = np.zeros(12)
    for i in range(12):
        def at(delta):
            md = make_model(case["levels"], case["depth"], case["K"])
            grp, k = divmod(i, 3)
            owner = md["pairs"] if grp == 1 else md["modes"]
            if k >= len(owner):
                return None
            cubic = md["modes"][0]["potential"] == "cubic"
            key = ("g3_cm" if cubic else "morse_D_cm", "g_s2t_cm", "V_SL", "gamma_cm")[grp]
            step = 1e-3 * max(abs(owner[k][key]), 1.0)
            owner[k][key] += delta * step
            p = plain_model(md)
            return step, [p[x] for x in PARTS] + [kron({s: v}, p["dims"]) for s, v in enumerate(p["V"])]
        if at(0) is None:
            continue
        step = at(0)[0]
        p1, m1, p2, m2 = (at(x)[1] for x in (1, -1, 2, -2))
        out[i] = sum(float(np.sum(g * (8 * (a - b) - (c - e)))) for g, a, b, c, e in
                     zip(grads, p1, m1, p2, m2)) / (12 * step)
    return float(loss.detach()), out
