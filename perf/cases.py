"""The work that users of the library have it do, as cases with seeded inputs.

Whole calls: the thermal state and C(t) of a chain on the complex128 path (the default), C(t) of a
prepared chain on the mixed path (complex64 contractions on the tensor cores), a batch of
instances, and the gradient of a real-time correlation.  Single operations, each through its own
entry point: the H_eff product, the environment update, the gauge QR, the bond exponential and the
reverse pass of a site exponential.  Sizes come from the chains of the tests and of the benchmark
(one and two modes per molecule, 2 to 8 levels, bond dimensions up to 128) and from ragged
neighbours of them.

The mixed path's results are returned as complex64, the precision its contractions have; the
complex128 path's as complex128.  The chains of the complex128 path are taken at full bond
dimension, where C(t) has an exact value (below it, C(t) follows the rounding of the smallest
singular values).
"""
import numpy as np
import torch

from paper_2003_13245_gb300 import Model, PREC_C64_3XTF32, binding

DW = 7            # bond dimension of the Hamiltonian MPO of the periodic chain


def listed():
    return [
        # one small chain from the infinite-temperature state to C(t): latency and launches count
        {"name": "chain_n3_c128", "kind": "chain", "nmax": 2, "V": 1.0, "kT": 5.0, "points": 3},
        # the same call at the largest bond dimension that is exact for three levels per mode
        {"name": "chain_n3_wide_c128", "kind": "chain", "nmax": 3, "V": 1.0, "kT": 5.0,
         "points": 2},
        # the benchmark's two-mode chain (shorter), real-time steps of both states, mixed path
        {"name": "chain_n6_mixed", "kind": "mixed", "N": 6, "modes": 2, "nmax": 8, "M": 128,
         "V": 0.5, "points": 3},
        # a parameter sweep: instances of uneven length and bond dimension stepped together
        {"name": "batch_mixed", "kind": "batch", "nmax": 6, "instances": 4, "N": 8, "M": 32,
         "V": 0.5, "points": 2},
        # a training step on given states: C(t), the gradients of both states and of the parameters
        {"name": "gradient_c128", "kind": "grad", "nmax": 3, "M": 16, "V": 0.5},
        # H_eff at the bulk site of the adjoint's chain, and at the benchmark's bulk site
        {"name": "heff_c128", "kind": "heff", "mixed": False, "Ml": 96, "Mr": 96, "d": 6},
        {"name": "heff_mixed", "kind": "heff", "mixed": True, "Ml": 128, "Mr": 128, "d": 8},
        # environment update at uneven, odd bond dimensions
        {"name": "env_left_c128", "kind": "env", "Ml": 70, "Mr": 61, "d": 5},
        # gauge shift of the benchmark's bulk site; of a narrow site with skipped columns
        {"name": "gauge_qr_bulk", "kind": "qr", "m": 8192, "n": 128, "rank": 128},
        {"name": "gauge_qr_ragged", "kind": "qr", "m": 1000, "n": 100, "rank": 93},
        # bond back-step of the benchmark's chain (mixed path)
        {"name": "bond_exp_mixed", "kind": "bond", "M": 128},
        # reverse pass of one site exponential
        {"name": "site_exp_vjp_c128", "kind": "site_vjp", "Ml": 32, "Mr": 40, "d": 3},
    ]


def _log(rng, lo, hi):
    return int(round(lo * (hi / lo) ** rng.random()))


def draw(rng):
    kind = rng.choice(["chain", "mixed", "batch", "heff", "heff", "heff", "env", "env", "qr", "qr",
                       "qr", "bond", "bond", "site_vjp"])
    V = round(rng.uniform(0.3, 2.0), 3)
    if kind == "chain":
        nmax = rng.choice([2, 2, 3])
        return {"kind": kind, "nmax": nmax, "V": V, "kT": rng.choice([5.0, 10.0]),
                "points": rng.choice([2, 3]) if nmax == 2 else 2}
    if kind == "mixed":
        return {"kind": kind, "N": rng.choice([4, 5, 6]), "modes": rng.choice([1, 2]),
                "nmax": rng.choice([5, 6, 7, 8]), "M": _log(rng, 32, 100), "V": V, "points": 2}
    if kind == "batch":
        return {"kind": kind, "nmax": rng.choice([4, 5, 6]), "instances": rng.choice([2, 3, 4]),
                "N": rng.choice([4, 6, 8]), "M": _log(rng, 20, 32), "V": V, "points": 2}
    if kind == "heff":
        mixed = rng.random() < 0.5
        hi = 128 if mixed else 96
        return {"kind": kind, "mixed": mixed, "Ml": _log(rng, 8, hi), "Mr": _log(rng, 8, hi),
                "d": rng.choice([2, 3, 4, 5, 6])}
    if kind == "env":
        return {"kind": kind, "Ml": _log(rng, 8, 96), "Mr": _log(rng, 8, 96),
                "d": rng.choice([2, 3, 4, 5, 6])}
    if kind == "qr":
        n = _log(rng, 12, 128)
        m = min(8192, n * _log(rng, 2, 80))
        rank = n if rng.random() < 0.6 else max(2, int(n * rng.uniform(0.85, 0.99)))
        return {"kind": kind, "m": m, "n": n, "rank": rank}
    if kind == "bond":
        return {"kind": kind, "M": _log(rng, 12, 128)}
    return {"kind": kind, "Ml": _log(rng, 8, 36), "Mr": _log(rng, 8, 36), "d": rng.choice([2, 3])}


# ---------------------------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------------------------
def _randc(rng, shape):
    return rng.standard_normal(shape) + 1j * rng.standard_normal(shape)


def _mpo_site(rng, d):
    """A vibrational site of the chain's MPO: every channel passes on, channel 0 picks up the
    oscillator's energy and the channel that carries the site's occupation picks up the coupling."""
    w, g = rng.uniform(0.2, 1.5), rng.uniform(0.2, 1.5)
    b = np.diag(np.sqrt(np.arange(1, d)), 1)
    W = np.zeros((DW, DW, d, d), dtype=complex)
    for c in range(DW):
        W[c, c] = np.eye(d)
    W[0, DW - 1] += w * (b.T @ b)
    W[5, DW - 1] += g * w * (b + b.T)
    return W


def _env(rng, M):
    """Environments of a Hermitian MPO: the identity channel, and Hermitian blocks of unit scale."""
    X = _randc(rng, (DW, M, M))
    E = (X + np.conj(np.swapaxes(X, 1, 2))) / (2.0 * np.sqrt(M))
    E[0] = np.eye(M)
    return E


def _site(rng, Ml, D, Mr):
    """A center tensor with decaying singular values, normalised."""
    A = _randc(rng, (Ml, D, Mr))
    A *= np.exp(-6.0 * np.arange(Ml) / Ml)[:, None, None]
    A *= np.exp(-6.0 * np.arange(Mr) / Mr)[None, None, :]
    return A / np.linalg.norm(A)


def _heff_inputs(case, seed):
    rng = np.random.default_rng(seed)
    d = case["d"]
    return (_env(rng, case["Ml"]), _mpo_site(rng, d), _env(rng, case["Mr"]),
            _site(rng, case["Ml"], d * d, case["Mr"]), rng)


def _qr_inputs(case, seed):
    """A center matrix (decaying singular values, mixed columns) and completion candidates."""
    rng = np.random.default_rng(seed)
    m, n, r = case["m"], case["n"], case["rank"]
    U, _ = np.linalg.qr(_randc(rng, (r, r)))
    Y = _randc(rng, (m, r)) @ (np.exp(-9.0 * np.arange(r) / r)[:, None] * U.conj().T)
    E = None
    if r < n:
        Y = np.concatenate([Y, Y[:, :n - r] @ _randc(rng, (n - r, n - r))], axis=1)
        E = _randc(rng, (m, 2 * (n - r)))
    return Y / np.linalg.norm(Y), E


def _bond_inputs(case, seed):
    rng = np.random.default_rng(seed)
    M = case["M"]
    C = _site(rng, M, 1, M).reshape(M, M)
    return _env(rng, M), _env(rng, M), C


def _jitter(rng, x):
    return [float(v) * rng.uniform(0.95, 1.05) for v in x]


def _chain_parameters(case, seed):
    rng = np.random.default_rng(seed)
    return _jitter(rng, [1.0]), _jitter(rng, [1.0]), _jitter(rng, [case["V"]])[0]


def _states(rng, dims, M):
    """Two states with the center at site 0, the other sites right-orthonormal and shared."""
    L = len(dims)
    left, right = [1], [1]
    for x in dims:
        left.append(left[-1] * x)
    for x in reversed(dims):
        right.append(right[-1] * x)
    Mb = [min(M, left[k], right[L - k]) for k in range(L + 1)]
    sites = []
    for k in range(1, L):
        q, _ = np.linalg.qr(_randc(rng, (dims[k] * Mb[k + 1], Mb[k])))
        sites.append(np.ascontiguousarray(q.T).reshape(Mb[k], dims[k], Mb[k + 1]))
    out = []
    for _ in range(2):
        c = _randc(rng, (1, dims[0], Mb[1]))
        out.append([c / np.linalg.norm(c)] + sites)
    return out


def _dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).to("cuda")


TAU = -0.025j      # half a real-time step of 0.05
DT = 0.05


# ---------------------------------------------------------------------------------------------
# what a program has in hand, and one pass
# ---------------------------------------------------------------------------------------------
def prepare(case, seed):
    kind = case["kind"]
    s = {"case": case}
    if kind == "chain":
        om, g, V = _chain_parameters(case, seed)
        s["model"] = Model(3, om, g, [case["nmax"]], V)
    elif kind == "mixed":
        rng = np.random.default_rng(seed)
        om, g = _jitter(rng, [0.2, 1.0]), _jitter(rng, [1.5, 0.8])
        nm = [case["nmax"], 4]
        k = case["modes"]
        s["model"] = Model(case["N"], om[2 - k:], g[2 - k:], nm[:k],
                           _jitter(rng, [case["V"]])[0], precision=PREC_C64_3XTF32)
        s["model"].thermal_prepare(0.1, 0.05, case["M"])
    elif kind == "batch":
        rng = np.random.default_rng(seed)
        s["models"] = []
        for i in range(case["instances"]):
            m = Model(case["N"] if i % 2 else 3, [1.0], [1.0], [case["nmax"]],
                      _jitter(rng, [case["V"] * 2.0 ** i])[0], precision=PREC_C64_3XTF32,
                      krylov=(1e-7, 32, 8))
            m.thermal_prepare(0.1, 0.05, case["M"] + 8 * (i % 3))
            m.realtime_init()
            s["models"].append(m)
        s["batch"] = binding.Batch(s["models"])
    elif kind == "grad":
        rng = np.random.default_rng(seed)
        n = case["nmax"]
        s["model"] = Model(3, _jitter(rng, [1.0]), _jitter(rng, [1.0]), [n],
                           _jitter(rng, [case["V"]])[0])
        s["model"].set_adjoint_krylov_basis(True)
        p1, p2 = _states(rng, [4, n * n] * 3, case["M"])
        s["psi1"], s["psi2"] = [_dev(a) for a in p1], [_dev(a) for a in p2]
        s["cbar"] = np.array([0.5, 0.5])
    elif kind == "heff":
        L, W, R, A, _ = _heff_inputs(case, seed)
        s.update(L=_dev(L), W=W, R=_dev(R), A=_dev(A))
        s["out"] = torch.empty_like(s["A"])
        if case["mixed"]:
            nf = binding.heff_workspace_floats(case["Ml"], case["Mr"], case["d"], DW, DW)
            s["ws32"] = torch.empty(nf, dtype=torch.float32, device="cuda")
        else:
            s["X"] = torch.empty(DW * A.size, dtype=torch.complex128, device="cuda")
            s["Y"] = torch.empty_like(s["X"])
    elif kind == "env":
        L, W, _, ket, rng = _heff_inputs(case, seed)
        s.update(L=_dev(L), W=W, ket=_dev(ket), bra=_dev(_site(rng, *ket.shape)))
        s["X"] = torch.empty(DW * ket.size, dtype=torch.complex128, device="cuda")
        s["Y"] = torch.empty_like(s["X"])
        s["out"] = torch.empty((DW, case["Mr"], case["Mr"]), dtype=torch.complex128, device="cuda")
    elif kind == "qr":
        Y, E = _qr_inputs(case, seed)
        s.update(Y=_dev(Y), E=None if E is None else _dev(E))
        s["Q"] = torch.empty_like(s["Y"])
        s["R"] = torch.empty((case["n"], case["n"]), dtype=torch.complex128, device="cuda")
    elif kind == "bond":
        L, R, C = _bond_inputs(case, seed)
        s.update(L=_dev(L), R=_dev(R), C=_dev(C))
        s["out"] = torch.empty_like(s["C"])
    else:
        L, W, R, A, rng = _heff_inputs(case, seed)
        s.update(L=_dev(L), W=W, R=_dev(R), A=_dev(A), ybar=_dev(_site(rng, *A.shape)))
        s["outs"] = [torch.empty_like(s[k]) for k in ("A", "L", "R")]
    return s


def run(s):
    case = s["case"]
    kind = case["kind"]
    if kind == "chain":
        m = s["model"]
        m.thermal_prepare(1.0 / case["kT"], 0.05, 144)
        C = m.correlation(np.arange(case["points"]) * DT, DT)
        return {"C": C, "logz": m.logz(), "sigma": m.reduced_density()}
    if kind == "mixed":
        C = s["model"].correlation(np.arange(case["points"]) * DT, DT)
        return {"C": C.astype(np.complex64),
                "sigma": s["model"].reduced_density().astype(np.complex64)}
    if kind == "batch":
        return {"C": s["batch"].correlation(np.arange(case["points"]) * DT,
                                            DT).astype(np.complex64)}
    if kind == "grad":
        C, g1, g2, theta = s["model"].correlation_states_vjp(case["M"], s["psi1"], s["psi2"], DT,
                                                             1, s["cbar"])
        return {"C": C, "g1": g1, "g2": g2, "theta": theta}
    if kind == "heff":
        if case["mixed"]:
            binding.kernel_heff(s["L"], s["W"], s["R"], s["A"], s["out"], None, None, case["d"],
                                precision=PREC_C64_3XTF32, ws32=s["ws32"])
            return s["out"].to(torch.complex64)
        binding.kernel_heff(s["L"], s["W"], s["R"], s["A"], s["out"], s["X"], s["Y"], case["d"])
        return s["out"]
    if kind == "env":
        binding.kernel_env_left(s["L"], s["W"], s["bra"], s["ket"], s["out"], s["X"], s["Y"],
                                case["d"])
        return s["out"]
    if kind == "qr":
        binding.kernel_gauge_qr_blocked(s["Y"], s["Q"], s["R"], s["E"])
        return {"Q": s["Q"], "R": s["R"]}
    if kind == "bond":
        binding.kernel_bond_exp(s["L"], s["R"], s["C"], s["out"], TAU)
        return s["out"].to(torch.complex64)
    binding.kernel_site_exp_vjp(s["L"], s["W"], s["R"], s["A"], s["ybar"], TAU, *s["outs"],
                                case["d"])
    return s["outs"]


# ---------------------------------------------------------------------------------------------
# the bytes and operations a pass cannot do without
# ---------------------------------------------------------------------------------------------
def _heff_flops(Ml, D, Mr, Dl=DW, Dr=DW):
    return 8.0 * (Dl * Ml * Ml * D * Mr + Dr * Ml * D * Mr * Mr)


def _sweep(dims, M, krylov=6):
    """(bytes, flops) of one projector-splitting step: two passes over the sites, `krylov` H_eff
    products and one gauge QR each."""
    L = len(dims)
    left, right = [1.0], [1.0]
    for x in dims:
        left.append(left[-1] * x)
    for x in reversed(dims):
        right.append(right[-1] * x)
    Mb = [min(M, left[k], right[L - k]) for k in range(L + 1)]
    by = fl = 0.0
    for k in range(L):
        Ml, D, Mr = Mb[k], dims[k], Mb[k + 1]
        by += 2 * 16.0 * (2 * Ml * D * Mr + DW * (Ml * Ml + Mr * Mr))
        fl += 2 * (krylov * _heff_flops(Ml, D, Mr) + 8.0 * Ml * D * Mr * Mr)
    return by, fl


def work(case):
    kind = case["kind"]
    if kind in ("chain", "mixed", "batch"):
        if kind == "chain":
            n = [[4, case["nmax"] ** 2] * 3]
            M, steps = [144], round(1.0 / case["kT"] / 0.1) + 2 * (case["points"] - 1)
        elif kind == "mixed":
            n = [([4] + [x * x for x in [case["nmax"], 4][:case["modes"]]]) * case["N"]]
            M, steps = [case["M"]], 2 * (case["points"] - 1)
        else:
            n = [[4, case["nmax"] ** 2] * (case["N"] if i % 2 else 3)
                 for i in range(case["instances"])]
            M = [case["M"] + 8 * (i % 3) for i in range(case["instances"])]
            steps = 2 * (case["points"] - 1)
        both = [_sweep(a, b) for a, b in zip(n, M)]
        return {"bytes": steps * sum(b for b, _ in both), "flops": steps * sum(f for _, f in both)}
    if kind == "grad":
        by, fl = _sweep([4, case["nmax"] ** 2] * 3, case["M"])
        return {"bytes": 8 * by, "flops": 8 * fl}
    if kind == "qr":
        m, n = case["m"], case["n"]
        return {"bytes": 16.0 * (2 * m * n + n * n), "flops": 8.0 * m * n * n}
    if kind == "bond":
        M = case["M"]
        return {"bytes": 16.0 * (2 * DW * M * M + 2 * M * M), "flops": 6 * 16.0 * DW * M ** 3}
    Ml, Mr, D = case["Ml"], case["Mr"], case["d"] ** 2
    env = DW * (Ml * Ml + Mr * Mr)
    if kind == "heff":
        return {"bytes": 16.0 * (env + 2 * Ml * D * Mr), "flops": _heff_flops(Ml, D, Mr)}
    if kind == "env":
        return {"bytes": 16.0 * (env + 2 * Ml * D * Mr), "flops": _heff_flops(Ml, D, Mr)}
    # the two Krylov runs and the environment updates of eight quadrature nodes
    return {"bytes": 16.0 * (2 * env + 3 * Ml * D * Mr), "flops": 28 * _heff_flops(Ml, D, Mr)}


# ---------------------------------------------------------------------------------------------
# the same results in 64 bits by numpy
# ---------------------------------------------------------------------------------------------
def _heff(L, W, R, A, d):
    Ml, D, Mr = A.shape
    X = np.tensordot(L, A.reshape(Ml, d, d, Mr), axes=(2, 0))          # w a u t c
    Y = np.einsum("wvsu,wautc->vastc", W, X, optimize=True)
    return np.tensordot(Y, R, axes=([0, 4], [0, 2])).reshape(Ml, D, Mr)


def _env_left(L, W, bra, ket, d):
    """out[v, b, c] = sum conj(bra[a,s,t,b]) L[w,a,y] W[w,v,s,u] ket[y,u,t,c]"""
    Ml, _, Mr = ket.shape
    X = np.tensordot(L, ket.reshape(Ml, d, d, Mr), axes=(2, 0))
    Y = np.einsum("wvsu,wautc->vastc", W, X, optimize=True).reshape(DW, -1, ket.shape[2])
    return np.einsum("xb,vxc->vbc", bra.reshape(-1, bra.shape[2]).conj(), Y, optimize=True)


def _env_right(R, W, bra, ket, d):
    """out[w, a, y] = sum conj(bra[a,s,t,b]) R[v,b,c] W[w,v,s,u] ket[y,u,t,c]"""
    Ml, _, Mr = ket.shape
    X = np.tensordot(ket.reshape(Ml, d, d, Mr), R, axes=(3, 2))        # y u t v b
    Y = np.einsum("wvsu,yutvb->wystb", W, X, optimize=True)
    return np.einsum("ax,wyx->way", bra.reshape(bra.shape[0], -1).conj(),
                     Y.reshape(DW, Ml, -1), optimize=True)


def _taylor(op, v, tau):
    """exp(tau op) v for a small |tau| times the spectral radius, as four Taylor sub-steps."""
    out = v
    for _ in range(4):
        term, acc = out, out.copy()
        for q in range(1, 40):
            term = op(term) * (tau / 4 / q)
            acc = acc + term
            if np.linalg.norm(term) < 1e-18 * np.linalg.norm(acc):
                break
        out = acc
    return out


def _chain_exact(case, seed):
    """Exact diagonalisation of the one-carrier sector of the ring of three molecules."""
    om, g, V = _chain_parameters(case, seed)
    nm, beta = case["nmax"], 1.0 / case["kT"]
    b = np.diag(np.sqrt(np.arange(1, nm)), 1)
    eye = np.eye(nm)

    def local(op, i):
        ops = [op if k == i else eye for k in range(3)]
        return np.kron(np.kron(ops[0], ops[1]), ops[2])

    P = nm ** 3
    H = np.zeros((3 * P, 3 * P), dtype=complex)
    J = np.zeros_like(H)
    bath = sum(om[0] * local(b.T @ b, i) for i in range(3))
    for i in range(3):
        blk = slice(i * P, (i + 1) * P)
        H[blk, blk] += bath + g[0] * om[0] * local(b + b.T, i)
        nxt = slice((i + 1) % 3 * P, ((i + 1) % 3 + 1) * P)
        H[nxt, blk] += V * np.eye(P)
        H[blk, nxt] += V * np.eye(P)
        J[nxt, blk] += V / 1j * np.eye(P)
        J[blk, nxt] -= V / 1j * np.eye(P)
    e, U = np.linalg.eigh(H)
    p = np.exp(-beta * (e - e[0]))
    Z = p.sum()
    j2 = np.abs(U.conj().T @ J @ U) ** 2
    C = [np.sum((p / Z)[:, None] * np.exp(1j * t * (e[:, None] - e[None, :])) * j2)
         for t in np.arange(case["points"]) * DT]
    rho = (U * (p / Z)) @ U.conj().T
    sigma = np.trace(rho.reshape(3, P, 3, P), axis1=1, axis2=3).T     # <c+_i c_j>
    return {"C": np.array(C), "logz": float(np.log(Z) - beta * e[0]), "sigma": sigma}


def _qr_exact(case, seed):
    Y, E = _qr_inputs(case, seed)
    n, r = case["n"], case["rank"]
    Z = Y if E is None else np.concatenate([Y[:, :r], E[:, :n - r]], axis=1)
    Q, R = np.linalg.qr(Z)
    ph = np.diag(R) / np.abs(np.diag(R))
    Q = Q * ph
    S = np.triu(Q.conj().T @ Y)
    S[r:] = 0.0
    return {"Q": Q, "R": S}


def exact(case, seed):
    kind = case["kind"]
    if kind == "chain":
        return _chain_exact(case, seed)
    if kind in ("mixed", "batch", "grad"):
        return None           # no closed form below full bond dimension
    if kind == "qr":
        return _qr_exact(case, seed)
    if kind == "bond":
        L, R, C = _bond_inputs(case, seed)
        return _taylor(lambda X: np.matmul(np.matmul(L, X), np.swapaxes(R, 1, 2)).sum(0), C, TAU)
    L, W, R, A, rng = _heff_inputs(case, seed)
    d = case["d"]
    if kind == "heff":
        return _heff(L, W, R, A, d)
    if kind == "env":
        return _env_left(L, W, _site(rng, *A.shape), A, d)
    yb = _site(rng, *A.shape)

    def op(x):
        return _heff(L, W, R, x, d)

    tb = np.conj(TAU)
    x, w = np.polynomial.legendre.leggauss(12)
    Lb, Rb = np.zeros_like(L), np.zeros_like(R)
    for s, k in zip((x + 1) / 2, w / 2):
        a, c = _taylor(op, yb, (1 - s) * tb), _taylor(op, A, s * TAU)
        # Hbar = sum k tb a c^H: the cotangents of L and R are conjugated environment updates
        Lb += k * tb * np.conj(_env_right(R, W, a, c, d))
        Rb += k * tb * np.conj(_env_left(L, W, a, c, d))
    return [_taylor(op, yb, tb), Lb, Rb]
