"""The Krylov dimension at which an exponential stops is decided by the FP64 estimate
beta_{k+1} |(exp(tau T_k) e_1)_k| < tol, whatever is left out before it: the count equals that of
a plain Lanczos run with the estimate evaluated at every step."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_2003_13245_gb300.build import build_library
    build_library()
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")


def dimension(H, v, tau, tol, kmax):
    """(k, margin): the first k whose estimate is below tol and how far (as a factor) the estimates
    around it stay away from tol."""
    q = [v / np.linalg.norm(v)]
    al, be, est = [], [], []
    for j in range(min(kmax, len(v))):
        w = H @ q[-1]
        al.append((q[-1].conj() @ w).real)
        for _ in range(2):
            for x in q:
                w = w - x * (x.conj() @ w)
        b = np.linalg.norm(w)
        T = np.diag(al) + np.diag(be, 1) + np.diag(be, -1)
        e, U = np.linalg.eigh(T)
        y = U @ (np.exp(tau * e) * U[0])
        est.append(b * abs(y[-1]))
        if est[-1] < tol or b <= 1e-12 * np.abs(T).max():
            break
        be.append(b)
        q.append(w / b)
    near = [max(x / tol, tol / x) if x > 0 else np.inf for x in est[-2:]]
    return len(al), min(near)


@pytest.mark.parametrize("n", [17, 64, 300])
@pytest.mark.parametrize("tau", [-0.01j, -0.3j, -2.0j, -0.1, 0.2, 0.05 - 0.2j])
@pytest.mark.parametrize("tol", [1e-12, 1e-7, 1e-3])
def test_dimension_matches_plain_lanczos(n, tau, tol):
    from paper_2003_13245_gb300 import binding
    rng = np.random.default_rng(n)
    A = rng.standard_normal((n, n)) + 1j * rng.standard_normal((n, n))
    H = (A + A.conj().T) / np.sqrt(n) + 7.0 * np.eye(n)
    v = rng.standard_normal(n) + 1j * rng.standard_normal(n)
    k, margin = dimension(H, v, tau, tol, 32)
    out = torch.empty(n, dtype=torch.complex128, device="cuda")
    got = binding.kernel_krylov_dense(torch.from_numpy(H).cuda(), torch.from_numpy(v).cuda(), out,
                                      tau, tol=tol, kmax=32)
    # (the eigendecomposition knows small entries to 1e-16 of the largest: skip where tol is there)
    if margin > 1.05 and tol > 1e-13 * np.exp(abs(np.real(tau)) * 12):
        assert got == k
    w = np.linalg.eigh(H)
    ref = w[1] @ (np.exp(tau * w[0]) * (w[1].conj().T @ v))
    assert np.abs(out.cpu().numpy() - ref).max() <= 20 * max(tol, 1e-13) * np.linalg.norm(ref)
