"""The reverse of the gauge QR where R's columns fall over many decades and the cotangent of R rises as
they fall: the terms of R Rbar^H then stay of one size although the rows of R and of Rbar do not, and
the solve with R carries each of them into Ybar."""
import numpy as np
import pytest

from tests.inputs import random_complex

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_2003_13245_gb300.build import build_library
    build_library()
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")


def dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).to("cuda")


def case(m, n, span):
    rng = np.random.default_rng(m * n)
    g = np.exp(-span * np.arange(n) / n)
    Q, _ = np.linalg.qr(random_complex(rng, (m, n)))
    U = np.eye(n) + 0.1 * np.triu(random_complex(rng, (n, n)), 1)
    Rbar = np.triu(random_complex(rng, (n, n))) / g
    Qbar = random_complex(rng, (m, n))
    return Q, U * g, Qbar, Rbar


@pytest.mark.parametrize("m,n", [(24, 24), (200, 40), (300, 130)])
@pytest.mark.parametrize("span", [3.0, 28.0])
def test_full_rank(m, n, span):
    """Columns of Ybar against numpy's.  Both sides round sums of at most m + 2 n terms and solve with a
    factor whose columns, scaled to one size, are well conditioned (off-diagonal entries around 0.1,
    inverse below 1e3 at n = 130): (m + 2 n) 2^-53 1e3 < 1e-10."""
    from oracle import adjoint
    from paper_2003_13245_gb300 import binding
    Q, R, Qbar, Rbar = case(m, n, span)
    Ybar = torch.zeros((m, n), dtype=torch.complex128, device="cuda")
    binding.kernel_qr_vjp(dev(Q), dev(R), dev(Qbar), dev(Rbar), Ybar)
    ref = adjoint.qr_vjp(Q, R, Qbar, Rbar)
    err = np.linalg.norm(Ybar.cpu().numpy() - ref, axis=0)
    assert np.all(err <= 1e-10 * np.linalg.norm(ref, axis=0))


@pytest.mark.parametrize("m,n,rank", [(60, 24, 20), (300, 60, 40)])
def test_completed(m, n, rank):
    """The same with completed columns, whose rows of R are zero."""
    from oracle import adjoint
    from paper_2003_13245_gb300 import binding
    Q, R, Qbar, Rbar = case(m, n, 28.0)
    acc = np.zeros(n, dtype=int)
    acc[:rank] = 1
    R = R * acc[:, None]
    X = Q[:, rank:] + 0.1 * Q[:, :rank] @ random_complex(np.random.default_rng(1), (rank, n - rank))
    Ybar = torch.zeros((m, n), dtype=torch.complex128, device="cuda")
    Xbar = torch.zeros((m, n - rank), dtype=torch.complex128, device="cuda")
    binding.kernel_qr_vjp_completed(acc, dev(Q), dev(R), dev(X), dev(Qbar), dev(Rbar), Ybar, Xbar)
    ref, xref = adjoint.qr_vjp_completed(Q, R, Qbar, Rbar, X)
    for got, want in ((Ybar, ref), (Xbar, xref)):
        err = np.linalg.norm(got.cpu().numpy() - want, axis=0)
        assert np.all(err <= 1e-10 * np.linalg.norm(want, axis=0))
