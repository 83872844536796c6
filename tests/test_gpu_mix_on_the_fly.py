"""H_eff and the environment updates with the MPO mixing done where the operand is split into
digits: identity, real and complex entries, empty channels, odd extents, every operand layout."""
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


def site(rng, Dl, Dr, d, kind):
    W = np.zeros((Dl, Dr, d, d), dtype=complex)
    for c in range(min(Dl, Dr)):
        W[c, c] = np.eye(d)
    if kind != "identity":
        W[0, Dr - 1] = rng.standard_normal((d, d))
    if kind == "complex":
        W[Dl // 2, 0] += random_complex(rng, (d, d))
        W[Dl - 1, Dr - 1] = 1j * np.eye(d)[::-1]
    if kind == "empty" and Dr > 1:
        W[:, Dr // 2] = 0.0
        W[Dl // 2, :, 0] = 0.0
    return W


@pytest.mark.parametrize("kind", ["identity", "real", "complex", "empty"])
@pytest.mark.parametrize("Ml,Mr,d,Dl,Dr", [(1, 5, 2, 1, 3), (33, 17, 3, 4, 7), (40, 131, 2, 7, 7),
                                           (129, 31, 5, 3, 2)])
def test_heff_and_its_reverse(Ml, Mr, d, Dl, Dr, kind):
    """H_eff A, and through its reverse pass both environment updates (Lbar, Rbar), against numpy;
    sums of at most Dl Ml and Dr Mr d products, each rounded: 1e-12 of the largest entry."""
    from oracle import adjoint, tdvp
    from paper_2003_13245_gb300 import binding
    rng = np.random.default_rng(Ml * 7 + Mr)
    L, R = random_complex(rng, (Dl, Ml, Ml)), random_complex(rng, (Dr, Mr, Mr))
    A, yb = random_complex(rng, (Ml, d * d, Mr)), random_complex(rng, (Ml, d * d, Mr))
    W = site(rng, Dl, Dr, d, kind)
    ref = tdvp.heff(L, W, R, A, d)
    Ar, Lr, _, Rr = adjoint.heff_vjp(L, W, R, A, d, yb)
    X = torch.zeros(max(Dl, Dr) * A.size, dtype=torch.complex128, device="cuda")
    Y = torch.zeros_like(X)
    out = torch.zeros(A.shape, dtype=torch.complex128, device="cuda")
    binding.kernel_heff(dev(L), W, dev(R), dev(A), out, X, Y, d)
    Ab, Lb, Rb = torch.zeros_like(out), torch.zeros_like(dev(L)), torch.zeros_like(dev(R))
    binding.kernel_heff_vjp(dev(L), W, dev(R), dev(A), dev(yb), Ab, Lb, Rb, X, Y, d)
    for got, want in ((out, ref), (Ab, Ar), (Lb, Lr), (Rb, Rr)):
        assert np.abs(got.cpu().numpy() - want).max() <= 1e-12 * max(np.abs(want).max(), 1e-300)
