"""The bond exponential's FP32 copy of a Krylov vector is scaled by a power of two taken from its
norm: a bond matrix scaled by a power of two far outside the FP32 range gives the same result,
scaled, bit for bit."""
import numpy as np
import pytest

from tests.inputs import random_complex

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("M", [1, 2, 33, 64])
@pytest.mark.parametrize("p", [-400, -64, 130, 400])
def test_scaled_by_a_power_of_two(M, p):
    from paper_2003_13245_gb300 import binding
    from paper_2003_13245_gb300.build import build_library
    build_library()
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    rng = np.random.default_rng(M)

    def herm(D):
        X = random_complex(rng, (D, M, M))
        return (X + np.conj(np.swapaxes(X, 1, 2))) / (4.0 * np.sqrt(M))

    L, R, C = herm(2), herm(2), random_complex(rng, (M, M))

    def run(c):
        out = torch.zeros((M, M), dtype=torch.complex128, device="cuda")
        binding.kernel_bond_exp(*(torch.from_numpy(x).to("cuda") for x in (L, R, c)), out, -0.05j)
        return out.cpu().numpy()

    ref = run(C)
    assert np.isfinite(ref).all() and np.abs(ref).max() > 0
    assert np.array_equal(run(C * 2.0 ** p), ref * 2.0 ** p)
