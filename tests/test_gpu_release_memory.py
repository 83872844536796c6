"""Callers of the kernel-level entry points without a model can give the pool's memory back."""
import numpy as np
import pytest

from tests.inputs import random_complex

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def test_pool_memory_goes_back_to_the_device():
    from paper_2003_13245_gb300 import binding
    from paper_2003_13245_gb300.build import build_library
    build_library()
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    rng = np.random.default_rng(1)
    M, d = 96, 6
    dev = lambda a: torch.from_numpy(np.ascontiguousarray(a)).to("cuda")   # noqa: E731
    L, R, A = (dev(random_complex(rng, (7, M, M))), dev(random_complex(rng, (7, M, M))),
               dev(random_complex(rng, (M, d * d, M))))
    W = random_complex(rng, (7, 7, d, d))
    X = torch.zeros(7 * A.numel(), dtype=torch.complex128, device="cuda")
    Y, out = torch.zeros_like(X), torch.zeros_like(A)
    binding.kernel_heff(L, W, R, A, out, X, Y, d)        # (loads the kernels)
    binding.release_memory()
    free0 = torch.cuda.mem_get_info()[0]
    binding.kernel_heff(L, W, R, A, out, X, Y, d)
    torch.cuda.synchronize()
    held = free0 - torch.cuda.mem_get_info()[0]
    assert held >= 32 << 20                              # the digits alone are 63 MB
    binding.release_memory()
    assert free0 - torch.cuda.mem_get_info()[0] <= 2 << 20
    binding.release_memory()                             # nothing left: still fine
