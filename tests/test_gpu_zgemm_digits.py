"""The FP64 contractions by digit products (tensor cores) at the edges of their tiles (128 x 32
outputs, 16-deep k steps, 128-deep chunks), through the H_eff product of a site without physical
levels, out = sum_w,v L_w W[w,v] A R_v^T."""
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


def heff(L, W, R, A):
    from paper_2003_13245_gb300 import binding
    Ml, Mr = A.shape
    n = max(L.shape[0], R.shape[0]) * Ml * Mr
    X = torch.zeros(n, dtype=torch.complex128, device="cuda")
    Y = torch.zeros_like(X)
    out = torch.zeros((Ml, 1, Mr), dtype=torch.complex128, device="cuda")
    binding.kernel_heff(dev(L), W, dev(R), dev(A.reshape(Ml, 1, Mr)), out, X, Y, 1)
    return out.cpu().numpy()[:, 0, :]


SHAPES = [(1, 2, 1, 1), (2, 1, 1, 2), (15, 33, 2, 3), (16, 32, 1, 1), (17, 31, 3, 1),
          (127, 129, 1, 2), (128, 128, 2, 1), (129, 127, 1, 1), (257, 40, 7, 7), (5, 300, 2, 7)]


@pytest.mark.parametrize("Ml,Mr,Dl,Dr", SHAPES)
def test_integers_are_exact(Ml, Mr, Dl, Dr):
    """Integer entries below 2^7 with sums below 2^53: every digit product and sum is an integer
    that the scheme holds exactly, so the result equals the integer product bit for bit."""
    rng = np.random.default_rng(Ml * 1000 + Mr)

    def ints(shape):
        return rng.integers(-100, 101, shape) + 1j * rng.integers(-100, 101, shape)

    L, R, A = ints((Dl, Ml, Ml)), ints((Dr, Mr, Mr)), ints((Ml, Mr))
    W = rng.integers(-4, 5, (Dl, Dr, 1, 1)) + 0j
    X = np.einsum("way,yc->wac", L, A)
    Y = np.einsum("wv,wac->vac", W[:, :, 0, 0], X)
    ref = np.einsum("vac,vbc->ab", Y, R)
    assert np.abs(ref).max() < 2.0 ** 53
    assert np.array_equal(heff(L, W, R, A), ref)


@pytest.mark.parametrize("Ml,Mr,Dl,Dr", [(400, 530, 1, 1), (513, 561, 1, 1), (497, 640, 1, 1),
                                         (260, 257, 7, 2)])
def test_tile_widths(Ml, Mr, Dl, Dr):
    """The 32-column tiles are taken where 16-column ones would be more than the SMs: sizes on both
    sides of that line, with 1, 2, 17 and 32 columns in the last tile."""
    test_integers_are_exact(Ml, Mr, Dl, Dr)


@pytest.mark.parametrize("Ml,Mr,Dl,Dr", SHAPES)
def test_matches_numpy(Ml, Mr, Dl, Dr):
    """Rows and columns of very different size.  Both sides round sums of Ml and Dr Mr products:
    an entry is off by at most (Ml + Dr Mr + 8) 2^-52 of the sum of the absolute products (numpy)
    plus as much of the row and column maxima (the digits' common scale)."""
    rng = np.random.default_rng(Ml * 1000 + Mr + 1)
    L, R = random_complex(rng, (Dl, Ml, Ml)), random_complex(rng, (Dr, Mr, Mr))
    A = random_complex(rng, (Ml, Mr)) * np.exp(-9.0 * rng.random((Ml, 1)))
    L *= np.exp(-9.0 * rng.random((1, Ml, 1)))
    R *= np.exp(9.0 * rng.random((1, Mr, 1)))
    W = random_complex(rng, (Dl, Dr, 1, 1))
    X = np.einsum("way,yc->wac", L, A)
    Y = np.einsum("wv,wac->vac", W[:, :, 0, 0], X)
    ref = np.einsum("vac,vbc->ab", Y, R)
    # the same chain with every factor replaced by its row or column maximum
    Xm = np.abs(L).max(2)[:, :, None] * np.abs(A).max(0)[None, None, :] * Ml
    Ym = np.einsum("wv,wac->vac", np.abs(W[:, :, 0, 0]), Xm)
    big = np.einsum("va,vb->ab", Ym.max(2), np.abs(R).max(2)) * Mr
    assert np.all(np.abs(heff(L, W, R, A) - ref) <= 2 * (Ml + Dr * Mr + 8) * 2.0 ** -52 * big)


@pytest.mark.parametrize("p,q", [(500, -300), (-400, -400), (0, -1000), (300, 300)])
def test_powers_of_two_scale_exactly(p, q):
    """The digits are relative to the largest entry of a row, so scaling an operand by a power
    of two scales the result by it, bit for bit, while nothing leaves the normal range."""
    rng = np.random.default_rng(5)
    L, R, A = (random_complex(rng, (2, 40, 40)), random_complex(rng, (3, 50, 50)),
               random_complex(rng, (40, 50)))
    W = random_complex(rng, (2, 3, 1, 1))
    ref = heff(L, W, R, A)
    got = heff(L * 2.0 ** p, W, R, A * 2.0 ** q)
    assert np.array_equal(got, ref * 2.0 ** (p + q))


@pytest.mark.parametrize("bad", [np.inf, -np.inf, np.nan])
def test_nonfinite_entries_stay_visible(bad):
    """An Inf or NaN entry of A reaches its own column of X and so, through a dense R, the rows it
    contributes to: nothing finite may come out where the FP64 sum has a non-finite term."""
    rng = np.random.default_rng(6)
    L, R, A = (random_complex(rng, (1, 140, 140)), random_complex(rng, (1, 36, 36)),
               random_complex(rng, (140, 36)))
    W = np.ones((1, 1, 1, 1), dtype=complex)
    A[131, 7] = bad
    assert not np.isfinite(heff(L, W, R, A)).any()
    # an untouched row: L does not couple row 3 to the entry, but 0 * Inf is NaN in the sum too
    R0 = R.copy()
    R0[0, :, 7] = 0.0
    assert not np.isfinite(heff(L, W, R0, A)).any()


def test_zero_rows_and_subnormals():
    rng = np.random.default_rng(7)
    L, R, A = (random_complex(rng, (1, 33, 33)), random_complex(rng, (1, 17, 17)),
               random_complex(rng, (33, 17)))
    W = np.ones((1, 1, 1, 1), dtype=complex)
    L[0, 5] = 0.0
    got = heff(L, W, R, A)
    assert not got[5].any() and np.isfinite(got).all()
    # entries below the normal range: the result is subnormal too and keeps absolute accuracy
    tiny = heff(L * 2.0 ** -600, W, R * 2.0 ** -450, A)
    assert np.abs(tiny * 2.0 ** 1000 - got * 2.0 ** -50).max() <= 2.0 ** -1073 * 2.0 ** 1000
