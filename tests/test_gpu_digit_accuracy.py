"""What the FP64 contractions by digit products guarantee, against exact integer arithmetic.  With one
channel, R = 1 and identity operators on d levels the H_eff product is out = L A for A of d^2 columns
(the mixing and the product with R are exact).  Every entry is an integer times 2^-S, so the exact
product is a product of Python integers.

The bound of one component of an entry, from the scheme alone, over chunks c of 128 k, 2^EA and 2^EB
the powers of two above the largest component of the row of L and the column of A in the chunk:
 operands    sum_k 2^(EA-56) |b|_1 + 2^(EB-56) |a|_1       (rounded to 56 bits below 2^E)
 products    2^-60 per k of 2^(EA+EB)                      (digit pairs below level 7)
 rounding    n 2^-53 sum_c |chunk sum|, n chunks           (each chunk once, and their sum)
with 1 % on top for products of these errors.  Level sums stay below 2^24 for such entries (they are
random), so nothing is lost in their FP32 accumulation."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

S = 120                    # entries are integers times 2^-S


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_2003_13245_gb300.build import build_library
    build_library()
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")


def dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).to("cuda")


def product(L, A):
    """L A on the device for A of d^2 columns."""
    from paper_2003_13245_gb300 import binding
    m, n = A.shape
    d = int(round(n ** 0.5))
    X = torch.zeros(m * n, dtype=torch.complex128, device="cuda")
    Y = torch.zeros_like(X)
    out = torch.zeros((m, n, 1), dtype=torch.complex128, device="cuda")
    W = np.eye(d).reshape(1, 1, d, d) + 0j
    binding.kernel_heff(dev(L.reshape(1, m, m)), W, dev(np.ones((1, 1, 1), complex)),
                        dev(A.reshape(m, n, 1)), out, X, Y, d)
    return out.cpu().numpy()[:, :, 0]


def full_mantissas(rng, shape, down):
    """Doubles with all 53 bits in use and exponents from -down to 0, and both signs."""
    m = rng.integers(1 << 52, 1 << 53, shape).astype(np.float64)
    return np.ldexp(m * rng.choice([-1.0, 1.0], shape), -53 - rng.integers(0, down + 1, shape))


def as_ints(x):
    """x 2^S as Python integers."""
    m, e = np.frexp(x)
    m = np.ldexp(m, 53).astype(np.int64)
    f = np.frompyfunc(lambda a, b: int(a) << int(b), 2, 1)
    return f(m, e - 53 + S)


def parts(L, A):
    return [as_ints(x) for x in (L.real, L.imag, A.real, A.imag)]


def check(L, A, got, rows):
    """Every entry of the given rows of got = L A, against the bound of the module's docstring."""
    L, got = L[rows], got[rows]
    K = L.shape[1]
    n = (K + 127) // 128
    lr, li, ar, ai = parts(L, A)
    re, im = lr.dot(ar) - li.dot(ai), lr.dot(ai) + li.dot(ar)
    absre = np.zeros(got.shape)
    absim = np.zeros(got.shape)
    tol = np.zeros(got.shape)
    for c in range(n):
        k = slice(128 * c, min(K, 128 * c + 128))
        cr = lr[:, k].dot(ar[k]) - li[:, k].dot(ai[k])
        ci = lr[:, k].dot(ai[k]) + li[:, k].dot(ar[k])
        absre += np.abs(cr / 4.0 ** S).astype(float)
        absim += np.abs(ci / 4.0 ** S).astype(float)
        a1 = np.abs(L[:, k].real) + np.abs(L[:, k].imag)
        b1 = np.abs(A[k].real) + np.abs(A[k].imag)
        ea = np.frexp(np.maximum(np.abs(L[:, k].real), np.abs(L[:, k].imag)).max(1))[1]
        eb = np.frexp(np.maximum(np.abs(A[k].real), np.abs(A[k].imag)).max(0))[1]
        pa, pb = np.ldexp(1.0, ea)[:, None], np.ldexp(1.0, eb)[None, :]
        tol += 2.0 ** -56 * (pa * b1.sum(0)[None, :] + pb * a1.sum(1)[:, None])
        tol += 2.0 ** -60 * a1.shape[1] * pa * pb
    for have, want, mag in ((got.real, re, absre), (got.imag, im, absim)):
        err = np.abs((as_ints2(have) - want) / 4.0 ** S).astype(float)
        assert np.all(err <= 1.01 * (tol + n * 2.0 ** -53 * mag))


def as_ints2(x):
    """x 4^S as Python integers (x a sum of products)."""
    m, e = np.frexp(x)
    m = np.ldexp(m, 53).astype(np.int64)
    f = np.frompyfunc(lambda a, b: int(a) << int(b) if b >= 0 else int(a) >> int(-b), 2, 1)
    return f(m, e - 53 + 2 * S)


# 16-column tiles, one chunk and its remainder, several chunks; (900, 8): 32-column tiles
@pytest.mark.parametrize("m,d", [(16, 4), (17, 3), (128, 8), (129, 8), (300, 8), (900, 8)])
@pytest.mark.parametrize("down", [2, 20])
def test_full_mantissas(m, d, down):
    """All seven digits of every entry, over several k steps and chunks.  Exponents over three
    binades (down = 2) leave the operands exact; over twenty, the small entries are rounded."""
    rng = np.random.default_rng(m * 100 + down)
    L = full_mantissas(rng, (m, m), down) + 1j * full_mantissas(rng, (m, m), down)
    A = full_mantissas(rng, (m, d * d), down) + 1j * full_mantissas(rng, (m, d * d), down)
    check(L, A, product(L, A), np.unique(np.r_[0, m // 2, m - 1, rng.integers(0, m, 29)]))


@pytest.mark.parametrize("span", [9, 28, 45])
def test_opposite_grading(span):
    """Rows of L fall by 2^-span along k while the columns of A rise: every term of the sum is about
    2^-span.  The error is relative to the largest entries of a row and a column, not to the terms."""
    m, d = 128, 4
    rng = np.random.default_rng(span)
    g = np.ldexp(1.0, -(span * np.arange(m) // (m - 1)))
    L = (full_mantissas(rng, (m, m), 0) + 1j * full_mantissas(rng, (m, m), 0)) * g[None, :]
    A = (full_mantissas(rng, (m, d * d), 0) + 1j * full_mantissas(rng, (m, d * d), 0)) * g[::-1, None]
    check(L, A, product(L, A), np.arange(0, m, 5))


@pytest.mark.parametrize("m", [64, 128, 256])
def test_aligned_digits(m):
    """Every digit near its largest value and every product of one sign: the sums of levels 4 to 7
    (5, 6, 7 and 6 digit pairs) pass 2^24 from about 80 k on, where FP32 holds only even numbers.  A
    chunk then loses at most two units of level 4, 2^-46 2^(EA+EB), in each of the at most 92 steps of
    8 k that follow: below 2^-39 2^(EA+EB), and as every component is above 0.99 2^(E-1), below 2^-44
    of the sum of the absolute products (with the rounding of the result)."""
    v = float(0x7f7f7f7f7f7f7c) * 2.0 ** -56
    L = np.full((m, m), v + 1j * v)
    A = np.full((m, 16), v - 1j * v)
    got = product(L, A)
    want = 2 * m * int(np.ldexp(v, 56)) ** 2
    err = max(abs(int(np.ldexp(x, 60)) * 2 ** 52 - want) for x in got.real.ravel())
    assert err <= 2.0 ** -44 * want
    assert np.abs(got.imag).max() <= 2.0 ** -44 * 2 * m * v * v
