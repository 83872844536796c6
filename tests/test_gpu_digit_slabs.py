"""FP64 contractions whose digits do not fit the workspace: slabs of the batches, of the rows of either
operand, and FP64 FMAs where not even one tile of each fits, with and without the MPO mixing on the
fly.  Integer entries with sums below 2^53 make every route exact, so all give the same bits."""
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


def dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).to("cuda")


def ints(rng, shape, hi=30):
    return rng.integers(-hi, hi + 1, shape) + 1j * rng.integers(-hi, hi + 1, shape)


def site(rng, Dl, Dr, d):
    W = rng.integers(-2, 3, (Dl, Dr, d, d)) + 0j
    W[0, 0] = np.eye(d)
    W[Dl - 1, :, 0] = 0.0
    return W


# a tile of a 128-row operand takes 57,344 bytes per 16 k (and 512 per 128 k), one of the other operand a
# quarter or an eighth of that.  H_eff: K = 150 (10 steps) for 450 x 560, then K = 140 (9 steps) summed
# over 4 channels for 600 x 140; environment: K = 150 again, then K = 600 (38 steps) in 4 batches.
WORK = [0, 300_000, 700_000, 1_000_000, 2_000_000, 2_900_000, 4_000_000, 6_500_000, 12_000_000,
        1 << 30]


@pytest.mark.parametrize("work", WORK)
def test_heff(work):
    from paper_2003_13245_gb300 import binding
    rng = np.random.default_rng(1)
    Ml, Mr, d, Dl, Dr = 150, 140, 2, 3, 4
    L, R, A = ints(rng, (Dl, Ml, Ml)), ints(rng, (Dr, Mr, Mr)), ints(rng, (Ml, d, d, Mr))
    W = site(rng, Dl, Dr, d)
    X = np.einsum("way,yutc->wautc", L, A, optimize=True)
    Y = np.einsum("wvsu,wautc->vastc", W, X, optimize=True)
    ref = np.einsum("vastc,vbc->astb", Y, R, optimize=True)
    assert np.abs(ref).max() < 2.0 ** 52
    out = torch.full((Ml, d * d, Mr), float("nan"), dtype=torch.complex128, device="cuda")
    x = torch.zeros(max(Dl, Dr) * A.size, dtype=torch.complex128, device="cuda")
    binding.kernel_heff_work(dev(L), W, dev(R), dev(A.reshape(Ml, d * d, Mr)), out, x,
                             torch.zeros_like(x), d, work)
    assert np.array_equal(out.cpu().numpy(), ref.reshape(Ml, d * d, Mr))


@pytest.mark.parametrize("work", WORK)
def test_env_left(work):
    from paper_2003_13245_gb300 import binding
    rng = np.random.default_rng(2)
    Ml, Mr1, Mr2, d, Dl, Dr = 150, 290, 140, 2, 3, 4
    L, bra, ket = ints(rng, (Dl, Ml, Ml)), ints(rng, (Ml, d, d, Mr1)), ints(rng, (Ml, d, d, Mr2))
    W = site(rng, Dl, Dr, d)
    X = np.einsum("way,yutc->wautc", L, ket, optimize=True)
    Y = np.einsum("wvsu,wautc->vastc", W, X, optimize=True)
    ref = np.einsum("astb,vastc->vbc", bra.conj(), Y, optimize=True)
    assert np.abs(ref).max() < 2.0 ** 52
    out = torch.full((Dr, Mr1, Mr2), float("nan"), dtype=torch.complex128, device="cuda")
    x = torch.zeros(max(Dl, Dr) * ket.size, dtype=torch.complex128, device="cuda")
    binding.kernel_env_left_work(dev(L), W, dev(bra.reshape(Ml, d * d, Mr1)),
                                 dev(ket.reshape(Ml, d * d, Mr2)), out, x, torch.zeros_like(x), d,
                                 work)
    assert np.array_equal(out.cpu().numpy(), ref)


def test_no_workspace_means_fmas():
    """Without a workspace the error is relative to the sum of the absolute products: opposite
    gradings over 2^60, which the digits cannot hold, stay exact to rounding."""
    from paper_2003_13245_gb300 import binding
    rng = np.random.default_rng(3)
    m, d = 64, 2
    g = 2.0 ** -(60.0 * np.arange(m) / m)
    L = (rng.standard_normal((1, m, m)) + 1j * rng.standard_normal((1, m, m))) * g
    A = (rng.standard_normal((m, d * d, 1)) + 1j * rng.standard_normal((m, d * d, 1))) * g[::-1, None, None]
    out = torch.zeros((m, d * d, 1), dtype=torch.complex128, device="cuda")
    x = torch.zeros(m * d * d, dtype=torch.complex128, device="cuda")
    one = np.ones((1, 1, 1), complex)
    binding.kernel_heff_work(dev(L), np.eye(d).reshape(1, 1, d, d) + 0j, dev(one), dev(A), out, x,
                             torch.zeros_like(x), d, 0)
    scale = np.abs(L[0]) @ np.abs(A[:, :, 0])
    err = np.abs(out.cpu().numpy()[:, :, 0] - L[0] @ A[:, :, 0])
    assert np.all(err <= 4 * m * 2.0 ** -53 * scale)     # two sums of 2 m rounded products


def test_many_channels():
    """More pairs of output channel and level than a grid has rows (65535)."""
    from paper_2003_13245_gb300 import binding
    rng = np.random.default_rng(4)
    d, Dr = 2, 33000
    L, R, A = ints(rng, (1, 1, 1)), ints(rng, (Dr, 1, 1)), ints(rng, (1, d, d, 1))
    W = rng.integers(-2, 3, (1, Dr, d, d)) + 0j
    ref = np.einsum("w,wvsu,ut,v->st", L[:, 0, 0], W, A[0, :, :, 0], R[:, 0, 0], optimize=True)
    out = torch.zeros((1, d * d, 1), dtype=torch.complex128, device="cuda")
    x = torch.zeros(Dr * d * d, dtype=torch.complex128, device="cuda")
    binding.kernel_heff_work(dev(L), W, dev(R), dev(A.reshape(1, d * d, 1)), out, x,
                             torch.zeros_like(x), d, 0)
    assert np.array_equal(out.cpu().numpy()[0, :, 0], ref.reshape(-1))


@pytest.mark.parametrize("bad", [np.inf, -np.inf, np.nan, complex(0.0, np.inf)])
@pytest.mark.parametrize("where", ["L", "A", "R"])
def test_nonfinite_entries_as_with_fmas(where, bad):
    """An Inf or NaN of an operand reaches the same entries on both routes, and as NaN on both: the FMA
    sums of a complex product mix re and im, and alpha = 1 + 0 i multiplies both parts."""
    from paper_2003_13245_gb300 import binding
    rng = np.random.default_rng(5)
    m, n, d = 140, 30, 2
    ops = {"L": ints(rng, (1, m, m)), "R": ints(rng, (1, n, n)), "A": ints(rng, (m, d * d, n))}
    ops[where][(0, 7, 3) if where != "A" else (131, 2, 7)] = bad
    W = np.eye(d).reshape(1, 1, d, d) + 0j
    got = []
    for work in (0, 1 << 30):
        out = torch.zeros((m, d * d, n), dtype=torch.complex128, device="cuda")
        x = torch.zeros(ops["A"].size, dtype=torch.complex128, device="cuda")
        binding.kernel_heff_work(dev(ops["L"]), W, dev(ops["R"]), dev(ops["A"]), out, x,
                                 torch.zeros_like(x), d, work)
        got.append(out.cpu().numpy())
    assert not np.isfinite(got[0]).all()
    for part in (np.real, np.imag):
        assert np.array_equal(part(got[0]), part(got[1]), equal_nan=True)
