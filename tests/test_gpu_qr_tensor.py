"""The tensor-core gauge QR at the edges of its tiling (blocks of 16 columns, row slices of 32 to
128 rows per CTA, tiles of 128 accepted vectors, at most 256 columns), with the column layouts the sweep uses, rank deficiency
with candidates in and out of the span, and columns near the rank threshold."""
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


def run(Y, E=None):
    from paper_2003_13245_gb300 import binding
    m, n = Y.shape
    Q = torch.full((m, n), float("nan"), dtype=torch.complex128, device="cuda")
    R = torch.full((n, n), float("nan"), dtype=torch.complex128, device="cuda")
    binding.kernel_gauge_qr_blocked(dev(Y), Q, R, dev(E) if E is not None else None)
    return Q.cpu().numpy(), R.cpu().numpy()


@pytest.mark.parametrize("m,n", [(1, 1), (2, 2), (16, 16), (17, 17), (33, 15), (31, 31), (65, 32),
                                 (128, 128), (129, 127), (1000, 33), (4097, 113), (19000, 100), (129, 129), (300, 144),
                                 (2000, 256), (256, 255)])
def test_full_rank(m, n):
    """Columns of very different size, mixed: Q has orthonormal columns, QR = Y to rounding and R
    is upper triangular with a positive diagonal, which fixes both uniquely.  Both products round
    sums of at most m terms: 1e-13 for the sizes here (m 2^-53 = 2e-12 only in the worst case)."""
    rng = np.random.default_rng(m + n)
    Y = random_complex(rng, (m, n)) * np.exp(-12.0 * rng.random(n))
    Q, R = run(Y)
    assert np.abs(Q.conj().T @ Q - np.eye(n)).max() < 1e-13
    assert np.abs(Q @ R - Y).max() < 1e-13 * np.abs(Y).max()
    assert np.abs(np.tril(R, -1)).max() == 0.0
    assert np.all(np.diag(R).real > 0) and np.abs(np.diag(R).imag).max() == 0.0


@pytest.mark.parametrize("m,n,rank", [(20, 16, 1), (40, 17, 16), (300, 48, 20), (2000, 128, 65), (700, 200, 30), (600, 256, 140),
                                      (513, 96, 0)])
def test_completion_follows_the_candidates(m, n, rank):
    """Columns beyond the rank are skipped (their residual is rounding); the skipped positions are
    filled in order by the candidates that are not in the span: here every other candidate is a
    combination of the accepted columns and the ones between are random, so the completed columns
    span exactly the random ones, in order."""
    rng = np.random.default_rng(m * 3 + n)
    B = random_complex(rng, (m, max(rank, 1)))
    Y = B @ random_complex(rng, (max(rank, 1), n)) if rank else np.zeros((m, n), complex)
    free = random_complex(rng, (m, n - rank))
    E = np.zeros((m, 2 * (n - rank)), complex)
    E[:, 1::2] = free
    if rank:
        E[:, 0::2] = B @ random_complex(rng, (rank, n - rank))
    Q, R = run(Y, E)
    acc = np.abs(np.diag(R)) > 0
    assert acc.sum() == rank and acc[:rank].all()
    assert np.abs(Q.conj().T @ Q - np.eye(n)).max() < 1e-12
    if rank:
        assert np.abs(Q @ R - Y).max() < 1e-12 * np.abs(Y).max()
    assert not R[rank:].any()
    # Gram-Schmidt of [accepted | free] in order, by numpy's QR with a positive diagonal
    ref, tri = np.linalg.qr(np.concatenate([Q[:, :rank], free], axis=1))
    ref = ref * (np.diag(tri) / np.abs(np.diag(tri)))
    assert np.abs(Q[:, rank:] - ref[:, rank:]).max() < 1e-10


def test_unit_vectors_complete_an_empty_span():
    """No candidates: unit vectors fill the positions in order."""
    Q, R = run(np.zeros((50, 20), complex))
    assert not R.any()
    assert np.abs(Q - np.eye(50)[:, :20]).max() < 1e-14


def test_sparse_columns():
    """Unit-vector columns (entries of 1 among zeros): a row's scale grows with later columns."""
    rng = np.random.default_rng(3)
    m, n = 400, 64
    Y = np.zeros((m, n), complex)
    Y[rng.permutation(m)[:n], np.arange(n)] = 2.0 ** rng.integers(-20, 20, n)
    Y[:, 40:] += 1e-3 * random_complex(rng, (m, n - 40))
    Q, R = run(Y)
    assert np.abs(Q.conj().T @ Q - np.eye(n)).max() < 1e-13
    assert np.abs(Q @ R - Y).max() < 1e-13 * np.abs(Y).max()


def test_columns_near_the_rank_threshold():
    """Residuals a little above 1e-12 ||Y|| are taken (and orthonormal), a little below skipped."""
    rng = np.random.default_rng(4)
    m, n = 600, 24
    U, _ = np.linalg.qr(random_complex(rng, (m, n)))
    Y = np.zeros((m, n), complex)
    Y[:, :16] = U[:, :16]
    norm = 4.0                                  # ||Y||_F of the 16 orthonormal columns
    for k in range(16, n):
        Y[:, k] = U[:, k - 16] + U[:, k] * norm * (4e-12 if k % 2 else 2.5e-13)
    scale = np.sqrt(np.linalg.norm(Y) ** 2) / norm
    assert 1.0 < scale < 1.3                    # the threshold lies between the two residuals
    Q, R = run(Y, random_complex(rng, (m, 8)))
    acc = np.abs(np.diag(R)) > 0
    assert acc[:16].all() and acc[17::2].all() and not acc[16::2].any()
    assert np.abs(Q.conj().T @ Q - np.eye(n)).max() < 1e-12
    assert np.abs(Q @ R - Y).max() < 1e-11


@pytest.mark.parametrize("bad", [np.nan, np.inf])
def test_nonfinite_input_takes_nothing(bad):
    """The norm of Y is not finite: no column passes the threshold, as before; the candidates fill
    every position and a candidate that is not finite is never taken."""
    rng = np.random.default_rng(5)
    Y = random_complex(rng, (100, 20))
    Y[3, 4] = bad
    E = random_complex(rng, (100, 30))
    E[7, 2] = bad
    Q, R = run(Y, E)
    assert not R.any()
    assert np.abs(Q.conj().T @ Q - np.eye(20)).max() < 1e-13
    ref, tri = np.linalg.qr(np.delete(E, 2, axis=1)[:, :20])
    ref = ref * (np.diag(tri) / np.abs(np.diag(tri)))
    assert np.abs(Q - ref).max() < 1e-10


@pytest.mark.parametrize("span", [0.5, 3.0, 9.0, 20.0])
@pytest.mark.parametrize("m,n", [(16, 16), (40, 17), (257, 40), (1200, 130)])
def test_graded(m, n, span):
    """Singular values from 1 to e^-span, mixed over the columns: what is left of a column inside its
    block lies above a quarter, above 1e-8 (a second round) and below it (the next block).  Entries
    of both products round sums of rows and columns of norm <= 1: 1e-13 as in test_full_rank."""
    rng = np.random.default_rng(m + n)
    U, _ = np.linalg.qr(random_complex(rng, (n, n)))
    Y = np.linalg.qr(random_complex(rng, (m, n)))[0] @ (np.exp(-span * np.arange(n) / n)[:, None] * U)
    Q, R = run(Y)
    assert np.abs(Q.conj().T @ Q - np.eye(n)).max() < 1e-13
    assert np.abs(Q @ R - Y).max() < 1e-13 * np.linalg.norm(Y, axis=0).max()
    assert np.abs(np.tril(R, -1)).max() == 0.0
    assert np.all(np.diag(R).real > 0) and np.abs(np.diag(R).imag).max() == 0.0
