"""GPU: tensor-core products of graded operands, where the largest entries of a row and of a
column over a range of 512 summands lie in different places: a row that falls while a column
rises, rows and columns that peak in different blocks, a Gram product of localised columns.

Bar per entry, as for digits of 49 bits aligned over blocks of 64 summands: 2^-44 of
(largest of the row) x (largest of the column) in each block, for each of its summands, and
2^-52 K of the sum of |products| for the sums of the ranges and of the reference."""
import numpy as np
import pytest

from tests.test_gpu_split import _run

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    from paper_1702_00339_gb300 import build, fock
    build.build()
    c = fock.Context(0)
    yield c
    c.close()


def _check(C, A, B):
    K = A.shape[1]
    bar = 2.0 ** -52 * K * (np.abs(A) @ np.abs(B))
    for k in range(0, K, 64):
        n = min(64, K - k)
        bar += n * 2.0 ** -44 * np.max(np.abs(A[:, k:k + 64]), axis=1)[:, None] * np.max(np.abs(B[k:k + 64]), axis=0)[None, :]
    assert np.all(np.abs(C - A @ B) <= bar), np.max(np.abs(C - A @ B) / bar)


@pytest.mark.parametrize("layout", [(True, True), (False, True), (True, False), (False, False)])
@pytest.mark.parametrize("bits", [4, 20, 40, 300])
@pytest.mark.parametrize("M,N,K,ks", [(5, 3, 512, 1), (130, 70, 700, 1), (40, 20, 1500, 2), (3, 9, 65, 1)])
def test_falling_rows_and_rising_columns(ctx, M, N, K, ks, bits, layout):
    rng = np.random.default_rng(K + bits)
    g = 2.0 ** (-bits * np.arange(K) / K)
    A = rng.standard_normal((M, K)) * g
    B = rng.standard_normal((K, N)) / g[:, None]
    _check(_run(ctx, A, B, *layout, ksplit=ks), A, B)


@pytest.mark.parametrize("ks", [1, 4])
@pytest.mark.parametrize("layout", [(True, True), (False, False)])
def test_rows_and_columns_that_peak_apart(ctx, layout, ks):
    """One row among smooth ones makes its tile take the blocks: both kinds of tile in one product."""
    rng = np.random.default_rng(7)
    K = 1024
    A, B = rng.standard_normal((200, K)), rng.standard_normal((K, 150))
    A[17] *= 2.0 ** (-60.0 * (np.arange(K) % 512) / 512)
    B[:, 100] *= 2.0 ** (50.0 * (np.arange(K) % 512) / 512)
    A[150, 64:] = 0.0
    B[:448, 3] = 0.0
    _check(_run(ctx, A, B, *layout, ksplit=ks), A, B)


def test_gram_of_localised_columns(ctx):
    rng = np.random.default_rng(9)
    n, K = 90, 2048
    Y = rng.standard_normal((n, K)) * np.exp(-0.02 * np.abs(np.arange(K)[None, :] - rng.integers(0, K, n)[:, None]))
    C = _run(ctx, Y, Y.T.copy(), True, True, ksplit=4, sym=True)
    assert np.array_equal(C, C.T)
    _check(C, Y, Y.T)


def test_more_ranges_than_are_looked_at(ctx):
    """One CTA with more than 2048 ranges takes those past them in blocks, graded or not."""
    rng = np.random.default_rng(11)
    K = 2048 * 512 + 700
    A, B = rng.standard_normal((3, K)), rng.standard_normal((K, 2))
    B[-600:] *= 2.0 ** (-60.0 * np.arange(600) / 600)[:, None]
    A[:, -600:] *= 2.0 ** (60.0 * np.arange(600) / 600)
    _check(_run(ctx, A, B, True, True), A, B)
