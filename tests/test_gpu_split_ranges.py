"""GPU: the tensor-core FP64 product at the edges of its ranges, stages and
tiles: summation lengths about 32, 64 and 512 (one range, two, a range per
K split), both operand layouts, the skipped lower tiles of a symmetric
product, and operands at the limits of the digits (every mantissa bit set over
a full range, zeros, exponents across the whole normal range, subnormals).

Bar per entry: an operand is rounded to 2^-56 of the power of two above its
row's largest (two operands: 2^-55), the dropped levels hold at most 7 x 64^2 x
128^6 of 2^110 (2^-53.1) and the sum of a range keeps 2^-53 of that scale; with
the powers of two up to twice the largest (a factor 4) this is below 2^-50 K
rowmax colmax, and the reference's own FP64 sums add 2^-53 K: 2^-49 in all."""
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


def _bar(A, B):
    return 2.0 ** -49 * A.shape[1] * np.max(np.abs(A), axis=1)[:, None] * np.max(np.abs(B), axis=0)[None, :]


@pytest.mark.parametrize("layout", [(True, True), (False, True), (True, False), (False, False)])
@pytest.mark.parametrize("M,N,K,ks", [(1, 1, 31, 1), (129, 65, 33, 1), (127, 63, 511, 1), (128, 64, 512, 1),
                                      (40, 70, 513, 1), (16, 130, 1100, 2), (216, 72, 1024, 2), (9, 9, 4000, 32)])
def test_ranges_against_fp64(ctx, M, N, K, ks, layout):
    rng = np.random.default_rng(M + N + K)
    A, B = rng.standard_normal((M, K)), rng.standard_normal((K, N)) * np.exp(rng.uniform(-9, 9, size=(K, 1)))
    C = _run(ctx, A, B, *layout, ksplit=ks)
    assert np.all(np.abs(C - A @ B) <= _bar(A, B))


@pytest.mark.parametrize("n,K,ks", [(63, 700, 2), (216, 640, 5), (257, 512, 1)])
def test_symmetric_product_is_whole(ctx, n, K, ks):
    A = np.random.default_rng(n).standard_normal((n, K))
    C = _run(ctx, A, A.T.copy(), True, True, ksplit=ks, sym=True)
    assert np.array_equal(C, C.T) and np.all(np.abs(C - A @ A.T) <= _bar(A, A.T))


@pytest.mark.parametrize("value", [2.0 - 2.0 ** -52, -(2.0 - 2.0 ** -52), 1.0, 2.0 ** 500, 2.0 ** -500, 2.0 ** -1060, 0.0])
def test_digit_limits(ctx, value):
    K = 512
    A, B = np.full((130, K), value), np.full((K, 66), 2.0 - 2.0 ** -52)
    B[:, 1] = 0.0
    B[::2, 2] *= 2.0 ** -40
    C = _run(ctx, A, B, True, True)
    assert np.all(np.abs(C - A @ B) <= np.maximum(_bar(A, B), 2.0 ** -1074))
