"""The split FP64 GEMM by element: an output whose products are small against
its row's and column's largest elements keeps the accuracy of FP64 FMAs.

Bound, element by element and without the largest elements in it:
(K_total + 4) 2^-53 |A||B| |alpha| + 2^-52 |C0|, the a priori bound of a loop of
FMAs with a few roundings more for the sums of pieces and the last addition."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    from paper_2609_09990_gb300 import build, gbdmrg
    build.build()
    c = gbdmrg.Context(0)
    yield c
    c.close()


def check(ctx, A, B, flags, alpha=1.0, C0=None):
    """A [t, M, K], B [t, K, N] as multiplied; the storage follows flags."""
    got = ctx.gemm_f64(np.swapaxes(A, 1, 2) if flags & 1 else A, np.swapaxes(B, 1, 2) if flags & 2 else B, flags, alpha, C0)
    ld = np.longdouble
    ref = alpha * sum(a.astype(ld) @ b.astype(ld) for a, b in zip(A, B)) + (0 if C0 is None else C0)
    bound = 2.0 ** -53 * (A.shape[0] * A.shape[2] + 4) * abs(alpha) * sum(np.abs(a) @ np.abs(b) for a, b in zip(A, B))
    bound += 0 if C0 is None else 2.0 ** -52 * np.abs(C0)
    err = np.abs((got - ref).astype(float))
    assert np.all(err <= bound), (err / np.maximum(bound, 1e-300)).max()


def operands(kind, t, M, N, K, rng):
    A, B = rng.normal(size=(t, M, K)), rng.normal(size=(t, K, N))
    decades = np.arange(K) / max(K - 1, 1)
    if kind.startswith("apart"):      # graded in opposite directions
        g = 10.0 ** (-float(kind[5:]) * decades)
        return A * g, B / g[:, None]
    if kind == "graded x diagonal":
        return A * 10.0 ** (-6 * decades), np.eye(K, N) + 1e-12 * B
    if kind == "graded x near diagonal":
        return A * 10.0 ** (-2 * decades), np.eye(K, N) + 0.02 * B
    if kind == "sparse":
        return A * (rng.random(A.shape) < 0.1), B * (rng.random(B.shape) < 0.1)
    assert kind == "wild"
    return A * 10.0 ** rng.uniform(-6, 0, A.shape), B * 10.0 ** rng.uniform(-6, 0, B.shape)


KINDS = ["apart0.5", "apart1", "apart2", "apart3", "apart4", "apart8", "graded x diagonal", "graded x near diagonal",
         "sparse", "wild"]


# K at the edges of the 16- and 32-column steps, M and N at those of the 64 x 64
# tile and its 16 x 8 blocks; 1000 columns in one term are cut into pieces
@pytest.mark.parametrize("kind", KINDS)
@pytest.mark.parametrize("t,M,N,K", [(1, 64, 65, 3), (1, 63, 64, 16), (1, 65, 63, 17), (1, 40, 50, 32), (3, 33, 72, 33),
                                     (1, 17, 130, 64), (7, 48, 24, 20), (1, 30, 40, 1000)])
def test_by_element(ctx, kind, t, M, N, K):
    rng = np.random.default_rng(K + M)
    A, B = operands(kind, t, M, N, K, rng)
    check(ctx, A, B, 4 + (M + K) % 4)
    check(ctx, A, B, 4 + (M + K + 1) % 4, -0.3, rng.normal(size=(M, N)) * np.abs(A[0]).max() * 1e-3)


def test_many_pieces_of_work(ctx):
    """More tiles than the device has multiprocessors, some outputs weak."""
    rng = np.random.default_rng(8)
    A, B = operands("wild", 1, 1000, 1000, 40, rng)
    check(ctx, A, B, 4)


def test_cut_chains_with_rows_outside_the_range_and_c0(ctx):
    """Pieces of a chain, added to C0, some of whose rows go through FMAs and some of whose outputs are weak."""
    rng = np.random.default_rng(9)
    A, B = operands("apart4", 1, 70, 90, 1500, rng)
    A[0, 5] *= 1e-200
    A[0, 66] *= 1e150
    A[0, 20] = 0.0
    B[0, :, 70] = 0.0
    check(ctx, A, B, 4, 0.7, rng.normal(size=(70, 90)))
    check(ctx, A, B, 7, 0.7, rng.normal(size=(70, 90)))


def test_a_second_product_of_other_operands(ctx):
    """The marks of one product are not those of the next."""
    rng = np.random.default_rng(10)
    for kind in ("wild", "apart1", "sparse", "apart8", "wild"):
        A, B = operands(kind, 2, 96, 80, 64, rng)
        check(ctx, A, B, 4)
