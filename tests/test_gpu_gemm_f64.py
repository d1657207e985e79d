"""The FP64 grouped GEMM (plans of results: the tensor-core kernel with split
operands, except for small outputs; others: the FMA kernels) against products
in extended precision.

Elementwise bound: a chunk of 32 columns rounds each operand to 2^-56 of
twice its row's (column's) largest element, 2^-53 amax bmax a product, and
its sum once more; adding the chunks, or the plain FMA loop, rounds at
2^-53 of the running sum, at most |A||B|.  So
|error| <= 2^-53 (K_total + 4) (amax bmax + |A||B|) |alpha| + 2^-52 |C0|."""
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
    sa = np.swapaxes(A, 1, 2) if flags & 1 else A
    sb = np.swapaxes(B, 1, 2) if flags & 2 else B
    got = ctx.gemm_f64(sa, sb, flags, alpha, C0)
    ld = np.longdouble
    ref = alpha * sum(a.astype(ld) @ b.astype(ld) for a, b in zip(A, B)) + (0 if C0 is None else C0)
    aa = sum(np.abs(a) @ np.abs(b) for a, b in zip(A, B))
    mm = np.abs(A).max((0, 2))[:, None] * np.abs(B).max((0, 1))[None, :]
    bound = 2.0 ** -53 * (A.shape[0] * A.shape[2] + 4) * (aa + mm) * abs(alpha)
    bound += 0 if C0 is None else 2.0 ** -52 * np.abs(C0)
    assert np.all(np.abs((got - ref).astype(float)) <= bound)
    return got, ref


# every storage order; K at the edges of the 16- and 32-column steps; outputs
# at the edges of the 16 x 8 fragments and of the 32 x 64 tile
@pytest.mark.parametrize("flags", [0, 1, 2, 3, 4, 5, 6, 7])
@pytest.mark.parametrize("M,N,K,terms", [(32, 64, 32, 1), (33, 65, 33, 2), (31, 63, 31, 1), (16, 8, 64, 40),
                                         (17, 9, 95, 7), (100, 130, 16, 1), (130, 100, 17, 3), (1, 300, 500, 1),
                                         (300, 1, 500, 1), (40, 40, 15, 5), (75, 20, 1, 2), (3, 2, 5, 1),
                                         (96, 40, 1000, 1)])
def test_matches_extended_precision(ctx, M, N, K, terms, flags):
    rng = np.random.default_rng(M * 1000 + N + K + flags)
    A, B = rng.normal(size=(terms, M, K)), rng.normal(size=(terms, K, N))
    check(ctx, A, B, flags)
    check(ctx, A, B, flags, -0.3, rng.normal(size=(M, N)))


def test_error_not_above_the_fma_loops(ctx):
    """Relative 2-norm errors on operands like the sweep's, against FP64 sums rounded at every product."""
    rng = np.random.default_rng(3)
    M, N = 60, 70
    for K in (32, 64, 256):
        grade = np.exp(-20.0 * np.arange(K) / K)
        for A, B in [(rng.normal(size=(M, K)), rng.normal(size=(K, N))),
                     (rng.normal(size=(M, K)) * grade, rng.normal(size=(K, N)) * grade[:, None]),
                     (5 * np.eye(M, K) + 1e-3 * rng.normal(size=(M, K)), rng.normal(size=(K, N)))]:
            got, ref = check(ctx, A[None], B[None], 4)
            loop = np.zeros((M, N))
            for k in range(K):
                loop = (loop + A[:, k:k + 1].astype(np.longdouble) * B[k:k + 1]).astype(float)
            assert np.linalg.norm((got - ref).astype(float)) <= np.linalg.norm((loop - ref).astype(float))


@pytest.mark.parametrize("value", [np.inf, -np.inf, np.nan, 1e-200, 1e200, 1e-310, 0.0])
def test_rows_outside_the_split_range(ctx, value):
    rng = np.random.default_rng(5)
    A, B = rng.normal(size=(1, 40, 50)), rng.normal(size=(1, 50, 60))
    A[0, 3, 5] = value
    A[0, 9, :] = value
    B[0, :, 11] = 0.0
    with np.errstate(all="ignore"):
        got, ref, aa = ctx.gemm_f64(A, B, 4), A[0] @ B[0], np.abs(A[0]) @ np.abs(B[0])
    assert np.array_equal(np.isnan(got), np.isnan(ref))
    ok = np.isfinite(ref)
    assert np.array_equal(got[~ok & ~np.isnan(ref)], ref[~ok & ~np.isnan(ref)])
    assert np.all(np.abs(got[ok] - ref[ok]) <= 2.0 ** -52 * 54 * aa[ok])


def test_bad_arguments_are_refused(ctx):
    from paper_2609_09990_gb300 import gbdmrg
    with pytest.raises(gbdmrg.GbdError, match="GBD_ERR_ARG"):
        ctx.gemm_f64(np.ones((1, 2, 2)), np.ones((1, 2, 2)), 8)
